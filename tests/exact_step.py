"""Steps in 64 bits whose only rounding is the one that the state is defined with: the projector is (1 + 2^-7) I, the entries of the gradients are
+-(1 + a 2^-7), so that R is exact in fp32, and a history in bf16 rounds all of them down, by 0.4 of the last place on average (a row of the
Gram matrix that is not worked out again for the rounded slot is off by a third of a percent, in the same direction for every entry).
Without moments (beta1 = beta2 = 0) u = n / sqrt(n^2 + eps) follows the natural gradient n.  W starts from zero in every step."""
import torch

SCALE = 1.0 + 2.0 ** -7
# u in fp16, 2^-11 of an entry; beside it the fp32 products of the Gram matrix, a few 2^-24 of it, times its condition number, at most about 40
# here (half of every gradient is shared): 1e-5.
BOUND = 2.0 ** -11 + 2e-5


def scale_bound(n):
    """... and of the factor between an update and the exact one: the roundings of n entries (of 500 different ones at most), each of a standard
    deviation of 2^-11 / sqrt(3), average out; six times what is left of them.  (A row for the slot as it was before it was rounded: 8e-4.)"""
    return 6.0 * 2.0 ** -11 / 3.0 ** 0.5 / min(n, 500) ** 0.5 + 2e-5


def gradients(shapes, steps, device, seed):
    gen = torch.Generator(device=device).manual_seed(seed)
    common = [torch.sign(torch.randn(x, generator=gen, device=device)) for x in shapes]
    for _ in range(steps):
        out = []
        for x, c in zip(shapes, common):
            a = torch.randint(40, 64, x, generator=gen, device=device)
            flip = torch.rand(x, generator=gen, device=device) < 0.25
            out.append((torch.where(flip, -c, c) * (1.0 + a / 128.0)).bfloat16())
        yield out


def hyper(shapes, r):
    """lambda and eps of a size with K and with n^2 for the largest matrix."""
    rn = max(min(r, M, N) * N for M, N in shapes)
    return 0.25 * rn, (16.0 / rn) ** 2


def exact_update(ring, cur, lam, eps):
    """-u of the step whose low-rank gradients are ring (64 bits, c of them)."""
    H = torch.stack([x.flatten() for x in ring])
    c = H.shape[0]
    K = H @ H.T / c + lam * torch.eye(c, dtype=H.dtype, device=H.device)
    e = torch.zeros(c, dtype=H.dtype, device=H.device)
    e[cur] = 1.0
    n = (torch.linalg.solve(K, e)[:, None] * H).sum(0).view_as(ring[0])
    return -n / torch.sqrt(n * n + eps)


def largest_errors(shapes, r, s, steps, rounded, seed=3, **kw):
    """Over all steps and matrices, as parts of the bounds above: the largest error of an update against 64 bits, and of its scale from the second
    step on (the entries of the first have 24 sizes)."""
    from paper_2410_16029_b200.ngalore import NGaLore

    lam, eps = hyper(shapes, r)
    opt = NGaLore(shapes, r, s, 0, lam=lam, lr=1.0, beta1=0.0, beta2=0.0, eps=eps, history_bf16=rounded, **kw)
    for i, (M, N) in enumerate(shapes):
        opt.set_subspace(i, SCALE * torch.eye(M, min(r, M, N), device="cuda"))
    rings = [[] for _ in shapes]
    worst = scale = 0.0
    for k, G in enumerate(gradients(shapes, steps, "cuda", seed)):
        W = [torch.zeros(x, device="cuda") for x in shapes]
        opt.step(W, G)
        for i, (M, N) in enumerate(shapes):
            R = SCALE * G[i][: min(r, M, N)].double()
            if len(rings[i]) < s:
                rings[i].append(R)
            else:
                rings[i][k % s] = R
            want = SCALE * exact_update(rings[i], k % s, lam, eps)
            got = W[i][: min(r, M, N)].double()
            assert torch.count_nonzero(W[i][min(r, M, N):]).item() == 0
            worst = max(worst, (torch.linalg.norm(got - want) / torch.linalg.norm(want)).item() / BOUND)
            if k > 0:
                scale = max(scale, abs(((got * want).sum() / (want * want).sum()).item() - 1.0) / scale_bound(want.numel()))
            if rounded:
                rings[i][k % s] = R.float().bfloat16().double()
    assert opt.poll_status()[0] == 0
    opt.close()
    return worst, scale
