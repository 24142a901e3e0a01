"""_bind.so holds the layout of one torch's tensors and of one Python's objects: it is built again for another, and not taken with another."""
import os
import sys

import pytest
import torch


def test_it_is_built_again_for_another_torch_or_python(tmp_path):
    from paper_2410_16029_b200 import build

    build._build_bind(False)
    stamp = build._bind_stamp()
    python = ".".join(map(str, sys.version_info[:3]))
    assert torch.__version__ in stamp and python in stamp
    assert build._bind_current(build.BIND_OUT, stamp)
    out = str(tmp_path / "_bind.so")
    assert not build._bind_current(out, stamp)                  # nothing there
    open(out, "w").close()
    assert not build._bind_current(out, stamp)                  # built by what did not say for what
    with open(out + ".stamp", "w") as f:
        f.write(stamp)
    assert build._bind_current(out, stamp)
    assert not build._bind_current(out, stamp.replace(torch.__version__, "1.0"))
    assert not build._bind_current(out, stamp.replace(python, "3.0.0"))
    os.utime(out, (1, 1))                                       # older than its source
    assert not build._bind_current(out, stamp)


def test_it_is_not_taken_with_another_torch_or_python():
    import __graft_entry__ as entry

    entry.build()
    from paper_2410_16029_b200 import _bind, ngalore

    version, major, minor = _bind.built_for
    ngalore._check_built_for(_bind.built_for)
    for other in [(), ("1.0.0", major, minor), (version, major, minor + 1), (version, major + 1, minor)]:
        with pytest.raises(ImportError):
            ngalore._check_built_for(other)
