"""What makes a compiled translation unit stale."""
import os
import shutil

import pytest

from paper_2310_03921_gb300 import build as B


@pytest.mark.parametrize("header", sorted(f for f in os.listdir(B.CSRC) if not f.endswith(".cu")))
def test_every_internal_header_is_a_dependency(header, tmp_path, monkeypatch):
    """An object older than any header of the sources' folder is rebuilt, a newer one is not."""
    csrc = tmp_path / "csrc"
    shutil.copytree(B.CSRC, csrc)
    monkeypatch.setattr(B, "CSRC", str(csrc))
    monkeypatch.setattr(B, "HERE", str(tmp_path))
    src, obj = str(csrc / "tc_gemm.cu"), str(tmp_path / "tc_gemm.o")
    open(obj, "w").close()
    for f in csrc.iterdir():
        os.utime(f, (1000, 1000))
    os.utime(obj, (2000, 2000))
    assert not B._stale(obj, src)
    os.utime(csrc / header, (3000, 3000))
    assert B._stale(obj, src)
