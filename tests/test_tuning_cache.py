"""Host-side checks of the tuning cache's key (autotune.py)."""
import shutil
from types import SimpleNamespace

from paper_1702_01335_gb300 import autotune as AT
from paper_1702_01335_gb300 import lbs as L


def key(*instances):
    return AT.signature(SimpleNamespace(instances=list(instances), precision=1))


def test_signature_tells_the_marches_apart():
    """V = 4 (and V = 1 in FP64) runs the grouped march where every Qy is a multiple of four, another
    one elsewhere: batches of the same (Nz, Q) on either side have keys of their own."""
    a, b = L.Instance(Qx=8, Qy=8, Qz=16, Nz=64), L.Instance(Qx=16, Qy=2, Qz=32, Nz=64)
    assert a.Q == b.Q and key(a) != key(b) and key(a, a) != key(a, b)
    c = L.Instance(Qx=16, Qy=4, Qz=16, Nz=64)  # grouped too
    assert c.Q == a.Q and key(a) == key(c)
    r = L.Instance(Qx=16, Qy=0, Qz=32, Nz=64)
    assert r.Q == a.Q and len({key(a), key(b), key(r)}) == 3


def test_kernel_hash_covers_the_choice_of_the_kernel(monkeypatch, tmp_path):
    """A change of the sources that decide which kernel a tiling runs (the layouts and the
    finalisation's rule, api.cu) or of the kernels' own makes the cached choices stale."""
    csrc = tmp_path / "csrc"
    shutil.copytree(AT._CSRC, csrc)
    monkeypatch.setattr(AT, "_CSRC", str(csrc))
    seen = {AT.kernel_hash()}
    for f in ("api.cu", "kernels.cuh", "finalize.cuh", "pdl.cuh", "kernels.cu", "lbs_internal.h"):
        with open(csrc / f, "a") as out:
            out.write("// changed\n")
        seen.add(AT.kernel_hash())
    assert len(seen) == 7
