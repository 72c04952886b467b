"""Cell build around the one-launch radix sort (up to 8192 keys in one CTA) on the
GPU against the oracle's canonical order, bit-exact: one key, sizes off a multiple
of a warp and of the CTA, the largest size that takes it and the first that does
not, coincident particles (stability decides), runs of equal keys, and several
halos (an eighth digit pass)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_sort import _built, _check  # noqa: E402,F401


@pytest.mark.parametrize("halos", [
    [("uniform", 1)],
    [("clump", 31)],
    [("clump", 1025)],
    [("lattice", 8191)],
    [("coincident", 8192)],
    [("clump", 8192)],
    [("clump", 8193)],
    [("lattice", 33)] * 40,
    [("uniform", 1000), ("coincident", 3001), ("clump", 4191)],
], ids=lambda h: f"{len(h)}x{h[0][0]}{sum(n for _, n in h)}")
def test_small_build_order_matches_canonical_order(halos):
    _check(halos, 91)
