"""Per-particle sums of P: in a halo of two particles the sum is one P, and its
FP32 bits are those of the P that the plain draw records with its event (both
form it from the same table sums in the same order)."""
import numpy as np
import pytest

from paper_2506_06269_gb300 import ics, sidm
from gpu_helpers import gpu_step

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2506_06269_gb300 import build
    build.build()


@pytest.mark.parametrize("flags", [0, sidm.SIDM_FLAG_DRAG])
def test_sum_of_one_pair_is_the_recorded_probability(flags):
    rng = np.random.default_rng(5)
    H = 600
    halos = [ics.Halo(pos=rng.normal(size=(3, 2)), vel=rng.normal(size=(3, 2)), ids=np.arange(2, dtype=np.uint32), mass=1.0)
             for _ in range(H)]
    b = ics.batch(halos)
    ks, xs, dts = [1] * H, [(1, 1e6, 1.0)] * H, [1.0] * H      # P far above 1: every pair fires
    plain = gpu_step(b, ks, xs, dts, 3, 0)
    ctx = sidm.Context(n_max=b.n, halo_max=H, ngb_max=1, event_cap=4 * b.n, flags=sidm.SIDM_FLAG_SUM_P | flags)
    got = gpu_step(b, ks, xs, dts, 3, 0, ctx=ctx)
    sums = np.empty(b.n, np.float32)
    sums[got["perm"]] = ctx.sum_p(b.n).cpu().numpy()
    ev = plain["events"]
    assert plain["status"] == 0 and got["status"] == 0 and len(ev) == H
    assert np.array_equal(sums[ev["i"]], ev["P"]) and np.array_equal(sums[ev["j"]], ev["P"])
