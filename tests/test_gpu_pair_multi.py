"""The cases of test_gpu_pair_batches: the oracle's events, except for at most the
draws that lie within 1e-6 of their probability (one, in the largest case), and
the number of particles in more than one of them."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2506_06269_gb300 import ics
from gpu_helpers import gpu_step
from test_gpu_pair_batches import CASES, _clumps

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2506_06269_gb300 import build
    build.build()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("kind,n,k", CASES)
def test_events_and_multiple_hits_match_oracle(kind, n, k, precision):
    halo = {"uniform": lambda: ics.uniform_box(n, 3), "hernquist": lambda: ics.hernquist(n, 4),
            "clumps": lambda: _clumps(n, 5), "nfw": lambda: ics.nfw(n, 6)}[kind]()
    b = ics.batch([halo, ics.hernquist(40, 7)])
    ks, xs, dts = [k, 8], [(0, 10.0, 1.0), (1, 100.0, 0.4)], [2e-7 if kind == "clumps" else 0.05, 0.05]
    g = gpu_step(b, ks, xs, dts, 17, 2, precision=precision)
    o = O.step(b.pos, g["vel_in"], b.ids, b.offsets, ks, b.mass, xs, dts, 17, 2, O.MODE_MIXED if precision == "mixed" else O.MODE_FP64)
    assert g["status"] == 0
    assert len(np.setxor1d(g["events"]["key"], o["events"]["key"])) <= g["stats"].n_near
    hits = np.bincount(np.concatenate([g["events"]["i"], g["events"]["j"]]).astype(np.int64), minlength=b.n)
    assert g["stats"].n_multi == int((hits > 1).sum())
