"""The pair kernel's batches, queues and runs of queries at the sizes where they
can go wrong: halos around a leaf (32), a batch of candidates (16) and a list of
leaves, and leaves whose particles lie far apart, against the oracle.

Checked exactly: the number of in-range pairs, the events (these sizes draw
tens of events, none within 1e-6 of its probability) and the number of
particles hit more than once; kernel sizes bit for bit.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2506_06269_gb300 import ics
from gpu_helpers import gpu_step

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2506_06269_gb300 import build
    build.build()


def _clumps(n, seed):
    """Tight clumps of 1 to 40 particles a thousand of their sizes apart: most leaves span several."""
    rng = np.random.default_rng(seed)
    sizes = []
    while sum(sizes) < n:
        sizes.append(int(min(rng.integers(1, 41), n - sum(sizes))))
    centre = np.repeat(rng.uniform(-10.0, 10.0, (3, len(sizes))), sizes, axis=1)
    pos = centre + 0.01 * rng.standard_normal((3, n))
    return ics.Halo(pos=pos, vel=0.3 * rng.standard_normal((3, n)), ids=rng.permutation(n).astype(np.uint32), mass=1.0 / n)


CASES = [("uniform", 17, 4), ("uniform", 33, 16), ("uniform", 48, 31), ("uniform", 65, 7), ("hernquist", 1023, 16),
         ("hernquist", 1057, 128), ("clumps", 700, 5), ("clumps", 3000, 24), ("nfw", 33000, 3)]


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("kind,n,k", CASES)
def test_pair_counts_and_events_match_oracle(kind, n, k, precision):
    halo = {"uniform": lambda: ics.uniform_box(n, 3), "hernquist": lambda: ics.hernquist(n, 4),
            "clumps": lambda: _clumps(n, 5), "nfw": lambda: ics.nfw(n, 6)}[kind]()
    other = ics.hernquist(40, 7)                       # a second halo behind the first
    b = ics.batch([halo, other])
    ks, xs, dts = [k, 8], [(0, 10.0, 1.0), (1, 100.0, 0.4)], [2e-7 if kind == "clumps" else 0.05, 0.05]
    g = gpu_step(b, ks, xs, dts, 17, 2, precision=precision)
    vin = g["vel_in"]
    o = O.step(b.pos, vin, b.ids, b.offsets, ks, b.mass, xs, dts, 17, 2, O.MODE_MIXED if precision == "mixed" else O.MODE_FP64)
    assert g["status"] == 0
    assert np.array_equal(g["h"], o["h"])
    assert g["stats"].n_pairs == sum(int(s["n_pairs"]) for s in o["stats"])
    assert sum(int(s["n_near"]) for s in o["stats"]) == g["stats"].n_near
    if g["stats"].n_near == 0:
        assert np.array_equal(np.sort(g["events"]["key"]), np.sort(o["events"]["key"]))
