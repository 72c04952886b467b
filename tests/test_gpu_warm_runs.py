"""Warm-started kernel sizes where the search can go wrong, against a cold
context bit for bit and, for the first step, against the oracle: leaves of
far-apart clumps (runs of queries), guesses that are too small (wider bounds)
and far too small (the redo), N_ngb from 1 to 128 at halos around a leaf, and
lattices, whose equal distances the FP64 form's FP32 search cannot order.
Small halos share a leaf among warps; the 40,000-particle one does not.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2506_06269_gb300 import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2506_06269_gb300 import build
    build.build()


def _positions(kind, n):
    rng = np.random.default_rng(n)
    if kind == "lattice":
        m = int(np.ceil(n ** (1.0 / 3.0)))
        g = np.stack(np.meshgrid(*[np.arange(m, dtype=np.float64)] * 3, indexing="ij")).reshape(3, -1)[:, :n]
        return 0.25 * g[:, rng.permutation(n)]
    if kind == "clumps":
        sizes = []
        while sum(sizes) < n:
            sizes.append(int(min(rng.integers(1, 41), n - sum(sizes))))
        return np.repeat(rng.uniform(-10.0, 10.0, (3, len(sizes))), sizes, axis=1) + 0.01 * rng.standard_normal((3, n))
    if kind == "far":                                    # a small halo at a large distance
        return ics.hernquist(n, 3).pos + np.array([[1e6], [-3e5], [7e5]])
    return ics.hernquist(n, 3).pos


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("kind,n,k", [("plain", 33, 1), ("plain", 65, 31), ("plain", 257, 128), ("plain", 40000, 24),
                                      ("clumps", 900, 6), ("clumps", 5000, 32), ("lattice", 1000, 18), ("lattice", 4096, 64),
                                      ("far", 3000, 32)])
def test_warm_equals_cold_and_oracle(kind, n, k, precision):
    from paper_2506_06269_gb300 import sidm
    x = np.ascontiguousarray(_positions(kind, n))
    ids = np.random.default_rng(1).permutation(n).astype(np.int64)
    out = []
    for warm in (True, False):
        ctx = sidm.Context(n_max=n, halo_max=1, ngb_max=128, precision=precision)
        ctx.warm_start(warm)
        pos = torch.tensor(x, device=ctx.device)
        vel = torch.zeros((3, n), dtype=ctx.vdtype, device=ctx.device)
        idt = torch.tensor(ids, device=ctx.device).to(torch.int32)
        h = torch.zeros(n, dtype=ctx.vdtype, device=ctx.device)
        got = []
        # the same positions, a stretch by 1.3 and one by 50 (guesses 1.2 and 47 times too small), and back
        for scale in (1.0, 1.0, 1.3, 50.0, 1.0 / 65.0):
            if scale != 1.0:
                pos *= scale
            ctx.build_cells([0, n], pos, vel, idt)
            ctx.kernel_sizes([k], h)
            assert ctx.status() == 0
            got.append((idt.cpu().numpy().copy(), h.cpu().numpy().copy(), pos.cpu().numpy().copy()))
        out.append(got)
        ctx.close()
    for (i0, h0, _), (i1, h1, _) in zip(*out):
        assert np.array_equal(i0, i1) and np.array_equal(h0, h1)
    i1, h1, p1 = out[0][1]
    ref, _, _ = O.knn(p1, i1.astype(np.uint32), k, O.MODE_MIXED if precision == "mixed" else O.MODE_FP64)
    assert np.array_equal(h1, ref.astype(h1.dtype))
