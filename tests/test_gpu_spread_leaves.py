"""Halos whose leaves are hard on the fixed-bound search and the pair search: a core
denser than the cells that order it, with sparse outliers whose kernels reach it; a
steep cusp; a dense halo beside a wide one; clumps far apart.  They take the paths
that ordinary leaves do not: whole leaves, the redo of many runs, leaves left to
teams, rests of the pair kernel, guesses of mixed leaves.

Kernel sizes (first, warm-started, after a stretch) and neighbour lists bit for bit
against the per-lane search, pairs and events against the kernel that forms every P,
densities of the mixed form against a direct FP64 sum over the canonical distances of
a sample: d / h and 1 - d / h are FP32 there, each term off by at most 1e-6 of W and of
its slope.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2506_06269_gb300 import ics, sidm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2506_06269_gb300 import build
    build.build()


def _positions(kind, n):
    r = np.random.default_rng(n)
    if kind == "core":
        x = 1e-3 * r.standard_normal((3, n))
        x[:, : n // 100] = r.uniform(-10.0, 10.0, (3, n // 100))
        return x
    if kind == "cusp":
        d = r.standard_normal((3, n))
        return 10.0 * r.random(n) ** 2.5 * d / np.sqrt((d * d).sum(0))
    if kind == "two":
        x = ics.hernquist(n, 3).pos
        x[:, : n // 2] = 1e-3 * x[:, : n // 2] + 200.0
        return x
    if kind == "clumps":
        return np.repeat(r.uniform(-10.0, 10.0, (3, n // 20)), 20, axis=1) + 0.01 * r.standard_normal((3, n))
    return ics.hernquist(n, 3).pos


CASES = [("core", 60000, 16), ("core", 40000, 100), ("core", 200000, 16), ("cusp", 300000, 16), ("two", 400000, 32), ("cusp", 50000, 24), ("two", 60000, 32), ("clumps", 40000, 48),
         ("hernquist", 120000, 128)]


def _run(kind, n, k, precision, **kw):
    x = np.ascontiguousarray(_positions(kind, n))
    v = np.random.default_rng(2).standard_normal((3, n)).astype(np.float32)
    ctx = sidm.Context(n_max=n, halo_max=1, ngb_max=128, precision=precision, event_cap=4 * n, **kw)
    pos, vel = torch.tensor(x, device=ctx.device), torch.tensor(v, dtype=ctx.vdtype, device=ctx.device)
    ids = torch.arange(n, dtype=torch.int32, device=ctx.device)
    h = torch.zeros(n, dtype=ctx.vdtype, device=ctx.device)
    got = {}
    for step, scale in enumerate((1.0, 1.0, 1.3, 1.0 / 1.3)):
        pos *= scale
        ctx.build_cells([0, n], pos, vel, ids)
        ctx.kernel_sizes([k], h)
        got["h%d" % step] = h.cpu().numpy().copy()
    if precision == "mixed":
        got["lists"] = ctx.neighbours([k], n, k).cpu().numpy()
    dt = 0.02 * float(torch.quantile(h.double(), 0.001)) ** 3 * n        # P near one for the densest thousandth only
    xs, mass = ctx.xs_tensor([(0, 1.0, 1.0)]), ctx.f64([1.0 / n])
    got["pos"], got["sizes"], got["v"] = pos.clone(), h.clone(), vel.clone()
    if kw.get("flags", 0) & sidm.SIDM_FLAG_LOCAL_DIAG:
        got["rho"] = ctx.local_diagnostics(xs, mass, vel, n)["rho"].double()
    ctx.scatter_step(3, 1, xs, ctx.f64([dt]), mass, vel)
    assert ctx.status() == 0
    st = ctx.stats()
    ev = np.sort(ctx.events()[1], order="key")
    got["counts"] = np.array([st.n_pairs, st.n_events, st.n_near, st.n_p_gt1, st.n_multi])
    got["keys"], got["P"], got["vel"] = ev["key"].copy(), ev["P"].copy(), vel.cpu().numpy()
    ctx.close()
    return got


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("kind,n,k", CASES)
def test_spread_leaves_equal_the_per_lane_search_and_every_probability(kind, n, k, precision):
    got = _run(kind, n, k, precision, flags=sidm.SIDM_FLAG_LOCAL_DIAG)
    ref = _run(kind, n, k, precision, flags=sidm.SIDM_FLAG_SUM_P, knn_batch=2)
    for key in ref:
        if key not in ("pos", "sizes", "v"):
            assert np.array_equal(got[key], ref[key]), key
    assert len(ref["keys"]) > 10
    if precision == "mixed":
        x, h = got["pos"].cpu().numpy(), got["sizes"].double().cpu().numpy()
        pick = np.concatenate([np.random.default_rng(1).choice(n, 30, replace=False), np.argsort(h)[-20:]])
        for i in pick:
            q = np.sqrt(O.d2_mixed(x, np.full(n, i), np.arange(n)).astype(np.float64)) / h[i]
            w = np.where(q < 0.5, 1.0 - 6.0 * q * q * (1.0 - q), 2.0 * np.maximum(1.0 - q, 0.0) ** 3)
            slope = np.where(q < 0.5, 12.0 * q, 6.0 * np.maximum(1.0 - q, 0.0) ** 2)
            norm = (8.0 / np.pi) / n / h[i] ** 3
            assert abs(float(got["rho"][i]) - norm * w.sum()) <= 1e-6 * norm * (w + slope).sum(), i
