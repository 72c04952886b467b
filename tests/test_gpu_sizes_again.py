"""Kernel sizes found several times on one build (a sweep over N_ngb): the last
call's sizes, and the scatter that follows, are those of a context that called
once, bit for bit."""
import numpy as np
import pytest

from paper_2506_06269_gb300 import ics, sidm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2506_06269_gb300 import build
    build.build()


def _clumps(n):
    """Clumps of 1 to 40 particles a thousand of their sizes apart: leaves whose offsets dwarf their kernel sizes."""
    rng = np.random.default_rng(n)
    sizes = []
    while sum(sizes) < n:
        sizes.append(int(min(rng.integers(1, 41), n - sum(sizes))))
    return np.repeat(rng.uniform(-10.0, 10.0, (3, len(sizes))), sizes, axis=1) + 1e-4 * rng.standard_normal((3, n))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("kind,n,last,dt", [("hernquist", 3000, 32, 0.5), ("hernquist", 40000, 32, 0.1), ("clumps", 3000, 20, 5e-10)])
def test_repeated_sizes_equal_one_call(kind, n, last, dt, precision):
    x = np.ascontiguousarray(_clumps(n) if kind == "clumps" else ics.hernquist(n, 3).pos)
    v = np.random.default_rng(2).standard_normal((3, n)).astype(np.float32)
    out = []
    for calls in ([16, 64, 8, last], [last]):
        ctx = sidm.Context(n_max=n, halo_max=1, ngb_max=64, precision=precision, event_cap=20 * n)
        pos = torch.tensor(x, device=ctx.device)
        vel = torch.tensor(v, dtype=ctx.vdtype, device=ctx.device)
        ids = torch.arange(n, dtype=torch.int32, device=ctx.device)
        h = torch.zeros(n, dtype=ctx.vdtype, device=ctx.device)
        ctx.build_cells([0, n], pos, vel, ids)
        for k in calls:
            ctx.kernel_sizes([k], h)
        ctx.scatter_step(3, 1, ctx.xs_tensor([(0, 10.0, 1.0)]), ctx.f64([dt]), ctx.f64([1.0 / n]), vel)
        assert ctx.status() == 0
        out.append((h.cpu().numpy(), ctx.stats().n_pairs, np.sort(ctx.events()[1]["key"]), vel.cpu().numpy()))
        ctx.close()
    assert len(out[1][2]) > 10
    for a, b in zip(*out):
        assert np.array_equal(a, b)
