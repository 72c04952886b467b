"""Local diagnostics of the mixed form: leaves shared by the warps of a CTA (few
leaves) against one warp per leaf (the same halo with one CTA), where the lanes'
queues differ in length: clumps smaller and larger than N_ngb, full kernels.

Both add the same FP64 terms, in another order, and round to FP32 once: 1e-6
allows for a few FP32 steps in the quantities formed from them."""
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
    rng = np.random.default_rng(n)
    sizes = []
    while sum(sizes) < n:
        sizes.append(int(min(rng.integers(1, 41), n - sum(sizes))))
    return np.repeat(rng.uniform(-10.0, 10.0, (3, len(sizes))), sizes, axis=1) + 0.01 * rng.standard_normal((3, n))


@pytest.mark.parametrize("kind,n,k", [("clumps", 900, 6), ("clumps", 3000, 24), ("hernquist", 1023, 64), ("hernquist", 300, 128)])
def test_shared_leaves_give_the_moments_of_one_warp(kind, n, k):
    x = np.ascontiguousarray(_clumps(n) if kind == "clumps" else ics.hernquist(n, 3).pos)
    v = np.random.default_rng(2).standard_normal((3, n)).astype(np.float32)
    out = []
    for ctas in (0, 1):
        ctx = sidm.Context(n_max=n, halo_max=1, ngb_max=128, flags=sidm.SIDM_FLAG_LOCAL_DIAG, grid_ctas=ctas)
        pos, vel = torch.tensor(x, device=ctx.device), torch.tensor(v, device=ctx.device)
        ids = torch.arange(n, dtype=torch.int32, device=ctx.device)
        ctx.build_cells([0, n], pos, vel, ids)
        ctx.kernel_sizes([k], torch.zeros(n, device=ctx.device))
        got = ctx.local_diagnostics(ctx.xs_tensor([(1, 100.0, 0.5)]), ctx.f64([1.0 / n]), vel, n)
        assert ctx.status() == 0
        out.append({q: t.cpu().numpy().copy() for q, t in got.items()})
        ctx.close()
    for q in out[0]:
        np.testing.assert_allclose(out[0][q], out[1][q], rtol=1e-6, atol=0, err_msg=q)
