"""FP64 energy and momentum sums at the edges of their chunks of 16384 particles and
around the number of chunks where the sums go from a cluster per chunk to a CTA per
chunk, against correctly rounded sums on the host (math.fsum of the same terms).

Bound: a compensated sum S' of n terms is within 2 u |S| + n^2 u^2 sum|x| of S (u =
2^-53); the factor m or m/2 and the final rounding add u |S| each."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

C = 16384


@pytest.mark.parametrize("sizes", [[1], [31, 33, 255, 257], [C - 1, C, C + 1], [3 * C + 77] * 3,
                                   [1] * 151, [1] * 152, [40] * 153],
                         ids=lambda s: f"{len(s)}x{s[0]}")
def test_fp64_sums_match_host_sums(sizes):
    from paper_2506_06269_gb300 import build, sidm
    build.build()
    rng = np.random.default_rng(17)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n, H = int(off[-1]), len(sizes)
    ctx = sidm.Context(n_max=n, halo_max=H, ngb_max=8, event_cap=1 << 12, precision="fp64")
    pos = torch.tensor(rng.random((3, n)), device="cuda")
    vel = torch.tensor(rng.standard_normal((3, n)) * 10.0 ** rng.integers(-3, 4, (3, n)), device="cuda")
    ids = torch.cat([torch.arange(s, dtype=torch.int32) for s in sizes]).cuda()
    ctx.build_cells(off, pos, vel, ids)
    mass = rng.random(H) + 0.5
    out = torch.full((H, 4), float("nan"), dtype=torch.float64, device="cuda")
    ctx.energy_momentum(ctx.f64(mass), vel, out)
    got = out.cpu().numpy()
    assert ctx.status() == 0
    ctx.close()
    v = vel.cpu().numpy()
    q = v[0] * v[0] + v[1] * v[1] + v[2] * v[2]
    u = 2.0 ** -53
    for h in range(H):
        a, b = int(off[h]), int(off[h + 1])
        for k, (x, f) in enumerate([(q, 0.5 * mass[h]), (v[0], mass[h]), (v[1], mass[h]), (v[2], mass[h])]):
            s, m = math.fsum(x[a:b]), math.fsum(np.abs(x[a:b]))
            bound = f * (4 * u * abs(s) + (b - a) ** 2 * u * u * m)
            assert abs(got[h, k] - f * s) <= bound, (h, k)
