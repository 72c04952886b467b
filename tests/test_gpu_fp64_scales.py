"""The FP64 form in any unit of length: a scaling of all lengths by a power of
two (the cross-section by its cube) is exact in FP64, so kernel sizes scale
exactly and pairs, events and velocities stay the same bits, from the oracle's
values at scale 1 to scales whose squares leave FP32's range on both sides.
The plain draw and the kernel that forms every P; first and warm-started sizes.
"""
import functools

import numpy as np
import pytest

from oracle import oracle as O
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


KS, DTS = [32, 6, 16], [0.3, 1e-10, 0.3]


def _batch(s):
    rng = np.random.default_rng(4)
    n = 700
    centre = np.repeat(rng.uniform(-10.0, 10.0, (3, 70)), 10, axis=1)
    clumps = ics.Halo(pos=centre + 1e-4 * rng.standard_normal((3, n)), vel=rng.standard_normal((3, n)),
                      ids=rng.permutation(n).astype(np.uint32), mass=1.0 / n)
    halos = [ics.hernquist(1500, 3), clumps, ics.uniform_box(33, 5)]
    for h in halos:
        h.pos = np.ldexp(h.pos, s)
    return ics.batch(halos)


def _xs(s):
    return [(1, float(np.ldexp(10.0, 3 * s)), 0.4), (0, float(np.ldexp(10.0, 3 * s)), 1.0), (0, float(np.ldexp(10.0, 3 * s)), 1.0)]


def _steps(s, flags):
    b = _batch(s)
    ctx = sidm.Context(n_max=b.n, halo_max=3, ngb_max=32, precision="fp64", event_cap=60 * b.n, flags=flags)
    got = [gpu_step(b, KS, _xs(s), DTS, 9, 1, precision="fp64", ctx=ctx) for _ in range(2)]
    ctx.close()
    return got


@functools.lru_cache(maxsize=None)
def _base(flags):
    return _steps(0, flags)


@pytest.mark.parametrize("flags", [0, sidm.SIDM_FLAG_SUM_P])
def test_scale_one_matches_oracle(flags):
    b = _batch(0)
    o = O.step(b.pos, b.vel, b.ids, b.offsets, KS, b.mass, _xs(0), DTS, 9, 1, O.MODE_FP64)
    for g in _base(flags):
        assert g["status"] == 0
        assert np.array_equal(g["h"], o["h"])
        assert g["stats"].n_pairs == sum(int(x["n_pairs"]) for x in o["stats"])


@pytest.mark.parametrize("flags", [0, sidm.SIDM_FLAG_SUM_P])
@pytest.mark.parametrize("s", [-300, -100, -66, -40, 50, 62, 70, 100, 300])
def test_scaled_lengths_give_the_same_bits(s, flags):
    for g, r in zip(_steps(s, flags), _base(flags)):
        assert g["status"] == 0
        assert np.array_equal(g["h"], np.ldexp(r["h"], s))
        assert g["stats"].n_pairs == r["stats"].n_pairs
        assert len(r["events"]) > 10 and np.array_equal(g["events"]["key"], r["events"]["key"])
        assert np.array_equal(g["events"]["P"], r["events"]["P"])
        assert np.array_equal(g["vel"], r["vel"])
