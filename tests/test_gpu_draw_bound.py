"""The integer bound that spares most pairs their P must keep every pair that can
fire, whatever the units of length, speed and time: the plain draw's events
against those of a context that forms every P (per-particle sums of P), and in
the FP64 form, where scaling by powers of two is exact, against scale 1."""
import functools

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


def _events(s, u, precision, flags):
    """Lengths times 2^s (cross-sections 2^3s), speeds times 2^u, time steps times 2^-u."""
    halos = [ics.hernquist(1500, 3), ics.nfw(700, 4), ics.uniform_box(33, 5)]
    for h in halos:
        h.pos, h.vel = np.ldexp(h.pos, s), np.ldexp(h.vel, u)
    b = ics.batch(halos)
    s0 = float(np.ldexp(10.0, 3 * s))
    xs = [(1, s0, float(np.ldexp(0.4, u))), (0, s0, 1.0), (0, s0, 1.0)]
    g = gpu_step(b, [32, 16, 8], xs, [float(np.ldexp(0.3, -u))] * 3, 9, 1, precision=precision, event_cap=60 * b.n,
                 ctx_kw=dict(flags=flags))
    assert g["status"] == 0
    return g


@functools.lru_cache(maxsize=None)
def _base():
    return _events(0, 0, "fp64", 0)


@pytest.mark.parametrize("s,u", [(56, 40), (0, -70), (0, -160), (0, 70), (-40, 30), (40, -30)])
def test_fp64_events_do_not_depend_on_the_units(s, u):
    g, r = _events(s, u, "fp64", 0), _base()
    assert len(r["events"]) > 10
    assert np.array_equal(g["events"]["key"], r["events"]["key"]) and np.array_equal(g["events"]["P"], r["events"]["P"])
    assert g["stats"].n_near == r["stats"].n_near
    assert np.array_equal(g["vel"], np.ldexp(r["vel"], u))


@pytest.mark.parametrize("s,u", [(0, 0), (0, -62), (0, -66), (0, -70), (30, 0), (-30, 0), (38, 0), (40, 30), (-38, -20)])
def test_mixed_events_are_those_of_every_probability_formed(s, u):
    g, r = _events(s, u, "mixed", 0), _events(s, u, "mixed", sidm.SIDM_FLAG_SUM_P)
    assert np.array_equal(g["events"]["key"], r["events"]["key"]) and np.array_equal(g["events"]["P"], r["events"]["P"])
    assert g["stats"].n_near == r["stats"].n_near and g["stats"].n_pairs == r["stats"].n_pairs
