"""Forward-dominated scattering at the particle numbers that pick each form of
the list resolve: one CTA, a cluster of two, the most a cluster holds and one
particle more (a cooperative launch); a context made for more particles than one
thread each on the device takes lists of active particles instead, with the same
bits.  Against the oracle's sequential application: the interacting pairs exactly, the velocities to the tolerance of
the forward-dominated parity test (1e-5 of each particle's largest step-start
pair speed in the mixed form, 1e-10 in FP64), and the booked energy change
against the change of the exact sums (1e-12 of the energy).
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


def _run(b, ks, xs, dts, vin, precision, k, n_max):
    from paper_2506_06269_gb300 import sidm
    ctx = sidm.Context(n_max=n_max, halo_max=2, ngb_max=16, precision=precision, event_cap=16 * b.n * k,
                       flags=sidm.SIDM_FLAG_DRAG)
    pos = torch.tensor(b.pos, device=ctx.device)
    vel = torch.tensor(vin, dtype=ctx.vdtype, device=ctx.device)
    ids = torch.tensor(b.ids.astype(np.int64), device=ctx.device).to(torch.int32)
    h = torch.zeros(b.n, dtype=ctx.vdtype, device=ctx.device)
    mass = ctx.f64(b.mass)
    E = torch.zeros((2, 2, 4), dtype=torch.float64, device=ctx.device)
    ctx.build_cells(b.offsets, pos, vel, ids)
    perm = ctx.perm(b.n).cpu().numpy().astype(np.int64)
    ctx.kernel_sizes(ks, h)
    ctx.energy_momentum(mass, vel, E[0])
    ctx.scatter_step(5, 2, ctx.xs_tensor(xs), ctx.f64(dts), mass, vel)
    ctx.energy_momentum(mass, vel, E[1])
    assert ctx.status() == 0
    st = ctx.stats()
    n_ev, ev = ctx.events()
    got = np.empty((3, b.n))
    got[:, perm] = vel.cpu().numpy().astype(np.float64)
    ctx.close()
    return ev, n_ev, got, st, E


@pytest.mark.parametrize("precision,n,k", [("mixed", 1000, 12), ("fp64", 1025, 12), ("mixed", 16384, 6), ("mixed", 16385, 6),
                                           ("fp64", 20000, 4)])
def test_every_resolve_form_matches_oracle(precision, n, k):
    halos = [ics.hernquist(n - 300, 71), ics.hernquist(300, 72)]
    b = ics.batch(halos)
    ks, xs, dts = [k, 8], [(1, 20.0, 0.5, 1), (0, 10.0, 1.0)], [0.002, 0.2]     # forward-dominated beside isotropic
    vin = b.vel.astype(np.float32).astype(np.float64) if precision == "mixed" else b.vel
    ev, n_ev, got, st, E = _run(b, ks, xs, dts, vin, precision, k, b.n)
    _, _, lists, st2, _ = _run(b, ks, xs, dts, vin, precision, k, 400000)
    assert np.array_equal(got, lists) and st.d_energy == st2.d_energy
    assert (st.rounds, st.n_multi, st.n_events) == (st2.rounds, st2.n_multi, st2.n_events)
    o = O.step(b.pos, vin, b.ids, b.offsets, ks, b.mass, xs, dts, 5, 2, O.MODE_MIXED if precision == "mixed" else O.MODE_FP64)
    gk, ok = np.sort(ev["key"]), np.sort(o["events"]["key"])
    assert n_ev == ok.size and np.array_equal(gk, ok)
    sp = np.linalg.norm(vin, axis=0)
    scale = sp.copy()
    s = sp[o["events"]["i"]] + sp[o["events"]["j"]]
    np.maximum.at(scale, o["events"]["i"], s)
    np.maximum.at(scale, o["events"]["j"], s)
    err = np.abs(got - o["vel_out"]).max(axis=0)
    assert np.all(err <= (1e-5 if precision == "mixed" else 1e-10) * scale)
    e0, e1 = E[0, :, 0].sum().item(), E[1, :, 0].sum().item()
    assert abs((e1 - e0) - st.d_energy) <= 1e-12 * e0
