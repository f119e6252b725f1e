"""Mechanisms whose fixed-point coefficients and gather list do not fit in shared
memory beside one cell: the block keeps the thermo coefficients alone, the
reactions run in the direct form and the species rows are read from global memory.
Source term, J v and one short step at every precision level that fits against the
FP64 oracle; the levels whose own arrays do not fit are refused on the host.
Bars as in the parity tests: 1e-11 of the row scale (1e-10 in double-float, 1e-4 in
FP32), |dY| <= 1e-8 + 1e-6 |Y| and |dT| <= 1e-6 K for the replayed step."""

import functools

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

P = 101325.0


@pytest.fixture(scope="module")
def rk():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1712_00953_gb300 as rk

    return rk


@functools.lru_cache(maxsize=None)
def _mech(ns, nr, n_pressure):
    from oracle.kinetics import Kinetics
    from synth.mechanism import generate_mechanism

    mech = generate_mechanism(ns, nr, seed=5, n_third_body=n_pressure, n_troe=n_pressure)
    return mech, Kinetics(mech)


def _states(mech, n=3):
    rng = np.random.default_rng(8)
    return np.concatenate([rng.dirichlet(np.full(mech.n_species, 0.5), n), rng.uniform(900.0, 1500.0, (n, 1))], 1)


# (150 / 2500): no level's list fits; (120 / 1000 with 80 pressure-dependent reactions):
# it fits at levels 0 and 6 and not at levels 1 and 3, whose prefix or slot is larger
@pytest.mark.parametrize("size,mode,bar", [((150, 2500, 0), 0, 1e-11), ((150, 2500, 0), 5, 1e-4),
                                           ((120, 1000, 40), 3, 1e-10), ((120, 1000, 40), 5, 1e-4)])
def test_source_term_and_products(rk, size, mode, bar):
    mech, kin = _mech(*size)
    U = _states(mech)
    V = np.random.default_rng(9).normal(size=U.shape)
    m = rk.mech_load(mech)
    Ug = torch.tensor(U, device="cuda")
    for got, ref, b in ((rk.chem_rhs(m, Ug, P), [kin.rhs(u, P) for u in U], 1e-11),
                        (rk.chem_jvp(m, Ug, torch.tensor(V, device="cuda"), P, mode=mode),
                         [kin.jvp(u, P, v) for u, v in zip(U, V)], bar)):
        got, ref = got.cpu().numpy(), np.array(ref)
        assert np.max(np.abs(got - ref) / np.max(np.abs(ref), axis=1, keepdims=True)) < b


@pytest.mark.parametrize("size,precision", [((150, 2500, 0), 0), ((150, 2500, 0), 5), ((150, 2500, 0), 6),
                                            ((120, 1000, 40), 1), ((120, 1000, 40), 3), ((120, 1000, 40), 6)])
def test_one_step(rk, size, precision):
    from oracle import rok4e as orok

    mech, kin = _mech(*size)
    U = _states(mech)
    m = rk.mech_load(mech)
    Y = torch.tensor(U, device="cuda")
    stats = torch.zeros(len(U), 4, dtype=torch.int32, device="cuda")
    trace = torch.zeros(len(U), 512, dtype=torch.float64, device="cuda")
    dt = 2e-8
    rk.rok4e_integrate(m, Y, dt, 1e-6, 1e-10, 4, stats=stats, opts=rk.Opts(trace=trace, precision=precision))
    assert (stats[:, 3] == 0).all()
    replay = [[(abs(h), h > 0) for h in r if h != 0.0] for r in trace.cpu().numpy()]
    ref, _ = orok.integrate_cells(kin, U, P, dt, 1e-6, 1e-10, 4, replay=replay)
    got = Y.cpu().numpy()
    assert np.all(np.abs(got[:, :-1] - ref[:, :-1]) <= 1e-8 + 1e-6 * np.abs(ref[:, :-1]))
    assert np.max(np.abs(got[:, -1] - ref[:, -1])) <= 1e-6


@pytest.mark.parametrize("size,precision", [((150, 2500, 0), 1), ((150, 2500, 0), 2), ((150, 2500, 0), 3),
                                            ((150, 2500, 0), 4), ((120, 1000, 40), 2), ((120, 1000, 40), 4)])
def test_levels_that_do_not_fit_are_refused(rk, size, precision):
    mech, _ = _mech(*size)
    m = rk.mech_load(mech)
    Y = torch.tensor(_states(mech), device="cuda")
    with pytest.raises(rk.RokError, match="shared memory"):
        rk.rok4e_integrate(m, Y, 2e-8, 1e-6, 1e-10, 4, opts=rk.Opts(precision=precision))
