"""The fixed-point form of the reactions and of the species gather, where it can
go wrong: the ends of its temperature range, Gibbs factors and Arrhenius
coefficients that send a cell to the direct form, zero, tiny and negative mass
fractions, few and many cells to a block.  Bars as in the parity tests: the
source term and J v within 1e-11 of the row scale of the FP64 oracle; the
launch shape never changes a bit."""

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


def _mech(name):
    from synth.fields import WORKLOADS, mechanism_for
    from synth.mechanism import generate_mechanism

    if name == "pressure":  # more pressure-dependent reactions than the group sums together
        return generate_mechanism(30, 150, seed=1002, n_third_body=9, n_troe=3, k_cap=1e8, T_window=(300.0, 2200.0))
    return mechanism_for(WORKLOADS[name])


def _check(rk, mech, U, bar=1e-11):
    from oracle.kinetics import Kinetics

    kin = Kinetics(mech)
    m = rk.mech_load(mech)
    V = np.random.default_rng(5).normal(size=U.shape)
    Ug, Vg = torch.tensor(U, device="cuda"), torch.tensor(V, device="cuda")
    for got, ref in ((rk.chem_rhs(m, Ug, P), [kin.rhs(u, P) for u in U]),
                     (rk.chem_jvp(m, Ug, Vg, P), [kin.jvp(u, P, v) for u, v in zip(U, V)])):
        got, ref = got.cpu().numpy(), np.array(ref)
        scale = np.max(np.abs(ref), axis=1, keepdims=True)
        assert np.all(np.isfinite(got))
        assert np.all(np.abs(got - ref) <= bar * scale)  # (a species alone does not react: both zero)


@pytest.mark.parametrize("name", ["small", "flame1d", "pressure", "batched"])
def test_temperatures_around_the_range(rk, name):
    """150 K is the lower end of the fixed-point form; below it the direct form runs."""
    mech = _mech(name)
    T = np.array([120.0, 149.0, np.nextafter(150.0, 0), 150.0, np.nextafter(150.0, 151), 256.0, 511.9999, 1024.0, 4000.0])
    U = np.concatenate([np.random.default_rng(1).dirichlet(np.full(mech.n_species, 0.5), len(T)), T[:, None]], 1)
    _check(rk, mech, U)


@pytest.mark.parametrize("name", ["small", "flame1d", "batched"])
def test_zero_tiny_and_negative_mass_fractions(rk, name):
    mech = _mech(name)
    rng = np.random.default_rng(2)
    Y = rng.dirichlet(np.full(mech.n_species, 0.5), 8)
    Y[0, ::2] = 0.0
    Y[1, 1:] = 0.0
    Y[2, ::3] = 1e-300
    Y[3, ::3] = 5e-324
    Y[4, ::4] = -1e-9
    Y[5] = 10.0 ** rng.uniform(-150, 0, mech.n_species)
    Y[6, :] = 0.0
    Y[6, 3] = 1.0
    _check(rk, mech, np.concatenate([Y, rng.uniform(400.0, 2500.0, (8, 1))], 1))


@pytest.mark.parametrize("name", ["small", "flame1d", "batched"])
def test_large_gibbs_factors_take_the_direct_form(rk, name):
    """An element-additive shift of the enthalpies cancels from every reaction but
    carries |g/RT| past 170 in the cold cells."""
    mech = _mech(name)
    mech.nasa[:, 8] -= 60000.0 * mech.elem[:, 1]
    mech.nasa[:, 15] -= 60000.0 * mech.elem[:, 1]
    T = np.linspace(300.0, 2500.0, 9)
    U = np.concatenate([np.random.default_rng(3).dirichlet(np.full(mech.n_species, 0.5), len(T)), T[:, None]], 1)
    _check(rk, mech, U)


@pytest.mark.parametrize("change", ["b", "A", "Ea"])
def test_coefficients_outside_the_fixed_point_range(rk, change):
    mech = _mech("small")
    if change == "b":
        mech.arrh[3, 1] = 20.0
        mech.arrh[3, 0] *= 1e-60
    elif change == "A":
        mech.arrh[3, 0] = 1e-140
    else:
        mech.arrh[3, 2] = 2.0e6
    T = np.linspace(300.0, 2500.0, 7)
    U = np.concatenate([np.random.default_rng(4).dirichlet(np.full(mech.n_species, 0.5), len(T)), T[:, None]], 1)
    _check(rk, mech, U)


def test_non_finite_states_give_non_finite_rates(rk):
    mech = _mech("batched")
    m = rk.mech_load(mech)
    U = np.concatenate([np.random.default_rng(6).dirichlet(np.full(mech.n_species, 0.5), 4), np.full((4, 1), 900.0)], 1)
    U[0, 5] = np.nan
    U[1, -1] = np.nan
    U[2, 7] = np.inf
    out = rk.chem_rhs(m, torch.tensor(U, device="cuda"), P).cpu().numpy()
    assert not np.isfinite(out[:3, -1]).any() and np.isfinite(out[3]).all()


@pytest.mark.parametrize("name,precision", [("small", 0), ("flame1d", 0), ("batched", 0), ("batched", 6)])
def test_cells_per_block_never_change_a_bit(rk, name, precision):
    """One, eight (256 threads), ten (384) and sixteen cells a block (512 where they
    fit), more cells than the device holds at once."""
    mech = _mech(name)
    m = rk.mech_load(mech)
    n = 8 * torch.cuda.get_device_properties(0).multi_processor_count + 37
    rng = np.random.default_rng(7)
    U = np.concatenate([rng.dirichlet(np.full(mech.n_species, 0.5), n), rng.uniform(900.0, 1500.0, (n, 1))], 1)
    ref = None
    for cells in (0, 1, 8, 10, 16):
        Y = torch.tensor(U, device="cuda")
        h = torch.zeros(n, dtype=torch.float64, device="cuda")
        stats = torch.zeros(n, 4, dtype=torch.int32, device="cuda")
        for _ in range(2):
            rk.rok4e_integrate(m, Y, 2e-8, 1e-6, 1e-10, 4, h_cell=h, stats=stats,
                               opts=rk.Opts(cells_per_block=cells, precision=precision))
        got = (Y, h, stats)
        ref = ref or got
        assert all(torch.equal(a, b) for a, b in zip(got, ref)), cells


def test_cells_that_are_no_state_are_not_finite_and_fail(rk):
    """All mass fractions zero or tiny (an unset cell; sum Y/W at or below the smallest
    number whose reciprocal the right-hand side forms), a zero temperature: the source term
    is not finite, the integrators say so and touch no other cell."""
    for name in ("small", "batched"):
        mech = _mech(name)
        m = rk.mech_load(mech)
        ns = mech.n_species
        U = np.concatenate([np.random.default_rng(11).dirichlet(np.full(ns, 0.5), 6), np.full((6, 1), 1100.0)], 1)
        U[0, :-1] = 0.0
        U[1, :-1] = 1e-60
        U[2, -1] = 0.0
        U[3, :-1] = -0.0
        U[4, :-1] = 5e-324
        Ug = torch.tensor(U, device="cuda")
        out = rk.chem_rhs(m, Ug, P).cpu().numpy()
        assert not np.isfinite(out[:5, -1]).any() and np.isfinite(out[5]).all()
        rho = torch.full((6,), 0.2, dtype=torch.float64, device="cuda")
        out = rk.chem_rhs_cv(m, Ug, rho).cpu().numpy()  # (fixed density: the mixture's heat capacity is what is zero)
        assert not np.isfinite(out[:5, -1]).any() and np.isfinite(out[5]).all()
        for run in (lambda y, st: rk.rok4e_integrate(m, y, 1e-8, 1e-6, 1e-10, 4, stats=st),
                    lambda y, st: rk.rkdp_integrate(m, y, 1e-8, 1e-6, 1e-10, stats=st)):
            Y, stats = Ug.clone(), torch.zeros(6, 4, dtype=torch.int32, device="cuda")
            run(Y, stats)
            alone, one = Ug[5:].clone(), torch.zeros(1, 4, dtype=torch.int32, device="cuda")
            run(alone, one)
            st = stats.cpu().numpy()
            assert (st[:5, 3] != 0).all() and st[5, 3] == 0
            assert torch.equal(Y[5:], alone)


def _terms(kin, u, v):
    """Each entry's sum of the magnitudes of its terms: of the source term's species rows
    and of the Jacobian-vector product's (elementary reactions only for the latter)."""
    st = kin.state(u, P)
    nu, W, ns = np.abs(kin.nu), kin.W, kin.ns
    f, b = st["m"] * st["k"] * st["Pf"], st["m"] * st["kr"] * st["Pb"]
    rhs = W / st["rho"] * (nu.T @ (f + b))
    drr = np.sum(np.abs(v[:ns]) / W) / st["S"] + abs(v[ns]) / st["T"]
    dC = st["rho"] / W * np.abs(v[:ns]) + st["C"] * drr

    def dprod(n):  # sum over factors of |dC| times the others
        out = np.zeros(len(n), dtype=dC.dtype)
        for j, row in enumerate(n):
            ks = [k for k in np.flatnonzero(row) for _ in range(int(row[k]))]
            for i, k in enumerate(ks):
                out[j] += dC[k] * np.prod([st["C"][q] for q in ks[:i] + ks[i + 1:]])
        return out

    dT = np.abs(st["dlnk"]) * (f + b) + np.abs(st["dlnKc"]) * b
    dq = st["m"] * (st["k"] * dprod(kin.nu_f) + st["kr"] * dprod(kin.nu_r)) + dT * abs(v[ns])
    return rhs, W / st["rho"] * (nu.T @ (dq + drr * (f + b)))


@pytest.mark.parametrize("name", ["flame1d", "batched", "adjoint"])
@pytest.mark.parametrize("T", [200.0, 300.0, 600.0])
def test_slow_rows_of_unburnt_mixtures_entry_by_entry(rk, name, T):
    """Six species present, the others zero: the rows of the first radicals lie tens of
    orders of magnitude below the fastest.  Every entry within 1e-12 of its own terms'
    magnitudes: exponents of at most ~300 in all with about ten roundings of 2^-53 of that on
    either side (3.4e-13), and the sums' own."""
    from oracle.kinetics import Kinetics

    mech = _mech(name)
    kin = Kinetics(mech)
    m = rk.mech_load(mech)
    rng = np.random.default_rng(12)
    U = np.zeros((24, mech.n_species + 1))
    for u in U:
        u[rng.permutation(mech.n_species)[:6]] = rng.dirichlet(np.full(6, 0.5))
    U[:, -1] = T
    V = rng.normal(size=U.shape) * (U != 0)  # along what is there
    Ug = torch.tensor(U, device="cuda")
    f = rk.chem_rhs(m, Ug, P).cpu().numpy()
    jv = rk.chem_jvp(m, Ug, torch.tensor(V, device="cuda"), P).cpu().numpy()
    for c, (u, v) in enumerate(zip(U, V)):
        sf, sj = _terms(kin, u, v)
        assert np.all(np.abs(f[c, :-1] - kin.rhs(u, P)[:-1]) <= 1e-12 * sf)
        if not (mech.kind > 0).any():
            assert np.all(np.abs(jv[c, :-1] - kin.jvp(u, P, v)[:-1]) <= 1e-12 * sj)


def _extended(kin):
    """The oracle with its arrays in numpy's long double (15-bit exponents)."""
    import copy

    ext = copy.copy(kin)
    for name, v in vars(kin).items():
        if isinstance(v, np.ndarray) and v.dtype == np.float64:
            setattr(ext, name, v.astype(np.longdouble))
    return ext


def test_sums_past_the_largest_double(rk):
    """Rates just below the largest double, three quarters of them of one reaction written many
    times: a species row past the largest double is not finite, one whose terms stay below it is
    right.  (1e-11: as the parity tests, of the magnitudes of the row's terms.)"""
    from oracle.kinetics import Kinetics

    mech = _mech("batched")
    mech.arrh[:, 0] *= 1e34
    U = np.concatenate([np.random.default_rng(13).dirichlet(np.full(53, 0.5), 4), np.full((4, 1), 1400.0)], 1)
    fastest = int(np.argmax(np.abs(Kinetics(mech).rop(U[0], 1e60))))
    for a in (mech.rxn_sp, mech.rxn_nu, mech.arrh, mech.reversible, mech.kind):
        a[80:] = a[fastest]
    kin = Kinetics(mech)
    ext = _extended(kin)
    m = rk.mech_load(mech)
    past = 0
    for u in U:
        lo, hi = 90.0, 145.0  # the pressure's exponent that puts the largest rate at ~1.5e308
        for _ in range(40):
            mid = 0.5 * (lo + hi)
            over = np.max(np.abs(ext.state(u.astype(np.longdouble), np.longdouble(10.0) ** mid)["q"])) > np.longdouble("1.5e308")
            lo, hi = (lo, mid) if over else (mid, hi)
        p = 10.0 ** lo
        st = ext.state(u.astype(np.longdouble), np.longdouble(p))
        terms = np.abs(kin.nu).T @ np.abs(st["q"])
        scale = kin.W / st["rho"] * (np.abs(kin.nu).T @ (st["m"] * (st["k"] * st["Pf"] + st["kr"] * st["Pb"])))
        f = rk.chem_rhs(m, torch.tensor(u[None], device="cuda"), p).cpu().numpy()[0, :-1]
        ref = ext.rhs(u.astype(np.longdouble), np.longdouble(p))[:-1]
        far, within = np.abs(st["omega"]) > np.finfo(float).max, terms < 0.5 * np.finfo(float).max
        past += far.sum()
        assert not np.isfinite(f[far]).any()
        assert np.all(np.abs(f[within] - ref[within]) <= 1e-11 * scale[within])
    assert past >= 8


@pytest.mark.parametrize("p", [P, 1e-100])
def test_rates_below_the_normal_range(rk, p):
    """Irreversible reactions with rate constants near 2^-350 and a mixture of a few species with 1e-102 of the others, or
    all of them at a pressure of 1e-100 Pa: rates of progress among the subnormal numbers, alone
    in their rows or all a cell has.  1e-11 of the terms' magnitudes and 64 units of the
    smallest double a row for their own rounding."""
    from oracle.kinetics import Kinetics

    mech = _mech("batched")
    mech.arrh[:, 0] *= 1e-40
    mech.arrh[:, 2] = 3.8e5
    mech.reversible[:] = 0
    kin = Kinetics(mech)
    ext = _extended(kin)
    rng = np.random.default_rng(14)
    U = np.concatenate([rng.dirichlet(np.full(53, 0.5), 8), np.full((8, 1), 300.0)], 1)
    if p == P:
        for u in U:
            u[rng.permutation(53)[6:]] *= 1e-102
    got = rk.chem_rhs(rk.mech_load(mech), torch.tensor(U, device="cuda"), p).cpu().numpy()[:, :-1]
    below = 0
    for g, u in zip(got, U):
        st = ext.state(u.astype(np.longdouble), np.longdouble(p))
        ref = kin.W / st["rho"] * st["omega"]
        terms = np.abs(kin.nu).T @ (st["k"] * st["Pf"] + st["kr"] * st["Pb"])
        below += np.sum((np.abs(st["omega"]) < 2.2e-308) & (np.abs(st["omega"]) > 1e-315))
        assert np.all(np.abs(g - ref) <= kin.W / st["rho"] * (1e-11 * terms + 64 * 5e-324) + 5e-324)
    assert below >= 8


@pytest.mark.parametrize("case", ["cold", "thin"])
def test_small_rate_constants_and_fractions_with_extreme_gibbs_factors(rk, case):
    """An element-additive enthalpy shift carries g/RT to +-160.  cold: rate constants of
    ~2^-800, so that k / (E E) is below the normal range where k C C is not.  thin: fractions
    of 1e-120, so that the products of C E are.  Every entry within 1e-12 of its terms'
    magnitudes times twice the exponents of the mixtures above (E of up to 160: 2e-12 with
    g/RT's own rounding, five operations on terms of up to ~200)."""
    from oracle.kinetics import Kinetics

    mech = _mech("batched")
    T = 160.0 if case == "cold" else 300.0
    atoms = mech.elem.sum(1)
    kin0 = Kinetics(mech)
    _, h, s, _ = kin0.thermo(T)
    c = (1.0 if case == "cold" else -1.0) * min((160.0 - abs(x)) * T / n for x, n in zip(h - s + np.log(T / 1.2e4), atoms))
    mech.nasa[:, 8] += c * atoms
    mech.nasa[:, 15] += c * atoms
    mech.reversible[:] = 0
    rng = np.random.default_rng(15)
    U = np.concatenate([rng.dirichlet(np.full(53, 0.5), 8), np.full((8, 1), T)], 1)
    if case == "cold":
        mech.arrh[:, 0] *= 1e-40
        mech.arrh[:, 2] = 6.8e5
    else:
        for u in U:
            u[rng.permutation(53)[6:]] *= 1e-120
    assert rk.mech_validate(mech) == ""
    kin = Kinetics(mech)
    ext = _extended(kin)
    V = rng.normal(size=U.shape) * U
    m = rk.mech_load(mech)
    Ug = torch.tensor(U, device="cuda")
    f = rk.chem_rhs(m, Ug, P).cpu().numpy()
    jv = rk.chem_jvp(m, Ug, torch.tensor(V, device="cuda"), P).cpu().numpy()
    for g, j, u, v in zip(f, jv, U.astype(np.longdouble), V.astype(np.longdouble)):
        sf, sj = _terms(ext, u, v)
        assert np.all(np.abs(g[:-1] - ext.rhs(u, np.longdouble(P))[:-1]) <= 2e-12 * sf)
        assert np.all(np.abs(j[:-1] - ext.jvp(u, np.longdouble(P), v)[:-1]) <= 2e-12 * sj)


def test_temperature_direction_of_the_fp32_product(rk):
    """J v of precision 6 along T: every reaction and the density take the same FP32 factor
    vT / T, so its rounding scales the whole row, the median over the species being hardly
    touched by their own.  Rounded once it is off by 0.36 x 2^-24 on average, as a product of
    rounded factors by 0.58; the line is between the two."""
    mech = _mech("batched")
    m = rk.mech_load(mech)
    n = 4000
    rng = np.random.default_rng(16)
    U = np.concatenate([rng.dirichlet(np.full(53, 0.5), n), rng.uniform(900.0, 2500.0, (n, 1))], 1)
    V = np.zeros_like(U)
    V[:, -1] = rng.uniform(0.5, 1.0, n)
    Ug, Vg = torch.tensor(U, device="cuda"), torch.tensor(V, device="cuda")
    a, b = (rk.chem_jvp(m, Ug, Vg, P, mode=k).cpu().numpy()[:, :-1] for k in (0, 5))
    factor = np.median(b / a - 1.0, axis=1)
    assert np.mean(np.abs(factor)) < 0.47 * 2.0 ** -24
