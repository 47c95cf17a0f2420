"""Forms of mechanism that the loader accepts and that the synthetic mechanisms do not have, in every
integrator kernel, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_2312_13513_gb300 as cg  # noqa: E402

from gpu_common import assert_parity, to_dev  # noqa: E402
from helpers import random_states, with_inert_species  # noqa: E402

pytestmark = pytest.mark.gpu


def _states(base, m, n, seed, fuel):
    """Seeded states of the base mechanism, with a little of every species appended to it."""
    T, p, Y = random_states(base, n, seed, fuel, Tlo=300.0, Thi=2600.0)
    Y = np.vstack([Y, np.full((m.ns - base.ns, n), 1e-3)])
    return T, p, Y / Y.sum(axis=0)


def _rate_magnitudes(om, m, T, p, Y):
    """Of each component of f, the sum of its terms' magnitudes: forward and reverse rates apart."""
    _, _, kf, kr = om.rates(T, p, Y)
    cp, h, _, _ = om.thermo(T)
    rho = p / (om.RU * T * np.sum(Y / m.W))
    C = np.append(rho * Y / m.W, 1.0)                  # an empty slot reads 1
    r = kf * C[m.reac].prod(1) + kr * C[m.prod].prod(1)
    r = np.where(m.rtype == 1, (m.eff * C[:-1]).sum(1), 1.0) * r
    w = np.zeros(m.ns + 1)
    for s in (m.reac, m.prod):
        for i in range(3):
            np.add.at(w, s[:, i], r)
    w = w[:-1]
    return np.r_[T * (np.abs(h) @ w) / (rho * (cp @ (Y / m.W))), m.W * w / rho]


def _assert_rhs_jac(m, T, p, Y, cancel=False):
    """f and the Jacobian against the oracle: 1e-10 of each rate and of each column's largest entry (the
    sums of up to a few hundred terms, each good to about 1e-13), as in test_rhs_and_jacobian_parity;
    cancel: 1e-12 of the magnitudes summed in each rate, where forward and reverse ones nearly cancel."""
    om, N = oracle.OracleMech(m), m.ns + 1
    f, J = (a.cpu().numpy() for a in cg.eval_rhs_jac(cg.Mechanism(m), *to_dev(T, p, Y)))
    for c in range(T.size):
        y = np.r_[T[c], Y[:, c]]
        fr, Jr = om.rhs(p[c], y), om.jacobian(p[c], y)
        tol = 1e-10 * (np.abs(fr) + 1e-12 * np.max(np.abs(fr))) + 1e-300
        if cancel:
            tol = np.maximum(tol, 1e-12 * _rate_magnitudes(om, m, T[c], p[c], Y[:, c]))
        assert np.all(np.abs(f[:, c] - fr) <= tol), (c, T[c])
        sc = np.max(np.abs(Jr), axis=0) + 1e-300
        assert np.all(np.abs(J[:, c].reshape(N, N) - Jr) <= 1e-10 * sc), (c, T[c])


def _assert_advance(m, T, p, Y, dt, group):
    Td, pd, Yd = to_dev(T, p, Y)
    st = torch.full((T.size,), -1, dtype=torch.int8, device="cuda")
    cg.advance(cg.Mechanism(m), Td, pd, Yd, dt, status=st, opts=cg.options(group_threads=group) if group else None)
    assert torch.all(st == 0)
    assert_parity(oracle.OracleMech(m), T, p, Y, Td.cpu().numpy(), Yd.cpu().numpy(), dt, 1e-6, 1e-10)


def _shuffled_slots(m, seed):
    """The same reactions with the species of each side in any of its three places."""
    m = m.copy()
    rng = np.random.default_rng(seed)
    m.reac, m.prod = rng.permuted(m.reac, axis=1), rng.permuted(m.prod, axis=1)
    return m


@pytest.mark.parametrize("base,inert", [("h2", 0), ("h2", 7), ("ch4", 0), ("ch4", 1), ("ch4", 12)])
def test_empty_slots_in_any_place(base, inert, request):
    """An empty slot before a species: odd and even species counts, each integrator kernel."""
    b = request.getfixturevalue(base)
    m = _shuffled_slots(with_inert_species(b, inert) if inert else b, 70 + inert)
    assert np.any(m.reac[:, 0] < 0) and np.any(m.prod[:, 0] < 0)
    T, p, Y = _states(b, m, 37, 71 + inert, base.upper())
    _assert_rhs_jac(m, T, p, Y)
    for group in (0, 64):
        _assert_advance(m, T, p, Y, 5e-7, group)


def _without_reactions(m):
    m = m.copy()
    for a in ("rtype", "reac", "prod", "A", "b", "Ea", "troe", "has_t2", "eff"):
        setattr(m, a, getattr(m, a)[:0].copy())
    return m


@pytest.mark.parametrize("form", ["none", "no net production"])
@pytest.mark.parametrize("base,inert", [("h2", 0), ("h2", 7), ("ch4", 0)])
def test_mechanism_that_changes_nothing(base, inert, form, request):
    """No reactions at all, or none with a net production: no entry in the Jacobian's programs.  Every
    rate is an exact zero, so the state comes back as it was."""
    b = request.getfixturevalue(base)
    m = with_inert_species(b, inert) if inert else b.copy()
    if form == "none":
        m = _without_reactions(m)
    else:
        m.prod = m.reac.copy()
    T, p, Y = _states(b, m, 19, 72, base.upper())
    dm = cg.Mechanism(m)
    f, J = cg.eval_rhs_jac(dm, *to_dev(T, p, Y))
    assert torch.all(f == 0.0) and torch.all(J == 0.0)
    for group in (0, 64):
        Td, pd, Yd = to_dev(T, p, Y)
        st = torch.full((T.size,), -1, dtype=torch.int8, device="cuda")
        cg.advance(dm, Td, pd, Yd, 1e-6, status=st, opts=cg.options(group_threads=group) if group else None)
        assert torch.all(st == 0)
        assert np.array_equal(Td.cpu().numpy(), T) and np.array_equal(Yd.cpu().numpy(), Y)


@pytest.mark.parametrize("ns", [139, 140, 141])
def test_largest_mechanisms(h2, ns):
    """Where one cell's workspace is all the shared memory of a block (227 KB): 139 species are the last
    that fit in fixed point (16 bytes short), 140 the last that fit in FP64, 141 are refused."""
    m = with_inert_species(h2, ns - h2.ns)
    T, p, Y = _states(h2, m, 9, 73, "H2")
    if ns > 140:
        with pytest.raises(cg.ChemError):
            cg.eval_rhs_jac(cg.Mechanism(m), *to_dev(T, p, Y))
        return
    _assert_rhs_jac(m, T, p, Y)
    _assert_advance(m, T, p, Y, 5e-7, 0)


@pytest.mark.parametrize("base", ["h2", "ch4"])
def test_low_pressure_limit_far_below_the_other(base, request):
    """k0 = 2^-2296 and kinf = 2^989 at 130 K: their ratio is beyond the range of a fixed-point exponent
    by more than its width.  k0 is 0 in FP64, and so is the rate."""
    b = request.getfixturevalue(base)
    m = b.copy()
    j = int(np.nonzero(m.rtype == 2)[0][0])
    m.A[j], m.b[j], m.Ea[j] = 1e150, 0.0, -8.8e4
    m.troe[j, :3] = 1e-170, 0.0, 3.1e5
    T, p, Y = _states(b, m, 12, 74, base.upper())
    _assert_rhs_jac(m, np.linspace(129.0, 133.0, T.size), p, Y)


def _three_a_side(m, base_ns, seed, balanced):
    """The mechanism with a third species on one or both sides of most reactions of every type: the same one
    on both (balanced), or also others, which make up to six net species."""
    m = m.copy()
    rng = np.random.default_rng(seed)
    for j in range(m.nr):
        kind = rng.integers(0, 2 if balanced else 4)
        k = rng.permutation(base_ns)
        k = k[~np.isin(k, np.r_[m.reac[j], m.prod[j]])]
        room = m.reac[j, 2] < 0 and m.prod[j, 2] < 0
        if kind == 0 or not room:
            continue
        m.reac[j, np.argmin(m.reac[j])] = k[0]
        m.A[j] *= 1e5                                # over a concentration of 1e-5 mol / cm^3
        m.troe[j, 0] *= 1e5
        if kind < 3:
            m.prod[j, np.argmin(m.prod[j])] = k[kind - 1]
    return m


@pytest.mark.parametrize("base,inert", [("h2", 0), ("h2", 2), ("h2", 7), ("ch4", 0)])
def test_three_species_on_a_side(base, inert, request):
    """Reactions of the general form in every kernel: any type, three species a side, six net species; inside
    and outside the fixed-point range."""
    b = request.getfixturevalue(base)
    wide = with_inert_species(b, inert) if inert else b
    m = _three_a_side(wide, b.ns, 75, False)
    three = (m.reac[:, 2] >= 0) | (m.prod[:, 2] >= 0)
    net = [len(set(np.r_[m.reac[j], m.prod[j]]) - {-1}) for j in range(m.nr)]
    assert all(np.any(three & (m.rtype == t)) for t in range(3)) and max(net) == 6 and not np.all(three)
    T, p, Y = _states(b, m, 31, 76, base.upper())
    _assert_rhs_jac(m, np.where(np.arange(T.size) % 5 == 0, 4500.0, T), p, Y, cancel=True)
    m = _three_a_side(wide, b.ns, 78, True)
    _assert_rhs_jac(m, np.where(np.arange(T.size) % 5 == 0, 110.0, T), p, Y, cancel=True)
    for group in (0, 64):
        _assert_advance(m, T, p, Y, 1e-7, group)
