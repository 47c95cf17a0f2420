"""GPU parity of the thermophysical and transport property kernels against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2312_13513_gb300 as cg  # noqa: E402
from oracle import transport as ot  # noqa: E402
from synth.states import les_field, load_table, quasi_dns_field  # noqa: E402
from synth.transport import generate_transport  # noqa: E402

from gpu_common import to_dev  # noqa: E402
from helpers import random_states, with_inert_species  # noqa: E402

pytestmark = pytest.mark.gpu


def _states(kind, mech, n, seed):
    if kind == "h2":
        f = quasi_dns_field(load_table("h2_flamelet.npz"), n=n, seed=seed)
    else:
        f = les_field(load_table("ch4_flamelet.npz"), n=n, seed=seed)
    return f["T"], f["p"], f["Y"]


@pytest.mark.parametrize("kind", ["h2", "ch4"])
def test_transport_matches_oracle(kind, h2, ch4):
    mech = h2 if kind == "h2" else ch4
    tr = generate_transport(mech)
    T, p, Y = _states(kind, mech, 700, 41)
    p = p * np.linspace(0.5, 3.0, p.size)              # pressure varies across cells
    dm = cg.Mechanism(mech)
    gt = cg.Transport(dm, tr)
    Td, pd, Yd = to_dev(T, p, Y)
    mu = torch.empty_like(Td); lam = torch.empty_like(Td); D = torch.empty_like(Yd)
    gt(Td, pd, Yd, mu, lam, D)
    torch.cuda.synchronize()
    mu_r, lam_r, D_r = ot.mixture_cells(tr, mech.W, T, p, Y)
    assert np.allclose(mu.cpu().numpy(), mu_r, rtol=1e-11, atol=0)
    assert np.allclose(lam.cpu().numpy(), lam_r, rtol=1e-11, atol=0)
    assert np.allclose(D.cpu().numpy(), D_r, rtol=1e-11, atol=0)


def test_transport_pure_species_and_optional_outputs(h2):
    tr = generate_transport(h2)
    n = h2.ns
    Y = np.eye(n)                                      # cell k holds species k alone
    T = np.linspace(400.0, 2800.0, n)
    p = np.full(n, 1.01325e6)
    dm = cg.Mechanism(h2)
    gt = cg.Transport(dm, tr)
    Td, pd, Yd = to_dev(T, p, Y)
    D = torch.empty_like(Yd)
    gt(Td, pd, Yd, D=D)                                # viscosity and conductivity not requested
    torch.cuda.synchronize()
    for k in range(n):
        _, _, Djk = ot.pure_species(tr, T[k], p[k])
        assert D[k, k].item() == pytest.approx(Djk[k, k], rel=1e-12)


def test_mixture_thermo_matches_oracle(h2, om_h2):
    T, p, Y = random_states(h2, 500, 43, "H2", Tlo=300.0, Thi=2900.0)
    dm = cg.Mechanism(h2)
    Td, _, Yd = to_dev(T, p, Y)
    h = torch.empty_like(Td); cp = torch.empty_like(Td)
    cg.mixture_thermo(dm, Td, Yd, h, cp)
    torch.cuda.synchronize()
    h_r = np.array([om_h2.enthalpy_mass(T[i], Y[:, i]) for i in range(T.size)])
    cp_r = np.array([om_h2.cp_mass(T[i], Y[:, i]) for i in range(T.size)])
    assert np.allclose(h.cpu().numpy(), h_r, rtol=1e-12, atol=1e-6 * np.abs(h_r).max())
    assert np.allclose(cp.cpu().numpy(), cp_r, rtol=1e-12, atol=0)


def test_temperature_from_enthalpy_recovers_temperature(ch4, om_ch4):
    T, p, Y = _states("ch4", ch4, 400, 44)
    h0 = np.array([om_ch4.enthalpy_mass(T[i], Y[:, i]) for i in range(T.size)])
    dm = cg.Mechanism(ch4)
    guess = T + np.where(np.arange(T.size) % 2 == 0, 250.0, -150.0)
    guess = np.clip(guess, 250.0, 3000.0)
    Td, _, Yd = to_dev(guess, p, Y)
    hd = torch.tensor(h0, device="cuda")
    st = torch.full((T.size,), 7, dtype=torch.int8, device="cuda")
    cg.temperature_from_enthalpy(dm, hd, Yd, Td, st)
    torch.cuda.synchronize()
    assert int(st.abs().sum()) == 0
    assert np.allclose(Td.cpu().numpy(), T, rtol=1e-9, atol=0)


def test_temperature_from_enthalpy_flags_failures(h2):
    dm = cg.Mechanism(h2)
    T, p, Y = random_states(h2, 4, 45, "H2", Tlo=800.0, Thi=1200.0)
    Td, _, Yd = to_dev(T, p, Y)
    h = torch.tensor([np.nan, 1e30, -1e30, 0.0], device="cuda", dtype=torch.float64)
    st = torch.zeros(4, dtype=torch.int8, device="cuda")
    before = Td.clone()
    cg.temperature_from_enthalpy(dm, h, Yd, Td, st)
    torch.cuda.synchronize()
    s = st.cpu().numpy()
    assert s[0] == 1 and s[1] == 1 and s[2] == 1
    assert torch.equal(Td[:3], before[:3])             # unconverged cells keep their temperature


@pytest.mark.parametrize("ns", [9, 15, 16])
def test_transport_at_the_edges_of_its_ranges(h2, ns):
    """Both kernels (one thread per cell up to 15 species, a warp per cell beyond) inside, at and
    outside the temperatures of the fixed-point fits, [1, 65536), in odd numbers of cells."""
    mech = with_inert_species(h2, ns - h2.ns) if ns > h2.ns else h2
    tr = generate_transport(mech)
    T = np.array([0.5, np.nextafter(1.0, 0.0), 1.0, 250.0, 1000.0, 3500.0, np.nextafter(65536.0, 0.0), 65536.0, 2e5] * 5)[:41]
    rng = np.random.default_rng(47)
    Y = rng.dirichlet(np.full(mech.ns, 0.4), T.size).T.copy()
    Y[:, 40] = 0.0; Y[0, 40] = 1.0                      # one species alone
    p = np.full(T.size, 1.01325e6)
    dm = cg.Mechanism(mech)
    gt = cg.Transport(dm, tr)
    Td, pd, Yd = to_dev(T, p, Y)
    mu = torch.empty_like(Td); lam = torch.empty_like(Td); D = torch.empty_like(Yd)
    gt(Td, pd, Yd, mu, lam, D)
    torch.cuda.synchronize()
    mu_r, lam_r, D_r = ot.mixture_cells(tr, mech.W, T, p, Y)
    for got, ref in ((mu, mu_r), (lam, lam_r), (D, D_r)):
        assert np.allclose(got.cpu().numpy(), ref, rtol=1e-11, atol=0)


@pytest.mark.parametrize("kind", ["h2", "ch4"])
def test_enthalpies_at_the_edges_of_the_fixed_point_range(kind, h2, ch4):
    """Mixture h, cp and heat release at the ends of both polynomial ranges and of the fixed-point
    range [128, 4096), and outside it, against the NASA polynomials in extended precision."""
    mech = h2 if kind == "h2" else ch4
    T = np.array([90.0, np.nextafter(128.0, 0), 128.0, 298.15, np.nextafter(1000.0, 0), 1000.0, 1023.5, 1024.0, 2900.0,
                  np.nextafter(4096.0, 0), 4096.0, 5500.0] * 3)[:35]
    rng = np.random.default_rng(48)
    Y = rng.dirichlet(np.full(mech.ns, 0.4), T.size).T.copy()
    Y1 = rng.dirichlet(np.full(mech.ns, 0.4), T.size).T.copy()
    p = np.full(T.size, 1.01325e6)
    dm = cg.Mechanism(mech)
    Td, pd, Yd = to_dev(T, p, Y)
    h = torch.empty_like(Td); cp = torch.empty_like(Td)
    cg.mixture_thermo(dm, Td, Yd, h, cp)
    q = cg.heat_release(dm, Td, pd, Yd, to_dev(T, p, Y1)[2], 1e-6)
    torch.cuda.synchronize()
    L = np.longdouble
    a = np.where((T < 1000.0)[None, None], mech.nasa_lo[:, :, None], mech.nasa_hi[:, :, None]).astype(L)   # [ns, 7, n]
    t = T.astype(L)
    terms = np.stack([a[:, 5]] + [a[:, i] * t ** (i + 1) / (i + 1) for i in range(5)])
    cterms = np.stack([a[:, i] * t ** i for i in range(5)])
    w = 1.0 / mech.W.astype(L)[:, None]
    ru = L(8.314462618e7)
    # 1e-13 of the magnitudes that are summed: 2^-42 K times a dozen units in fixed point (about
    # 3e-12 K against hundreds), about ten roundings of 1.1e-16 in FP64
    for got, ref, mag in ((h, ru * (terms.sum(0) * Y * w).sum(0), ru * (np.abs(terms).sum(0) * Y * w).sum(0)),
                          (cp, ru * (cterms.sum(0) * Y * w).sum(0), ru * (np.abs(cterms).sum(0) * Y * w).sum(0)),
                          (q, -(p / (t * (Y * w).sum(0))) * (terms.sum(0) * (Y1.astype(L) - Y) * w).sum(0) / L(1e-6),
                           p / (t * (Y * w).sum(0)) * (np.abs(terms).sum(0) * (Y1 + Y) * w).sum(0) / L(1e-6))):
        assert np.all(np.abs(got.cpu().numpy() - ref) <= 1e-13 * mag)
