"""Fixed-point exponentials, logarithms and reciprocals (fixed.cuh) and the cell-per-thread
integrator built on them: the functions against long double on the host, the kernel against the
group kernels and the oracle at its edges."""
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2312_13513_gb300", "csrc")

HOST = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "fixed.cuh"
using namespace chem::fx;
static const u64 E[256] = {CHEM_FX_EXP2_VALUES};
static const uint32_t R[128] = {CHEM_FX_RCP_VALUES};
static const u64 G[128] = {CHEM_FX_LOG2_VALUES};
int main() {
  std::mt19937_64 g(3);
  std::uniform_real_distribution<double> U(0, 1);
  double m[6] = {0, 0, 0, 0, 0, 0};
  auto up = [&](int i, long double v) { if (!(v <= m[i])) m[i] = (double)v; };
  for (int i = 0; i < 400000; ++i) {
    const i64 X = i < 2045 ? (i64)(i - 1022) << 52 : q52(U(g) * 2044.9 - 1022.0);   // whole powers first
    if (!exp2_in_range(X)) continue;
    const long double r = exp2l((long double)X / 4503599627370496.0L);
    const double y = exp2_q52(X, E);
    up(0, fabsl(y - r) / (nextafter((double)r, INFINITY) - (double)r));
    double x = (U(g) - 0.5) * (i & 1 ? 1400.0 : 40.0);
    const long double e = expl((long double)x);
    up(1, fabsl(exp2_q52(mulhi_su(q52(x) * 2, kLog2e), E) - e) / (nextafter((double)e, INFINITY) - (double)e));
    u64 mt = g() | 0x8000000000000000ull;
    if (i < 1000) mt = 0x8000000000000000ull + i;
    else if (i < 2000) mt = ~0ull - (i - 1000);
    const long double v = (long double)mt / 9223372036854775808.0L;
    up(2, fabsl((long double)(i64)log2_mant_q60(mt, R, G) - log2l(v) * 1152921504606846976.0L));
    up(3, fabsl((long double)rcp_mant(mt, R) - 18446744073709551616.0L / v));
    x = (U(g) - 0.5) * exp2(U(g) * 70 - 59);
    up(4, fabsl((long double)q52(x) - (long double)x * 4503599627370496.0L));
    const i64 w = (i64)g() >> (g() & 63);
    const long double wl = ldexpl((long double)w, -52);
    up(5, w ? fabsl((long double)to_double(w, 52) - wl) / (fabsl(wl) * 0x1p-53L) : (to_double(w, 52) == 0.0 ? 0 : 9));
  }
  printf("%.17g %.17g %.17g %.17g %.17g %.17g\n", m[0], m[1], m[2], m[3], m[4], m[5]);
}
"""


def test_tables_are_the_generator_output():
    out = subprocess.run([sys.executable, os.path.join(CSRC, "gen_fixed_tables.py")], capture_output=True,
                         text=True, check=True).stdout
    assert open(os.path.join(CSRC, "fixed_tables.h")).read().strip() == out.strip()


def test_functions_against_long_double(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(HOST)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    exp2_ulp, exp_ulp, log2_u, rcp_u, q_u, d_h = map(float, subprocess.run([exe], capture_output=True, text=True,
                                                                           check=True).stdout.split())
    # half an ulp of rounding plus 2^-58 / 2^-53 of truncation; exp adds two Q.52 truncations of
    # the exponent (ln 2 each, up to two ulps at the bottom of a binade)
    assert exp2_ulp <= 0.55 and exp_ulp <= 0.55 + 4 * np.log(2.0)
    # Taylor truncation plus one unit per product and table entry; Newton's last step
    assert log2_u <= 8.0 and rcp_u <= 8.0
    assert q_u <= 0.5 and d_h <= 1.0 + 1e-9


def _without_last_species(m):
    """The mechanism without its (inert) last species."""
    m = m.copy()
    m.species, m.W, m.comp = m.species[:-1], m.W[:-1], m.comp[:-1]
    m.nasa_lo, m.nasa_hi, m.eff = m.nasa_lo[:-1], m.nasa_hi[:-1], m.eff[:, :-1].copy()
    return m


def _mechs(h2):
    from helpers import with_inert_argon, with_inert_species
    fast = h2.copy()
    slow = h2.copy()
    slow.b[3], slow.Ea[5], slow.A[7] = 40.0, 0.0, 0.0            # outside the formats; no rate at all
    slow.A[3] = 1e-110
    return {"8": _without_last_species(fast), "9": fast, "10": with_inert_argon(fast),
            "11": with_inert_species(fast, 2), "slow": slow}


@pytest.mark.gpu
@pytest.mark.parametrize("which", ["8", "9", "10", "11", "slow"])
def test_rhs_and_jacobian_over_the_temperature_range(h2, which):
    """Both sides of every switch of the fixed-point range: 128, 1000 and 4096 K."""
    import oracle
    import paper_2312_13513_gb300 as cg
    from gpu_common import to_dev
    from helpers import random_states
    m = _mechs(h2)[which]
    om, dm = oracle.OracleMech(m), cg.Mechanism(m)
    T, p, Y = random_states(h2, 40, 5, "H2")
    Y = np.vstack([Y, np.full((max(0, m.ns - h2.ns), 40), 1e-3)])[:m.ns]
    edges = np.array([128.0, 1000.0, 4096.0])
    T = np.concatenate([np.nextafter(edges, 0), edges, np.geomspace(150.0, 5500.0, 34)])
    f, J = (a.cpu().numpy() for a in cg.eval_rhs_jac(dm, *to_dev(T, p, Y)))
    N = m.ns + 1
    for c in range(T.size):
        y = np.r_[T[c], Y[:, c]]
        fr, Jr = om.rhs(p[c], y), om.jacobian(p[c], y)
        assert np.all(np.abs(f[:, c] - fr) <= 1e-10 * (np.abs(fr) + 1e-12 * np.max(np.abs(fr))) + 1e-300), (which, T[c])
        sc = np.max(np.abs(Jr), axis=0) + 1e-300
        assert np.all(np.abs(J[:, c].reshape(N, N) - Jr) <= 1e-10 * sc), (which, T[c])


@pytest.mark.gpu
@pytest.mark.parametrize("which,n", [("8", 33), ("9", 1), ("9", 31), ("9", 32), ("9", 33), ("9", 20011), ("10", 129),
                                     ("11", 65), ("slow", 257)])
def test_advance_agrees_with_the_group_kernel(h2, which, n):
    """One thread per cell against two lanes per cell (the general kernel): the same method, so
    within the parity contract cell by cell, whatever fills the last warp."""
    import torch
    import paper_2312_13513_gb300 as cg
    from gpu_common import to_dev, within
    from helpers import random_states
    m = _mechs(h2)[which]
    dm = cg.Mechanism(m)
    T, p, Y = random_states(h2, n, 6 + n, "H2", Tlo=300.0, Thi=2600.0)
    Y = np.vstack([Y, np.full((max(0, m.ns - h2.ns), n), 1e-3)])[:m.ns]
    got = []
    for opts in (None, cg.options(group_threads=2)):
        Td, pd, Yd = to_dev(T, p, Y)
        st = torch.full((n,), -1, dtype=torch.int8, device="cuda")
        cg.advance(dm, Td, pd, Yd, 5e-7, status=st, opts=opts)
        got.append((Td.cpu().numpy(), Yd.cpu().numpy(), st.cpu().numpy()))
    # (two cells of "slow" end in H_UNDERFLOW, in the oracle too: a rate with T^40)
    assert np.array_equal(got[0][2], got[1][2]) and np.mean(got[0][2] == 0) > 0.99 - 1.0 / n
    assert np.all(within(got[1][0], got[1][1], got[0][0], got[0][1]))


@pytest.mark.gpu
@pytest.mark.parametrize("which,per_sm,extra,big_sm", [("8", 0, 1, 104), ("9", 0, 5, 104), ("9", 28, 0, 104),
                                                       ("9", 28, 1, 104), ("9", 104, 0, 104), ("10", 28, 3, 104),
                                                       ("11", 0, 129, 104), ("11", 30, 0, 104), ("slow", 0, 65, 104),
                                                       ("slow", 29, 0, 104), ("9", 120, 7, 420), ("8", 28, 0, 420),
                                                       ("11", 104, 1, 420), ("slow", 110, 0, 420)])
def test_launch_size_does_not_change_a_cell(h2, which, per_sm, extra, big_sm):
    """Launches of few cells (16 or 8 lanes a cell up to 28 and 104 cells per SM) and of many (eight
    warps an SM from 416 cells per SM on) against one thread per cell in between: the same
    operations, so the same bits."""
    import torch
    import paper_2312_13513_gb300 as cg
    from gpu_common import to_dev
    from helpers import random_states
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n, big = per_sm * sms + extra, big_sm * sms + 33
    m = _mechs(h2)[which]
    dm = cg.Mechanism(m)
    T, p, Y = random_states(h2, big, 60 + n, "H2", Tlo=300.0, Thi=2600.0)
    Y = np.vstack([Y, np.full((max(0, m.ns - h2.ns), big), 1e-3)])[:m.ns]
    Tb, pb, Yb = to_dev(T, p, Y)
    sb = torch.full((big,), -1, dtype=torch.int8, device="cuda"); kb = torch.zeros(big, dtype=torch.int32, device="cuda")
    cg.advance(dm, Tb, pb, Yb, 5e-7, status=sb, nsub=kb)
    Ts, ps, Ys = to_dev(T[:n].copy(), p[:n].copy(), Y[:, :n].copy())
    ss = torch.full((n,), -1, dtype=torch.int8, device="cuda"); ks = torch.zeros(n, dtype=torch.int32, device="cuda")
    cg.advance(dm, Ts, ps, Ys, 5e-7, status=ss, nsub=ks)
    assert torch.equal(ss, sb[:n]) and torch.equal(ks, kb[:n])
    assert torch.equal(Ts, Tb[:n]) and torch.equal(Ys, Yb[:, :n])


@pytest.mark.gpu
def test_cells_beyond_the_temperature_range_are_not_slower(h2):
    """Cells above 4096 K take the FP64 forms cell by cell: no slower than the group kernel, which has
    no other (0.91 of its time measured, 1.36 with the library's exponentials and logarithms)."""
    import torch
    import paper_2312_13513_gb300 as cg
    from gpu_common import to_dev
    from helpers import random_states
    n = 100003
    T, p, Y = random_states(h2, n, 5, "H2", Tlo=4100.0, Thi=5500.0)
    T0, pd, Y0 = to_dev(T, p, Y)
    Td, Yd = T0.clone(), Y0.clone()
    dm = cg.Mechanism(h2)
    best = [np.inf, np.inf]
    for _ in range(2):
        for i, opts in enumerate((None, cg.options(group_threads=2))):
            Td.copy_(T0), Yd.copy_(Y0)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            cg.advance(dm, Td, pd, Yd, 1e-8, opts=opts)
            b.record()
            torch.cuda.synchronize()
            best[i] = min(best[i], a.elapsed_time(b))
    assert best[0] <= 1.2 * best[1], best
