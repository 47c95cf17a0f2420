"""Calls of different sizes from several host threads, each on its own stream: what one call sets up for its
kernels does not touch another's."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2312_13513_gb300 as cg  # noqa: E402
from synth.transport import generate_transport  # noqa: E402

from gpu_common import to_dev  # noqa: E402
from helpers import random_states, with_inert_species  # noqa: E402

pytestmark = pytest.mark.gpu


def _together(calls, reps):
    """Each call over and over in its own thread and stream; every repetition gives the first one's bits."""
    errors = []

    def work(make):
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                run = make()
                ref = [t.clone() for t in run(st)]
                barrier.wait(timeout=60)
                for _ in range(reps):
                    out = run(st)
                st.synchronize()
                assert all(torch.equal(a, b) for a, b in zip(out, ref))
        except BaseException as e:  # noqa: BLE001 (a thread's failure is the test's)
            errors.append(e)
            barrier.abort()

    barrier = threading.Barrier(len(calls))
    ts = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors


@pytest.mark.parametrize("base,inert", [("h2", 0), ("h2", 7)])
def test_transport_of_small_and_large_fields(base, inert, request):
    b = request.getfixturevalue(base)
    m = with_inert_species(b, inert) if inert else b
    dm = cg.Mechanism(m)

    def call(n, ns):
        def make():
            mm = dm if ns == m.ns else cg.Mechanism(with_inert_species(b, ns - b.ns))
            tr = cg.Transport(mm, generate_transport(m if ns == m.ns else with_inert_species(b, ns - b.ns)))
            T, p, Y = random_states(b, n, n, "H2")
            Y = np.vstack([Y, np.full((ns - b.ns, n), 1e-3)])
            Td, pd, Yd = to_dev(T, p, Y)
            mu, lam, D = torch.empty_like(Td), torch.empty_like(Td), torch.empty_like(Yd)

            def run(st):
                tr(Td, pd, Yd, mu, lam, D, stream=st)
                return mu, lam, D
            return run
        return make

    other = m.ns + 1 if inert else m.ns              # the warp kernel's size depends on the species alone
    _together([call(33, m.ns), call(19001, other), call(1003, m.ns), call(19456, m.ns)], 6000)


@pytest.mark.parametrize("base,n", [("h2", 33), ("h2", 20011), ("ch4", 9)])
def test_advance_of_two_mechanisms(base, n, request):
    """Mechanisms that share a kernel instance and need different amounts of shared memory."""
    b = request.getfixturevalue(base)
    few = b.copy()
    for a in ("rtype", "reac", "prod", "A", "b", "Ea", "troe", "has_t2", "eff"):
        setattr(few, a, getattr(b, a)[: b.nr - 6].copy())

    def call(m):
        def make():
            dm = cg.Mechanism(m)
            T, p, Y = random_states(b, n, n, base.upper(), Tlo=300.0, Thi=600.0)
            T0, pd, Y0 = to_dev(T, p, Y)
            Td, Yd = T0.clone(), Y0.clone()

            def run(st):
                Td.copy_(T0)
                Yd.copy_(Y0)
                cg.advance(dm, Td, pd, Yd, 1e-9, stream=st)
                return Td, Yd
            return run
        return make

    _together([call(b), call(few), call(b), call(few)], 1500 if n < 100 else 300)
