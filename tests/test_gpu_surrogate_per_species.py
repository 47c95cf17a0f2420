"""GPU parity of the paper's per-species surrogate variant (one GELU network per species, run layer
by layer on the tcgen05 GEMM with its activation epilogue) and of the variable-width trainer."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2312_13513_gb300 as cg  # noqa: E402
from oracle import mlp as omlp  # noqa: E402
from oracle import surrogate as osur  # noqa: E402

from gpu_common import to_dev  # noqa: E402
from helpers import random_states  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,gelu", [(300, 200, 192, True), (128, 1600, 64, True), (1000, 400, 800, False),
                                        (16384, 800, 1600, True), (777, 12800, 64, True), (4096, 300, 400, True)])
def test_gemm_activation_epilogue_matches_torch(M, N, K, gelu):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, device="cuda", generator=g).to(torch.bfloat16)
    B = (torch.randn(N, K, device="cuda", generator=g) / np.sqrt(K)).to(torch.bfloat16)
    bias = torch.randn(N, device="cuda", generator=g)
    C = cg.gemm_bf16_act(A, B, bias, gelu=gelu)
    z = (A.double() @ B.double().T + bias.double()).cpu().numpy()
    ref = omlp.bf16_round(omlp.gelu(z) if gelu else z)
    got = C.float().cpu().numpy().astype(np.float64)
    # one BF16 rounding of nearly the same value: the tensor cores' FP32 sums differ from the FP64
    # reference by ~1e-4 of the largest entry (as in the FP32-output test), which near zero
    # dominates; elsewhere values that straddle a rounding boundary land one BF16 ulp apart
    tol = 2.0 ** -7 * np.maximum(np.abs(ref), np.abs(got)) + 1e-4 * np.max(np.abs(ref))
    assert np.all(np.abs(got - ref) <= tol), np.max(np.abs(got - ref) - tol)
    assert np.mean(got == ref) > 0.95


def _ps_params(mech, x, seed, hidden, inert=()):
    rng = np.random.default_rng(seed)
    nin = mech.ns + 2
    dims = [nin] + list(hidden) + [1]
    nets = {}
    for k in range(mech.ns):
        if k in inert:
            continue
        W = [rng.standard_normal((dims[i + 1], dims[i])) / np.sqrt(dims[i]) for i in range(4)]
        b = [0.1 * rng.standard_normal(dims[i + 1]) for i in range(4)]
        nets[k] = {"W": W, "b": b}
    sd = x.std(axis=0)
    sd = np.where(sd > 1e-6 * np.maximum(1.0, np.abs(x.mean(axis=0))), sd, 1.0)
    y_std = np.array([0.0 if k in inert else 0.05 + 0.01 * k for k in range(mech.ns)])
    return {"hidden": list(hidden), "nets": nets, "dt": 5e-7, "x_mean": x.mean(axis=0), "x_std": sd,
            "y_mean": np.where(y_std > 0, 0.01 * np.arange(mech.ns), 0.0), "y_std": y_std,
            "box_lo": x.min(axis=0) - 1.0, "box_hi": x.max(axis=0) + 1.0}


def _oracle_z(prm, T, p, Y, ns):
    xz = (osur.features(T, p, Y) - prm["x_mean"]) / prm["x_std"]
    z = np.zeros((ns, T.size))
    for k, net in prm["nets"].items():
        W32 = [np.asarray(w, np.float32).astype(np.float64) for w in net["W"]]
        b32 = [np.asarray(v, np.float32).astype(np.float64) for v in net["b"]]
        out, _ = omlp.forward(W32, b32, xz, emulate_bf16=True)
        z[k] = out[:, 0]
    return z


@pytest.mark.parametrize("hidden,n", [((256, 200, 136), 300), ((1600, 800, 400), 1000),
                                      ((128, 136, 128), 5),              # below one 128-row tile
                                      ((256, 200, 136), 16384 + 77)])    # two chunks, ragged tail
def test_per_species_forward_matches_oracle(h2, hidden, n):
    dm = cg.Mechanism(h2)
    T, p, Y = random_states(h2, n, 31, "H2", Tlo=300.0, Thi=2500.0)
    x = osur.features(T, p, Y)
    inert = (h2.ns - 1,)                                   # N2: no network
    prm = _ps_params(h2, x, 5, hidden, inert=inert)
    prm["box_hi"][0] = 2000.0
    model = cg.Surrogate(dm, prm)
    ynet, z, box = cg.surrogate_forward(model, *to_dev(T, p, Y), with_z=True)
    torch.cuda.synchronize()
    z = z.cpu().numpy().astype(np.float64)
    zr = _oracle_z(prm, T, p, Y, h2.ns)
    tol = 1e-2 * np.maximum(1.0, np.abs(zr))
    assert np.all(np.abs(z - zr) <= tol), np.max(np.abs(z - zr))
    assert np.all(z[list(inert)] == 0.0)
    assert np.array_equal(box.cpu().numpy().astype(bool), T > 2000.0)
    yr = osur.boxcox_inv(osur.boxcox(Y) + zr * prm["y_std"][:, None] + prm["y_mean"][:, None])
    yg = ynet.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(yg - yr) <= 0.05 * np.abs(yr) + 1e-6)


def test_per_species_model_file_roundtrip(h2, tmp_path):
    from paper_2312_13513_gb300.train import save_model_per_species
    dm = cg.Mechanism(h2)
    T, p, Y = random_states(h2, 500, 32, "H2", Tlo=600.0, Thi=2400.0)
    prm = _ps_params(h2, osur.features(T, p, Y), 6, (256, 128, 128), inert=(h2.ns - 1,))
    path = str(tmp_path / "ps.chemsur")
    save_model_per_species(prm, path)
    a = cg.Surrogate(dm, prm)
    b = cg.Surrogate(dm, path=path)
    ya, za, _ = cg.surrogate_forward(a, *to_dev(T, p, Y), with_z=True)
    yb, zb, _ = cg.surrogate_forward(b, *to_dev(T, p, Y), with_z=True)
    torch.cuda.synchronize()
    assert torch.equal(za, zb) and torch.equal(ya, yb)


def test_per_species_identity_networks_through_projection_and_newton(h2, om_h2):
    """Networks that predict no change: every cell takes the network route and keeps its
    elements, enthalpy and temperature (the same post-processing as the single network)."""
    dm = cg.Mechanism(h2)
    T, p, Y = random_states(h2, 600, 33, "H2", Tlo=400.0, Thi=2400.0)
    prm = _ps_params(h2, osur.features(T, p, Y), 7, (128, 128, 128), inert=(h2.ns - 1,))
    for net in prm["nets"].values():
        net["W"][3] = np.zeros_like(net["W"][3])
        net["b"][3] = np.zeros(1)
    prm["y_mean"] = np.zeros(h2.ns)
    model = cg.Surrogate(dm, prm)
    Td, pd, Yd = to_dev(T, p, Y)
    route = torch.full((T.size,), -1, dtype=torch.int8, device="cuda")
    cg.surrogate_advance(model, Td, pd, Yd, prm["dt"], route=route)
    torch.cuda.synchronize()
    assert np.all(route.cpu().numpy() == 0)
    Tg, Yg = Td.cpu().numpy(), Yd.cpu().numpy()
    A = osur.element_mass_matrix(h2)
    assert np.max(np.abs(A @ Yg - A @ Y)) <= 1e-9
    assert np.max(np.abs(Tg - T) / T) <= 1e-5


def test_trainer_with_per_species_widths_matches_oracle():
    """The variable-width trainer (ragged widths 200 and 136 exercise the K and N tile edges):
    forward, loss and gradients against the FP64 oracle."""
    from paper_2312_13513_gb300.train import PAD, Trainer
    rng = np.random.default_rng(41)
    B, nin, nout = 256, 11, 1
    hidden = [200, 136, 160]
    dims = [nin] + hidden + [nout]
    W = [omlp.bf16_round(rng.standard_normal((dims[i + 1], dims[i])) / np.sqrt(dims[i])) for i in range(4)]
    b = [np.float32(0.1 * rng.standard_normal(dims[i + 1])).astype(np.float64) for i in range(4)]
    X = omlp.bf16_round(rng.standard_normal((B, nin)))
    T = rng.standard_normal((B, nout))
    tr = Trainer(nin, nout, B, W=W, b=b, hidden=hidden)
    Xd = torch.zeros((B, PAD), dtype=torch.bfloat16, device="cuda")
    Xd[:, :nin] = torch.tensor(X, dtype=torch.float32).to(torch.bfloat16)
    Td = torch.tensor(T, dtype=torch.float32, device="cuda")
    out = torch.empty((B, nout), dtype=torch.float32, device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    tr.forward(Xd, out)
    tr.backward(Td, loss)
    dW, db = tr.get(1)
    o_out, cache = omlp.forward(W, b, X, emulate_bf16=True)
    assert np.max(np.abs(out.cpu().numpy() - o_out)) <= 1e-2 * max(1.0, np.max(np.abs(o_out)))
    assert abs(loss.item() - omlp.mse_loss(o_out, T)) <= 1e-3 * omlp.mse_loss(o_out, T)
    gW, gb = omlp.backward(W, b, cache, o_out, T)
    for l in range(4):
        rel = np.linalg.norm(dW[l] - gW[l]) / np.linalg.norm(gW[l])
        relb = np.linalg.norm(db[l] - gb[l]) / np.linalg.norm(gb[l])
        assert rel < 2e-2 and relb < 2e-2, (l, rel, relb)


@pytest.mark.parametrize("M,N,K,ldc", [(128, 128, 64, 128), (300, 160, 64, 160), (385, 208, 128, 208), (257, 400, 192, 400),
                                       (20000, 400, 64, 400), (20000, 800, 64, 801), (20000, 833, 64, 840),
                                       (20000, 1600, 64, 1608), (129, 513, 70, 513)])
def test_gemm_tile_widths_and_store_widths(M, N, K, ldc):
    """Every tile width the dispatch picks (128 to 256 columns), ragged edges in M, N and K, and
    outputs whose pitch allows 32-byte, 16-byte and single stores, against FP32 torch."""
    import ctypes
    from paper_2312_13513_gb300 import _lib
    g = torch.Generator(device="cuda").manual_seed(M + N)
    lda = (K + 7) // 8 * 8
    A = torch.randn(M, lda, device="cuda", generator=g).bfloat16()
    B = (torch.randn(N, lda, device="cuda", generator=g) / K ** 0.5).bfloat16()
    bias = torch.randn(N, device="cuda", generator=g)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    C = torch.full((M, ldc), 7.0, device="cuda")
    Cb = torch.full((M, ldc), 7.0, device="cuda", dtype=torch.bfloat16)
    L = _lib.load()
    assert L.chem_gemm_bf16(p(A), lda, p(B), lda, p(C), ldc, p(bias), M, N, K, p(err), st) == 0
    assert L.chem_gemm_bf16_act(p(A), lda, p(B), lda, p(Cb), ldc, p(bias), 1, M, N, K, p(err), st) == 0
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    ref = A[:, :K].double() @ B[:, :K].double().T + bias.double()
    # FP32 accumulation of K products of size O(1 / sqrt K): K additions at 2^-24 of at most ~6
    assert torch.allclose(C[:, :N].double(), ref, rtol=0, atol=6 * K * 2.0 ** -24)
    act = torch.nn.functional.gelu(ref)
    # one BF16 rounding (2^-9 relative) and the GELU form's 5e-7
    assert torch.all((Cb[:, :N].double() - act).abs() <= 2.0 ** -8 * act.abs() + 1e-5)
    assert torch.all(C[:, N:] == 7.0) and torch.all(Cb[:, N:] == 7.0)         # nothing beyond column N


@pytest.mark.parametrize("hidden,B", [((2048, 2048), 256), ((4096, 4096), 8192)])
def test_trainer_with_wide_layers(hidden, B):
    """Layers whose weight-gradient products have a tile for every SM (not split: straight to the
    gradient), and activations beyond 128 MB (transposed one layer at a time into one buffer): gradients
    of a batch that repeats 128 rows against those of the 128 rows, and the memory that they take."""
    from paper_2312_13513_gb300.train import PAD, Trainer
    rng = np.random.default_rng(43)
    nin, nout, rep = 11, 9, B // 128
    dims = [nin, *hidden, nout]
    W = [rng.standard_normal((dims[i + 1], dims[i])).astype(np.float32) / np.sqrt(dims[i]) for i in range(3)]
    b = [0.1 * rng.standard_normal(dims[i + 1]).astype(np.float32) for i in range(3)]
    X = torch.zeros((128, PAD), dtype=torch.bfloat16, device="cuda")
    X[:, :nin] = torch.tensor(rng.standard_normal((128, nin)), dtype=torch.float32, device="cuda").bfloat16()
    T = torch.tensor(rng.standard_normal((128, nout)), dtype=torch.float32, device="cuda")
    got = []
    for n in (1, rep):
        Xn, Tn = X.repeat(n, 1).contiguous(), T.repeat(n, 1).contiguous()
        out = torch.empty((128 * n, nout), dtype=torch.float32, device="cuda")
        loss = torch.zeros(1, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        tr = Trainer(nin, nout, 128 * n, W=W, b=b, hidden=list(hidden))
        used = free - torch.cuda.mem_get_info()[0]
        for _ in range(2):
            tr.forward(Xn, out)
            tr.backward(Tn, loss)
        got.append((*tr.get(1), loss.item(), used))
        del tr
    (gW, gb, gl, _), (dW, db, l1, used) = got
    assert abs(l1 - gl) <= 1e-6 * gl
    # the same products, scaled by a power of two: FP32 sums of up to 8192 terms in another order
    for l in range(3):
        assert np.linalg.norm(dW[l] - gW[l]) <= 1e-3 * np.linalg.norm(gW[l]), l
        assert np.linalg.norm(db[l] - gb[l]) <= 1e-3 * np.linalg.norm(gb[l]), l
    # parameters, two moments and the gradient in FP32, two BF16 copies; Z and A of each layer; three working
    # arrays and one A^T of the widest; 96 MB for partials and the allocator's rounding
    ins, outs = [PAD, *hidden], [*hidden, PAD]
    need = sum(20 * i * o for i, o in zip(ins, outs)) + B * (sum(4 * o for o in outs) + sum(2 * i for i in hidden) + 10 * max(outs))
    assert used <= need + (96 << 20), (used / 2 ** 20, need / 2 ** 20)


@pytest.mark.parametrize("M,N,K,ldc,width", [(20000, 160, 64, 160, 160), (20000, 130, 128, 131, 160), (20000, 320, 128, 328, 160),
                                             (20000, 301, 70, 301, 160), (20000, 208, 64, 208, 208)])
def test_gemm_160_column_tiles(M, N, K, ldc, width):
    """The 160-column tiles (five stages, ten 16-column units over four epilogue warps), and a single
    208-column one: enough rows for a tile on every SM, whole and ragged columns, each width of store."""
    import ctypes
    from paper_2312_13513_gb300 import _lib
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cost = {w: -(-N // w) * (128 + w) for w in (256, 208, 160, 128)}           # the dispatch's rule
    assert min(cost, key=cost.get) == width and -(-M // 128) * -(-N // width) >= sms
    g = torch.Generator(device="cuda").manual_seed(M + N)
    lda = (K + 7) // 8 * 8
    A = torch.randn(M, lda, device="cuda", generator=g).bfloat16()
    B = (torch.randn(N, lda, device="cuda", generator=g) / K ** 0.5).bfloat16()
    bias = torch.randn(N, device="cuda", generator=g)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    C = torch.full((M, ldc), 7.0, device="cuda")
    Cb = torch.full((M, ldc), 7.0, device="cuda", dtype=torch.bfloat16)
    L = _lib.load()
    assert L.chem_gemm_bf16(p(A), lda, p(B), lda, p(C), ldc, p(bias), M, N, K, p(err), st) == 0
    assert L.chem_gemm_bf16_act(p(A), lda, p(B), lda, p(Cb), ldc, p(bias), 1, M, N, K, p(err), st) == 0
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    ref = A[:, :K].double() @ B[:, :K].double().T + bias.double()
    # FP32 accumulation of K products of size O(1 / sqrt K): K additions at 2^-24 of at most ~6
    assert torch.allclose(C[:, :N].double(), ref, rtol=0, atol=6 * K * 2.0 ** -24)
    act = torch.nn.functional.gelu(ref)
    # one BF16 rounding (2^-9 relative) and the GELU form's 5e-7
    assert torch.all((Cb[:, :N].double() - act).abs() <= 2.0 ** -8 * act.abs() + 1e-5)
    assert torch.all(C[:, N:] == 7.0) and torch.all(Cb[:, N:] == 7.0)         # nothing beyond column N
