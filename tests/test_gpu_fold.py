"""Folded layouts (several instances per warp, several columns per lane) at the sizes where
they can go wrong: batches that end inside a warp or a block, sizes at both ends of a bucket.

Tolerance: the FP32 detector's bound of 1e-5 relative (Frobenius) against the FP64 oracle.
"""
import numpy as np
import pytest
import torch

from oracle import taser_oracle as O
from synth import make_jed, make_mimo

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_01797_gb300 as taser
    return taser


def problem(n, N, seed):
    U = N - 1
    w = make_mimo(n, max(2 * U, 4), U, np.linspace(0, 15, n), "bpsk", seed=seed)
    r = O.detect("mimo_bpsk", w["H"], w["y"], 0.5, 1)
    return r["T_tilde"].astype(np.float32), r["D"].astype(np.float32), r["tau"].astype(np.float32)


@pytest.mark.parametrize("N", [2, 8, 9, 10, 13, 14, 16, 17, 18, 21, 22, 25, 26, 29, 30, 32, 33])
@pytest.mark.parametrize("n", [1, 3, 7, 9, 33])
def test_fp32_ragged_batches(T, N, n):
    Tt, D, tau = problem(n, N, 9000 + N)
    guard = 77
    s = torch.full((n + 1, N - 1), guard, dtype=torch.int8, device="cuda")
    L = torch.full((n + 1, N, N), float(guard), device="cuda")
    T.detect(*(torch.from_numpy(x).cuda() for x in (Tt, D, tau)), 6, "fp32", out_s=s, out_L=L)
    torch.cuda.synchronize()
    Lo, _ = O.taser(Tt.astype(np.float64), D.astype(np.float64), tau.astype(np.float64), 6)
    got = L.cpu().numpy().astype(np.float64)
    err = np.linalg.norm(got[:n] - Lo, axis=(1, 2)) / np.linalg.norm(Lo, axis=(1, 2))
    assert err.max() <= 1e-5
    row = Lo[:, -1, :]
    sure = np.abs(row[:, :-1]) > 1e-3 * np.linalg.norm(row, axis=1, keepdims=True)
    assert np.array_equal(s.cpu().numpy()[:n][sure], O.decisions(Lo)[sure])
    assert (got[n] == guard).all() and (s.cpu().numpy()[n] == guard).all()   # nothing past the batch


@pytest.mark.parametrize("kind,B,M", [("jed_bpsk", B, K) for K in (10, 15, 16, 17, 18, 31, 32, 33) for B in (1, 9, 16, 33)]
                         + [("mimo_bpsk", B, U) for U in (9, 15, 16, 17, 31, 32) for B in (8, 16, 35, 70)]
                         + [("mimo_qpsk", B, U) for U in (15, 17, 31, 32) for B in (16, 33)]
                         + [("jed_qpsk", B, K) for K in (10, 17, 18, 33) for B in (3, 16, 17, 40)])
def test_build_T_bucket_edges(T, kind, B, M):
    """build_T at the ends of its column buckets and of its staged row chunks, with odd column
    counts (8-byte copies), against FP64: the bounds of the parity tests (T~ 2e-5 absolute; D
    and tau 1e-5 relative)."""
    n = 9
    if kind.startswith("jed"):
        X, y = make_jed(n, B, M, 6.0, seed=50 + M, constellation=kind[4:])["Y"], None
    else:
        w = make_mimo(n, B, M, 8.0, kind[5:], seed=60 + M)
        X, y = w["H"], w["y"]
    out = T.build_T(kind, torch.from_numpy(X).cuda(), None if y is None else torch.from_numpy(y).cuda(), alpha=0.5)
    torch.cuda.synchronize()
    ref = O.detect(kind, X, y, 0.5, 1)
    got = {k: v.cpu().numpy().astype(np.float64) for k, v in out.items()}
    assert np.abs(got["T_tilde"] - ref["T_tilde"]).max() <= 2e-5
    for key in ("D", "tau"):
        assert (np.abs(got[key] - ref[key]) / np.abs(ref[key])).max() <= 1e-5


@pytest.mark.parametrize("N,t_max,spacings", [(33, 60, (8, 46, 47, 60)), (17, 200, (40, 79, 160, 200)), (9, 140, (20, 121, 140)),
                                              (25, 9, (4,)), (2, 3, (2,))])
@pytest.mark.parametrize("n", [1, 5, 17])
def test_unfolded_adjoint_any_spacing(T, N, t_max, spacings, n):
    """The adjoint holds as many instances per warp as their c + 1 iterates fit in shared memory;
    every spacing gives the same gradient bit for bit, for batches that end inside a warp, and it
    is the FP64 one within the adjoint's bound (1e-3 of the instance's largest entry)."""
    Tt, D, tau = problem(n, N, 300 + N)
    inv = (2.0 * tau).astype(np.float32)                       # tau = 0.5 / ||T~||
    rng = np.random.default_rng(N)
    alpha = rng.uniform(0.3, 0.6, size=t_max).astype(np.float32)
    g = (rng.standard_normal((n, N - 1)) * 1e-3).astype(np.float32)
    dT, dD, dinv, da, dg = (torch.from_numpy(x).cuda() for x in (Tt, D, inv, alpha, g))
    ref = None
    for c in spacings:
        _, _, ckpt = T.unfolded_forward(dT, dD, dinv, da, c)
        gt, _ = T.unfolded_backward(dT, dD, dinv, da, c, ckpt, dg)
        torch.cuda.synchronize()
        ref = gt if ref is None else ref
        assert torch.equal(gt, ref), c
    if t_max > 10:
        return                                                  # the oracle's bound is derived for short runs
    tau_t = alpha[None, :].astype(np.float64) * inv[:, None].astype(np.float64)
    T64, D64 = Tt.astype(np.float64), D.astype(np.float64)
    _, Ls = O.unfolded_forward(T64, D64, tau_t)
    go = O.unfolded_backward(T64, D64, tau_t, Ls, g.astype(np.float64))
    scale = np.abs(go).max(axis=1, keepdims=True) + 1e-30
    assert (np.abs(ref.cpu().numpy() - go) / scale).max() <= 1e-3


@pytest.mark.parametrize("N,n", [(9, 7), (10, 7), (13, 33), (14, 9), (17, 9), (18, 9), (25, 17), (26, 5), (33, 9), (34, 5),
                                 (47, 2000), (65, 1300)])
@pytest.mark.parametrize("structure", [-1, "mimo_bpsk"])
def test_step_size_layout_edges(T, N, n, structure):
    """||T~||_2 at the ends of the step-size kernels' layouts and beyond one wave at N > 33, against
    FP64: 1e-5 relative, the bound of the parity tests."""
    Tt = problem(min(n, 40), N, 700 + N)[0]
    ref = np.abs(np.linalg.eigvalsh(Tt.astype(np.float64))).max(axis=1)
    if structure == -1:
        Tt = Tt * np.where(np.arange(Tt.shape[0]) % 2, -1, 1)[:, None, None].astype(np.float32)   # either sign
    reps = -(-n // Tt.shape[0])
    dT = torch.from_numpy(np.ascontiguousarray(np.tile(Tt, (reps, 1, 1))[:n])).cuda()
    tau, nrm = T.step_size(dT, 0.5, structure)
    torch.cuda.synchronize()
    want = np.tile(ref, reps)[:n]
    got = nrm.cpu().numpy().astype(np.float64)
    assert (np.abs(got - want) / want).max() <= 1e-5
    assert (np.abs(tau.cpu().numpy() - 0.5 / want) * want / 0.5).max() <= 1e-5


@pytest.mark.parametrize("kind,M", [("mimo_qpsk", U) for U in (8, 9, 12, 13, 16, 17, 24, 25, 32)]
                         + [("jed_qpsk", K) for K in (9, 10, 13, 14, 18, 25, 26, 33)])
def test_step_size_complex_layout_edges(T, kind, M):
    """The complex form's layouts at their ends, from build_T's own T~: 1e-5 relative."""
    n, B = 11, 40
    if kind == "jed_qpsk":
        X, y = make_jed(n, B, M, 6.0, seed=80 + M, constellation="qpsk")["Y"], None
    else:
        w = make_mimo(n, B, M, 8.0, "qpsk", seed=90 + M)
        X, y = w["H"], w["y"]
    out = T.build_T(kind, torch.from_numpy(X).cuda(), None if y is None else torch.from_numpy(y).cuda(), alpha=0.5)
    torch.cuda.synchronize()
    want = np.abs(np.linalg.eigvalsh(out["T_tilde"].cpu().numpy().astype(np.float64))).max(axis=1)
    assert (np.abs(out["spec_norm"].cpu().numpy() - want) / want).max() <= 1e-5
