"""The FP32 adjoint of unfolded TASER over the range of D, and over long segments.

Tolerance: the adjoint's bound of 1e-3 of the instance's largest entry.  It covers the runs here by
their total step: an error made at one step reaches the others amplified by at most about
exp(2 sum alpha), and t_max steps make t_max of them, each of a few 2^-24.  With sum alpha = 1 that
is 200 * 4 * 2^-24 * 7.4 = 3.5e-4 at the longest run.
"""
import numpy as np
import pytest
import torch

from oracle import taser_oracle as O
from synth import make_mimo

pytestmark = pytest.mark.gpu
BOUND = 1e-3


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_01797_gb300 as taser
    return taser


def problem(n, N, t_max, seed):
    """T~, D in [1, 2), 1 / ||T~||, steps of sum 1 and a gradient of the soft outputs."""
    w = make_mimo(n, max(2 * (N - 1), 4), N - 1, np.linspace(0, 15, n), "bpsk", seed=seed)
    Tt = O.detect("mimo_bpsk", w["H"], w["y"], 0.5, 1)["T_tilde"].astype(np.float32)
    rng = np.random.default_rng(seed)
    alpha = rng.uniform(0.5, 1.5, t_max)
    return (Tt, rng.uniform(1.0, 2.0, (n, N)).astype(np.float32),
            (1.0 / O.spectral_norm(Tt.astype(np.float64))).astype(np.float32),
            (alpha / alpha.sum()).astype(np.float32), rng.standard_normal((n, N - 1)).astype(np.float32))


def gradients(T, Tt, D, inv, alpha, g, c):
    d = [torch.from_numpy(x).cuda() for x in (Tt, D, inv, alpha, g)]
    ckpt = T.unfolded_forward(*d[:4], c)[2]
    grad_tau, _ = T.unfolded_backward(*d[:4], c, ckpt, d[4])
    torch.cuda.synchronize()
    return grad_tau.cpu().numpy().astype(np.float64)


def oracle(Tt, D, inv, alpha, g):
    T64, D64 = Tt.astype(np.float64), D.astype(np.float64)
    tau = alpha[None, :].astype(np.float64) * inv[:, None].astype(np.float64)
    return O.unfolded_backward(T64, D64, tau, O.unfolded_forward(T64, D64, tau)[1], g.astype(np.float64))


@pytest.mark.parametrize("N", [9, 16, 17, 33])
@pytest.mark.parametrize("exponent,bound", [(-66, 5e-3), (-62, BOUND), (-30, BOUND), (0, BOUND), (30, BOUND), (60, BOUND)])
def test_gradient_does_not_depend_on_the_scale_of_D(T, N, exponent, bound):
    """The soft outputs do not depend on D's scale, so neither does the gradient.  The gradient of
    the soft outputs is large enough that a product with 1 / D^2 would overflow at 2^-62.  At 2^-66
    the squares of a column (about D^2 = 2^-132) are denormal: up to 33 of them, each rounded by
    2^-150, are 2^-14 of the scale at each of 8 steps, times 7.4: 4e-3 more."""
    Tt, D, inv, alpha, g = problem(9, N, 8, 30 + N)
    g *= np.float32(2.0 ** 14)
    want = oracle(Tt, D, inv, alpha, g)
    got = gradients(T, Tt, np.ldexp(D, exponent).astype(np.float32), inv, alpha, g, 3)
    assert np.isfinite(got).all()
    assert (np.abs(got - want) / np.abs(want).max(axis=1, keepdims=True)).max() <= bound


@pytest.mark.parametrize("N,t_max,spacings", [(33, 60, (8, 46, 47, 60)), (17, 200, (40, 79, 160, 200)),
                                              (9, 140, (20, 121, 140)), (25, 9, (2, 4, 9)), (2, 3, (1, 2, 3))])
def test_long_segments_against_fp64(T, N, t_max, spacings):
    p = problem(5, N, t_max, 60 + N)
    want = oracle(*p)
    for c in spacings:
        got = gradients(T, *p, c)
        assert (np.abs(got - want) / np.abs(want).max(axis=1, keepdims=True)).max() <= BOUND, c


@pytest.mark.parametrize("N,n,t_max,spacings", [(9, 9000, 5, (2, 5)), (10, 4100, 5, (3, 5)), (17, 4100, 9, (2, 9)),
                                                (20, 4100, 4, (2, 4)), (33, 4100, 9, (2, 9)), (33, 700, 26, (4, 25))])
def test_one_result_in_every_layout(T, N, n, t_max, spacings):
    """Columns a lane and instances a warp follow the batch and the spacing; an instance's soft
    outputs, checkpoints and gradient are the same bit for bit."""
    Tt, D, inv, alpha, g = problem(9, N, t_max, 90 + N)
    reps = -(-n // 9)
    Tt, D, inv, g = (np.ascontiguousarray(np.tile(x, (reps,) + (1,) * (x.ndim - 1))[:n]) for x in (Tt, D, inv, g))
    d = [torch.from_numpy(x).cuda() for x in (Tt, D, inv, alpha, g)]
    want = None
    for c in spacings:
        soft, s, ckpt = T.unfolded_forward(*d[:4], c)
        gt, _ = T.unfolded_backward(*d[:4], c, ckpt, d[4])
        want = (soft, s, gt) if want is None else want
        assert all(torch.equal(a, b) for a, b in zip((soft, s, gt), want)), c
        for at in (slice(0, 1), slice(4, 23), slice(n - 300, n)):
            p = [x[at].clone() for x in d[:3]]
            soft1, s1, ckpt1 = T.unfolded_forward(*p, d[3], c)
            gt1, _ = T.unfolded_backward(*p, d[3], c, ckpt1, d[4][at].clone())
            torch.cuda.synchronize()
            assert torch.equal(ckpt1, ckpt[at])
            assert all(torch.equal(a, b[at]) for a, b in zip((soft1, s1, gt1), want)), (c, at)
