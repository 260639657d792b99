"""The FP32 detector's layouts give one result: an instance may run in taser_detect, in
taser_detect_monitored or in an uneven batch, in layouts that differ in their column counts, and
L~, the decisions and the flags are the same bit for bit.

The inputs put V_NN of the last iteration at the rounding error of its own sum: T~_NN enters V_NN
alone, so it is set to cancel the other terms, taken from the kernel's own iterate.  The sign of
V_NN (flag, and sign of L~_NN in the literal mode) then follows from the order of the sum.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_01797_gb300 as taser
    return taser


STEPS, TAU = 3, 0.7


def cancelling(T, N, n):
    """n instances of size N whose V_NN is positive in iterations 1 and 2 and about 0 in iteration 3."""
    rng = np.random.default_rng(400 + N)
    parts, have = [], 0
    while have < n:
        m = 4096
        A = rng.standard_normal((m, N, N)) * 0.35
        Tt = ((A + A.transpose(0, 2, 1)) / 2).astype(np.float32)
        Tt[:, np.arange(N), np.arange(N)] = 1.0
        D = rng.uniform(0.5, 2.0, (m, N)).astype(np.float32)
        tau = np.full(m, TAU, np.float32)
        _, L, _ = T.detect(*(torch.from_numpy(x).cuda() for x in (Tt, D, tau)), STEPS - 1, "fp32")
        row = L.cpu().numpy()[:, -1, :-1].astype(np.float64)
        c = 2.0 * tau.astype(np.float64) * (row * Tt[:, :-1, -1].astype(np.float64)).sum(1)   # minus the sum
        keep = c > 0.05                      # V_NN = D_N (1 - 2 tau T_NN) > 0 until then
        Tt[:, -1, -1] = (1.0 - c / D[:, -1]) / (2.0 * tau)
        parts.append([x[keep] for x in (Tt, D, tau)])
        have += int(keep.sum())
    return [np.ascontiguousarray(np.concatenate(p)[:n]) for p in zip(*parts)]


def uneven(T, Tt, D, tau, mode):
    """The same instances as items of one uneven batch."""
    n, N = D.shape
    i = np.arange(n, dtype=np.int64)
    items = T.make_items(np.full(n, N), np.full(n, STEPS), i * N * N, i * N, i * (N - 1), l_off=i * N * N)
    s, L = torch.zeros((n, N - 1), dtype=torch.int8, device="cuda"), torch.zeros_like(Tt)
    flags = torch.zeros(n, dtype=torch.int32, device="cuda")
    ws = torch.empty(T.uneven_workspace_bytes(n), dtype=torch.uint8, device="cuda")
    T.detect_uneven(torch.from_numpy(items.view(np.uint8)).cuda(), Tt.view(-1), D.view(-1), tau, s.view(-1), ws,
                    precision="fp32", lnn_mode=mode, L_pool=L.view(-1), flags=flags)
    return s, L, flags


@pytest.mark.parametrize("mode", ["fixed", "literal"])
@pytest.mark.parametrize("N", [3, 9, 10, 12, 13, 14, 17, 18, 21, 25, 29, 33, 34, 65])
def test_one_result_in_every_layout(T, N, mode):
    n = 700
    Tt, D, tau = (torch.from_numpy(x).cuda() for x in cancelling(T, N, n))
    s, L, flags = T.detect(Tt, D, tau, STEPS, "fp32", lnn_mode=mode)
    ms, mL, mflags, _ = T.detect_monitored(Tt, D, tau, STEPS, "fp32", lnn_mode=mode, ascent_tol=1e30)
    us, uL, uflags = uneven(T, Tt, D, tau, mode)
    torch.cuda.synchronize()
    lnn_sign = 1 << 3
    assert 0 < int(((flags & lnn_sign) != 0).sum()) < n   # the inputs do what they are made for
    assert torch.equal(ms, s) and torch.equal(mL, L) and torch.equal(mflags, flags)
    assert torch.equal(us, s) and torch.equal(uL, L) and torch.equal(uflags, flags)


@pytest.mark.parametrize("mode", ["fixed", "literal"])
@pytest.mark.parametrize("N,n", [(9, 9800), (10, 5000), (13, 5000), (17, 5000), (18, 2500), (21, 2500), (25, 2500),
                                 (29, 2500), (33, 2500)])
def test_one_result_in_small_and_large_batches(T, N, n, mode):
    """Batches that leave the schedulers without a second warp run with one column a lane, larger
    ones with two: in taser_detect, monitored (with its objective) and in uneven batches."""
    Tt, D, tau = (torch.from_numpy(x).cuda() for x in cancelling(T, N, n))

    def results(at):
        a = [x[at].clone() for x in (Tt, D, tau)]
        return list(T.detect(*a, STEPS, "fp32", lnn_mode=mode)) + list(
            T.detect_monitored(*a, STEPS, "fp32", lnn_mode=mode)) + list(uneven(T, *a, mode))

    large = results(slice(0, n))
    for at in (slice(0, 1), slice(3, 40), slice(n - 600, n)):
        small = results(at)
        torch.cuda.synchronize()
        for a, b in zip(small, large):
            assert torch.equal(a, b[at])
