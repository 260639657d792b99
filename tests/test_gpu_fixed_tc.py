"""TASER_FIXED14 on the tensor cores (N <= 33): codes over their whole 14-bit range,
where the split products reach their largest sums, must still match the integer oracle bit by
bit: L~, decisions and flags."""
import numpy as np
import pytest
import torch

from oracle import taser_fixed_oracle as F

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_01797_gb300 as taser
    return taser


def inputs(case, N, n, seed):
    rng = np.random.default_rng(seed)
    tau = np.full(n, 0.5, np.float32)
    if case == "extremes":            # every code at an end of its range
        Tt = rng.choice([-4.0, 4.0], size=(n, N, N))
        D = rng.choice([-40.0, 40.0], size=(n, N))
    elif case == "wide":              # not symmetric, often saturated
        Tt = rng.uniform(-2.5, 2.5, size=(n, N, N))
        D = rng.uniform(-33.0, 33.0, size=(n, N))
    else:                             # "small": sums near the rounding half points
        Tt = rng.integers(-40, 41, size=(n, N, N)) / 4096.0
        D = rng.integers(0, 60, size=(n, N)) / 256.0
    return Tt.astype(np.float32), D.astype(np.float32), tau


@pytest.mark.parametrize("case", ["extremes", "wide", "small"])
@pytest.mark.parametrize("N", [2, 5, 9, 10, 15, 16, 17, 18, 25, 32, 33])
@pytest.mark.parametrize("n,t_max", [(1, 3), (41, 7)])
def test_fixed14_whole_code_range(T, case, N, n, t_max):
    Tt, D, tau = inputs(case, N, n, 7000 + N)
    s, L, flags = T.detect(*(torch.from_numpy(x).cuda() for x in (Tt, D, tau)), t_max, "fixed14")
    torch.cuda.synchronize()
    ref = F.taser_fixed(Tt, D, tau, t_max)
    np.testing.assert_array_equal(L.cpu().numpy(), ref["L_real"].astype(np.float32))
    np.testing.assert_array_equal(s.cpu().numpy(), ref["s_hat"])
    np.testing.assert_array_equal(flags.cpu().numpy().astype(np.uint32), ref["flags"])
