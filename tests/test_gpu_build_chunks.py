"""build_T where its staging ring wraps: antenna counts around whole chunks and several ring
lengths, in each kind of Gram (TF32 split up to 9 columns, FP16 split, real rows), with slot counts
whose last slot is staged by itself.  Against FP64, with the bounds of the parity tests (T~ 2e-5
absolute; D and tau 1e-5 relative)."""
import numpy as np
import pytest
import torch

from oracle import taser_oracle as O
from synth import make_jed, make_mimo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,M,B", [("jed_bpsk", K, B) for K in (11, 17, 33) for B in (15, 48, 49, 64, 65, 130)]
                         + [("jed_qpsk", K, B) for K in (18, 24, 33) for B in (31, 32, 33, 64, 97)]
                         + [("mimo_bpsk", U, B) for U in (4, 8) for B in (31, 32, 33, 63, 65, 200)]
                         + [("jed_qpsk", 7, B) for B in (7, 32, 39, 64, 65)])
def test_chunk_edges(kind, M, B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_01797_gb300 as T
    n = 5
    if kind.startswith("jed"):
        X, y = make_jed(n, B, M, 6.0, seed=70 + M + B, constellation=kind[4:])["Y"], None
    else:
        w = make_mimo(n, B, M, 8.0, kind[5:], seed=70 + M + B)
        X, y = w["H"], w["y"]
    out = T.build_T(kind, torch.from_numpy(X).cuda(), None if y is None else torch.from_numpy(y).cuda(), alpha=0.5)
    torch.cuda.synchronize()
    ref = O.detect(kind, X, y, 0.5, 1)
    got = {k: v.cpu().numpy().astype(np.float64) for k, v in out.items()}
    assert np.abs(got["T_tilde"] - ref["T_tilde"]).max() <= 2e-5
    for key in ("D", "tau"):
        assert (np.abs(got[key] - ref[key]) / np.abs(ref[key])).max() <= 1e-5
    assert (got["flags"] == 0).all()
