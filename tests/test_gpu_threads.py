"""Host threads that call the library at the same time, each on its own stream."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,precision,wide", [(33, "fp32", 12), (17, "fp32", 20), (33, "bf16_tc", 12)])
def test_adjoint_spacings_in_several_threads(N, precision, wide):
    """The adjoint's shared memory follows the checkpoint spacing: threads with a narrow and with a
    wide one (more than the 48 KB that need no opt-in) each get their own result, in every call.
    The loop calls the C entry with ready arguments, so that the calls overlap."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_01797_gb300 as T
    from paper_1609_01797_gb300._native import lib
    from paper_1609_01797_gb300.api import PRECISIONS, _ptr, _stream
    gen = torch.Generator(device="cuda")
    gen.manual_seed(N)
    A = torch.randn((2, N, N), generator=gen, device="cuda") * 0.1
    Tt = (A + A.transpose(1, 2)).contiguous()
    D, inv = torch.ones((2, N), device="cuda"), torch.full((2,), 0.5, device="cuda")
    g = torch.randn((2, N - 1), generator=gen, device="cuda")
    failures, start = [], threading.Barrier(4)
    call = lib().taser_unfolded_backward

    def work(c, calls):
        try:
            stream = torch.cuda.Stream()
            a = torch.full((c,), 0.5, device="cuda")
            ckpt = T.unfolded_forward(Tt, D, inv, a, c, precision=precision)[2]
            want, want_a = T.unfolded_backward(Tt, D, inv, a, c, ckpt, g, precision=precision)
            got, got_a = torch.zeros_like(want), torch.zeros_like(want_a)
            torch.cuda.synchronize()
            args = (2, N, _ptr(Tt), _ptr(D), _ptr(inv), _ptr(a), c, c, PRECISIONS[precision], _ptr(ckpt), _ptr(g),
                    _ptr(got), _ptr(got_a), _stream(stream))
            start.wait()
            bad = 0
            for k in range(calls):
                bad += call(*args) != 0
                if k % 256 == 255:
                    stream.synchronize()
            stream.synchronize()
            if bad or not torch.equal(got, want):
                failures.append("c = %d: %d of %d calls refused" % (c, bad, calls))
        except Exception as e:   # reported by the main thread
            start.abort()
            failures.append("c = %d: %s" % (c, e))

    threads = [threading.Thread(target=work, args=a) for a in ((wide, 4000), (1, 20000), (1, 20000), (1, 20000))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures
