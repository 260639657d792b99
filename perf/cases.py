"""Performance cases of the detector: what a receiver has it do, through the public calls.

Each case is one pass of one public call (or of the two calls that make up the whole
detector): the problem build with its step size, Algorithm 1 in each arithmetic, an uneven
batch, and a training step of unfolded TASER.  The layers take inputs made here with plain
torch, so that a layer is measured and compared on its own; the two whole passes run in
FP32, the default precision.  taser_run_host is the whole pass behind the host link, which
alone bounds it, and returns decisions only; it is left to bench.py.
"""
import math

import torch

import paper_1609_01797_gb300 as taser

ALPHA = 0.5
SNR_DB = (4.0, 16.0)      # uniform per instance, the uneven benchmark's range
UNEVEN_SHAPES = ((32, 4), (64, 8), (128, 16), (256, 32))   # (B, U), QPSK: N = 9, 17, 33, 65
UNEVEN_T = (10, 20)
PRECISIONS = ("fp32", "bf16_tc", "fp16_tc", "fixed14")


def listed():
    return [
        # The smallest call: one slot's worth of a small cell, where launches and latency count.
        {"name": "whole_slot_qpsk32x8", "op": "whole", "kind": "mimo_qpsk", "n": 64, "B": 32, "M": 8, "t_max": 10},
        # Blind (JED) QPSK bursts of 13 slots: an odd batch of an odd size inside its bucket.
        {"name": "whole_jed_qpsk16x13", "op": "whole", "kind": "jed_qpsk", "n": 10007, "B": 16, "M": 13, "t_max": 20},
        # Build and step size of the headline workload, QPSK 128x16.
        {"name": "build_qpsk128x16", "op": "build", "kind": "mimo_qpsk", "n": 65536, "B": 128, "M": 16},
        # The largest problem, QPSK 256x32 (N = 65).
        {"name": "build_qpsk256x32", "op": "build", "kind": "mimo_qpsk", "n": 16384, "B": 256, "M": 32},
        # The JED benchmark's longer burst.
        {"name": "build_jed_bpsk16x32", "op": "build", "kind": "jed_bpsk", "n": 131072, "B": 16, "M": 32},
        # Algorithm 1 of the headline workload on the tensor cores and in FP32.
        {"name": "detect_bf16_n33", "op": "detect", "precision": "bf16_tc", "n": 65536, "N": 33, "t_max": 20},
        {"name": "detect_fp32_n33", "op": "detect", "precision": "fp32", "n": 65536, "N": 33, "t_max": 20},
        # 32 QPSK users, the largest size, at the iteration count the trade-off benchmark ends with.
        {"name": "detect_bf16_n65", "op": "detect", "precision": "bf16_tc", "n": 16384, "N": 65, "t_max": 20},
        # Emulation of the fixed-point hardware (error-rate studies against the 14-bit designs).
        {"name": "detect_fixed14_n33", "op": "detect", "precision": "fixed14", "n": 8192, "N": 33, "t_max": 20},
        # Users of four cell sizes in one batch, as a scheduler hands them over.
        {"name": "uneven_bf16_50000", "op": "uneven", "precision": "bf16_tc", "n": 50000},
        # One training step of unfolded TASER: forward, loss, gradient of the step sizes.
        {"name": "train_fp32_n33", "op": "train", "precision": "fp32", "n": 8192, "N": 33, "t_max": 10, "c": 4},
        {"name": "train_bf16_n33", "op": "train", "precision": "bf16_tc", "n": 8192, "N": 33, "t_max": 10, "c": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(kind, M):
    return {"mimo_bpsk": M + 1, "mimo_qpsk": 2 * M + 1, "jed_bpsk": M, "jed_qpsk": 2 * M - 1}[kind]


def draw(rng):
    op = rng.choice(("whole", "build", "build", "detect", "detect", "detect", "uneven", "train"))
    if op in ("whole", "build"):
        kind = rng.choice(("mimo_qpsk", "mimo_qpsk", "mimo_bpsk", "jed_bpsk", "jed_qpsk"))
        M = _log(rng, 2, 32)
        B = _log(rng, 8, 32) if kind.startswith("jed") else max(M, min(256, _log(rng, 2, 9) * M))
        most = int(1.0e9 / (8 * B * (M + 1) + 8 * _size(kind, M) ** 2))
        if op == "build":
            return {"op": op, "kind": kind, "n": min(most, _log(rng, 64, 131072)), "B": B, "M": M}
        return {"op": op, "kind": kind, "n": min(most, _log(rng, 16, 16384)), "B": B, "M": M,
                "t_max": rng.randint(1, 20)}
    if op == "detect":
        N, t_max = _log(rng, 3, 65), rng.randint(1, 20)
        precision = rng.choice(PRECISIONS)
        most = 65536 if N <= 33 else 16384
        n = _log(rng, 64, most // 8 if precision == "fixed14" else most)
        return {"op": op, "precision": precision, "n": n, "N": N, "t_max": t_max}
    if op == "uneven":
        return {"op": op, "precision": rng.choice(("bf16_tc", "fp16_tc", "fp32")), "n": _log(rng, 500, 50000)}
    t_max = rng.randint(4, 16)
    return {"op": op, "precision": rng.choice(("fp32", "bf16_tc")), "n": _log(rng, 256, 8192),
            "N": rng.randint(9, 33), "t_max": t_max, "c": math.isqrt(t_max - 1) + 1}


# Inputs ------------------------------------------------------------------------------


def _cn(shape, gen):
    """i.i.d. CN(0, 1)."""
    return torch.view_as_complex(torch.normal(0.0, 0.5 ** 0.5, tuple(shape) + (2,), generator=gen, device="cuda"))


def _signs(shape, gen):
    return torch.randint(0, 2, shape, generator=gen, device="cuda").float() * 2 - 1


def _channel(kind, n, B, M, gen):
    """(H, y) of a MU-MIMO uplink or (Y, None) of JED bursts, and the transmitted signs."""
    qpsk = kind.endswith("qpsk")
    snr = SNR_DB[0] + (SNR_DB[1] - SNR_DB[0]) * torch.rand((n,), generator=gen, device="cuda")
    re, im = _signs((n, M), gen), _signs((n, M), gen)
    if kind.startswith("jed"):
        re[:, 0] = im[:, 0] = 1.0                       # the pilot slot
    s = torch.complex(re, im) * 0.5 ** 0.5 if qpsk else torch.complex(re, torch.zeros_like(re))
    truth = torch.cat([re, im], 1) if qpsk else re
    if kind.startswith("mimo"):
        H = _cn((n, B, M), gen)
        n0 = M / 10.0 ** (snr / 10.0)
        return H, torch.bmm(H, s.unsqueeze(2)).squeeze(2) + _cn((n, B), gen) * n0.sqrt()[:, None], truth
    n0 = 1.0 / 10.0 ** (snr / 10.0)
    Y = _cn((n, B), gen)[:, :, None] * s.conj()[:, None, :] + _cn((n, B, M), gen) * n0.sqrt()[:, None, None]
    return Y, None, truth


def _real_form(kind, X, y):
    """A with T = +-A^T A (Secs. II-A and II-B), in X's precision; the augmented column last."""
    if kind.startswith("jed"):
        X, y = X[:, :, 1:], X[:, :, 0] * ((1 + 1j) * 0.5 ** 0.5 if kind == "jed_qpsk" else 1)
    else:
        y = -y
    last = torch.cat([y.real, y.imag], 1).unsqueeze(2)
    if kind.endswith("bpsk"):
        return torch.cat([torch.cat([X.real, X.imag], 1), last], 2)
    X = X * 0.5 ** 0.5
    top, bottom = torch.cat([X.real, -X.imag], 2), torch.cat([X.imag, X.real], 2)
    return torch.cat([torch.cat([top, bottom], 1), last], 2)


def _norm2(T, doublings):
    """||T||_2 of symmetric matrices by repeated squaring: T^(2^k) tends to the projector on
    the top eigenspace, whose Rayleigh quotient is the norm."""
    P = T
    for _ in range(doublings):
        P = torch.bmm(P, P)
        P = P / P.diagonal(dim1=1, dim2=2).sum(1)[:, None, None]
    return (P * T).sum((1, 2)).abs() / P.diagonal(dim1=1, dim2=2).sum(1).abs()


def _preconditioned(kind, X, y, doublings):
    """(T~, D, ||T~||_2) in X's precision."""
    A = _real_form(kind, X, y)
    T = torch.bmm(A.transpose(1, 2), A)
    T = (T + T.transpose(1, 2)) * (-0.5 if kind.startswith("jed") else 0.5)
    D = T.diagonal(dim1=1, dim2=2).abs().sqrt()
    T = T / (D[:, :, None] * D[:, None, :])
    return T.contiguous(), D.contiguous(), _norm2(T, doublings)


def _problem(n, N, gen):
    """T~, D, 1 / ||T~||_2 and the transmitted signs of n MU-MIMO problems of size N, in FP32."""
    kind, U = ("mimo_qpsk", (N - 1) // 2) if N % 2 else ("mimo_bpsk", N - 1)
    parts = []
    for first in range(0, n, 16384):
        H, y, truth = _channel(kind, min(16384, n - first), 8 * U if N % 2 else 4 * U, U, gen)
        parts.append(_preconditioned(kind, H, y, 12) + (truth,))
    T, D, norm, truth = (torch.cat(p) for p in zip(*parts))
    return T, D, 1.0 / norm, truth


def _uneven(case, gen):
    """Items of four sizes, as many of each, in random order over shared pools."""
    n = case["n"]
    shape = torch.randperm(n, generator=gen, device="cuda") % 4
    t_max = torch.tensor(UNEVEN_T, device="cuda")[torch.randint(0, 2, (n,), generator=gen, device="cuda")]
    N = 2 * torch.tensor([u for _, u in UNEVEN_SHAPES], device="cuda")[shape] + 1
    size, d_size, s_size = N * N, N, N - 1
    T_pool, D_pool = (torch.empty(int(z.sum()), device="cuda") for z in (size, d_size))
    tau = torch.empty(n, device="cuda")
    t_off, d_off, s_off = (torch.cumsum(z, 0) - z for z in (size, d_size, s_size))
    groups = []
    for k, (B, U) in enumerate(UNEVEN_SHAPES):
        at, Nk = torch.nonzero(shape == k).flatten(), 2 * U + 1
        if not at.numel():
            continue
        T, D, inv, _ = _problem(at.numel(), Nk, gen)
        where = t_off[at][:, None] + torch.arange(Nk * Nk, device="cuda")
        T_pool[where] = T.reshape(at.numel(), -1)
        D_pool[d_off[at][:, None] + torch.arange(Nk, device="cuda")] = D
        tau[at] = ALPHA * inv
        groups.append((at, T, D, tau[at], t_max[at], where))
    host = [z.cpu().numpy() for z in (N, t_max, t_off, d_off, s_off)]
    items = taser.make_items(host[0], host[1], host[2], host[3], host[4], l_off=host[2])
    return {"items": torch.from_numpy(items.view("u1")).cuda(), "T_pool": T_pool, "D_pool": D_pool, "tau": tau,
            "s_pool": torch.empty(int(s_size.sum()), dtype=torch.int8, device="cuda"),
            "L_pool": torch.empty_like(T_pool), "flags": torch.zeros(n, dtype=torch.int32, device="cuda"),
            "workspace": torch.empty(taser.uneven_workspace_bytes(n), dtype=torch.uint8, device="cuda")}, groups


def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return gen


def prepare(case, seed):
    gen = _generator(seed)
    state = {"case": case}
    if case["op"] in ("whole", "build"):
        state["X"], state["y"], _ = _channel(case["kind"], case["n"], case["B"], case["M"], gen)
    elif case["op"] == "uneven":
        state.update(_uneven(case, gen)[0])
    else:
        T, D, inv, truth = _problem(case["n"], case["N"], gen)
        state.update(T=T, D=D, inv=inv, tau=ALPHA * inv)
        if case["op"] == "train":
            state["truth"] = truth
            state["alpha"] = (0.3 + 0.4 * torch.rand((case["t_max"],), generator=gen, device="cuda")).requires_grad_()
    return state


# One pass ----------------------------------------------------------------------------


def run(state):
    case, op = state["case"], state["case"]["op"]
    if op in ("whole", "build"):
        out = taser.build_T(case["kind"], state["X"], state["y"], alpha=ALPHA)
        if op == "build":
            return out
        s, L, flags = taser.detect(out["T_tilde"], out["D"], out["tau"], case["t_max"], flags=out["flags"])
        return {"s": s, "L": L, "flags": flags, "T_tilde": out["T_tilde"], "D": out["D"], "tau": out["tau"]}
    if op == "detect":
        s, L, flags = taser.detect(state["T"], state["D"], state["tau"], case["t_max"], case["precision"])
        return {"s": s, "L": L, "flags": flags}
    if op == "uneven":
        taser.detect_uneven(state["items"], state["T_pool"], state["D_pool"], state["tau"], state["s_pool"],
                            state["workspace"], precision=case["precision"], L_pool=state["L_pool"],
                            flags=state["flags"])
        return {"s": state["s_pool"], "L": state["L_pool"], "flags": state["flags"]}
    soft = taser.UnfoldedTASER.apply(state["alpha"], state["T"], state["D"], state["inv"], case["c"],
                                     case["precision"])
    loss = torch.nn.functional.mse_loss(soft, state["truth"])
    (grad,) = torch.autograd.grad(loss, state["alpha"])
    return {"soft": soft, "loss": loss, "grad_alpha": grad}


# What a pass cannot do without -------------------------------------------------------


def _iteration_flops(N):
    """One iteration with the triangular skip (Table I): products, column norms, rescaling."""
    return 2 * (N * (N + 1) * (2 * N + 1) // 6) + 3 * N * (N + 1) // 2 + N


def work(case):
    op, n = case["op"], case["n"]
    if op in ("whole", "build"):
        kind, B, M = case["kind"], case["B"], case["M"]
        N, mimo, qpsk = _size(kind, M), kind.startswith("mimo"), kind.endswith("qpsk")
        columns = M + 1 if mimo else M
        gram = (4 if qpsk else 2) * B * columns * (columns + 1)
        reduction = (16 if qpsk else 4) * columns ** 3 // 3     # to tridiagonal form, for ||T~||_2
        inputs = 8 * B * columns
        outputs = 4 * (N * N + N + 3)
        if op == "whole":
            outputs += 4 * N * N + N - 1
        return {"bytes": n * (inputs + outputs),
                "flops": n * (gram + reduction + (case["t_max"] * _iteration_flops(N) if op == "whole" else 0))}
    if op == "uneven":
        sizes, t = [2 * u + 1 for _, u in UNEVEN_SHAPES], sum(UNEVEN_T) / len(UNEVEN_T)
        return {"bytes": n * sum(8 * N * N + 5 * N + 47 for N in sizes) / 4,
                "flops": n * t * sum(_iteration_flops(N) for N in sizes) / 4}
    N, t = case["N"], case["t_max"]
    if op == "detect":
        return {"bytes": n * (8 * N * N + 5 * N + 7), "flops": n * t * _iteration_flops(N)}
    # Training: forward, and in reverse the same product once for G and once for the adjoint.
    return {"bytes": n * (4 * N * N + 4 * N + 8 * (N - 1) + 4), "flops": n * t * 3 * _iteration_flops(N)}


# The same in 64 bits -----------------------------------------------------------------


def _iterate(T, D, taus):
    """Algorithm 1 with step taus[t] ([n] each) at iteration t."""
    N = T.shape[1]
    L = torch.diag_embed(D)
    last = torch.zeros_like(L)
    last[:, N - 1, N - 1] = D[:, N - 1]
    live = torch.ones(N, dtype=T.dtype, device=T.device)
    live[N - 1] = 0
    for tau in taus:
        V = (L - torch.tril(torch.bmm(L, T) * (2 * tau)[:, None, None])) * live
        norm = torch.where(live > 0, V.square().sum(1), torch.ones_like(D)).sqrt()
        L = V * torch.where(norm > 0, D / norm, torch.zeros_like(D))[:, None, :] + last
    return L


def _batched(f, *args):
    parts = [f(*(a[i:i + 16384] for a in args)) for i in range(0, args[0].shape[0], 16384)]
    return torch.cat(parts) if torch.is_tensor(parts[0]) else tuple(torch.cat(p) for p in zip(*parts))


def exact(case, seed):
    gen = _generator(seed)
    op = case["op"]
    if case.get("precision") == "fixed14":
        return None                                     # whole-number arithmetic: compared bit by bit
    if op in ("whole", "build"):
        kind = case["kind"]
        X, y, _ = _channel(kind, case["n"], case["B"], case["M"], gen)
        if y is None:
            y = torch.zeros_like(X[:, :, 0])
        T, D, norm = _batched(lambda a, b: _preconditioned(kind, a.cdouble(), b.cdouble(), 34), X, y)
        out = {"T_tilde": T, "D": D, "tau": ALPHA / norm, "flags": None}
        if op == "build":
            return dict(out, spec_norm=norm)
        L = _batched(lambda t, d, s: _iterate(t, d, [s] * case["t_max"]), T, D, ALPHA / norm)
        return dict(out, s=None, L=L)
    if op == "uneven":
        state, groups = _uneven(case, gen)
        out = torch.zeros_like(state["L_pool"], dtype=torch.float64)
        for _, T, D, tau, t_max, where in groups:
            for t in UNEVEN_T:
                m = t_max == t
                if m.any():
                    L = _batched(lambda a, b, c: _iterate(a, b, [c] * t), T[m].double(), D[m].double(),
                                 tau[m].double())
                    out[where[m]] = L.reshape(L.shape[0], -1)
        return {"s": None, "L": out, "flags": None}
    T, D, inv, truth = _problem(case["n"], case["N"], gen)
    if op == "detect":
        L = _batched(lambda a, b, c: _iterate(a.double(), b.double(), [c.double()] * case["t_max"]), T, D, ALPHA * inv)
        return {"s": None, "L": L, "flags": None}
    alpha = (0.3 + 0.4 * torch.rand((case["t_max"],), generator=gen, device="cuda")).double().requires_grad_()
    softs, grad, total = [], torch.zeros_like(alpha), 0.0
    for i in range(0, case["n"], 4096):
        t, d, v, b = (x[i:i + 4096].double() for x in (T, D, inv, truth))
        soft = _iterate(t, d, [a * v for a in alpha])[:, -1, :-1] / d[:, :-1]
        loss = (soft - b).square().sum() / truth.numel()
        grad += torch.autograd.grad(loss, alpha)[0]
        total += loss.item()
        softs.append(soft.detach())
    return {"soft": torch.cat(softs), "loss": torch.tensor(total, dtype=torch.float64), "grad_alpha": grad}
