"""Timed workloads of the library, each through its public entry points.

listed() names twelve passes over the range a user runs: the smallest
instantiation, where launches and latency are all there is; FP64 and
complex64 brick walls from 7 to 12 qubits, with host and with device arrays;
the batched form over uneven blocks, large and small; the target product; the
allocation-free sweep; a layer of the learned warm start and its gradients.
draw() gives further passes of the same kinds and ranges, odd sizes included.

A circuit is a brick wall or a chain of general 2-qubit gates, its target the
product of Haar-random gates in the same structure, its training states and
starts Haar-random: the inputs the method is run on (workloads.py).  Runs have
a fixed budget of sweeps and a tolerance they do not reach, so that a pass is
the same work on every input; complex64 runs get few sweeps, because rounding
grows from sweep to sweep until two correct runs have little in common.
Complex64 sweeps hand out complex128 arrays that hold complex64-accurate
values; the passes keep them as complex64, as a program that stores them
would.  An FP64 cost 2 - 2 Re<U psi, C psi> is returned as the overlap
Re<U psi, C psi> = 1 - cost / 2 that it is formed from.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2405_12866_gb300 import learned, qfs
from paper_2405_12866_gb300 import workloads as w

_KEPT = {}


def _context():
    """The one context a program keeps for its lifetime."""
    if "ctx" not in _KEPT:
        _KEPT["ctx"] = qfs.Context(0)
    return _KEPT["ctx"]


def _model():
    if "ws" not in _KEPT:
        _KEPT["ws"] = qfs.WarmStart(_context(), seed=7, batch_cap=4096)
    return _KEPT["ws"]


# ------------------------------------------------------------------- cases

def listed():
    return [
        # The smallest block (3 qubits, 4 gates, one start, 200 sweeps): launch and update latency.
        dict(name="chain_n3_fp64", kind="instantiate", n=3, layers=0, L=4, M=4, S=1, sweeps=200, mixed=False, host=True),
        # Odd counts: 7 qubits, 21 gates, 24 states, 5 starts.
        dict(name="brick_n7_fp64", kind="instantiate", n=7, layers=7, L=21, M=24, S=5, sweeps=30, mixed=False, host=False),
        # The 8-qubit FP64 configuration: 28 gates, 16 states, 16 starts.
        dict(name="brick_n8_fp64", kind="instantiate", n=8, layers=8, L=28, M=16, S=16, sweeps=20, mixed=False, host=False),
        # FP64 at 10 qubits, the largest size of the comparison with full-unitary sweeps.
        dict(name="brick_n10_fp64", kind="instantiate", n=10, layers=4, L=18, M=32, S=8, sweeps=12, mixed=False, host=False),
        # The 8-qubit block in complex64 from host arrays: the call of the README.
        dict(name="brick_n8_mixed_host", kind="instantiate", n=8, layers=8, L=28, M=16, S=16, sweeps=4, mixed=True, host=True),
        # The headline configuration: 12 qubits, 17 gates, 32 states, 32 starts, complex64.
        dict(name="brick_n12_mixed", kind="instantiate", n=12, layers=3, L=17, M=32, S=32, sweeps=4, mixed=True, host=False),
        # The batched form over a thousand uneven 3-5 qubit blocks, 8 starts each, device arrays.
        dict(name="blocks_1024", kind="blocks", P=1024, S=8, sweeps=4, host=False),
        # A few blocks at a time from host arrays: too few units to fill the chip.
        dict(name="blocks_96_host", kind="blocks", P=96, S=8, sweeps=4, host=True),
        # Phi_L = U Psi at 12 qubits in FP64, the product every instantiation starts from.
        dict(name="product_n12_fp64", kind="product", n=12, M=32, mixed=False),
        # One allocation-free FP64 sweep, queued on the caller's stream.
        dict(name="noalloc_n6", kind="noalloc", n=6, layers=4, L=10, M=16, S=8),
        # A hidden layer of the warm-start network on a batch of 8192: GEMM, bias, GELU.
        dict(name="layer_8192", kind="gemm", rows=8192, cols=1024, depth=1024, gelu=True),
        # Loss and gradients of the warm-start network on a full batch: forward and backward.
        dict(name="grad_4096", kind="grad", count=4096),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["instantiate"] * 4 + ["blocks"] * 2 + ["product", "noalloc", "gemm", "grad"])
    if kind == "instantiate":
        mixed = rng.random() < 0.5
        n = rng.randint(3, 12) if mixed else rng.randint(3, 10)
        layers = rng.randint(4 if n < 7 else 3, 8)
        L = len(w.brick_pairs(n, layers))
        M = _log_int(rng, 4, min(1 << n, 48))
        S = _log_int(rng, 1, 32)
        # No more than the work of the largest listed pass (FP64 arithmetic runs at 1/64 of FP32's rate).
        per_sweep = (1 << n) * M * S * L * (1 if mixed else 12)
        cap = (1 << 12) * 32 * 32 * 17
        S = max(1, min(S, S * cap // per_sweep))
        # Few enough sweeps that no start of a small circuit has converged to rounding (equal costs have no best start).
        sweeps = max(2, min(4 if mixed else 6 if n < 7 else 10, cap * 4 // per_sweep))
        return dict(kind=kind, n=n, layers=layers, L=L, M=M, S=S, sweeps=sweeps, mixed=mixed, host=rng.random() < 0.3)
    if kind == "blocks":
        return dict(kind=kind, P=_log_int(rng, 24, 1024), S=rng.randint(2, 8), sweeps=rng.randint(2, 4), host=rng.random() < 0.5)
    if kind == "product":
        return dict(kind=kind, n=rng.randint(6, 12), M=_log_int(rng, 2, 48), mixed=rng.random() < 0.4)
    if kind == "noalloc":
        n, layers = rng.randint(3, 8), rng.randint(2, 6)
        L = len(w.brick_pairs(n, layers))
        M = _log_int(rng, 4, min(1 << n, 16))
        S = _log_int(rng, 1, 12)
        S = max(1, min(S, (12 << 20) // ((1 << n) * M * 16 * (L + 1))))
        return dict(kind=kind, n=n, layers=layers, L=L, M=M, S=S)
    if kind == "gemm":
        return dict(kind=kind, rows=128 * _log_int(rng, 2, 64), cols=256 * rng.randint(1, 4), depth=64 * _log_int(rng, 4, 16),
                    gelu=rng.random() < 0.7)
    return dict(kind=kind, count=_log_int(rng, 200, 4096))


def _pairs(case):
    return w.brick_pairs(case["n"], case["layers"]) if case["layers"] else w.chain_pairs(case["n"], case["L"])


# ------------------------------------------------------------------ inputs

def _apply(gate, pair, n, X):
    """(gate on `pair`, identity elsewhere) X, X of shape (..., N, K), gate (..., 4, 4); torch."""
    lead = X.dim() - 2
    a, b = pair
    T = X.reshape(X.shape[:lead] + (2,) * n + (X.shape[-1],))
    T = torch.movedim(T, (lead + a, lead + b), (lead, lead + 1))
    shape = T.shape
    T = (gate @ T.reshape(shape[:lead] + (4, -1))).reshape(shape)
    return torch.movedim(T, (lead, lead + 1), (lead + a, lead + b)).reshape(X.shape)


def _target(n, pairs, seed):
    """The target unitary on the GPU: the product of Haar-random gates in the structure."""
    g = torch.from_numpy(w.haar_gates_batched(seed, w.STREAM_TARGET_GATES, len(pairs))).cuda()
    U = torch.eye(1 << n, dtype=torch.complex128, device="cuda")
    for k, p in enumerate(pairs):
        U = _apply(g[k], p, n, U)
    return U.contiguous()


def _draws(case, seed):
    """Training states (N, M) and starts (S, L, 4, 4)."""
    S, L = case["S"], case["L"]
    return (w.sample_states(seed + 1, case["n"], case["M"]),
            w.haar_gates_batched(seed + 1, w.STREAM_INIT_GATES, S * L).reshape(S, L, 4, 4))


def _blocks(case, seed):
    """Uneven partition blocks in packed arrays: n uniform in 3..5, the first n + 1..10 gates of a brick wall.
    The structures belong to the case, the targets, states and starts to the seed."""
    P, S = case["P"], case["S"]
    ns = w.uniform_ints(4, w.STREAM_STRUCTURE, 0, P, 3, 5).astype(np.int32)
    Ls = (ns + 1 + w.uniform_ints(4, w.STREAM_STRUCTURE, P, P, 0, 1 << 20) % (10 - ns)).astype(np.int32)
    first = np.concatenate([[0], np.cumsum(Ls)])
    pairs = [w.brick_pairs(int(n), 10)[:L] for n, L in zip(ns, Ls)]
    tg = w.haar_gates_batched(seed, w.STREAM_TARGET_GATES, int(first[-1]))
    ig = w.haar_gates_batched(seed, w.STREAM_INIT_GATES, int(first[-1]) * S)
    z = w.complex_normals(seed, w.STREAM_SAMPLES, 0, int(np.sum(1 << (2 * ns.astype(np.int64) - 1))))
    targets, samples, at = [], [], 0
    for i in range(P):
        N, M = 1 << int(ns[i]), 1 << int(ns[i] - 1)
        targets.append(w.target_unitary(tg[first[i]:first[i + 1]], pairs[i], int(ns[i])).reshape(-1))
        samples.append(w.positive_qr_q(z[at:at + N * M].reshape(N, M)).reshape(-1))
        at += N * M
    return ns, Ls, np.array(sum(pairs, []), dtype=np.int32), np.concatenate(targets), np.concatenate(samples), ig.reshape(-1)


def _training_set(case, seed):
    """Targets of the learned structure and their gates in the canonical gauge."""
    n = case["count"]
    g = w.haar_gates_batched(seed, w.STREAM_TARGET_GATES, n * learned.L).reshape(n, learned.L, 4, 4)
    return w.target_unitaries(g, learned.PAIRS, 4), learned.gates_to_labels(learned.canonical_gauge(g))


def prepare(case, seed):
    kind, s = case["kind"], dict(case=case, ctx=_context())
    if kind == "instantiate":
        pairs = _pairs(case)
        U = _target(case["n"], pairs, seed)
        psi, g0 = _draws(case, seed)
        s["params"] = qfs.default_params(M=case["M"], multistarts=case["S"], max_sweeps=case["sweeps"], dist_tol=1e-30,
                                         precision=qfs.QFS_MIXED if case["mixed"] else qfs.QFS_FP64)
        if case["host"]:
            s.update(pairs=pairs, target=U.cpu().numpy(), samples=psi, starts=g0)
        else:
            s.update(pairs=pairs, target=U, samples=torch.from_numpy(psi).cuda(), starts=torch.from_numpy(g0).cuda(),
                     out=torch.empty((case["L"], 4, 4), dtype=torch.complex128, device="cuda"))
    elif kind == "blocks":
        ns, Ls, pairs, targets, samples, starts = _blocks(case, seed)
        s.update(ns=ns, Ls=Ls, pairs=np.ascontiguousarray(pairs.reshape(-1)), targets=targets, samples=samples, starts=starts)
        if not case["host"]:
            for k in ("targets", "samples", "starts"):
                s[k] = torch.from_numpy(s[k]).cuda()
            s["out"] = torch.empty(int(Ls.sum()) * 16, dtype=torch.complex128, device="cuda")
        s["params"] = qfs.default_params(M=0, multistarts=case["S"], max_sweeps=case["sweeps"], dist_tol=1e-30, refine_sweeps_max=0,
                                         precision=qfs.QFS_MIXED)
    elif kind == "product":
        s["target"] = _target(case["n"], w.brick_pairs(case["n"], 3), seed)
        s["samples"] = torch.from_numpy(w.sample_states(seed + 1, case["n"], case["M"])).cuda()
    elif kind == "noalloc":
        pairs = _pairs(case)
        psi, g0 = _draws(case, seed)
        s.update(pairs=np.ascontiguousarray(np.asarray(pairs, dtype=np.int32).reshape(-1)), target=_target(case["n"], pairs, seed),
                 samples=torch.from_numpy(psi).cuda(), starts=torch.from_numpy(g0).cuda())
        s["circuit"] = qfs.Circuit(case["n"], case["L"], s["pairs"].ctypes.data_as(ctypes.POINTER(ctypes.c_int32)))
        s["out"] = torch.empty_like(s["starts"])
        s["envs"] = torch.empty_like(s["starts"])
        s["costs"] = torch.empty(case["S"], dtype=torch.float64, device="cuda")
    elif kind == "gemm":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        a = torch.randn(case["rows"], case["depth"], generator=gen, device="cuda")
        s["A"] = torch.nn.functional.gelu(a).to(torch.bfloat16)
        s["B"] = (torch.randn(case["cols"], case["depth"], generator=gen, device="cuda") * math.sqrt(2.0 / case["depth"])).to(torch.bfloat16)
        s["bias"] = 0.1 * torch.randn(case["cols"], generator=gen, device="cuda")
    else:
        s["targets"], s["labels"] = _training_set(case, seed)
        s["model"] = _model()
    return s


# --------------------------------------------------------------------- run

def _kept(case, gates, costs):
    """Gates and costs at the accuracy the run has."""
    costs = np.asarray(costs)
    if not case.get("mixed", True):
        return dict(gates=gates, overlap=1.0 - 0.5 * costs)
    gates = gates.astype(np.complex64) if isinstance(gates, np.ndarray) else gates.to(torch.complex64)
    return dict(gates=gates, costs=costs.astype(np.float32))


def run(s):
    case, kind, ctx = s["case"], s["case"]["kind"], s["ctx"]
    if kind == "instantiate":
        if case["host"]:
            r = ctx.instantiate(case["n"], s["pairs"], s["target"], s["params"], samples=s["samples"], init_gates=s["starts"])
        else:
            r = ctx.instantiate_dev(case["n"], s["pairs"], s["target"], s["samples"], s["starts"], s["params"], s["out"])
        return _kept(case, r.gates, r.start_costs)
    if kind == "blocks":
        if case["host"]:
            gates, info = ctx.instantiate_batch_packed(s["ns"], s["Ls"], s["pairs"], s["targets"], s["samples"], s["starts"], s["params"])
        else:
            gates = s["out"]
            info = ctx.instantiate_batch_dev(s["ns"], s["Ls"], s["pairs"], s["targets"], s["samples"], s["starts"], s["params"], gates)
        return _kept(case, gates, [r["cost"] for r in info])
    if kind == "product":
        return ctx.target_product(case["n"], s["target"], s["samples"], qfs.QFS_MIXED if case["mixed"] else qfs.QFS_FP64)
    if kind == "noalloc":
        qfs._check(qfs.lib().qfs_sweep_once_noalloc(
            torch.cuda.current_stream().cuda_stream, ctypes.byref(s["circuit"]), s["target"].data_ptr(), s["samples"].data_ptr(),
            case["M"], case["S"], 0.0, s["starts"].data_ptr(), s["out"].data_ptr(), s["costs"].data_ptr(), s["envs"].data_ptr()))
        return dict(gates=s["out"], envs=s["envs"], costs=s["costs"])
    if kind == "gemm":
        return ctx.gemm_bf16(s["A"], s["B"], bias=s["bias"], gelu=case["gelu"], want_f32=False, want_bf16=True)[1]
    loss, grads = s["model"].loss_grad(s["targets"], s["labels"])
    return dict(loss=np.float32(loss), grads=grads)


# -------------------------------------------------------------------- work

def work(case):
    kind = case["kind"]
    if kind in ("instantiate", "noalloc"):
        N, M, S, L = 1 << case["n"], case["M"], case["S"], case["L"]
        sweeps = case.get("sweeps", 1)
        # Per sweep, gate and state entry: one forward product, one backward product, one environment term (4 complex FMAs each).
        gates_out = S * L if kind == "noalloc" else L
        return dict(bytes=16.0 * (N * N + N * M + S * L * 16 + gates_out * 16), flops=8.0 * N * N * M + 96.0 * sweeps * S * L * N * M)
    if kind == "blocks":
        # Means over the blocks' sizes: N^2 = 448, N M = 224, L = 7.5, L N M = 1760.
        P, S, sweeps = case["P"], case["S"], case["sweeps"]
        return dict(bytes=16.0 * P * (448 + 224 + 7.5 * 16 * (S + 1)), flops=P * S * sweeps * 96.0 * 1760 + P * 8.0 * (512 + 4096 + 32768) / 6)
    if kind == "product":
        N, M = 1 << case["n"], case["M"]
        return dict(bytes=16.0 * (N * N + 2 * N * M), flops=8.0 * N * N * M)
    if kind == "gemm":
        m, n, k = case["rows"], case["cols"], case["depth"]
        return dict(bytes=2.0 * (m * k + n * k + m * n) + 4.0 * n, flops=2.0 * m * n * k)
    weights = sum(a * b for a, b in qfs.WarmStart.DIMS)
    n = case["count"]
    return dict(bytes=n * (16.0 * 256 + 8.0 * 192) + 8.0 * weights, flops=6.0 * n * weights)


# ------------------------------------------------------------------- exact

def _polar(A):
    """Unitary polar factor of a stack of 4x4 matrices (host SVD)."""
    u, _, vh = np.linalg.svd(A.resolve_conj().cpu().numpy())
    return torch.from_numpy(u @ vh).to(A.device)


def _pair_major(X, pair, n):
    """(B, N, M) -> (B, 4, N M / 4), row = 2 bit_a + bit_b."""
    T = X.reshape((X.shape[0],) + (2,) * n + (X.shape[-1],))
    return torch.movedim(T, (1 + pair[0], 1 + pair[1]), (1, 2)).reshape(X.shape[0], 4, -1)


def _sweeps(n, pairs, phi, psi, gates, sweeps):
    """QFactor-Sample sweeps in 64 bits: phi and psi (B, N, M), gates (B, L, 4, 4).  Returns gates, environments, costs."""
    L, M = len(pairs), psi.shape[-1]
    gates = gates.clone()
    envs = torch.empty_like(gates)
    for _ in range(sweeps):
        B = [psi]
        for k in range(L - 1):
            B.append(_apply(gates[:, k], pairs[k], n, B[-1]))
        P = phi
        for k in range(L - 1, -1, -1):
            E = _pair_major(B[k], pairs[k], n) @ _pair_major(P, pairs[k], n).mH
            gates[:, k] = _polar(E.mH)
            envs[:, k] = E
            if k:
                P = _apply(gates[:, k].mH, pairs[k], n, P)
        cost = 2.0 - 2.0 / M * torch.einsum("bij,bji->b", gates[:, 0], envs[:, 0]).real
    return gates, envs, cost


def exact(case, seed):
    kind = case["kind"]
    if kind in ("instantiate", "noalloc"):
        n, pairs, S = case["n"], _pairs(case), case["S"]
        U = _target(n, pairs, seed)
        psi, g0 = (torch.from_numpy(x).cuda() for x in _draws(case, seed))
        g, envs, cost = _sweeps(n, pairs, (U @ psi).expand(S, -1, -1), psi.expand(S, -1, -1), g0, case.get("sweeps", 1))
        if kind == "noalloc":
            return dict(gates=g, envs=envs, costs=cost)
        best = g[int(torch.argmin(cost))]
        best, cost = best.cpu().numpy() if case["host"] else best, cost.cpu().numpy()
        return dict(gates=best, costs=cost) if case["mixed"] else dict(gates=best, overlap=1.0 - 0.5 * cost)
    if kind == "blocks":
        P, S = case["P"], case["S"]
        if P > 128:
            return None
        ns, Ls, pairs, targets, samples, starts = _blocks(case, seed)
        gates, costs, t, m, k = [], [], 0, 0, 0
        for i in range(P):
            n, L = int(ns[i]), int(Ls[i])
            N, M = 1 << n, 1 << (n - 1)
            U = torch.from_numpy(targets[t:t + N * N].reshape(N, N))
            psi = torch.from_numpy(samples[m:m + N * M].reshape(N, M))
            g0 = torch.from_numpy(starts[k * S * 16:(k + L) * S * 16].reshape(S, L, 4, 4))
            g, _, cost = _sweeps(n, pairs[k:k + L].tolist(), (U @ psi).expand(S, -1, -1), psi.expand(S, -1, -1), g0, case["sweeps"])
            best = int(torch.argmin(cost))
            gates.append(g[best].reshape(-1).numpy())
            costs.append(float(cost[best]))
            t, m, k = t + N * N, m + N * M, k + L
        gates = np.concatenate(gates)
        return dict(gates=gates if case["host"] else torch.from_numpy(gates), costs=np.array(costs))
    if kind == "product":
        U = _target(case["n"], w.brick_pairs(case["n"], 3), seed)
        psi = torch.from_numpy(w.sample_states(seed + 1, case["n"], case["M"])).cuda()
        return U @ psi
    if kind == "gemm":
        s = prepare(case, seed)
        y = s["A"].double() @ s["B"].double().T + s["bias"].double()
        return torch.nn.functional.gelu(y, approximate="tanh") if case["gelu"] else y
    return None
