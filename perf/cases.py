"""The work that programs built on this package have it do, case by case, through its public entry
points: decoding of channel LLRs (one code block at a time, a burst of blocks, simulation batches,
several codes together), weighted-BP training and inference, and encoding.

Sizes: lengths 32 .. 2048 at rates 1/4 .. 3/4 with CRC-8 up to N = 256 and CRC-24 above, Eb/N0
1 .. 4 dB, and the schedules of the benchmark (PP-BP s = 4, T = 10 with at most 300 iterations,
FP-BP of 10 trellises of 100 iterations, plain BP; min-sum and exact box-plus; CRC stop, CRC and
G-matrix stop).  FP64 weighted BP serves gradient checks only and is not listed.
"""
from __future__ import annotations

import math

import torch

from paper_1911_08868_gb300 import inputs, pcbp

DEV = "cuda"

# Mean iterations of PP-BP by Eb/N0 (dB), N = 1024, rate 1/2, at most 300: what the work counts use.
MEAN_ITERS = ((1.0, 220.0), (1.5, 135.0), (2.0, 54.0), (2.5, 21.0), (3.0, 9.9), (3.5, 6.2), (4.0, 4.8))


def listed():
    return [
        # one code block as it arrives from a demodulator: latency, not throughput
        dict(name="decode_n1024_one", kind="decode", N=1024, K=512, B=1, ebn0=3.5, mode="pp", f="minsum", stop="crc"),
        # the control-channel blocks of one slot: a small batch of a short code
        dict(name="decode_n256_burst", kind="decode", N=256, K=100, B=48, ebn0=3.0, mode="pp", f="minsum", stop="crc"),
        # short code in a Monte-Carlo simulation, a ragged number of frames
        dict(name="decode_n64", kind="decode", N=64, K=32, B=100003, ebn0=3.0, mode="pp", f="minsum", stop="crc"),
        # plain BP of the N = 256, K = 128, CRC-8 configuration, a ragged number of frames
        dict(name="decode_n256_plain", kind="decode", N=256, K=128, B=50021, ebn0=3.0, mode="bp", f="minsum",
             stop="crc"),
        # the benchmark's code, schedule and Eb/N0 (a quarter of its frames)
        dict(name="decode_n1024", kind="decode", N=1024, K=512, B=262144, ebn0=3.0, mode="pp", f="minsum",
             stop="crc"),
        # the longest code at low Eb/N0: many iterations and switches per frame
        dict(name="decode_n2048_low", kind="decode", N=2048, K=1024, B=16384, ebn0=2.0, mode="pp", f="minsum",
             stop="crc"),
        # high rate, CRC and G-matrix stop together
        dict(name="decode_n512_crc_g", kind="decode", N=512, K=384, B=32768, ebn0=3.5, mode="pp", f="minsum",
             stop="crc_g"),
        # exact box-plus in place of min-sum
        dict(name="decode_n1024_boxplus", kind="decode", N=1024, K=512, B=32768, ebn0=3.0, mode="pp", f="boxplus",
             stop="crc"),
        # traffic of five lengths at three rates in one sweep
        dict(name="decode_mixed", kind="mixed", B=65536, ebn0_lo=1.0, ebn0_hi=4.0, lo=7, hi=11),
        # a training step of the weighted-BP benchmark (forward, loss, backward)
        dict(name="wbp_train_n1024", kind="wbp", N=1024, K=512, T=5, B=4096, grad="w"),
        # the step of the weighted-BP training run
        dict(name="wbp_train_n256", kind="wbp", N=256, K=128, T=5, B=4096, grad="w"),
        # encoding of a simulation's payloads
        dict(name="encode_n1024", kind="encode", N=1024, K=512, B=262144),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("decode", "decode", "decode", "host", "mixed", "wbp", "wbp", "infer", "encode"))
    if kind == "mixed":
        lo = rng.randint(5, 9)
        return dict(kind="mixed", B=_log_int(rng, 256, 65536), ebn0_lo=round(rng.uniform(1.0, 2.5), 2), ebn0_hi=4.0,
                    lo=lo, hi=rng.randint(lo + 1, 11))
    if kind in ("wbp", "infer"):
        n = rng.randint(4, 10)
        N = 1 << n
        T = rng.randint(1, 20)
        most = min(16384, 4096 * 10 * 10 * 1024 // (T * n * N))
        return dict(kind="wbp", N=N, K=rng.randint(N // 4, 3 * N // 4), T=T, B=_log_int(rng, 16, most),
                    grad="none" if kind == "infer" else rng.choice(("w", "w", "w+llr")))
    n = rng.randint(5, 11)
    N = 1 << n
    K = rng.randint(max(N // 4, 12 if N <= 256 else 40), 3 * N // 4)
    if kind == "encode":
        return dict(kind="encode", N=N, K=K, B=_log_int(rng, 1, 262144 * 1024 // N))
    c = dict(kind=kind, N=N, K=K, B=1, ebn0=round(rng.uniform(1.5, 4.0), 2), mode=rng.choice(("pp", "pp", "fp", "bp")),
             f=rng.choice(("minsum", "minsum", "minsum", "boxplus")), stop=rng.choice(("crc", "crc", "crc_g")))
    # as much work as the largest listed batches at most (exact box-plus costs about three times as much)
    most = 2.0e10 / (_mean_iters(c) * n * N * (3 if c["f"] == "boxplus" else 1))
    return dict(c, B=_log_int(rng, 1, min(max(most, 2.0), 262144.0)))


def _crc(N):
    return (8, 0x9B) if N <= 256 else (24, 0x1B2B117)


def _sched(c, n, seed):
    stop = dict(stop_from=1, stop_kind=3 if c["stop"] == "crc_g" else 1, fkind=1 if c["f"] == "boxplus" else 0,
                alpha=0.9375, seed=seed)
    if c["mode"] == "fp":
        return pcbp.sched(mode=2, it_reset_full=100, q_max=10, **stop), 1000
    if c["mode"] == "bp":
        return pcbp.sched(mode=0, **stop), 300
    return pcbp.sched(mode=1, rho_range_fixed=4, P_level=n - 1, N_min=10, D=0, T0=10, **stop), 300


def _mean_iters(c):
    e = min(max(c["ebn0"], MEAN_ITERS[0][0]), MEAN_ITERS[-1][0])
    it = MEAN_ITERS[-1][1]
    for (a, x), (b, y) in zip(MEAN_ITERS, MEAN_ITERS[1:]):
        if a <= e <= b:
            it = x * (y / x) ** ((e - a) / (b - a))
            break
    return it * 3.0 if c["mode"] == "fp" else it


def _frames(code, gen, B, ebn0):
    """Payload bits and the LLRs of their codewords after the AWGN channel (Eb/N0 scalar or per frame)."""
    pay = inputs.payload_torch(gen, B, code.K - code.crc_len, DEV)
    x = torch.empty((B, code.N), dtype=torch.uint8, device=DEV)
    pcbp.pc_encode(code, pay, x)
    s2 = inputs.sigma2_of(ebn0, code.K, code.crc_len, code.N)
    return pay, inputs.bpsk_awgn_llr_torch(x, gen, s2).contiguous()


def _classes(c):
    """(N, K, frames) of the mixed case's classes, the longest work first."""
    sizes = [(1 << n, (1 << n) * q // 4) for n in range(c["lo"], c["hi"] + 1) for q in (1, 2, 3)]
    sizes = [(N, max(K, 12 if N <= 256 else 40)) for N, K in sizes]
    per, rest = divmod(c["B"], len(sizes))
    got = [(N, K, per + (1 if i < rest else 0)) for i, (N, K) in enumerate(sizes)]
    return sorted((g for g in got if g[2] > 0), key=lambda g: -g[0] * g[2])


def _uniform_ebn0(gen, B, lo, hi):
    return (lo + (hi - lo) * torch.rand(B, generator=gen, device=DEV, dtype=torch.float64)).cpu().numpy()


def _wbp_inputs(case, seed):
    """Code, LLRs, weights around the min-sum scale and the bits of a weighted-BP batch (Eb/N0 uniform on [1, 4] dB)."""
    N, K, T, B = case["N"], case["K"], case["T"], case["B"]
    n = N.bit_length() - 1
    code = pcbp.pc_construct(N, K)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    bits, llr = _frames(code, gen, B, _uniform_ebn0(gen, B, 1.0, 4.0))
    w = 0.9375 + 0.05 * torch.randn((T, n, N // 2, 4), generator=gen, device=DEV)
    return code, llr, w, bits


def prepare(case, seed):
    kind = case["kind"]
    gen = torch.Generator(device=DEV).manual_seed(seed)
    if kind == "wbp":
        code, llr, w, bits = _wbp_inputs(case, seed)
        return dict(kind=kind, code=code, T=case["T"], llr=llr.requires_grad_("llr" in case["grad"]),
                    w=w.requires_grad_(case["grad"] != "none"), target=bits.float(), grad=case["grad"])
    if kind == "mixed":
        parts = []
        for i, (N, K, B) in enumerate(_classes(case)):
            n = N.bit_length() - 1
            code = pcbp.pc_construct(N, K, *_crc(N))
            _, llr = _frames(code, gen, B, _uniform_ebn0(gen, B, case["ebn0_lo"], case["ebn0_hi"]))
            sch, most = _sched(dict(mode="pp", f="minsum", stop="crc"), n, seed + i)
            parts.append((code, sch, most, llr, 0))
        return dict(kind=kind, decoder=pcbp.MixedDecoder(parts, DEV))
    N, K, B = case["N"], case["K"], case["B"]
    code = pcbp.pc_construct(N, K, *_crc(N))
    if kind == "encode":
        pay = inputs.payload_torch(gen, B, K - code.crc_len, DEV)
        return dict(kind=kind, code=code, payload=pay, x=torch.empty((B, N), dtype=torch.uint8, device=DEV))
    _, llr = _frames(code, gen, B, case["ebn0"])
    sch, most = _sched(case, N.bit_length() - 1, seed)
    if kind == "host":
        return dict(kind=kind, decoder=pcbp.HostDecoder(code, sch, most, DEV), llr=llr.cpu().pin_memory())
    return dict(kind=kind, decoder=pcbp.Decoder(code, sch, most, DEV), llr=llr)


def run(state):
    kind = state["kind"]
    if kind == "encode":
        pcbp.pc_encode(state["code"], state["payload"], state["x"])
        return state["x"]
    if kind == "mixed":
        return state["decoder"]()
    if kind != "wbp":
        return state["decoder"](state["llr"])
    llr, w, code, T = state["llr"], state["w"], state["code"], state["T"]
    if state["grad"] == "none":
        with torch.no_grad():
            return pcbp.wbp(llr, w, code, T)
    llr.grad = w.grad = None
    logits = pcbp.wbp(llr, w, code, T)
    loss = torch.nn.functional.binary_cross_entropy_with_logits(-logits, state["target"])
    loss.backward()
    grads = [w.grad] if llr.grad is None else [w.grad, llr.grad]
    return [logits.detach(), loss.detach(), *grads]


def work(case):
    kind = case["kind"]
    if kind == "encode":
        N, K, B = case["N"], case["K"], case["B"]
        return {"bytes": B * (K - _crc(N)[0] + N), "flops": B * N // 2 * (N.bit_length() - 1)}
    if kind == "wbp":
        N, K, T, B = case["N"], case["K"], case["T"], case["B"]
        n = N.bit_length() - 1
        stages = T * n + (T - 1) * (n - 1)
        weights = 4 * T * n * 2 * N
        train = case["grad"] != "none"
        # per processing element and stage 8 operations forward, 16 in the adjoint
        flops = B * stages * (N // 2) * (24 if train else 8)
        moved = B * (4 * N + 4 * K) + weights
        if train:
            moved += B * 4 * K + weights + (B * 4 * N if "llr" in case["grad"] else 0)
        return {"bytes": moved, "flops": flops}
    # decoding: LLRs in, packed bits, iterations and CRC flags out; 8 operations per processing
    # element in each half sweep
    if kind == "mixed":
        mid = dict(ebn0=0.5 * (case["ebn0_lo"] + case["ebn0_hi"]) - 0.3, mode="pp")
        parts = [(N, K, B, _mean_iters(mid)) for N, K, B in _classes(case)]
    else:
        parts = [(case["N"], case["K"], case["B"], _mean_iters(case))]
    return {"bytes": sum(B * (4 * N + 4 * ((K + 31) // 32) + 5) for N, K, B, _ in parts),
            "flops": sum(B * it * 8 * (N.bit_length() - 1) * N for N, _, B, it in parts)}


def _f(u, v, w):
    """f_w(a, b) = w sign(a) sign(b) min(|a|, |b|) of operand pairs (64-bit value, 32-bit value).  f is
    linear once the minimum (the first operand on ties; it takes the gradient) and the signs are
    known; the 32-bit values choose them, since a near-tie may fall the other way in 64 bits and
    with it the gradient of everything behind, and the 64-bit values are what is computed."""
    first = u[1].abs() <= v[1].abs()
    su, sv = torch.sign(u[1]), torch.sign(v[1])
    return (w[0] * torch.where(first, u[0] * sv, v[0] * su), w[1] * torch.where(first, u[1] * sv, v[1] * su))


def _add(u, v):
    return u[0] + v[0], u[1] + v[1]


def _wbp64(llr, w, frozen, T):
    """L at the last level after T iterations of weighted BP; llr and w are pairs (64-bit, 32-bit values).
    Frozen priors are infinite, and a large finite number where autograd would multiply them by 0."""
    B, N = llr[0].shape
    n = N.bit_length() - 1
    prior = ((frozen.double() * 1e200).expand(B, N), torch.where(frozen, math.inf, 0.0).expand(B, N))
    R = [tuple(torch.zeros_like(x) for x in prior)] * n + [prior]
    L = [llr] + [None] * n

    def halves(x, s):
        top, bot = zip(*(y.reshape(B, 1 << s, 2, N >> (s + 1)).unbind(2) for y in x))
        return top, bot

    def weights(it, s, k):
        return tuple(x[it, s, :, k].reshape(1 << s, N >> (s + 1)) for x in w)

    def joined(top, bot):
        return tuple(torch.stack(x, 2).reshape(B, N) for x in zip(top, bot))

    for it in range(T):
        for s in range(n):
            (lt, lb), (rt, rb) = halves(L[s], s), halves(R[s + 1], s)
            L[s + 1] = joined(_f(lt, _add(lb, rb), weights(it, s, 0)), _add(_f(rt, lt, weights(it, s, 1)), lb))
        if it == T - 1:
            break
        R = list(R)
        for s in range(n - 1, 0, -1):
            (lt, lb), (rt, rb) = halves(L[s], s), halves(R[s + 1], s)
            R[s] = joined(_f(rt, _add(lb, rb), weights(it, s, 2)), _add(_f(rt, lt, weights(it, s, 3)), rb))
    return L[n][0]


# Unrolled BP grows the messages and, more so, their gradients from iteration to iteration, and the
# rounding of 32 bits with them: after this many iterations it can be of the result's own size.
EXACT_LOGITS_T, EXACT_GRAD_T = 8, 6


def exact(case, seed):
    """Weighted BP in 64 bits, up to the iterations above; decoding and encoding give whole numbers."""
    if case["kind"] != "wbp" or case["T"] > EXACT_LOGITS_T:
        return None
    code, llr, w, bits = _wbp_inputs(case, seed)
    B, N = llr.shape
    K = code.K
    frozen = torch.tensor(code.frozen(), dtype=torch.bool, device=DEV)
    train = case["grad"] != "none"
    grads = case["T"] <= EXACT_GRAD_T
    w32, w = w, w.double().requires_grad_(train)
    logits = torch.empty((B, K), dtype=torch.float64, device=DEV)
    loss = torch.zeros((), dtype=torch.float64, device=DEV)
    gllr = torch.zeros((B, N), dtype=torch.float64, device=DEV)
    step = max(1, (1 << 19) // N)
    for lo in range(0, B, step):
        x = llr[lo:lo + step].double().requires_grad_(train)
        with torch.set_grad_enabled(train):
            y = _wbp64((x, llr[lo:lo + step]), (w, w32), frozen, case["T"])[:, ~frozen]
            part = torch.nn.functional.binary_cross_entropy_with_logits(-y, bits[lo:lo + step].double(),
                                                                        reduction="sum") / (B * K)
        logits[lo:lo + step] = y.detach()
        if train:
            part.backward()
            loss += part.detach()
            gllr[lo:lo + step] = x.grad
    if not train:
        return logits
    return [logits, loss, w.grad if grads else None] + ([gllr if grads else None] if "llr" in case["grad"] else [])
