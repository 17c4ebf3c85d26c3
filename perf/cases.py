"""The work that users of this library have it do, as a list of measurable cases.

Every case goes through the public entry points of paper_2608_13426_b200 (binding.py) on torch CUDA tensors.  Kinds:

  product     Y, idx = rmm(A, B, rho): scores, selection and reduced product in one call (prefill of a projection for
              many rows, a decode step for one row or a small batch of them), bf16 or fp32 operands
  mlp_block   up projection that scores its own output, selection on those energies, reduced down projection
  product_q8  scores and selection on bf16 activations, reduced product with e4m3 operands
  attention   rmm_reduced_attn: prefill (causal, with or without token reduction or an additive mask) and decode
              (few query rows against a long key/value cache)
"""
import math

import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import synth


def listed():
    return [
        # the smallest benchmark configuration: a call is launch latency and little else
        {"name": "product_small", "kind": "product", "M": 64, "K": 512, "N": 256, "rho": 0.5, "dtype": "bf16"},
        # 1B-class MLP down projection, prefill of 2048 tokens
        {"name": "product_1b_down", "kind": "product", "M": 2048, "K": 8192, "N": 2048, "rho": 0.5, "dtype": "bf16"},
        # 70B-class MLP down projection, prefill of 32768 tokens: the largest product the library is quoted on
        {"name": "product_70b_down", "kind": "product", "M": 32768, "K": 28672, "N": 8192, "rho": 0.5, "dtype": "bf16"},
        # fp32 operands (the 1e-5 accuracy path) at sizes that no tile divides
        {"name": "product_fp32", "kind": "product", "M": 777, "K": 3000, "N": 1500, "rho": 0.5, "dtype": "fp32"},
        # one decode step through a 70B-class gate/up projection
        {"name": "decode_row", "kind": "product", "M": 1, "K": 8192, "N": 28672, "rho": 0.5, "dtype": "bf16"},
        # a decode step of a batch of sequences through the same projection
        {"name": "decode_batch", "kind": "product", "M": 24, "K": 8192, "N": 28672, "rho": 0.25, "dtype": "bf16"},
        # whole MLP block on a ragged number of tokens: no score pass over the intermediate activations
        {"name": "mlp_block_ragged", "kind": "mlp_block", "M": 1531, "K": 4096, "F": 14336, "rho": 0.5},
        # quantised weights and activations on the fp8 tensor cores
        {"name": "product_q8", "kind": "product_q8", "M": 4096, "K": 8192, "N": 8192, "rho": 0.5},
        # 7B-class attention prefill, grouped-query heads, feature reduction
        {"name": "attn_prefill", "kind": "attention", "B": 1, "Hq": 32, "Hkv": 8, "Lq": 4096, "Lk": 4096, "Dh": 128,
         "causal": True, "rho_d": 0.5, "rho_t": 1.0, "mask": False},
        # prefill with feature and token reduction at the paper's own ratios, odd length
        {"name": "attn_tokens", "kind": "attention", "B": 1, "Hq": 32, "Hkv": 32, "Lq": 3001, "Lk": 3001, "Dh": 128,
         "causal": True, "rho_d": 0.8, "rho_t": 0.8, "mask": False},
        # two padded sequences: the padding comes as an additive mask shared by the heads
        {"name": "attn_masked", "kind": "attention", "B": 2, "Hq": 16, "Hkv": 4, "Lq": 2048, "Lk": 2048, "Dh": 128,
         "causal": True, "rho_d": 0.5, "rho_t": 1.0, "mask": True},
        # one decode step of eight sequences against their caches
        {"name": "attn_decode", "kind": "attention", "B": 8, "Hq": 32, "Hkv": 8, "Lq": 1, "Lk": 4096, "Dh": 128,
         "causal": True, "rho_d": 0.5, "rho_t": 1.0, "mask": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mult(x, q):
    return max(q, x // q * q)


def draw(rng):
    kind = rng.choice(["product", "product", "decode", "fp32", "mlp_block", "product_q8", "prefill", "tokens", "masked",
                       "attn_decode"])
    rho = rng.choice([0.25, 0.5, 0.75, round(rng.uniform(0.2, 0.9), 3)])
    if kind == "product":
        # rows and contraction axis of any size (odd ones too), output columns in the multiples of 8 that weights have
        M, K, N = _log(rng, 64, 32768), _log(rng, 512, 28672), _mult(_log(rng, 256, 8192), 8)
        if rng.random() < 0.75:
            K = _mult(K, 8)
        return {"kind": "product", "M": M, "K": K, "N": N, "rho": rho, "dtype": "bf16"}
    if kind == "decode":
        M = rng.choice([1, 1, 2, 4, _log(rng, 5, 64)])
        return {"kind": "product", "M": M, "K": _mult(_log(rng, 1024, 28672), 64), "N": _mult(_log(rng, 1024, 28672), 64),
                "rho": rho, "dtype": "bf16"}
    if kind == "fp32":
        return {"kind": "product", "M": _log(rng, 32, 2048), "K": _log(rng, 256, 8192), "N": _log(rng, 64, 4096), "rho": rho,
                "dtype": "fp32"}
    if kind == "mlp_block":
        return {"kind": "mlp_block", "M": _log(rng, 300, 4096), "K": _mult(_log(rng, 1024, 8192), 64),
                "F": _mult(_log(rng, 2048, 28672), 64), "rho": rho}
    if kind == "product_q8":
        return {"kind": "product_q8", "M": _log(rng, 256, 16384), "K": _mult(_log(rng, 1024, 28672), 64),
                "N": _mult(_log(rng, 1024, 8192), 64), "rho": rho}
    Dh = rng.choice([64, 128, 128, 128, 256])
    Hkv = rng.choice([2, 4, 8])
    Hq = Hkv * rng.choice([1, 2, 4])
    rho_d = rng.choice([0.25, 0.5, 0.5, 0.8]) if Dh <= 128 else 0.5
    case = {"kind": "attention", "B": 1, "Hq": Hq, "Hkv": Hkv, "Lq": 0, "Lk": 0, "Dh": Dh, "causal": True, "rho_d": rho_d,
            "rho_t": 1.0, "mask": False}
    if kind == "attn_decode":
        case.update(B=_log(rng, 1, 16), Lq=rng.choice([1, 1, 1, 2, 4]), Lk=_log(rng, 512, 32768))
        return case
    L = _log(rng, 512, 8192)
    case.update(B=rng.choice([1, 1, 2]), Lq=L, Lk=L)
    if kind == "prefill":
        case["causal"] = rng.random() < 0.8
        if rng.random() < 0.25:  # a chunk of a longer prompt: earlier keys are in the cache
            case["Lk"] = L + _log(rng, 256, 4096)
    elif kind == "tokens":
        case["rho_t"] = rng.choice([0.25, 0.5, 0.8])
    else:
        L = min(L, 4096)
        if rng.random() < 0.75:  # masks are usually allocated with rows of whole vectors
            L = _mult(L, 4)
        case.update(Lq=L, Lk=L, mask=True, causal=rng.random() < 0.7)
    return case


def prepare(case, seed):
    kind, dev = case["kind"], "cuda"
    if kind == "product":
        dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
        A, B = synth.mlp_product(case["M"], case["K"], case["N"], seed=4 * seed, dtype=dt, device=dev)
        return {"kind": kind, "A": A, "B": B, "rho": case["rho"]}
    if kind == "mlp_block":
        # normalised hidden states; the up projection's output is the activation that the down projection contracts over
        X = synth.heavy_tailed_activations(case["M"], case["K"], 4 * seed, device=dev)
        return {"kind": kind, "X": X, "up": synth.weight(case["K"], case["F"], 4 * seed + 1, device=dev),
                "down": synth.weight(case["F"], case["K"], 4 * seed + 2, device=dev), "rho": case["rho"]}
    if kind == "product_q8":
        A = synth.heavy_tailed_activations(case["M"], case["K"], 4 * seed, device=dev)
        W = synth.weight(case["N"], case["K"], 4 * seed + 1, dtype=torch.float32, device=dev)
        step = float(W.abs().max()) / 448.0
        return {"kind": kind, "A": A, "Wq": (W / step).to(torch.float8_e4m3fn), "step": step, "rho": case["rho"]}
    Q, K, V = synth.attention_qkv(case["B"], case["Hq"], case["Hkv"], case["Lq"], case["Lk"], case["Dh"], seed=4 * seed,
                                  device=dev)
    mask = None
    if case["mask"]:
        # sequence b is padded on the right from its own length on
        mask = torch.zeros(case["B"], 1, case["Lq"], case["Lk"], dtype=torch.float32, device=dev)
        g = torch.Generator().manual_seed(4 * seed + 3)
        for b in range(case["B"]):
            n = int(torch.randint(case["Lk"] // 2, case["Lk"], (1,), generator=g))
            mask[b, :, :, n:] = float("-inf")
    return {"kind": kind, "Q": Q, "K": K, "V": V, "mask": mask, "causal": case["causal"], "rho_d": case["rho_d"],
            "rho_t": case["rho_t"]}


def run(state):
    kind = state["kind"]
    if kind == "product":
        return rmm.rmm(state["A"], state["B"], state["rho"])
    if kind == "mlp_block":
        H, energy = rmm.rmm_reduced_gemm(state["X"], state["up"], None, want_energy=True)
        idx = rmm.rmm_select(energy, rho=state["rho"])
        return rmm.rmm_reduced_gemm(H, state["down"], idx)
    if kind == "product_q8":
        idx = rmm.rmm_score_select(state["A"], rho=state["rho"])[0]
        return rmm.rmm_reduced_gemm_q8(state["A"], state["Wq"], state["step"], idx)
    return rmm.rmm_reduced_attn(state["Q"], state["K"], state["V"], state["causal"], state["rho_d"], state["rho_t"],
                                mask=state["mask"])


def work(case):
    kind = case["kind"]
    if kind == "product":
        M, K, N, e = case["M"], case["K"], case["N"], 2 if case["dtype"] == "bf16" else 4
        k = rmm.rmm_keep_count(case["rho"], K)
        return {"bytes": e * (M * K + k * N + M * N) + 4 * k, "flops": 2 * M * k * N}
    if kind == "mlp_block":
        # the intermediate activations are written by one call and read by another
        M, K, F = case["M"], case["K"], case["F"]
        k = rmm.rmm_keep_count(case["rho"], F)
        return {"bytes": 2 * (M * K + K * F + M * F + M * k + k * K + M * K), "flops": 2 * M * K * (F + k)}
    if kind == "product_q8":
        M, K, N = case["M"], case["K"], case["N"]
        k = rmm.rmm_keep_count(case["rho"], K)
        return {"bytes": 2 * M * K + k * N + 2 * M * N, "flops": 2 * M * k * N}
    B, Hq, Hkv, Lq, Lk, Dh = (case[x] for x in ("B", "Hq", "Hkv", "Lq", "Lk", "Dh"))
    kd = rmm.rmm_keep_count(case["rho_d"], Dh)
    pairs = Lq * Lk
    if case["causal"]:
        pairs = sum(max(0, min(Lk, i + 1 + Lk - Lq)) for i in range(Lq))
    nbytes = 2 * B * Dh * (2 * Hq * Lq + 2 * Hkv * Lk)
    if case["mask"]:
        nbytes += 4 * B * pairs
    return {"bytes": nbytes, "flops": 2 * B * Hq * pairs * (kd + case["rho_t"] * Dh)}


def tolerance(case):
    # about four times the distance seen from the same path evaluated in 64 bits on the same index sets
    if case["kind"] == "product":
        # bf16 outputs: 1.7e-3, which is the rounding of the result itself
        return {"rel": 7e-3} if case["dtype"] == "bf16" else {"rel": 2e-6}
    if case["kind"] == "product_q8":
        return {"rel": 1e-2}
    if case["kind"] == "attention":
        return {"rel": 8e-3}
    # The intermediate activations are rounded to bf16 and then ranked: a rounding that falls the other way moves single
    # indices across the threshold.  Taken in 64 bits up to that rounding, the block differs by 2.3e-2.
    return {"rel": 3e-2}


def _kept(energy, rho):
    """The ceil(rho K) indices of largest energy, equal energies to the lower index, ascending."""
    k = rmm.rmm_keep_count(rho, energy.numel())
    return torch.sort(energy, descending=True, stable=True).indices[:k].sort().values


def _exact_attention(st):
    Q, K, V, causal = st["Q"], st["K"], st["V"], st["causal"]
    B, Hq, Lq, Dh = Q.shape
    Hkv, Lk = K.shape[1], K.shape[2]
    hidden = torch.ones(Lq, Lk, dtype=torch.bool, device=Q.device).triu(1 + Lk - Lq) if causal else None
    O = torch.empty(B, Hq, Lq, Dh, dtype=torch.float64, device=Q.device)
    for b in range(B):
        for h in range(Hq):
            q, k, v = Q[b, h].double(), K[b, h // (Hq // Hkv)].double(), V[b, h // (Hq // Hkv)].double()
            idx = _kept(q.square().sum(0), st["rho_d"])
            S = q[:, idx] @ k[:, idx].T / math.sqrt(Dh)
            if st["mask"] is not None:
                S += st["mask"][b, 0].double()
            if causal:
                S.masked_fill_(hidden, float("-inf"))
            P = torch.softmax(S, -1)
            if st["rho_t"] < 1.0:
                # tokens are scored on the probabilities as they are stored
                t = _kept(P.to(torch.bfloat16).double().square().sum(0), st["rho_t"])
                P, v = P[:, t], v[t]
            O[b, h] = P @ v
    return O


def exact(case, seed):
    st, kind = prepare(case, seed), case["kind"]
    if kind == "attention":
        return _exact_attention(st)
    if kind == "mlp_block":
        # the intermediate activations are bf16 numbers: they are an output of the first call and an input of the next
        H = (st["X"].double() @ st["up"].double()).to(torch.bfloat16).double()
        idx = _kept(H.square().sum(0), st["rho"])
        return H[:, idx] @ st["down"].double()[idx]
    A = st["A"].double()
    idx = _kept(A.square().sum(0), st["rho"])
    if kind == "product_q8":
        return A[:, idx] @ (st["Wq"].double()[:, idx] * st["step"]).T
    return A[:, idx] @ st["B"][idx].double(), idx.to(torch.int32)
