"""What a user of this library has it do, as cases to be timed and compared.

Each case is one pass through the public entry points: a single masked linear (``spl_*`` calls), one
step of a decoder layer or stack (``MaskedLayer`` / ``MaskedStack``, replayed from the CUDA graphs their
own ``capture`` methods record, as a serving loop does), a refill of a correction bank, the mask alone,
or the Down projection in binary64.  Layers and stacks hold the six projections that the paper offloads
in binary32 (Q|K|V, O, Gate|Up; Sec. 5.5 keeps Down apart, because its noise needs binary64).

A pass recovers Y = X W^T from the masked product, so its exact value needs no noise; corrections
C = eta W^T and masked inputs X~ = X + eta are compared with the noise drawn again here in 64 bits.
"""

import math

import torch

from paper_2609_15039_gb300 import spl
from paper_2609_15039_gb300.layer import MaskedLayer, MaskedStack
from paper_2609_15039_gb300.workloads import LLAMA_3_2_3B, QWEN3_4B, WEIGHT_STD, ModelShape

MODELS = {"llama": LLAMA_3_2_3B, "qwen": QWEN3_4B}
DEV = "cuda"
CYCLE = 2   # bank cycle of the timed step (even: parity 0)
STEP_DRAWS = {"stacked": 2, "online": 3}  # draws of a layer's bank: the timed step is never the cycle's last


class Offloaded(ModelShape):
    """The projections of a model that run on the GPU in binary32: all but Down."""

    def projections(self):
        return [p for p in super().projections() if p[0] != "down"]


def offloaded(name):
    m = MODELS[name]
    return Offloaded(m.name, m.layers, m.d_model, m.d_ff, m.q_out, m.kv_out, m.vocab)


# ---------------------------------------------------------------------------------- the cases
def listed():
    return [
        # one small masked linear, the call's latency: 16 unit rows, 256 -> 512, Laplace, Delta = 2
        {"name": "linear_16x256x512", "kind": "linear", "M": 16, "K": 256, "N": 512, "norm": "unit", "delta": 2.0,
         "mech": "laplace", "eps": 1.0},
        # decode, one token: two layers, each call also computing the next cycle's correction row
        {"name": "decode_llama_1", "kind": "stacked", "model": "llama", "layers": 2, "M": 1, "mech": "laplace",
         "eps": 1.0},
        # decode of a few sequences with a bank of corrections
        {"name": "decode_qwen_4", "kind": "online", "model": "qwen", "M": 4, "mech": "gaussian", "eps": 1.0},
        # decode of a server batch (the paper's is 15 prompts, Sec. 6.1)
        {"name": "batch_qwen_15", "kind": "online", "model": "qwen", "M": 15, "mech": "gaussian", "eps": 1.0},
        # a short prompt, or a large decode batch, of no round size
        {"name": "batch_qwen_61", "kind": "online", "model": "qwen", "M": 61, "mech": "gaussian", "eps": 1.0},
        # prefill of 128 tokens through a layer, each product with the next cycle's 128 noise rows
        {"name": "prefill_llama_128", "kind": "stacked", "model": "llama", "layers": 1, "M": 128, "mech": "gaussian",
         "eps": 0.5},
        # prefill of 512 tokens, the same schedule (1024 rows a product)
        {"name": "prefill_llama_512", "kind": "stacked", "model": "llama", "layers": 1, "M": 512, "mech": "laplace",
         "eps": 1.0},
        # a long prefill against a bank computed earlier
        {"name": "prefill_qwen_2048", "kind": "online", "model": "qwen", "M": 2048, "mech": "gaussian", "eps": 1.0},
        # the offline side: the bank of one layer, 8 draws of 128 rows
        {"name": "refill_llama_8x128", "kind": "refill", "model": "llama", "draws": 8, "M": 128, "mech": "laplace",
         "eps": 1.0},
        # the LM head over a ragged batch of positions
        {"name": "lm_head_llama_509", "kind": "linear", "M": 509, "K": 3072, "N": 128256, "norm": "rms",
         "delta": 825.0, "mech": "gaussian", "eps": 1.0},
        # the mask alone on a large activation (a whole batch of long prompts)
        {"name": "mask_1e8", "kind": "mask", "M": 32768, "K": 3072, "delta": 825.0, "mech": "gaussian", "eps": 1.0},
        # the Down projection in binary64 (Sec. 5.5) for a prompt of 128 tokens
        {"name": "down64_llama_128", "kind": "down64", "model": "llama", "M": 128, "mech": "gaussian", "eps": 1.0},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["linear", "linear", "stacked", "stacked", "online", "online", "online", "refill", "mask",
                       "down64"])
    case = {"kind": kind, "mech": rng.choice(["laplace", "gaussian"]),
            "eps": round(math.exp(rng.uniform(math.log(0.1), math.log(10.0))), 3)}
    if kind == "linear":
        K = 4 * _log_int(rng, 16, 2432)  # 64 .. 9728; odd multiples of 4 run without the fp16 split
        M, N = _log_int(rng, 1, 2048), _log_int(rng, 64, 32768)
        N = max(1, min(N, int(1.5e11 / (M * K))))
        case.update(M=M, K=K, N=N, norm="rms", delta=round(2.0 * K ** 0.75, 1))
    elif kind == "mask":
        K = 4 * _log_int(rng, 16, 2432)
        case.update(M=max(1, _log_int(rng, 10 ** 4, 10 ** 8) // K), K=K, delta=round(2.0 * K ** 0.75, 1))
    elif kind == "down64":
        case.update(model=rng.choice(list(MODELS)), M=_log_int(rng, 1, 128))
    elif kind == "refill":
        case.update(model=rng.choice(list(MODELS)), draws=rng.choice([2, 4, 8]), M=_log_int(rng, 1, 256))
    elif kind == "stacked":
        M = _log_int(rng, 1, 1024)
        case.update(model=rng.choice(list(MODELS)), layers=rng.choice([1, 2]) if M <= 512 else 1,
                    M=M if M <= 4 else (M + 3) // 4 * 4)
    else:
        case.update(model=rng.choice(list(MODELS)), M=_log_int(rng, 1, 2048))
    return case


# ---------------------------------------------------------------------------------- inputs
def _randn(shape, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.float32)


def _weight(N, K, seed):
    return _randn((N, K), seed).mul_(WEIGHT_STD)


def _rows(M, K, seed, norm="rms"):
    x = _randn((M, K), seed)
    n = torch.linalg.vector_norm(x.double(), dim=1, keepdim=True)
    s = math.sqrt(K) / n if norm == "rms" else torch.clamp(1.0 / n, max=1.0)
    return (x.double() * s).float().contiguous()


def _shapes(case):
    """(name, K, [(projection, N)]) of each input group of an offloaded layer."""
    m = offloaded(case["model"])
    width = {p: n for p, _k, n, _g in m.projections()}
    return [(g, K, [(p, width[p]) for p in names]) for g, K, names in m.input_groups()]


def _seeds(seed, layer, i):
    return (seed * 1_000_003 + layer * 101 + i) % 2 ** 62


def _layer_weights(case, seed, li):
    return {p: _weight(n, K, _seeds(seed, li, 10 * gi + pi))
            for gi, (_g, K, ps) in enumerate(_shapes(case)) for pi, (p, n) in enumerate(ps)}


def _layer_inputs(case, seed, li):
    return {g: _rows(case["M"], K, _seeds(seed, li, 50 + gi)) for gi, (g, K, _p) in enumerate(_shapes(case))}


def _norm_bound(n, k):
    """Largest singular value of an n x k matrix of N(0, WEIGHT_STD^2) entries (its edge for large n, k)."""
    return WEIGHT_STD * (math.sqrt(n) + math.sqrt(k))


def _deltas(case):
    """Global sensitivities of a layer's inputs for unit norm weights (Thms. 1 and 2)."""
    m = MODELS[case["model"]]
    ln = 2.0 * m.d_model ** 0.75
    return {"qkv": ln, "gateup": ln, "o": ln * _norm_bound(m.kv_out, m.d_model)}


def _delta_down(case):
    """Thm. 3 for the input of Down."""
    m = MODELS[case["model"]]
    return 2.0 * math.sqrt(m.d_ff) * m.d_model ** 1.5 * _norm_bound(m.d_ff, m.d_model) ** 2


def _noise_args(case, seed):
    return case["delta"], case["eps"], case["mech"], seed


# ---------------------------------------------------------------------------------- prepare
def prepare(case, seed):
    return {"linear": _prepare_linear, "stacked": _prepare_stacked, "online": _prepare_online,
            "refill": _prepare_refill, "mask": _prepare_mask, "down64": _prepare_down64}[case["kind"]](case, seed)


def _prepare_linear(case, seed):
    M, K, N = case["M"], case["K"], case["N"]
    W = spl.Weight.prepare(_weight(N, K, _seeds(seed, 0, 1)))
    ws = spl.workspace(max(spl.spl_linear_workspace_bytes(M, K, N),
                           spl.spl_precompute_matched_workspace_bytes(M, K, N, M)), DEV)
    eta, C = torch.empty((M, K), device=DEV), torch.empty((M, N), device=DEV)
    spl.spl_noise(eta, *_noise_args(case, seed))
    spl.spl_precompute_noise_product_matched(C, eta, W, M, workspace=ws)
    return {"case": case, "seed": seed, "X": _rows(M, K, _seeds(seed, 0, 2), case["norm"]), "W": W, "C": C, "ws": ws,
            "Y": torch.empty((M, N), device=DEV), "Xt": eta}


def _prepare_layer(case, seed, li):
    layer = MaskedLayer.from_weights(offloaded(case["model"]), _layer_weights(case, seed, li), device=DEV)
    layer.deltas = _deltas(case)
    return layer


def _prepare_stacked(case, seed):
    M, D = case["M"], STEP_DRAWS["stacked"]
    layers = [_prepare_layer(case, seed, li) for li in range(case["layers"])]
    for layer in layers:
        layer.allocate_stacked(M, D)
    stack = MaskedStack(layers, [_seeds(seed, li, 99) for li in range(len(layers))])
    inputs = [_layer_inputs(case, seed, li) for li in range(len(layers))]
    for layer, x, s in zip(layers, inputs, stack.seeds):  # every call once before the capture
        layer.stacked_step(x, case["eps"], case["mech"], s, 0, 0)
    graphs, _ = stack.capture_stacked(inputs, case["eps"], case["mech"])
    stack.start_stacked(CYCLE, graphs)
    return {"case": case, "stack": stack, "inputs": inputs, "graphs": graphs}


def _prepare_online(case, seed):
    M, D = case["M"], STEP_DRAWS["online"]
    layer, x = _prepare_layer(case, seed, 0), _layer_inputs(case, seed, 0)
    layer.allocate(M, D)
    args = (case["eps"], case["mech"], seed)
    layer.refill(*args, CYCLE)
    out = layer.online(x, *args, CYCLE, 0)
    layer.set_cycle(CYCLE)
    graphs, _ = layer.capture(x, *args)
    graphs[0].replay()  # the bank of the cycle, and its first step
    return {"case": case, "layer": layer, "inputs": x, "graphs": graphs, "out": out}


def _prepare_refill(case, seed):
    layer = _prepare_layer(case, seed, 0)
    layer.allocate(case["M"], case["draws"])
    return {"case": case, "layer": layer, "seed": seed}


def _prepare_mask(case, seed):
    X = _rows(case["M"], case["K"], _seeds(seed, 0, 2))
    return {"case": case, "seed": seed, "X": X, "Xt": torch.empty_like(X)}


def _prepare_down64(case, seed):
    m = MODELS[case["model"]]
    M, K, N = case["M"], m.d_ff, m.d_model
    W = _weight(N, K, _seeds(seed, 0, 1))
    ws = spl.workspace(spl.spl_f64_workspace_bytes(M, K, N), DEV)
    eta, C = torch.empty((M, K), device=DEV), torch.empty((M, N), device=DEV, dtype=torch.float64)
    spl.spl_noise(eta, _delta_down(case), case["eps"], case["mech"], seed)
    spl.spl_precompute_noise_product_f64(C, eta, W, workspace=ws)
    return {"case": case, "seed": seed, "X": _rows(M, K, _seeds(seed, 0, 2)), "W": W, "C": C, "ws": ws,
            "Y": torch.empty((M, N), device=DEV), "Xt": torch.empty((M, K), device=DEV, dtype=torch.float64)}


# ---------------------------------------------------------------------------------- run
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "linear":  # noise, mask, product, unmask
        spl.spl_noise_mask_linear_unmask(s["Y"], s["Xt"], s["X"], s["W"], s["C"], *_noise_args(case, s["seed"]),
                                         workspace=s["ws"])
        return {"Y": s["Y"], "Xt": s["Xt"]}
    if kind == "stacked":  # step 0 of an even cycle: Y of the step and the next cycle's corrections
        stack, M = s["stack"], case["M"]
        stack.replay_stacked(s["graphs"], CYCLE * stack.draws)
        return {"Y": stack.step_outputs(0, 0),
                "C": [{g.name: l.stacked[g.name]["out"][1][0][M:] for g in l.groups} for l in stack.layers]}
    if kind == "online":
        s["graphs"][1].replay()
        return {"Y": s["out"]}
    if kind == "refill":
        layer = s["layer"]
        layer.refill(case["eps"], case["mech"], s["seed"], CYCLE, parallel=True)
        return {"C": {g.name: layer.bank[g.name]["C"] for g in layer.groups}}
    if kind == "mask":
        spl.spl_noise_mask(s["Xt"], None, s["X"], *_noise_args(case, s["seed"]))
        return {"Xt": s["Xt"]}
    spl.spl_noise_mask_f64(s["Xt"], s["X"], _delta_down(case), case["eps"], case["mech"], s["seed"])
    spl.spl_masked_linear_unmask_f64(s["Y"], s["Xt"], s["W"], s["C"], workspace=s["ws"])
    return {"Y": s["Y"], "Xt": s["Xt"]}


# ---------------------------------------------------------------------------------- work
def work(case):
    """Bytes and flops of one pass: the fp32 weight, the input and the correction read once, the results
    written once; the products of the path at 2 flops a term (the splits' extra products are not counted)."""
    kind, M = case["kind"], case["M"]
    if kind == "mask":
        return {"bytes": 8 * M * case["K"], "flops": 0}
    if kind == "linear":
        K, N = case["K"], case["N"]
        return {"bytes": 4 * (N * K + 2 * M * K + 2 * M * N), "flops": 2 * M * K * N}
    if kind == "down64":
        m = MODELS[case["model"]]
        K, N = m.d_ff, m.d_model
        return {"bytes": 4 * N * K + 12 * M * K + 12 * M * N, "flops": 2 * M * K * N}
    b = f = 0
    for _g, K, ps in _shapes(case):
        N = sum(n for _p, n in ps)
        if kind == "stacked":  # X and C in, Y and the next C out; 2M rows multiplied
            b += 4 * (N * K + M * K + 3 * M * N)
            f += 4 * M * K * N
        elif kind == "online":
            b += 4 * (N * K + M * K + 2 * M * N)
            f += 2 * M * K * N
        else:
            rows = case["draws"] * M
            b += 4 * (N * K + rows * N)
            f += 2 * rows * K * N
    n = case.get("layers", 1)
    return {"bytes": n * b, "flops": n * f}


# ---------------------------------------------------------------------------------- exact values
def _philox(count, offset, seed, stream_id):
    """Words 0-3 of Philox4x32-10 blocks offset .. offset + count - 1 (Salmon et al., SC'11), as int64."""
    mask = 0xFFFFFFFF
    j = torch.arange(count, device=DEV, dtype=torch.int64) + offset
    c = [j & mask, (j >> 32) & mask, torch.full_like(j, stream_id & mask), torch.full_like(j, (stream_id >> 32) & mask)]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # low 64 bits: all that is needed
        c = [((p1 >> 32) & mask) ^ c[1] ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _noise(rows, cols, delta, eps, mech, seed, stream_id=0, offset=0):
    """eta [rows, cols] in 64 bits at scale fl32(delta / eps): the transforms that include/spl.h states."""
    n = rows * cols
    b = float(torch.tensor(delta / eps, dtype=torch.float32))
    w = _philox((n + 3) // 4, offset, seed % 2 ** 64, stream_id)
    if mech == "laplace":
        v = [torch.log(((x & 0xFFFFFF) + 1).double() * 2.0 ** -24) * torch.where(x >> 31 != 0, b, -b).double()
             for x in w]
    else:
        v = []
        for a, c in ((w[0], w[1]), (w[2], w[3])):
            r = b * torch.sqrt(-2.0 * torch.log(((a >> 8) + 1).double() * 2.0 ** -24))
            t = 2.0 * math.pi * ((c >> 8).double() * 2.0 ** -24)
            v += [r * torch.cos(t), r * torch.sin(t)]
    return torch.stack(v, dim=1).reshape(-1)[:n].reshape(rows, cols)


def _product(A, W):
    """A W^T in 64 bits, W in blocks of rows so that its 64-bit copy stays small."""
    step = max(1, 2 ** 27 // W.shape[1])
    return torch.cat([A.double() @ W[i:i + step].double().T for i in range(0, W.shape[0], step)], dim=1)


def exact(case, seed):
    kind, M = case["kind"], case["M"]
    if kind in ("linear", "down64"):
        m = MODELS.get(case.get("model"))
        K, N = (case["K"], case["N"]) if kind == "linear" else (m.d_ff, m.d_model)
        X, W = _rows(M, K, _seeds(seed, 0, 2), case.get("norm", "rms")), _weight(N, K, _seeds(seed, 0, 1))
        delta = case["delta"] if kind == "linear" else _delta_down(case)
        return {"Y": _product(X, W), "Xt": X.double() + _noise(M, K, delta, case["eps"], case["mech"], seed)}
    if kind == "mask":
        X = _rows(M, case["K"], _seeds(seed, 0, 2))
        return {"Xt": X.double() + _noise(M, case["K"], *_noise_args(case, seed))}
    deltas = _deltas(case)

    def group_weights(li):
        weights = _layer_weights(case, seed, li)
        return {g: torch.cat([weights[p] for p, _n in ps]) for g, _K, ps in _shapes(case)}

    def recovered(li):
        W, x = group_weights(li), _layer_inputs(case, seed, li)
        return {g: _product(x[g], W[g]) for g in W}

    def corrections(li, rows, noise_seed, blocks_of):
        W = group_weights(li)
        return {g: _product(_noise(rows, K, deltas[g], case["eps"], case["mech"], noise_seed, gi, blocks_of(K)), W[g])
                for gi, (g, K, _p) in enumerate(_shapes(case))}

    if kind == "online":
        return {"Y": recovered(0)}
    if kind == "refill":
        D = case["draws"]
        return {"C": corrections(0, D * M, seed, lambda K: CYCLE * D * (M * K // 4))}
    D, layers = STEP_DRAWS["stacked"], range(case["layers"])
    return {"Y": [recovered(li) for li in layers],
            "C": [corrections(li, M, _seeds(seed, li, 99), lambda K: (CYCLE + 1) * D * (M * K // 4))
                  for li in layers]}


# ---------------------------------------------------------------------------------- tolerance
def tolerance(case):
    """Largest relative error of a pass.  The recovered Y = fl(x~ W^T) - C keeps the rounding of sums that
    are noise / input times larger than it: a few 2^-24 of that ratio, more with longer accumulation chains
    (coefficient: four times the 1.1e-3 measured at 2048 x 4096 by 2560, eps = 1).  Corrections are good to
    3e-6, masked inputs to 6e-8, the binary64 path to 9e-8 (its result is binary32)."""
    kind = case["kind"]
    if kind in ("refill", "mask", "down64"):
        return {"rel": {"refill": 1.3e-5, "mask": 3e-7, "down64": 4e-7}[kind]}
    K = case["K"] if kind == "linear" else min(K for _g, K, _p in _shapes(case))
    delta = case["delta"] if kind == "linear" else max(_deltas(case).values())
    rms = 1.0 / math.sqrt(K) if case.get("norm") == "unit" else 1.0
    rel = 1e-5 + 50.0 * math.sqrt(min(1.0, K / 1024)) * 2.0 ** -24 * delta / case["eps"] / rms
    return {"rel": min(0.03, rel), "max": min(1.0 - 2.0 ** -10, 100.0 * rel)}
