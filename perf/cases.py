"""The work that a program using libdamp has it do, as measurable cases.

A case is one call of the binding: a decode step of one layer on the packed state (the six
low tiers, GDN and KDA, with and without slot indirection), the same step of a layer stored
as two head groups, the FP32-state step, a prefill or multi-token chunk, a calibration run,
and the hand-off between FP32 states and the packed cache.

    op        call                                       sizes
    decode    {gdn,kda}_decode_step                      B request slots
    groups    {gdn,kda}_decode_step_groups               B request slots, two K_hi
    fp32      fp32_{gdn,kda}_decode_step                 B request slots
    chunk     {gdn,kda}_prefill_chunk                    B request slots, T tokens each
    calib     calib_accumulate, calib_select             B documents, T tokens each
    store     quantize_state                             B request slots
    load      dequantize_state                           B request slots

Operands follow the recipe of workloads.py: unit q and k, normal v, sigmoid beta, softplus
gates (GDN) or a fixed per-channel decay profile (KDA).  The initial states are normal with
the variance that the recurrence has on each channel, and are packed from tiers that plain
torch computes, so that the 64-bit results start from the same stored values.
"""
import math

import torch

import paper_2608_27513_gb300 as damp

DEFAULTS = {"op": "decode", "kind": "kda", "B": 1, "T": 1, "H": 32, "Hqk": 32, "dk": 128, "dv": 128, "K": 16, "K2": 0,
            "fmt": 0, "bf16": True, "slots": False, "ragged": False}
U8, U4 = (0, 1), (3, 4)
HADAMARD = (0, 3)  # low tiers stored in the H_32 domain


def listed():
    return [
        # one user decoding: one step of one KDA layer at the paper's operating point, pure latency
        {"name": "decode_kda_b1", **DEFAULTS, "B": 1, "K": 16},
        # a moderate serving batch of a GDN layer with grouped q/k heads; slots are handed out by the engine
        {"name": "decode_gdn_b64_gqa", **DEFAULTS, "kind": "gdn", "B": 64, "Hqk": 16, "K": 8, "slots": True},
        # the full serving batch of the paper's KDA layer
        {"name": "decode_kda_b256", **DEFAULTS, "B": 256, "K": 10},
        # an odd batch on the four-bit tier
        {"name": "decode_gdn_u4_b100", **DEFAULTS, "kind": "gdn", "B": 100, "K": 16, "fmt": 3},
        # a GDN layer whose fast- and slow-decay heads keep different channel budgets
        {"name": "decode_groups_gdn_b256", **DEFAULTS, "op": "groups", "kind": "gdn", "B": 256, "K": 12, "K2": 20},
        # the FP32-state deployment that the packed state replaces
        {"name": "decode_fp32_gdn_b64", **DEFAULTS, "op": "fp32", "kind": "gdn", "B": 64},
        # speculative decoding: four tokens of every request slot verified in one launch
        {"name": "steps4_kda_b256", **DEFAULTS, "op": "chunk", "B": 256, "T": 4, "K": 10},
        # chunked prefill of a full batch
        {"name": "prefill_kda_b256_t64", **DEFAULTS, "op": "chunk", "B": 256, "T": 64, "K": 10},
        # a few prompts of different lengths prefilled together
        {"name": "prefill_gdn_b8_ragged", **DEFAULTS, "op": "chunk", "kind": "gdn", "B": 8, "T": 500, "Hqk": 16,
         "K": 16, "slots": True, "ragged": True},
        # one long prompt
        {"name": "prefill_kda_b1_t2048", **DEFAULTS, "op": "chunk", "B": 1, "T": 2048, "K": 16},
        # the calibration protocol of one layer: 32 documents of 256 tokens, every eighth state sampled
        {"name": "calibrate_kda_32x256", **DEFAULTS, "op": "calib", "B": 32, "T": 256, "K": 16},
        # FP32 prefix states written into the packed cache
        {"name": "store_gdn_b64", **DEFAULTS, "op": "store", "kind": "gdn", "B": 64, "K": 16},
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(("decode", "decode", "decode", "chunk", "chunk", "chunk", "groups", "fp32", "calib", "store", "load"))
    c = dict(DEFAULTS, op=op, kind=rng.choice(("gdn", "kda")))
    c["H"] = rng.choice((32, 32, 32, 16, 12))
    c["Hqk"] = rng.choice((c["H"], c["H"] // 2))
    c["B"] = _log(rng, 1, 256)
    c["K"] = rng.choice((0, 4, 8, 10, 16, 16, 32, rng.randint(1, 48)))
    c["slots"] = rng.random() < 0.4
    if op != "groups" and rng.random() < 0.15:
        c["dk"] = c["dv"] = 64
        c["K"] = min(c["K"], 32)
    if op in ("decode", "chunk", "store", "load", "calib"):
        c["fmt"] = rng.choice((0, 0, 0, 0, 1, 2, 3, 4, 5))
    if op in ("decode", "chunk", "fp32", "calib"):
        c["bf16"] = rng.random() < 0.85
    if op == "groups":
        c["fmt"] = rng.choice((0, 0, 1))
        c["K"], c["K2"] = rng.choice(((12, 20), (8, 24), (4, 28)))
    elif op == "chunk":
        c["T"] = _log(rng, 2, 1024)
        c["B"] = max(1, min(c["B"], 16384 // c["T"]))
        c["ragged"] = rng.random() < 0.4
    elif op == "calib":
        c["B"], c["T"], c["slots"] = _log(rng, 4, 32), _log(rng, 16, 256), False
    return c


# ---- inputs ----

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _generator(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(1_000_003 * int(seed) + 17)
    return g


def _operands(case, gen, lead):
    """q, k, v, g, beta of the leading shape `lead` ([B] or [B, T]; calibration [T, B])."""
    H, Hqk, dk, dv = case["H"], case["Hqk"], case["dk"], case["dv"]

    def n(*shape):
        return torch.randn(*shape, generator=gen, device=_device())

    q, k, v = n(*lead, Hqk, dk), n(*lead, Hqk, dk), n(*lead, H, dv)
    q /= q.norm(dim=-1, keepdim=True)
    k /= k.norm(dim=-1, keepdim=True)
    beta = torch.sigmoid(n(*lead, H))
    if case["kind"] == "gdn":
        g = -torch.nn.functional.softplus(n(*lead, H))
    else:
        g = -torch.exp(_profile(case))[(None,) * len(lead)] * (1.0 + 0.05 * n(*lead, H, dk))
    if case["bf16"]:
        q, k, v = q.bfloat16(), k.bfloat16(), v.bfloat16()
    return {"q": q, "k": k, "v": v, "g": g.contiguous(), "beta": beta}


def _profile(case):
    """The layer's log-log decay per channel [H, d_k], uniform in (-6, 0): a property of its weights."""
    gen = torch.Generator(device=_device())
    gen.manual_seed(4)
    return torch.rand(case["H"], case["dk"], generator=gen, device=_device()) * 6.0 - 6.0


def _states(case, gen, n):
    """n FP32 states [n, H, d_k, d_v] with the variance the recurrence gives each key channel."""
    S = torch.randn(n, case["H"], case["dk"], case["dv"], generator=gen, device=_device())
    a2 = torch.exp(-2.0 * torch.exp(_profile(case))) if case["kind"] == "kda" else torch.full(
        (case["H"], case["dk"]), 0.3, device=_device())
    return S * torch.sqrt(0.3 / case["dk"] / (1.0 - a2))[None, :, :, None]


def _lengths(case, seed):
    """Ragged lengths of a chunk: between an eighth of the chunk and all of it, the longest first."""
    g = torch.Generator()
    g.manual_seed(int(seed) + 91)
    n = (torch.rand(case["B"], generator=g) * 0.875 + 0.125) * case["T"]
    n = n.round().clamp(1, case["T"]).to(torch.int32)
    n[0] = case["T"]
    return n


def _slots(case, seed):
    """(slots in the pool, the slot of each batch row)."""
    if not case["slots"]:
        return case["B"], torch.arange(case["B"])
    g = torch.Generator()
    g.manual_seed(int(seed) + 57)
    n = case["B"] + case["B"] // 2 + 1
    return n, torch.randperm(n, generator=g)[:case["B"]]


def _perm(case, gen):
    return torch.argsort(torch.rand(case["H"], case["dk"], generator=gen, device=_device()), dim=1).to(torch.uint8)


def _groups(case):
    """[(K_hi, model heads)] of the layer: one group, or alternating heads in two."""
    H = case["H"]
    if case["op"] != "groups":
        return [(case["K"], list(range(H)))]
    return [(case["K"], list(range(0, H, 2))), (case["K2"], list(range(1, H, 2)))]


def _h32(dtype):
    i = torch.arange(32, device=_device())
    bits = (i[:, None] & i[None, :])
    parity = sum((bits >> b) & 1 for b in range(5)) & 1
    return ((1 - 2 * parity).to(dtype) / math.sqrt(32.0)).contiguous()


def _quantized(x, fmt):
    """Rows x [..., d_v] in blocks of 32 -> (codes as numbers, s, z) of a low tier, in x's precision."""
    y = x.reshape(*x.shape[:-1], -1, 32)
    if fmt in HADAMARD:
        y = y @ _h32(x.dtype)
    if fmt == 2:
        s = (y.abs().amax((-1, -2), keepdim=True) / 127.0)
        return torch.round(y / torch.where(s == 0, torch.ones_like(s), s)).clamp(-127, 127), s, torch.zeros_like(s)
    if fmt == 5:
        s = y.abs().amax(-1, keepdim=True).clamp(min=1e-10) / 448.0
        return (y / s).clamp(-448, 448).to(torch.float8_e4m3fn).to(x.dtype), s, torch.zeros_like(s)
    top = 15.0 if fmt in U4 else 255.0
    lo, hi = y.amin(-1, keepdim=True), y.amax(-1, keepdim=True)
    s = ((hi - lo) / top).half().to(x.dtype)
    z = torch.round(-lo / s).half().to(x.dtype)
    return (torch.round(y / s) + z).clamp(0, top), s, z


def _tiers(x, perm, K, fmt):
    """The logical tiers of states x [n, H, d_k, d_v] in calibrated order: hi, codes, meta as
    pack_tiers takes them, and the values that they stand for, in 64 bits and natural order."""
    n, H, dk, dv = x.shape
    order = perm.long()[None, :, :, None].expand(n, H, dk, dv)
    rows = torch.gather(x, 2, order)
    hi = rows[:, :, :K].half()
    code, s, z = _quantized(rows[:, :, K:], fmt)
    low = ((code.double() - z.double()) * s.double())
    if fmt in HADAMARD:
        low = low @ _h32(torch.float64)
    packed = torch.cat([hi.double(), low.reshape(n, H, dk - K, dv)], 2)
    values = torch.empty_like(packed).scatter_(2, order, packed)
    if fmt == 2:
        meta = s.reshape(n, H, dk - K).float()
        codes = code.reshape(n, H, dk - K, dv).to(torch.int8)
    elif fmt == 5:
        meta = s.reshape(n, H, dk - K, dv // 32).float()
        codes = code.reshape(n, H, dk - K, dv).to(torch.float8_e4m3fn).view(torch.uint8)
    else:
        meta = torch.cat([s, z], -1).half()
        codes = code.reshape(n, H, dk - K, dv).to(torch.uint8)
        if fmt in U4:
            codes = codes[..., 0::2] | (codes[..., 1::2] << 4)
    return (hi.contiguous(), codes.contiguous(), meta.contiguous()), values


def _drawn(case, seed):
    """Everything that both prepare and exact start from."""
    gen = _generator(seed)
    perm = _perm(case, gen)
    if case["op"] == "calib":
        return {"in": _operands(case, gen, (case["T"], case["B"]))}
    S = _states(case, gen, case["B"])
    if case["op"] in ("store", "load"):
        return {"perm": perm, "S": S}
    lead = (case["B"], case["T"]) if case["op"] == "chunk" else (case["B"],)
    return {"perm": perm, "S": S, "in": _operands(case, gen, lead)}


def _layouts(case):
    if case["op"] == "groups":
        of_head = [0] * case["H"]
        for K, heads in _groups(case):
            for h in heads:
                of_head[h] = K
        return [(lay, heads) for lay, heads in damp.head_groups(of_head, case["Hqk"], case["dk"], case["dv"], case["fmt"])]
    return [(damp.Layout(case["H"], case["Hqk"], case["dk"], case["dv"], case["K"], case["fmt"]), list(range(case["H"])))]


def prepare(case, seed):
    d = _drawn(case, seed)
    st = {"case": case, "in": d.get("in")}
    if case["op"] == "calib":
        st["layout"] = _layouts(case)[0][0]
        return st
    n, slots = _slots(case, seed)
    st["slot_idx"] = slots.to(torch.int32).cuda() if case["slots"] else None
    if case["op"] == "chunk":
        st["lengths"] = _lengths(case, seed).cuda() if case["ragged"] else None
    if case["op"] == "fp32":
        st["layout"] = _layouts(case)[0][0]
        st["state"] = damp.new_fp32_state(st["layout"], n)
        st["state"][slots.cuda()] = d["S"]
        return st
    st["groups"] = []
    for lay, heads in _layouts(case):
        perm = d["perm"][heads].contiguous()
        pool = damp.new_state(lay, n)
        if case["op"] != "store":
            for at in range(0, case["B"], 64):  # 64 slots at a time: the working copies stay small
                tiers, _ = _tiers(d["S"][at:at + 64, heads], perm, lay.k_hi, case["fmt"])
                rows = slots[at:at + 64].to(torch.int32).cuda()
                damp.pack_tiers(lay, *tiers, pool, slot_idx=rows)
        st["groups"].append((lay, pool, perm))
    if case["op"] == "store":
        st["S"] = d["S"]
    return st


def run(st):
    case, x = st["case"], st["in"]
    op, kda = case["op"], case["kind"] == "kda"
    if op == "calib":
        lay = st["layout"]
        S = damp.new_fp32_state(lay, case["B"])
        E = torch.zeros(lay.num_heads, lay.d_k, device=S.device)
        G = torch.zeros_like(E)
        samples, tokens = damp.calib_accumulate(lay, case["kind"], S, x["q"], x["k"], x["v"], x["g"], x["beta"], E, G, every=8)
        C, perm = damp.calib_select(lay, E, samples, G, tokens)
        return {"state": S, "energy": E, "log_decay": G, "scores": C, "perm": perm}
    idx = st["slot_idx"]
    if op == "fp32":
        step = damp.fp32_kda_decode_step if kda else damp.fp32_gdn_decode_step
        o = step(st["layout"], st["state"], x["q"], x["k"], x["v"], x["g"], x["beta"], slot_idx=idx)
        return {"o": o, "state": st["state"]}
    if op == "groups":
        step = damp.kda_decode_step_groups if kda else damp.gdn_decode_step_groups
        o = step(st["groups"], x["q"], x["k"], x["v"], x["g"], x["beta"], slot_idx=idx)
        return {"o": o, "state": [pool for _, pool, _ in st["groups"]]}
    lay, pool, perm = st["groups"][0]
    if op == "store":
        damp.quantize_state(lay, st["S"], perm, pool, slot_idx=idx)
        return {"state": pool}
    if op == "load":
        return {"S": damp.dequantize_state(lay, pool, perm, batch=case["B"], slot_idx=idx)}
    if op == "chunk":
        chunk = damp.kda_prefill_chunk if kda else damp.gdn_prefill_chunk
        o = chunk(lay, pool, perm, x["q"], x["k"], x["v"], x["g"], x["beta"], lengths=st["lengths"], slot_idx=idx)
    else:
        step = damp.kda_decode_step if kda else damp.gdn_decode_step
        o = step(lay, pool, perm, x["q"], x["k"], x["v"], x["g"], x["beta"], slot_idx=idx)
    return {"o": o, "state": pool}


def _tokens(case):
    """Tokens that a chunk runs, on average over the seeds."""
    if not case["ragged"]:
        return case["B"] * case["T"]
    return int((case["B"] - 1) * case["T"] * 0.5625) + case["T"]


def work(case):
    B, T, H, Hqk, dk, dv, op = (case[n] for n in ("B", "T", "H", "Hqk", "dk", "dv", "op"))
    esz, fmt = (2 if case["bf16"] else 4), case["fmt"]
    gate = 4 * (dk if case["kind"] == "kda" else 1) + 4
    per_token = 2 * Hqk * dk * esz + H * (dv * esz + gate + 4 * dv)  # q, k, v, gates read, o written
    meta = 4 if fmt == 2 else 4 * (dv // 32)
    row = dv // 2 if fmt in U4 else dv
    packed = sum(len(heads) * (2 * K * dv + (dk - K) * (row + meta)) for K, heads in _groups(case))
    full = 4 * H * dk * dv
    step = 7 * H * dk * dv  # decay, read, correction and output of one token
    if op == "calib":  # the trajectories need no o: the inputs once, the final states, sums, scores and pi
        return {"bytes": T * B * (per_token - 4 * H * dv) + B * full + 13 * H * dk,
                "flops": T * B * 5 * H * dk * dv + B * (T // 8) * 10 * H * dk * dv}
    if op in ("store", "load"):
        return {"bytes": B * (full + packed), "flops": B * 6 * H * dk * dv}
    if op == "fp32":
        return {"bytes": B * (2 * full + per_token), "flops": B * step}
    tokens = _tokens(case) if op == "chunk" else B
    return {"bytes": B * 2 * packed + tokens * per_token, "flops": tokens * step}


# ---- the same results in 64 bits ----

def _advance(S, q, k, v, g, beta, group):
    """One token of the recurrence on S [B, H, d_k, d_v] (64 bits, in place); returns o."""
    q, k = (t.repeat_interleave(group, dim=1) for t in (q, k))
    S *= torch.exp(g)[..., None] if g.dim() == 3 else torch.exp(g)[..., None, None]
    d = (v - torch.einsum("bhkv,bhk->bhv", S, k)) * beta[..., None]
    S += k[..., :, None] * d[..., None, :]
    return torch.einsum("bhkv,bhk->bhv", S, q)


def exact(case, seed):
    d = _drawn(case, seed)
    group = case["H"] // case["Hqk"]
    x = {n: t.double() for n, t in d["in"].items()} if "in" in d else None
    if case["op"] == "calib":
        return _exact_calibration(case, x, group)
    n, slots = _slots(case, seed)
    if case["op"] == "store":
        return None  # whole bytes
    S = torch.empty(d["S"].shape, dtype=torch.float64, device=d["S"].device)
    if case["op"] == "fp32":
        S.copy_(d["S"])
    else:
        for K, heads in _groups(case):
            for at in range(0, case["B"], 64):
                S[at:at + 64, heads] = _tiers(d["S"][at:at + 64, heads], d["perm"][heads], K, case["fmt"])[1]
    if case["op"] == "load":
        return {"S": S}
    if case["op"] != "chunk":
        o = _advance(S, x["q"], x["k"], x["v"], x["g"], x["beta"], group)
        if case["op"] == "fp32":
            pool = torch.zeros(n, *S.shape[1:], dtype=torch.float64, device=S.device)
            pool[slots.to(S.device)] = S
            return {"o": o, "state": pool}
        return {"o": o, "state": [None] * len(_groups(case)) if case["op"] == "groups" else None}
    o = torch.zeros(case["B"], case["T"], case["H"], case["dv"], dtype=torch.float64, device=S.device)
    left = _lengths(case, seed).to(S.device) if case["ragged"] else None
    for t in range(case["T"]):
        o[:, t] = _advance(S, *(x[m][:, t] for m in ("q", "k", "v", "g", "beta")), group)
    if left is not None:  # rows past a prompt's end stay zero
        o[torch.arange(case["T"], device=S.device)[None] >= left[:, None]] = 0.0
    return {"o": o, "state": None}


def _exact_calibration(case, x, group):
    B, T, H, dk, dv, fmt = (case[n] for n in ("B", "T", "H", "dk", "dv", "fmt"))
    S = torch.zeros(B, H, dk, dv, dtype=torch.float64, device=x["q"].device)
    energy = torch.zeros(H, dk, dtype=torch.float64, device=S.device)
    for t in range(T):
        _advance(S, *(x[m][t] for m in ("q", "k", "v", "g", "beta")), group)
        if (t + 1) % 8 == 0:
            code, s, z = _quantized(S, fmt)
            back = (code - z) * s
            rows = S.reshape(B, H, dk, -1, 32)
            energy += ((back - (rows @ _h32(torch.float64) if fmt in HADAMARD else rows)) ** 2).sum((0, 3, 4))
    log_a = x["g"].sum((0, 1))
    if log_a.dim() == 1:
        log_a = log_a[:, None].expand(H, dk)
    persistence = 1.0 / (-torch.expm1(2.0 * log_a / (B * T))).clamp(min=1e-4)
    return {"state": S, "energy": energy, "log_decay": log_a.contiguous(),
            "scores": energy / max(B * (T // 8), 1) * persistence, "perm": None}
