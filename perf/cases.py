"""The calls whose speed is followed from change to change: what programs that
use this library have it do, through its public entry points, over the range
of decoders, prefix lengths, block widths and batch sizes that it serves.

Weights are N(0, 0.02) in bf16 with norm gains 1 + N(0, 0.1), prefilled caches
N(0, 1) in bf16, tokens uniform over the vocabulary.  The work of a call does
not depend on how many candidates it accepts.  Every pass first takes the
state back to the prefix it was prepared with (as a program does that retries
from a committed prefix), so a pass can be repeated.
"""
import math
from dataclasses import dataclass

import numpy as np
import torch

import paper_2609_37617_gb300 as lib


@dataclass(frozen=True)
class Shape:
    n_layers: int
    hidden: int
    n_q: int
    n_kv: int
    head_dim: int
    ffn: int
    vocab: int
    rope_theta: float = 1.0e6
    rms_eps: float = 1.0e-6


# the decoders of the benchmark and the tests: the tiny one, the drafter-sized
# one, the target
MODELS = {"tiny": Shape(2, 256, 4, 2, 64, 704, 4096),
          "1.5b": Shape(28, 1536, 12, 2, 128, 8960, 151936),
          "7b": Shape(28, 3584, 28, 4, 128, 18944, 152064)}
ROOM = 64  # positions of the cache past the prefix and the call's own rows


def listed():
    return [
        # the smallest call: a two-layer decoder, where launches and latency are all
        {"name": "tiny-verify-k4", "model": "tiny", "entry": "verify", "lens": "200", "ks": "4"},
        # a drafter's (or a small target's) decode step over 30 s of audio and an instruction
        {"name": "1.5b-decode", "model": "1.5b", "entry": "decode", "lens": "814"},
        # the same step for programs that must not allocate; an odd prefix, a fuller cache
        {"name": "1.5b-static-decode", "model": "1.5b", "entry": "static", "lens": "1203"},
        # block verification with the drafter-sized decoder as the target
        {"name": "1.5b-verify-k8", "model": "1.5b", "entry": "verify", "lens": "814", "ks": "8"},
        # one round of a producer/verifier session: candidates published to a
        # buffer, verified, read back and aligned on the host
        {"name": "1.5b-session-call", "model": "1.5b", "entry": "buffers", "lens": "1187", "ks": "8"},
        # a long instruction behind a minute of audio, a ragged last pass
        {"name": "1.5b-prefill300", "model": "1.5b", "entry": "prefill", "lens": "1500", "n": 300},
        # as many requests as one call takes, short prefixes, mixed block widths
        {"name": "1.5b-batch64", "model": "1.5b", "entry": "verify",
         "lens": " ".join(str(250 + (i * 977) % 1751) for i in range(64)),
         "ks": " ".join(str((i * 7) % 17) for i in range(64))},
        # the target advancing alone by one token
        {"name": "7b-decode", "model": "7b", "entry": "decode", "lens": "1564"},
        # the headline: a block of 8 candidates over a minute of audio
        {"name": "7b-verify-k8", "model": "7b", "entry": "verify", "lens": "1564", "ks": "8"},
        # ten minutes of audio retained, the widest block
        {"name": "7b-long-k16", "model": "7b", "entry": "verify", "lens": "15128", "ks": "16"},
        # a server's round: 16 requests, prefixes of 10 s to 5 min, any block width
        {"name": "7b-ragged16", "model": "7b", "entry": "verify",
         "lens": "6130 6416 2466 5349 5631 376 2509 7495 1702 5900 3266 3948 5116 817 1839 2625",
         "ks": "4 13 16 11 2 13 5 16 13 9 11 3 5 5 15 14"},
        # the instruction that follows the retained audio
        {"name": "7b-prefill64", "model": "7b", "entry": "prefill", "lens": "1500", "n": 64},
    ]


def _ints(text):
    return [int(t) for t in text.split()]


def _rows(case):
    """(prefix lengths, rows of each request) of a call."""
    lens = _ints(case["lens"])
    if case["entry"] == "prefill":
        return lens, [case["n"]]
    if case["entry"] in ("decode", "static"):
        return lens, [1] * len(lens)
    return lens, [k + 1 for k in _ints(case["ks"])]


def _log_uniform(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        case = {"model": rng.choice(("tiny", "1.5b", "1.5b", "7b", "7b"))}
        entry = rng.choice(("verify", "verify", "verify", "decode", "prefill", "static", "buffers"))
        case["entry"] = entry
        if entry == "static":
            case["lens"] = str(_log_uniform(rng, 100, 4000))
        elif entry == "prefill":
            case["lens"] = str(_log_uniform(rng, 25, 15000))
            case["n"] = _log_uniform(rng, 1, 512)
        else:
            batch = 1 if rng.random() < 0.5 else _log_uniform(rng, 2, 64)
            top = 15128 if batch == 1 else 7500
            case["lens"] = " ".join(str(_log_uniform(rng, 100, top)) for _ in range(batch))
            if entry != "decode":
                case["ks"] = " ".join(str(rng.randint(0, 16)) for _ in range(batch))
            if entry == "buffers":  # a session gives every request the same budget
                case["ks"] = " ".join([str(rng.randint(1, 16))] * batch)
        if _cost(case) <= most:
            return case


# ---- inputs -----------------------------------------------------------------------

PER_LAYER = ("attn_norm", "w_q", "w_k", "w_v", "w_o", "mlp_norm", "w_gate", "w_up", "w_down")


def _dims(s, name):
    q, kv = s.n_q * s.head_dim, s.n_kv * s.head_dim
    return {"embed": (s.vocab, s.hidden), "lm_head": (s.vocab, s.hidden), "final_norm": (s.hidden,),
            "attn_norm": (s.hidden,), "mlp_norm": (s.hidden,), "w_q": (q, s.hidden),
            "w_k": (kv, s.hidden), "w_v": (kv, s.hidden), "w_o": (s.hidden, q),
            "w_gate": (s.ffn, s.hidden), "w_up": (s.ffn, s.hidden), "w_down": (s.hidden, s.ffn)}[name]


def _generator(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream) & 0x7FFFFFFFFFFFFFFF)
    return g


def _weight(s, seed, name, layer=0):
    """One weight tensor, a function of (seed, name, layer) alone."""
    names = ("embed", "lm_head", "final_norm") + PER_LAYER
    t = torch.empty(_dims(s, name), dtype=torch.bfloat16, device="cuda")
    g = _generator(seed, 16 + layer * 16 + names.index(name))
    return t.normal_(1.0, 0.1, generator=g) if "norm" in name else t.normal_(0.0, 0.02, generator=g)


def _caches(s, seed, batch, capacity):
    shape = (s.n_layers, batch, s.n_kv, capacity, s.head_dim)
    return [torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(generator=_generator(seed, i))
            for i in (1, 2)]


def _tokens(s, seed, batch, n):
    """(roots, n more tokens), uniform over the vocabulary."""
    t = torch.randint(0, s.vocab, (batch + n,), generator=torch.Generator().manual_seed(int(seed)),
                      dtype=torch.int32).tolist()
    return t[:batch], t[batch:]


def _capacity(case):
    lens, rows = _rows(case)
    if case["entry"] == "static":
        return min(4096, lens[0] + 2 * ROOM)
    return max(l + r for l, r in zip(lens, rows)) + ROOM


def _given(case, seed):
    """Roots, and candidates (or the instruction), of a call."""
    _, rows = _rows(case)
    extra = sum(rows) if case["entry"] == "prefill" else sum(rows) - len(rows)
    return _tokens(MODELS[case["model"]], seed, len(rows), extra)


def prepare(case, seed):
    s = MODELS[case["model"]]
    lens, rows = _rows(case)
    batch, cap = len(lens), _capacity(case)
    names = ("embed", "lm_head", "final_norm")
    w = {n: _weight(s, seed, n) for n in names}
    w.update({n: [_weight(s, seed, n, l) for l in range(s.n_layers)] for n in PER_LAYER})
    torch.cuda.synchronize()
    model = lib.Model(s, {n: t.data_ptr() if n in names else [x.data_ptr() for x in t]
                          for n, t in w.items()})
    del w
    kc, vc = _caches(s, seed, batch, cap)
    roots, extra = _given(case, seed)

    def out(*shape, dtype=torch.int32):
        return torch.zeros(shape, dtype=dtype, device="cuda")

    st = {"case": case, "entry": case["entry"], "model": model, "lens": lens, "roots": roots,
          "kc": kc, "vc": vc, "capacity": cap, "extra": extra,
          "tokens": torch.tensor(extra or [0], dtype=torch.int32, device="cuda"),
          "n": out(batch), "correction": out(batch)}
    # the entries that a call appends to the caches, as views of them
    st["appended"] = {f"{name}{b}": c[:, b, :, l:l + r] for name, c in (("k", kc), ("v", vc))
                      for b, (l, r) in enumerate(zip(lens, rows)) if batch <= 16}
    if batch > 16:  # too many requests for one output each
        longest = max(l + r for l, r in zip(lens, rows))
        st["appended"] = {"k": kc[:, :, :, min(lens):longest], "v": vc[:, :, :, min(lens):longest]}
    if st["entry"] == "static":
        st["start"] = torch.tensor([lens[0], roots[0]], dtype=torch.int32, device="cuda")
        st["now"] = st["start"].clone()
    else:
        st["kv"] = lib.State(model, lens, cap, kc, vc, roots)
    if st["entry"] in ("verify", "decode", "static"):
        st["greedy"] = out(sum(rows))
        st["logits"] = out(sum(rows), s.vocab, dtype=torch.float32)
    if st["entry"] in ("verify", "buffers"):
        st["ks"] = [r - 1 for r in rows]
    torch.cuda.synchronize()
    return st


def run(st):
    entry = st["entry"]
    if entry == "static":
        st["now"].copy_(st["start"])
        now = st["now"].data_ptr()
        status = lib.as2d_decode_step_static(
            st["model"].handle, st["kc"].data_ptr(), st["vc"].data_ptr(), st["capacity"], now, now + 4,
            st["correction"].data_ptr(), st["logits"].data_ptr())
        if status != lib.AS2D_OK:
            raise RuntimeError(lib.as2d_last_error())
        return {"logits": st["logits"], "correction": st["correction"], "state": st["now"],
                **st["appended"]}
    kv = st["kv"]
    kv.rollback(st["lens"], st["roots"])
    if entry == "prefill":
        kv.prefill(st["tokens"], st["correction"])
        return {"first": st["correction"], **st["appended"]}
    if entry == "buffers":
        bufs, at = [], 0
        for k in st["ks"]:
            buf = lib.CandidateBuffer()
            for i in range(0, k, lib.AS2D_CBUF_BATCH):
                buf.publish(st["extra"][at + i:at + min(k, i + lib.AS2D_CBUF_BATCH)], offset=i)
            at += k
            bufs.append(buf)
        used, committed = kv.verify_from_buffers(bufs, st["ks"][0])
        text = np.full((len(committed), st["ks"][0] + 1), -1, dtype=np.int32)
        for row, tokens in zip(text, committed):
            row[:len(tokens)] = tokens
        return {"used": np.array(used), "committed": text, **st["appended"]}
    if entry == "decode":
        kv.decode(st["n"], st["correction"], st["greedy"], st["logits"])
    else:
        kv.verify(st["tokens"], st["ks"], st["n"], st["correction"], st["greedy"], st["logits"])
    return {"logits": st["logits"], "greedy": st["greedy"], "n_accepted": st["n"],
            "correction": st["correction"], **st["appended"]}


# ---- what a call cannot do without -------------------------------------------------

def work(case):
    s = MODELS[case["model"]]
    lens, rows = _rows(case)
    total, q, kv = sum(rows), s.n_q * s.head_dim, s.n_kv * s.head_dim
    layer = s.hidden * (2 * q + 2 * kv) + 3 * s.hidden * s.ffn
    logit_rows = 1 if case["entry"] == "prefill" else total
    attended = sum(r * l + r * (r + 1) // 2 for l, r in zip(lens, rows))
    nbytes = 2 * (s.n_layers * (layer + 2 * s.hidden) + s.vocab * s.hidden + s.hidden)
    nbytes += 2 * total * s.hidden                                          # embedding rows
    nbytes += 2 * 2 * s.n_layers * kv * sum(l + r for l, r in zip(lens, rows))  # cache read and appended
    if case["entry"] in ("verify", "decode", "static"):
        nbytes += 4 * total * s.vocab                                       # logits
    flops = 2 * total * s.n_layers * layer + 2 * logit_rows * s.vocab * s.hidden
    flops += 4 * s.n_layers * q * attended
    return {"bytes": nbytes, "flops": flops}


def _cost(case):
    w = work(case)
    # about the time of a pass, in bytes: shallow calls cannot be dearer than
    # the listed ones, deep prefills stream the weights more than once
    return w["bytes"] + w["flops"] / 150


def tolerance(case):
    # The appended entries are bf16: a difference of 1e-5 in a value turns the
    # rounding of about one entry in 300 by one unit in the last place (up to
    # 2^-7 of the value), and those reach the layers that follow.
    # One greedy token of a large call may fall the other way at a tie.
    return {"rel": TOLERANCE[case["model"]], "max": 0.02, "differ": 0.0 if sum(_rows(case)[1]) < 100 else 0.01}


TOLERANCE = {"tiny": 1e-3, "1.5b": 2e-3, "7b": 2e-3}


# ---- the same in 64 bits ------------------------------------------------------------

def exact(case, seed):
    """Logits and appended cache entries by plain torch in 64 bits.  Keys and
    values are rounded to bf16 where the cache holds them: later rows of the
    call read the rounded entries."""
    s = MODELS[case["model"]]
    lens, rows = _rows(case)
    d, half, group = s.head_dim, s.head_dim // 2, s.n_q // s.n_kv
    cap, total = _capacity(case), sum(rows)
    roots, extra = _given(case, seed)
    tokens, at = [], 0
    for root, r in zip(roots, rows):
        if case["entry"] == "prefill":
            tokens += extra
        else:
            tokens += [root] + extra[at:at + r - 1]
            at += r - 1
    pos = torch.cat([torch.arange(l, l + r) for l, r in zip(lens, rows)]).cuda().double()
    freq = s.rope_theta ** (-2.0 * torch.arange(half, device="cuda").double() / d)
    cos, sin = torch.cos(pos[:, None] * freq)[:, None], torch.sin(pos[:, None] * freq)[:, None]

    def weight(name, layer=0):
        return _weight(s, seed, name, layer).double()

    def norm(x, gain):
        return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + s.rms_eps) * gain

    def rotate(x):
        a, b = x[..., :half], x[..., half:]
        return torch.cat([a * cos - b * sin, b * cos + a * sin], -1)

    kc, vc = _caches(s, seed, len(lens), cap)
    new = {}
    x = _weight(s, seed, "embed")[torch.tensor(tokens, device="cuda")].double()
    for layer in range(s.n_layers):
        y = norm(x, weight("attn_norm", layer))
        qh = rotate((y @ weight("w_q", layer).T).view(total, s.n_q, d))
        kh = rotate((y @ weight("w_k", layer).T).view(total, s.n_kv, d))
        vh = (y @ weight("w_v", layer).T).view(total, s.n_kv, d)
        o, r0 = torch.empty_like(qh), 0
        for b, (l, r) in enumerate(zip(lens, rows)):
            sl = slice(r0, r0 + r)
            new.setdefault(("k", b), []).append(kh[sl].transpose(0, 1))
            new.setdefault(("v", b), []).append(vh[sl].transpose(0, 1))
            keys = torch.cat([kc[layer, b, :, :l].double(), kh[sl].transpose(0, 1).bfloat16().double()], 1)
            vals = torch.cat([vc[layer, b, :, :l].double(), vh[sl].transpose(0, 1).bfloat16().double()], 1)
            qq = qh[sl].view(r, s.n_kv, group, d).permute(1, 2, 0, 3).reshape(s.n_kv, group * r, d)
            sc = (qq @ keys.transpose(1, 2) / math.sqrt(d)).view(s.n_kv, group, r, l + r)
            seen = torch.arange(l + r, device="cuda")[None] <= torch.arange(l, l + r, device="cuda")[:, None]
            p = sc.masked_fill(~seen, -math.inf).softmax(-1).view(s.n_kv, group * r, l + r)
            o[sl] = (p @ vals).view(s.n_kv, group, r, d).permute(2, 0, 1, 3).reshape(r, s.n_q, d)
            r0 += r
        x = x + o.reshape(total, -1) @ weight("w_o", layer).T
        y = norm(x, weight("mlp_norm", layer))
        y = torch.nn.functional.silu(y @ weight("w_gate", layer).T) * (y @ weight("w_up", layer).T)
        x = x + y @ weight("w_down", layer).T
    res = {}
    if case["entry"] in ("verify", "decode", "static"):
        res["logits"] = norm(x, weight("final_norm")) @ weight("lm_head").T
    if len(lens) <= 16:
        res.update({f"{name}{b}": torch.stack(t) for (name, b), t in new.items()})
    else:
        longest = max(l + r for l, r in zip(lens, rows))
        for name, c in (("k", kc), ("v", vc)):
            c = c.double()
            for b, (l, r) in enumerate(zip(lens, rows)):
                c[:, b, :, l:l + r] = torch.stack(new[name, b])
            res[name] = c[:, :, :, min(lens):longest]
    return res
