"""The work that users of the memory-pot library have it do, as cases that can be timed and compared.

Three kinds of calls make up a program that uses the library, and every case is one pass of one of them through
the public entry points of ``paper_2410_01518_b200.ipot``:

``cycle``    a prompt's tokens go into an empty pot (``ipot_append_chunk``) and are distilled to ``keep`` rows
             (``ipot_score_and_compress`` or, with the CaP's own keys in the softmax, ``..._cap``);
``novelty``  the logits of a chunk become the novelty scores that the cycle ranks (``ipot_nuc_scores``);
``decode``   one generated token attends to the pot (``ipot_decode_attention``).

Sizes are those of ``inputs.CONFIGS``, of the benchmark's workloads and of the tests, and generic odd ones.  A pass
starts from the same state every time (a cycle empties the pot first), so that its outputs depend on the inputs only.

Inputs: keys and values N(0, 1).  The queries of a catalyst prompt are not independent of one another - a head asks
the same thing from every position - so the rows of a query head share a direction, which concentrates the attention
on few keys as trained heads do.  Novelty ~ U(0, 1); logits and labels as in ``inputs.make_logits``.
"""
import math

import torch

from paper_2410_01518_b200 import ipot

# every listed cycle names all of these; "deferred": ipot_set_deferred_append; "rope": "" | "half" | "interleaved";
# "cap": the CaP's own keys join the softmax; "n" rows are appended, "keep" survive, "T" of them by novelty
_CYCLE = dict(kind="cycle", dtype="bf16", layers=1, batch=1, Hq=32, Hkv=8, d=128, n=4096, keep=2048, T=1024, P=32,
              deferred=False, rope="", cap=False)


def listed():
    return [
        # the smallest call: a toy model in fp32, where launches and host work are all there is
        dict(_CYCLE, name="cycle_tiny_f32", dtype="f32", Hq=8, Hkv=2, d=64, n=512, keep=256, T=128, P=16),
        # one layer of a 7B model at a time, as a model does that distils inside its layer loop
        dict(_CYCLE, name="cycle_one_layer"),
        # all 32 layers of that model in one call, the chunk read where it lies
        dict(_CYCLE, name="cycle_32_layers", layers=32, deferred=True),
        # the same in the paper's complete form: unrotated keys with positions reset, CaP keys in the softmax
        dict(_CYCLE, name="cycle_32_layers_rope_cap", layers=32, deferred=True, rope="half", cap=True),
        # a serving batch of 16 streams, library defaults
        dict(_CYCLE, name="cycle_batch16", batch=16, n=8192, P=64),
        # a layer of a 70B model, 8 long streams: many query rows per key
        dict(_CYCLE, name="cycle_batch8_70b", batch=8, Hq=64, n=16384, keep=4096, T=2048, P=64, deferred=True),
        # nothing is a multiple of anything
        dict(_CYCLE, name="cycle_ragged", layers=5, batch=3, Hq=12, Hkv=4, n=2999, keep=1003, T=401, P=19),
        # wide heads (256 channels), few query heads per key head
        dict(_CYCLE, name="cycle_wide_heads", layers=8, Hq=16, d=256),
        # novelty of a chunk over a large vocabulary, and over an odd one, whose rows start anywhere
        dict(name="novelty_128k", kind="novelty", dtype="bf16", batch=1, tokens=2048, vocab=128256),
        dict(name="novelty_ragged", kind="novelty", dtype="bf16", batch=1, tokens=777, vocab=50257),
        # a token of generation: one layer per call (the layer loop of a model), and a whole model's pot per call
        dict(name="decode_one_layer", kind="decode", dtype="bf16", layers=1, batch=1, Hq=32, Hkv=8, d=128, n=2048),
        dict(name="decode_32_layers", kind="decode", dtype="bf16", layers=32, batch=1, Hq=32, Hkv=8, d=128, n=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _heads(rng, most_rows_per_unit=0, P=0):
    while True:
        hkv, g = rng.choice((1, 2, 4, 4, 8, 8, 8)), rng.choice((1, 2, 3, 4, 4, 4, 5, 7, 8))
        if not most_rows_per_unit or g * P <= most_rows_per_unit:
            return hkv * g, hkv


def _draw_cycle(rng):
    n = _log_int(rng, 500, 16384)
    keep = max(16, int(n * rng.uniform(0.2, 0.6)))
    P = rng.choice((8, 16, 19, 32, 32, 48, 64))
    Hq, Hkv = _heads(rng, 512, P)
    f32 = rng.random() < 0.2
    return dict(_CYCLE, dtype="f32" if f32 else "bf16", layers=_log_int(rng, 1, 32), batch=_log_int(rng, 1, 16), Hq=Hq, Hkv=Hkv,
                d=rng.choice((32, 64, 128)) if f32 else rng.choice((64, 96, 128, 128, 128, 256)), n=n, keep=keep,
                T=rng.choice((0, keep // 2, keep // 2, int(keep * rng.random()))), P=P, deferred=rng.random() < 0.5,
                rope=rng.choice(("", "", "", "half", "interleaved")), cap=rng.random() < 0.25)


def _draw_novelty(rng):
    return dict(kind="novelty", dtype=rng.choice(("bf16", "bf16", "f32")), batch=rng.choice((1, 1, 2, 4)), tokens=_log_int(rng, 16, 2048),
                vocab=rng.choice((32000, 50257, 128256, 151936, _log_int(rng, 4000, 200000))))


def _draw_decode(rng):
    f32 = rng.random() < 0.2
    while True:
        Hq, Hkv = _heads(rng)
        if not f32 or Hq // Hkv in (1, 2, 4, 8):   # what the entry point takes
            break
    return dict(kind="decode", dtype="f32" if f32 else "bf16", layers=_log_int(rng, 1, 32), batch=_log_int(rng, 1, 16), Hq=Hq, Hkv=Hkv,
                d=rng.choice((64, 128, 128)), n=_log_int(rng, 100, 16384))


def _cost(c):
    """Rough seconds of a case, to keep drawn cases below the largest listed one."""
    w = work(c)
    if c["kind"] != "cycle":
        return w["bytes"] / 5e12
    copied = 0 if c["deferred"] else 4 * _units(c) * c["n"] * c["d"] * _elem(c)
    rate = 5e12 if c["dtype"] == "f32" else 4e14 if c["d"] in (64, 128) else 2.5e13
    return (w["bytes"] + copied) / 4e12 + w["flops"] / rate


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        c = rng.choice((_draw_cycle, _draw_cycle, _draw_cycle, _draw_novelty, _draw_decode))(rng)
        if _cost(c) <= most and work(c)["bytes"] <= max(work(x)["bytes"] for x in listed()):
            return c


def _units(c):
    return c["layers"] * c["batch"] * c["Hkv"]


def _elem(c):
    return 4 if c["dtype"] == "f32" else 2


def work(case):
    c, e = case, _elem(case)
    if c["kind"] == "novelty":
        logits = c["batch"] * c["tokens"] * c["vocab"]
        return {"bytes": logits * e + 8 * c["batch"] * c["tokens"], "flops": 3 * logits}
    units, G = _units(c), c["Hq"] // c["Hkv"]
    if c["kind"] == "decode":
        return {"bytes": units * (2 * c["n"] * c["d"] * e + G * (c["d"] * (e + 4) + 4)), "flops": 4 * units * G * c["n"] * c["d"]}
    M, row = G * c["P"], c["d"] * e
    rows = c["n"] + 3 * c["keep"] + M               # keys in; survivors' values in; survivors out; queries in
    flops = 2 * M * c["n"] * c["d"]
    if c["rope"]:
        rows += c["keep"] + c["keep"] / units       # the rotated survivors; the tables
    if c["cap"]:
        rows += c["P"]
        flops += M * c["P"] * c["d"]
    out = 4 * (c["n"] + c["keep"])                  # scores and index list
    return {"bytes": units * (rows * row + out) + 4 * c["batch"] * c["n"] * (c["T"] > 0), "flops": units * flops}


def tolerance(case):
    if case["kind"] == "cycle":
        # scores are fp32 sums of exponentials of fp32 logits; index lists and rows are whole numbers and bytes, in which
        # two scores that agree to fp32 rounding at the boundary of the selection may change places
        return {"rel": 1e-5, "differ": 0.01}
    return {"rel": 1e-5 if case["kind"] == "novelty" else 2e-5}


class _Pot:
    """A pot that is destroyed with the last object that refers to it: the case's state or a view of its memory."""

    def __init__(self, *args, **kw):
        self.h = None
        self.h = ipot.ipot_create_ex(*args, **kw)

    def __del__(self):
        if self.h is not None:
            ipot.ipot_destroy(self.h)

    def view(self, addr, shape, dtype):
        """A tensor over library-owned memory that keeps the pot alive."""
        memory = _Memory()
        memory.pot = self
        memory.__cuda_array_interface__ = {"shape": (math.prod(shape) * dtype.itemsize,), "typestr": "|u1", "data": (addr, False), "version": 2}
        return torch.as_tensor(memory, device="cuda").view(dtype).view(shape)


class _Memory:
    pass


class _State:
    """Device buffers of the caller and one pot."""


def _normal(g, shape, dtype):
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype)


def _pot(c, keep, T, P):
    return _Pot(c["n"], keep, c["layers"], c["Hq"], c["Hkv"], c["d"], batch=c["batch"],
                dtype=ipot.IPOT_F32 if c["dtype"] == "f32" else ipot.IPOT_BF16, nuc_slots=T, max_cap_rows=P)


def _prepare_cycle(c, g, dtype, s):
    L, B, n, d, P = c["layers"], c["batch"], c["n"], c["d"], c["P"]
    s.K, s.V = _normal(g, (L, B, c["Hkv"], n, d), dtype), _normal(g, (L, B, c["Hkv"], n, d), dtype)
    s.Q = (2.5 * _normal(g, (L, B, c["Hq"], 1, d), torch.float32) + _normal(g, (L, B, c["Hq"], P, d), torch.float32)).to(dtype)
    s.K_cap = _normal(g, (L, B, c["Hkv"], P, d), dtype) if c["cap"] else None
    s.aux = torch.rand((B, n), generator=g, device="cuda") if c["T"] > 0 else None
    s.n, s.P = n, P
    s.pot = _pot(c, c["keep"], c["T"], P)
    s.h = s.pot.h
    ipot.ipot_set_deferred_append(s.h, c["deferred"])
    if c["rope"]:
        half = d // 2
        ang = torch.arange(n, device="cuda", dtype=torch.float64)[:, None] * 10000.0 ** (-torch.arange(half, device="cuda", dtype=torch.float64) / half)
        s.cos, s.sin = ang.cos().to(dtype), ang.sin().to(dtype)
        ipot.ipot_enable_rope(s.h, s.cos, s.sin, ipot.IPOT_ROPE_HALF if c["rope"] == "half" else ipot.IPOT_ROPE_INTERLEAVED)
    # what the cycle leaves behind, seen through the library's own buffers: index lists and the pot's rows, the latter
    # as bit patterns (rows are moved, not computed)
    units, keep = _units(c), c["keep"]
    bits = torch.int32 if c["dtype"] == "f32" else torch.int16
    rows = lambda addr: s.pot.view(addr, (units, n, d), bits)[:, :keep]  # noqa: E731
    k_addr, v_addr, _ = ipot.ipot_view(s.h)
    s.out = {"idx": s.pot.view(ipot.ipot_last_indices(s.h), (units, keep), torch.int32), "K": rows(k_addr), "V": rows(v_addr)}
    if c["rope"]:
        s.out["K_rot"] = rows(ipot.ipot_view_rope(s.h))
    s.units, s.scores = units, {}


def _prepare_novelty(c, g, dtype, s):
    B, t, vocab = c["batch"], c["tokens"], c["vocab"]
    s.logits = _normal(g, (B * t, vocab), dtype).mul_(2.5)
    s.labels = torch.randint(0, vocab, (B * t,), generator=g, device="cuda", dtype=torch.int32)
    # about half of the tokens were predicted well
    boost = (0.6 + torch.rand(B * t, generator=g, device="cuda")) * (math.log(vocab) + 3.0)
    boost = torch.where(torch.rand(B * t, generator=g, device="cuda") < 0.5, boost, torch.zeros_like(boost))
    at = torch.arange(B * t, device="cuda"), s.labels.long()
    s.logits[at] = (s.logits[at].float() + boost).to(dtype)
    s.aux = torch.zeros((B, t), device="cuda")
    s.args = (ipot.IPOT_F32 if c["dtype"] == "f32" else ipot.IPOT_BF16, vocab, t, vocab)
    s.pot = _Pot(64, 32, 1, 1, 1, 64, batch=B)   # the pot whose cycle would use the result
    s.h = s.pot.h


def _prepare_decode(c, g, dtype, s):
    shape = (c["layers"], c["batch"], c["Hkv"], c["n"], c["d"])
    s.pot = _pot(c, max(1, c["n"] // 2), 0, 1)
    s.h = s.pot.h
    ipot.ipot_append_chunk(s.h, _normal(g, shape, dtype), _normal(g, shape, dtype), c["n"])
    ipot.ipot_sync_status(s.h)
    s.q = 1.5 * _normal(g, (c["layers"], c["batch"], c["Hq"], c["d"]), dtype)
    s.o = torch.zeros((c["layers"], c["batch"], c["Hq"], c["d"]), device="cuda")
    s.lse = torch.zeros((c["layers"], c["batch"], c["Hq"]), device="cuda")


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    s = _State()
    s.kind = case["kind"]
    dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    {"cycle": _prepare_cycle, "novelty": _prepare_novelty, "decode": _prepare_decode}[s.kind](case, g, dtype, s)
    return s


def run(state):
    s = state
    if s.kind == "novelty":
        dtype, stride, t, vocab = s.args
        ipot.ipot_nuc_scores(s.h, s.logits, dtype, stride, s.labels, t, vocab, s.aux, t, 0)
        return s.aux
    if s.kind == "decode":
        ipot.ipot_decode_attention(s.h, s.q, s.o, s.lse)
        return s.o, s.lse
    ipot.ipot_reset(s.h)
    ipot.ipot_append_chunk(s.h, s.K, s.V, s.n)
    if s.K_cap is None:
        ipot.ipot_score_and_compress(s.h, s.Q, s.P, s.aux)
    else:
        ipot.ipot_score_and_compress_cap(s.h, s.Q, s.K_cap, s.P, s.aux)
    addr, n = ipot.ipot_last_scores(s.h)
    if addr not in s.scores:   # a view of the library's score array, made once
        s.scores[addr] = s.pot.view(addr, (s.units, n), torch.float32)
    return dict(s.out, scores=s.scores[addr])
