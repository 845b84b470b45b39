"""What is measured: the calls that a streaming program makes on this library, over the
range of sizes that the workloads of synth/script.py and bench.py span.

A duplex unit (one second of speech) of a session is one chunk of 17 acoustic positions
(append + chunked-prefill attention of every layer), then about five single-token decode
rounds (append + decode attention of every layer), then one eviction.  The kinds:

  decode   the decode attention of every layer for one round: n sessions, one token each
  prefill  the chunked-prefill attention of every layer for n sessions' chunks
  unit     whole sessions: release, the history fed back in one append, eviction, then
           `steps` duplex units with every append, attention and eviction call in order
  restore  sessions moved onto this device: release, the history in one append, eviction,
           then the transcript export of each session

Every kind leaves the cache as it found it or starts from kvc_release, so a pass can be
repeated.  The histories' token counts, K, V and q all come from the seed.  The histories are token
streams with Poisson(3) transcript tokens a unit and a speaking turn of 20 to 80 text
tokens about every 60 units, evicted as they are fed, so that the caches are ragged:
compacted pages, partly consumed first live pages and partly filled last ones.

Attention inputs are N(0, 1), rounded to the cache's type.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_31224_gb300 import KVCache
from paper_2609_31224_gb300._lib import host_i32

ACOUSTIC, DELIM, TRANSCRIPT, TEXT, BEGIN = 0, 1, 2, 3, 0x80
UNIT_POSITIONS = 17        # acoustic positions of one unit: one prefill chunk
PER_UNIT = 22.8            # positions of an average unit, speaking turns included
KEPT_PER_UNIT = 3.8        # of these, transcript and text
FEED_UNITS = 32            # units of history fed between two evictions
BASE = 10000.0
DEV = "cuda"


def _case(name, kind, n, *, dtype="bf16", layers=32, heads=8, budget=4096, window=10, units=400,
          tokens=UNIT_POSITIONS, ragged=False, per_layer=False, steps=0):
    """name; kind (above); n sessions; layers; heads: KV heads (4 query heads each); budget
    and window of the eviction rule; units of history fed per session; tokens of the prefill
    chunk (ragged: 1 to that many, another number for each session); per_layer: K/V are
    written by the attention call of their layer, the order in which a model has them."""
    c = dict(name=name, kind=kind, n=n, dtype=dtype, layers=layers, heads=heads, budget=budget,
             window=window, units=units, tokens=tokens, ragged=ragged, per_layer=per_layer,
             steps=steps)
    if name is None:
        del c["name"]
    return c


def listed():
    return [
        # A whole one-minute session of the small binary32 shape (1 layer, 1 KV head): some
        # 800 calls of a few microseconds each, where launches and host work are the cost.
        _case("session_f32_tiny", "unit", 1, dtype="f32", layers=1, heads=1, budget=512, window=5,
              units=0, steps=60),
        # binary32 caches of a few sessions: one decode round and one chunk.
        _case("decode_f32_s6", "decode", 6, dtype="f32", layers=8, heads=8, budget=2048,
              units=200),
        _case("prefill_f32_s4", "prefill", 4, dtype="f32", layers=8, heads=8, budget=1024,
              units=100),
        # One conversation on the 32-layer shape: most decode rounds of a speaking turn, and
        # what one user waits for.
        _case("decode_s1", "decode", 1),
        _case("prefill_s1", "prefill", 1),
        # The round sizes between one session and the full batch, which a batch of sessions
        # passes through as their transcript segments end one after the other.
        _case("decode_s6_per_layer", "decode", 6, per_layer=True),
        _case("decode_s20", "decode", 20),
        _case("prefill_s9_per_layer", "prefill", 9, per_layer=True),
        # The full batch of 64 sessions.
        _case("decode_s64", "decode", 64),
        _case("prefill_s64", "prefill", 64),
        # Two sessions moved onto this device, and their transcripts read back.
        _case("restore_s2", "restore", 2, units=220),
        # Three conversations, two whole units each in the model's order (the later decode
        # rounds hold fewer sessions).
        _case("unit_s3_per_layer", "unit", 3, units=220, per_layer=True, steps=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "prefill", "prefill", "prefill", "unit",
                       "restore"])
    f32 = rng.random() < 0.25
    window = rng.choice([1, 5, 10, 20])
    budget = _log(rng, 256, 8192) if rng.random() < 0.9 else -1
    if kind in ("decode", "prefill"):
        n = _log(rng, 1, 64)
        units = _log(rng, 20, 500)
        most = 64 * 4096 // n                       # positions of a session, so that n of
        units = max(8, min(units, int(most / PER_UNIT) if budget < 0 else 500))  # them fit
        budget = min(budget, most)
        if budget >= 0:
            units = min(units, int(most / KEPT_PER_UNIT))
        return _case(None, kind, min(n, 24) if f32 else n, dtype="f32" if f32 else "bf16",
                     layers=rng.randint(2, 8) if f32 else rng.choice([16, 24, 28, 32]),
                     heads=rng.choice([1, 2, 4, 8]) if f32 else rng.choice([4, 8, 8]),
                     budget=budget, window=window, units=units,
                     tokens=rng.choice([17, 17, rng.randint(2, 32)]), ragged=rng.random() < 0.3,
                     per_layer=rng.random() < 0.4)
    n = rng.randint(1, 3)
    return _case(None, kind, n, dtype="f32" if f32 else "bf16",
                 layers=rng.randint(1, 8) if f32 else rng.choice([16, 24, 32]),
                 heads=rng.choice([1, 2, 4, 8]) if f32 else 8,
                 budget=budget, window=window, units=_log(rng, 20, 220),
                 per_layer=kind == "unit" and rng.random() < 0.6,
                 steps=rng.randint(1, 2) if kind == "unit" else 0)


# -- token streams and the positions that stay ------------------------------------------------
class _Stream:
    """One session's tokens and, under the eviction rule, its resident positions."""

    def __init__(self, rng, units, lengths):
        """History of `units` units, then units with segments of `lengths` transcript tokens,
        whose token types are kept apart."""
        types, cuts = [], [0]
        turn = int(rng.integers(20, 60))
        for u in range(units):
            types += [ACOUSTIC | BEGIN] + [ACOUSTIC] * (UNIT_POSITIONS - 1)
            types += [DELIM] + [TRANSCRIPT] * min(64, int(rng.poisson(3))) + [DELIM]
            if (u + turn) % 60 == 59:
                types += [TEXT] * int(rng.integers(20, 81))
            cuts.append(len(types))
        tails = [np.array([DELIM] + [TRANSCRIPT] * int(t) + [DELIM], np.uint8) for t in lengths]
        self.history = np.array(types, np.uint8)
        self.cuts, self.tails = cuts, tails
        self.n = 0
        self.unit_cur = -1
        self.type = np.zeros(0, np.uint8)
        self.unit = np.zeros(0, np.int64)
        self.res = np.zeros(0, np.int64)
        self.peak = 0

    def append(self, types):
        self.type = np.concatenate([self.type, types & 0x7F])
        units = self.unit_cur + np.cumsum((types & BEGIN) != 0)
        self.unit = np.concatenate([self.unit, units])
        self.unit_cur = int(units[-1])
        self.res = np.concatenate([self.res, np.arange(self.n, self.n + len(types))])
        self.n += len(types)
        self.peak = max(self.peak, len(self.res))

    def evict(self, budget, window):
        """While over budget: the acoustic and delimiter positions of the oldest unit
        outside the window that still has some."""
        over = len(self.res) - budget
        if budget < 0 or over <= 0:
            return
        u = self.unit[self.res]
        ev = (u >= 0) & (u <= self.unit_cur - window) & (self.type[self.res] <= DELIM)
        if not ev.any():
            return
        total = np.cumsum(np.bincount(u[ev], minlength=int(u.max()) + 1))
        last = int(np.searchsorted(total, over))
        self.res = self.res[~(ev & (u <= last))]


def _plan(case, seed):
    """The calls of one pass and before it: a list of ("append", tag, per-session types,
    positions fed before) and ("evict",), with, for every append, each session's resident
    positions after it; and the streams themselves."""
    kind, n = case["kind"], case["n"]
    streams, plan = [], []
    for i in range(n):
        rng = np.random.default_rng([seed, i])
        units = case["units"]
        if units and kind != "unit":
            units = max(1, int(round(units * rng.uniform(0.75, 1.0))))
        # The segments of a pass's own units are the same for every seed, and with them the
        # number of its decode rounds and the shapes of its outputs.
        lengths = np.random.default_rng([n, i]).poisson(3, size=case["steps"])
        streams.append(_Stream(rng, units, lengths))
    def append(tag, sessions, types):
        for s, t in zip(sessions, types):
            streams[s].append(t)
        plan.append(dict(op="append", tag=tag, sessions=list(sessions), types=list(types),
                         first=[streams[s].n - len(t) for s, t in zip(sessions, types)],
                         res=[streams[s].res for s in sessions]))

    def evict():
        for s in streams:
            s.evict(case["budget"], case["window"])
        plan.append(dict(op="evict", res=[s.res for s in streams]))

    every = range(n)
    if case["units"]:
        parts = 1 if kind in ("unit", "restore") else -(-case["units"] // FEED_UNITS)
        for p in range(parts):
            cut = [(s.cuts[(len(s.cuts) - 1) * p // parts], s.cuts[(len(s.cuts) - 1) * (p + 1) // parts])
                   for s in streams]
            who = [i for i in every if cut[i][1] > cut[i][0]]
            append("history", who, [streams[i].history[cut[i][0]:cut[i][1]] for i in who])
            evict()
    chunk = np.full(UNIT_POSITIONS, ACOUSTIC, np.uint8)
    chunk[0] |= BEGIN
    if kind == "prefill":
        most = case["tokens"]
        some = np.random.default_rng([n, most]).integers(1, most + 1, size=n)
        ts = [int(t) if case["ragged"] else most for t in some]
        types = [np.full(t, ACOUSTIC, np.uint8) for t in ts]
        for t in types:
            t[0] |= BEGIN
        append("prefill", every, types)
    elif kind == "decode":
        append("history", every, [chunk] * n)
        append("decode", every, [np.array([TRANSCRIPT], np.uint8)] * n)
    elif kind == "unit":
        for step in range(case["steps"]):
            append("prefill", every, [chunk] * n)
            tails = [s.tails[step] for s in streams]
            for r in range(max(len(t) for t in tails)):
                who = [i for i in every if len(tails[i]) > r]
                append("decode", who, [tails[i][r:r + 1] for i in who])
            evict()
    return streams, plan


# -- values -----------------------------------------------------------------------------------
def _dt(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _dim(case):
    return 128 if case["dtype"] == "bf16" else 64


def _normal(case, shape, *key):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(np.random.SeedSequence(key).generate_state(1, np.uint64)[0] >> np.uint64(1)))
    return torch.randn(shape, generator=g, device=DEV, dtype=_dt(case))


def _kv(case, seed, at, layer, total):
    """K and V of one layer for the plan's append number `at`: [2][total][heads][D]."""
    return _normal(case, (2, total, case["heads"], _dim(case)), seed, 1, at, layer)


def _q(case, seed, at, total):
    return _normal(case, (case["layers"], total, 4 * case["heads"], _dim(case)), seed, 2, at)


# -- the calls --------------------------------------------------------------------------------
class _Append:
    """Arguments of one append and of the attention calls that answer its queries, as a
    program that streams keeps them: host arrays with their pointers, device addresses."""

    def __init__(self, case, seed, at, op, keep_kv):
        self.tag = op["tag"]
        self.n = len(op["sessions"])
        lens = [len(t) for t in op["types"]]
        self.total = sum(lens)
        self.sess, self.sess_p = host_i32(op["sessions"])
        self.cu, self.cu_p = host_i32(np.concatenate([[0], np.cumsum(lens)]))
        self.types = torch.as_tensor(np.concatenate(op["types"]), device=DEV)
        self.k = self.v = None
        if keep_kv:
            shape = (case["layers"], self.total, case["heads"], _dim(case))
            self.k = torch.empty(shape, dtype=_dt(case), device=DEV)
            self.v = torch.empty_like(self.k)
            for layer in range(case["layers"]):
                kv = _kv(case, seed, at, layer, self.total)
                self.k[layer], self.v[layer] = kv[0], kv[1]
            self.k_ptr, self.v_ptr = self._layers(self.k), self._layers(self.v)
        if self.tag != "history":
            self.q = _q(case, seed, at, self.total)
            self.q_ptr = self._layers(self.q)

    @staticmethod
    def _layers(x):
        return [x.data_ptr() + i * x.stride(0) * x.element_size() for i in range(x.shape[0])]

    def into(self, out):
        """Outputs [layers][total][query heads][D] of this call."""
        self.out, self.out_ptr = out, self._layers(out)

    def feed(self, cache, stream, with_kv):
        cache.append_chunk_raw(self.n, self.sess_p, self.cu_p, self.types.data_ptr(),
                               self.k.data_ptr() if with_kv else None,
                               self.v.data_ptr() if with_kv else None, stream)

    def attend(self, cache, stream, per_layer):
        if per_layer:
            fn = cache.attn_decode_kv_raw if self.tag == "decode" else cache.attn_prefill_kv_raw
            for layer, (k, v, q, o) in enumerate(zip(self.k_ptr, self.v_ptr, self.q_ptr, self.out_ptr)):
                fn(layer, k, v, q, o, stream)
        else:
            fn = cache.attn_decode_raw if self.tag == "decode" else cache.attn_prefill_raw
            for layer, (q, o) in enumerate(zip(self.q_ptr, self.out_ptr)):
                fn(layer, q, o, stream)


def _cache(case, streams, plan):
    pages = [s.peak // 16 + s.peak // 32 + 8 for s in streams]
    tokens = max(sum(len(t) for t in op["types"]) for op in plan if op["op"] == "append")
    return KVCache(n_sessions=case["n"], layers=case["layers"], q_heads=4 * case["heads"],
                   kv_heads=case["heads"], head_dim=_dim(case), budget=case["budget"],
                   window=case["window"], dtype=case["dtype"], rope_base=BASE,
                   n_pages=sum(pages) + 16, max_pages_per_session=max(pages),
                   max_positions=max(s.n for s in streams) + 1, max_seq_per_call=case["n"],
                   max_tokens_per_call=tokens, device=DEV)


def _room(case):
    """Positions that a program leaves room for when it reads a session's transcript back."""
    return int(3 * case["units"] + 6 * math.sqrt(3 * case["units"])) + 8


def prepare(case, seed):
    streams, plan = _plan(case, seed)
    cache = _cache(case, streams, plan)
    stream = torch.cuda.current_stream().cuda_stream
    sessions = np.arange(case["n"], dtype=np.int32)
    state = dict(case=case, cache=cache, sessions=sessions)
    if case["kind"] in ("decode", "prefill"):
        # The cache as the calls before this one left it: the history, evicted as it came.
        for at, op in enumerate(plan):
            if op["op"] == "evict":
                cache.evict(sessions)
                continue
            last = at == len(plan) - 1
            a = _Append(case, seed, at, op, keep_kv=last)
            if last:
                a.feed(cache, stream, not case["per_layer"])
                a.into(torch.zeros(a.q.shape, dtype=a.q.dtype, device=DEV))
                state["call"] = a
            else:
                a.feed(cache, stream, False)
                for layer in range(case["layers"]):
                    kv = _kv(case, seed, at, layer, a.total)
                    cache.append_kv_layer(layer, kv[0], kv[1])
        return state
    calls = [op if op["op"] == "evict" else _Append(case, seed, at, op, keep_kv=True)
             for at, op in enumerate(plan)]
    state["calls"] = calls
    state["resident"] = torch.zeros((sum(op["op"] == "evict" for op in plan), case["n"]),
                                    dtype=torch.int64, device=DEV)
    if case["kind"] == "restore":
        return state
    # Outputs of every attention call, one buffer for each kind of call.
    row = case["layers"] * 4 * case["heads"] * _dim(case)
    for tag in ("prefill", "decode"):
        mine = [a for a in calls if isinstance(a, _Append) and a.tag == tag]
        flat = torch.zeros(sum(a.total for a in mine) * row, dtype=_dt(case), device=DEV)
        state[tag] = flat
        off = 0
        for a in mine:
            a.into(flat[off:off + a.total * row].view(a.q.shape))
            off += a.total * row
    return state


def run(state):
    case, cache = state["case"], state["cache"]
    stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] in ("decode", "prefill"):
        call = state["call"]
        call.attend(cache, stream, case["per_layer"])
        return call.out
    cache.release(state["sessions"])
    evicts = 0
    for a in state["calls"]:
        if not isinstance(a, _Append):
            cache.evict(state["sessions"], state["resident"][evicts])
            evicts += 1
        elif a.tag == "history":
            a.feed(cache, stream, True)
        else:
            a.feed(cache, stream, not case["per_layer"])
            a.attend(cache, stream, case["per_layer"])
    if case["kind"] == "unit":
        return {"prefill": state["prefill"], "decode": state["decode"],
                "resident": state["resident"]}
    got = [cache.export_transcript(s, _room(case)) for s in range(case["n"])]
    return {"resident": state["resident"], "transcripts": got}


# -- what a pass cannot do without -------------------------------------------------------------
def _resident(case, fed, units):
    """Expected resident positions of a session after `fed` positions in `units` units."""
    if case["budget"] < 0:
        return fed
    return min(fed, max(case["budget"], KEPT_PER_UNIT * units + 19 * case["window"]))


def work(case):
    n, esz, d = case["n"], 2 if case["dtype"] == "bf16" else 4, _dim(case)
    row = case["layers"] * case["heads"] * d * esz     # K (or V) of one position, all layers
    units = case["units"] * (0.875 if case["kind"] in ("decode", "prefill", "restore") else 1.0)
    fed = units * PER_UNIT
    res = _resident(case, fed, units)

    def attention(queries, keys, new):
        """bytes and flops of `queries` tokens of one session over `keys` positions (the
        `new` last ones handed over by the call itself when it writes its layer)."""
        b = 2 * keys * row + 2 * queries * 4 * row + (2 * new * row if case["per_layer"] else 0)
        return b, 4.0 * queries * keys * 4 * case["heads"] * d * case["layers"]

    if case["kind"] in ("decode", "prefill"):
        t = 1 if case["kind"] == "decode" else (case["tokens"] + 1) / 2 if case["ragged"] else case["tokens"]
        new = t
        keys = res + (UNIT_POSITIONS + 1 if case["kind"] == "decode" else t)
        b, f = attention(t, keys, new)
        return {"bytes": n * b, "flops": n * f}
    if case["kind"] == "restore":
        kept = 3.0 * units
        return {"bytes": n * (4 * fed * row + 4 * kept * row), "flops": 0}
    total_b, total_f = 4 * fed * row, 0.0
    for step in range(case["steps"]):
        keys = _resident(case, fed, units) + UNIT_POSITIONS
        b, f = attention(UNIT_POSITIONS, keys, 0)
        total_b += b + 4 * UNIT_POSITIONS * row
        total_f += f
        for r in range(5):
            b, f = attention(1, keys + r + 1, 0)
            total_b += b + 4 * row
            total_f += f
        fed, units = fed + PER_UNIT, units + 1
    return {"bytes": n * total_b, "flops": n * total_f}


def tolerance(case):
    """About four times what the calls are off exact().  bfloat16 (K stored rotated and
    rounded, q and the probabilities rounded for the tensor cores, outputs rounded): 3.4e-3,
    largest 0.032 of the root mean square.  binary32: 3.7e-7, largest 4e-6.  Stored keys
    read back: 1.7e-3, largest 4e-3 (bfloat16), 3.6e-8 (binary32)."""
    bf16 = case["dtype"] == "bf16"
    if case["kind"] == "restore":
        return {"rel": 6e-3, "max": 1.6e-2} if bf16 else {"rel": 1.5e-7, "max": 1e-6}
    return {"rel": 1e-2, "max": 0.1} if bf16 else {"rel": 2e-6, "max": 2e-5}


# -- the same in 64 bits -------------------------------------------------------------------------
def _rotate(x, pos):
    """Rotate-half RoPE of x [positions][heads][D] in binary64."""
    d = x.shape[-1]
    theta = BASE ** (-2.0 * torch.arange(d // 2, dtype=torch.float64, device=DEV) / d)
    ang = torch.as_tensor(pos, dtype=torch.float64, device=DEV)[:, None, None] * theta
    c, s = torch.cos(ang), torch.sin(ang)
    a, b = x[..., :d // 2], x[..., d // 2:]
    return torch.cat([a * c - b * s, b * c + a * s], dim=-1)


def _attention(q, qpos, k, v, kpos):
    """q [t][4 H][D] un-rotated, k rotated and v [keys][H][D]: causal in positions."""
    t, hq, d = q.shape
    h = k.shape[1]
    qr = _rotate(q, qpos).view(t, h, 4, d).permute(1, 0, 2, 3).reshape(h, t * 4, d)
    s = torch.bmm(qr, k.permute(1, 2, 0)) / math.sqrt(d)
    after = torch.as_tensor(kpos, device=DEV)[None, :] > torch.as_tensor(qpos, device=DEV)[:, None]
    s.masked_fill_(after.repeat_interleave(4, dim=0)[None], -math.inf)
    o = torch.bmm(torch.softmax(s, dim=-1), v.permute(1, 0, 2))
    return o.view(h, t, 4, d).permute(1, 0, 2, 3).reshape(t, hq, d)


def exact(case, seed):
    n, layers = case["n"], case["layers"]
    streams, plan = _plan(case, seed)
    ops = [(at, op) for at, op in enumerate(plan) if op["op"] == "append"]
    # Row of each session's position in the layer's K/V of all appends, one after another.
    rows = [np.zeros(s.n, np.int64) for s in streams]
    base = 0
    for at, op in ops:
        for s, first, t in zip(op["sessions"], op["first"], op["types"]):
            rows[s][first:first + len(t)] = np.arange(base, base + len(t))
            base += len(t)
    resident = torch.tensor([[len(r) for r in op["res"]] for op in plan if op["op"] == "evict"],
                            dtype=torch.int64)

    def layer_kv(layer):
        kv = torch.cat([_kv(case, seed, at, layer, sum(len(t) for t in op["types"]))
                        for at, op in ops], dim=1)
        return kv

    def session_kv(kv, s, pos):
        x = kv[:, torch.as_tensor(rows[s][pos], device=DEV)].double()
        return _rotate(x[0], pos), x[1]

    if case["kind"] == "restore":
        keep = [s.res[s.type[s.res] == TRANSCRIPT] for s in streams]
        k = [[] for _ in streams]
        v = [[] for _ in streams]
        for layer in range(layers):
            kv = layer_kv(layer)
            for s in range(n):
                a, b = session_kv(kv, s, keep[s])
                k[s].append(a)
                v[s].append(b)
        room = _room(case)

        def padded(x):  # [layers][positions][heads][D], zeros after the last position
            out = torch.zeros((layers, room, *x[0].shape[1:]), dtype=torch.float64, device=DEV)
            out[:, :x[0].shape[0]] = torch.stack(x)
            return out

        pos = torch.zeros((n, room), dtype=torch.int32)
        for s in range(n):
            pos[s, :len(keep[s])] = torch.as_tensor(keep[s])
        return {"resident": resident, "transcripts": [
            (pos[s], padded(k[s]), padded(v[s]), torch.tensor([len(keep[s])], dtype=torch.int32))
            for s in range(n)]}

    attended = [(at, op) for at, op in ops if op["tag"] != "history"]
    qs = {at: _q(case, seed, at, sum(len(t) for t in op["types"])) for at, op in attended}
    outs = {at: torch.zeros(qs[at].shape, dtype=torch.float64, device=DEV) for at, _ in attended}
    for layer in range(layers):
        kv = layer_kv(layer)
        for s in range(n):
            # Everything that any of the pass's queries sees, rotated once.
            seen = np.unique(np.concatenate([op["res"][op["sessions"].index(s)]
                                             for _, op in attended if s in op["sessions"]]))
            k, v = session_kv(kv, s, seen)
            for at, op in attended:
                if s not in op["sessions"]:
                    continue
                i = op["sessions"].index(s)
                off = sum(len(t) for t in op["types"][:i])
                t = len(op["types"][i])
                pos = op["res"][i]
                pick = slice(None) if len(pos) == len(seen) else torch.as_tensor(
                    np.searchsorted(seen, pos), device=DEV)
                outs[at][layer, off:off + t] = _attention(
                    qs[at][layer, off:off + t].double(),
                    np.arange(op["first"][i], op["first"][i] + t), k[pick], v[pick], pos)
    if case["kind"] != "unit":
        return outs[attended[0][0]]
    return {tag: torch.cat([outs[at].reshape(-1) for at, op in attended if op["tag"] == tag])
            for tag in ("prefill", "decode")} | {"resident": resident}
