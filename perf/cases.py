"""The work that users of this library have it do, as cases that can be timed
and compared: whole global steps of a parameter server (push the workers'
messages, apply them), and pulls of embedding rows, through the C ABI of
include/gba.h as its ctypes binding gives it.

A case is a dict of plain values:
  M, B        messages per global batch and local batch of a message
  ragged      local batches of B/2 .. B instead of B
  rows, dims, fields, per   per table, as texts "a,b,...": its rows, its width,
              the feature fields that look it up, and ids per field and sample
              (0: one id; else the Poisson mean)
  zipf        exponent of the ids' popularity law
  ids         "direct", "modulo" (hashed 64-bit ids folded into the rows) or
              "hash" (expandable hash table of 64-bit ids)
  opt, dense_opt            "adagrad" or "adam", of the tables / dense parameters
  D           dense parameters
  stale       staleness of the messages: "fresh", "geometric:mean:stragglers"
              (stragglers lag 5 .. 20 steps) or "pareto:alpha"
  iota, row_staleness, den, decay, drop_latest   the staleness rule
  push        "ref" (device buffers by reference), "copy" (device buffers) or
              "host" (pinned host buffers)
  eager       dense gradients summed at push time
  overlap     consecutive steps may overlap; a step's results are then there
              after a join or a synchronisation
  pulls       messages whose rows are pulled after the step (0: none)
  kind        "step", or "pull" for pulls alone

A program that trains has a server that has been running for a while: the
state is overwritten as from a checkpoint (weights, optimizer state and the
rows' step tags), and the step counter stands at START, so that staleness is
real from the first pass.  Every pass pushes the same messages with tokens that
lag the current step by the messages' staleness.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2205_11048_gb300 import binding as B

START = 24  # global steps applied before the first pass
MODES = {"direct": 0, "modulo": 1, "hash": 2}
OPTS = {"adagrad": 0, "adam": 1}
LR = {"adagrad": 0.01, "adam": 0.001}
B1, B2, EPS, ACC0 = 0.9, 0.999, 1e-8, 0.1
LAMBDA = 0.8

BASE = dict(kind="step", M=32, B=1024, ragged=False, rows="100000", dims="16", fields="26", per="0",
            zipf=1.05, ids="direct", opt="adagrad", dense_opt="adam", D=200_000,
            stale="geometric:1:0.1", iota=4, row_staleness=0, den=0, decay=0, drop_latest=0,
            push="ref", eager=False, overlap=False, pulls=0)


def _case(name, **kw):
    c = dict(BASE, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a small model on few workers: the time is the call's and the launches'
        _case("tiny", M=4, B=256, zipf=1.1, dense_opt="adagrad", stale="fresh"),
        # a click model with one-hot fields and one shared table
        _case("onehot-1e7x32", rows="10000000", dims="32", D=1_000_000),
        # sequence features: many ids per sample, four tables
        _case("multihot-4x1.25e7x16", M=64, rows=",".join(["12500000"] * 4), dims="16,16,16,16",
              fields="25,25,25,25", per="20,20,20,20", zipf=1.2, D=2_000_000, stale="geometric:2:0"),
        # a large dense network beside a small table
        _case("dense-heavy-64M", M=16, rows="1000000", dims="64", fields="40", D=64_000_000,
              stale="pareto:1.5"),
        # many workers, a large table of hashed ids, steps in flight one after another
        _case("large-5e7x64-overlap", M=128, rows="50000000", dims="64", fields="40", ids="modulo",
              D=8_000_000, stale="geometric:3:0.2", overlap=True),
        # 64-bit ids without a vocabulary: a step, then each worker's rows are pulled
        _case("hash-ids-step-pull", M=32, rows="8388608", dims="64", fields="40", ids="hash",
              D=2_000_000, stale="geometric:2:0.1", pulls=32),
        # dense gradients summed as they arrive, to hold few of them
        _case("eager-dense-16M", M=32, B=512, rows="2000000", dims="32", D=16_000_000, eager=True),
        # gradients that arrive in the host's memory
        _case("host-push-1e7x32", M=16, rows="10000000", dims="32", D=1_000_000, push="host"),
        # odd widths, uneven batches, weights that decay, Adam rows, late messages ignored
        _case("odd-widths-decay-copy", M=24, B=768, ragged=True, rows="1000003,200003,50021",
              dims="18,7,33", fields="12,9,5", per="0,3,0", opt="adam", D=300_007, decay=1, iota=6,
              row_staleness=1, den=1, drop_latest=2, push="copy"),
        # a table for each field
        _case("16-tables-1e5x16", M=8, B=512, rows=",".join(["100000"] * 16),
              dims=",".join(["16"] * 16), fields=",".join(["1"] * 16), per=",".join(["0"] * 16),
              D=400_000, zipf=1.1),
        # wide embeddings with Adam, averaged over all messages
        _case("wide-2e6x256-adam", M=32, B=512, rows="2000000", dims="256", fields="20", opt="adam",
              D=2_000_000, den=2, zipf=1.1),
        # one worker asks for the rows of its batch
        _case("pull-40960x64", kind="pull", M=1, rows="20000000", dims="64", fields="40", D=0,
              pulls=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("small", "mid", "mid", "large", "dense", "multihot", "odd", "tables", "wide", "hash",
                       "eager", "host", "pull"))
    stale = rng.choice(("fresh", "geometric:1:0.1", "geometric:2:0", "geometric:3:0.2", "pareto:1.5"))
    zipf = round(rng.uniform(1.02, 1.25), 3)
    c = _case(None, zipf=zipf, stale=stale, iota=rng.randrange(1, 9), dense_opt=rng.choice(("adagrad", "adam")),
              opt=rng.choice(("adagrad", "adagrad", "adam")), D=_log(rng, 5_000, 4_000_000),
              M=_log(rng, 2, 96), B=_log(rng, 32, 1024), rows=str(_log(rng, 2_000, 20_000_000)),
              dims=str(4 * _log(rng, 1, 32)), fields=str(_log(rng, 2, 48)),
              ids=rng.choice(("direct", "modulo")), push=rng.choice(("ref", "ref", "copy")),
              ragged=rng.random() < 0.3, overlap=rng.random() < 0.3, den=rng.randrange(3))
    if kind == "small":
        c.update(M=_log(rng, 1, 8), B=_log(rng, 16, 256), D=_log(rng, 64, 200_000),
                 rows=str(_log(rng, 500, 200_000)), dims=str(rng.randrange(4, 40)))
    elif kind == "large":
        c.update(M=_log(rng, 48, 128), B=1024, rows=str(_log(rng, 5_000_000, 40_000_000)), dims="64",
                 fields=str(rng.randrange(16, 41)), opt="adagrad", ids="modulo", push="ref")
    elif kind == "dense":
        c.update(M=_log(rng, 4, 32), D=_log(rng, 4_000_000, 32_000_003), rows=str(_log(rng, 10_000, 1_000_000)),
                 push="ref")
    elif kind == "multihot":
        t = rng.randrange(1, 5)
        c.update(M=_log(rng, 4, 32), rows=",".join(str(_log(rng, 100_000, 10_000_000)) for _ in range(t)),
                 dims=",".join(str(4 * rng.randrange(2, 9)) for _ in range(t)),
                 fields=",".join(str(rng.randrange(2, 20)) for _ in range(t)),
                 per=",".join(str(rng.randrange(0, 21)) for _ in range(t)))
    elif kind == "odd":
        t = rng.randrange(1, 4)
        c.update(rows=",".join(str(_log(rng, 1_000, 2_000_000)) for _ in range(t)),
                 dims=",".join(str(_log(rng, 1, 130)) for _ in range(t)),
                 fields=",".join(str(rng.randrange(1, 16)) for _ in range(t)),
                 per=",".join(str(rng.randrange(0, 4)) for _ in range(t)),
                 decay=rng.randrange(2), row_staleness=rng.randrange(2), drop_latest=rng.randrange(3))
    elif kind == "tables":
        t = rng.randrange(6, 16)
        c.update(M=_log(rng, 2, 16), opt="adagrad",
                 rows=",".join(str(_log(rng, 1_000, 1_000_000)) for _ in range(t)),
                 dims=",".join(str(8 * rng.randrange(1, 5)) for _ in range(t)),
                 fields=",".join(str(rng.randrange(1, 4)) for _ in range(t)))
    elif kind == "wide":
        c.update(M=_log(rng, 4, 32), B=_log(rng, 64, 512), dims=str(4 * rng.randrange(33, 65)),
                 rows=str(_log(rng, 10_000, 2_000_000)))
    elif kind == "hash":
        c.update(M=_log(rng, 2, 32), ids="hash", rows=str(1 << rng.randrange(18, 23)),
                 overlap=False, ragged=False)
        c["pulls"] = c["M"]
    elif kind == "eager":
        c.update(M=_log(rng, 4, 32), D=_log(rng, 100_000, 16_000_001), eager=True)
    elif kind == "host":
        c.update(M=_log(rng, 2, 16), push="host", D=_log(rng, 5_000, 1_000_000))
    elif kind == "pull":
        c.update(kind="pull", M=_log(rng, 1, 32), D=0, ragged=False, overlap=False, push="ref",
                 dims=str(_log(rng, 1, 256)))
        c["pulls"] = c["M"]
    # every per-table text has the tables' number of entries
    t = len(c["rows"].split(","))
    for k in ("dims", "fields", "per"):
        v = c[k].split(",")
        c[k] = ",".join(v if len(v) == t else (v * t)[:t])
    # no more ids and gradients than the largest listed case has
    while _input_bytes(c) > 3e9 and c["M"] > 1:
        c["M"] = max(1, c["M"] // 2)
        c["pulls"] = min(c["pulls"], c["M"])
    c["drop_latest"] = min(c["drop_latest"], c["M"] - 1)
    return c


# ---- the inputs, from the seed alone ---------------------------------------------------

def _ints(text):
    return [int(v) for v in text.split(",")]


def _tables(c):
    return list(zip(_ints(c["rows"]), _ints(c["dims"]), _ints(c["fields"]), _ints(c["per"])))


def _mean_ids(c, t):
    """Expected ids of a whole global batch for one table."""
    _, _, fields, per = t
    return c["M"] * c["B"] * (0.75 if c["ragged"] else 1.0) * fields * (per or 1)


def _input_bytes(c):
    return sum(_mean_ids(c, t) * (8 + 4 * t[1]) for t in _tables(c)) + 4.0 * c["M"] * c["D"]


def _staleness(c, rs):
    kind, *p = c["stale"].split(":")
    M = c["M"]
    if kind == "fresh":
        s = np.zeros(M)
    elif kind == "geometric":
        s = rs.geometric(1.0 / (1.0 + float(p[0])), M) - 1
        s = np.where(rs.rand(M) < float(p[1]), rs.randint(5, 21, M), s)
    else:  # Pareto(x_m = 1), whole steps
        s = np.floor((1.0 - rs.rand(M)) ** (-1.0 / float(p[0]))) - 1
    return np.minimum(s, START).astype(np.int64)


def _wrap(v):
    v &= (1 << 64) - 1
    return v - (1 << 64) if v >> 63 else v


def _mix(x):
    """SplitMix64's output for state x (int64 tensors, wrapping)."""
    def shr(z, s):
        return (z >> s) & ((1 << (64 - s)) - 1)
    z = x + _wrap(0x9E3779B97F4A7C15)
    z = (z ^ shr(z, 30)) * _wrap(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * _wrap(0x94D049BB133111EB)
    return z ^ shr(z, 31)


def _gen(seed, tag):
    return torch.Generator(device="cuda").manual_seed((seed * 1_000_003 + tag * 7_919 + 12345) & ((1 << 62) - 1))


def _inputs(c, seed):
    """The step's messages: local batches, staleness, per table the ids and
    gradient rows of all messages in a row with the messages' offsets, and the
    dense gradients (padded to 16 bytes).  Ids follow a bounded power law over
    popularity ranks, every field with its own order of the rows."""
    rs = np.random.RandomState(seed & 0x7FFFFFFF)
    M = c["M"]
    batch = rs.randint((c["B"] + 1) // 2, c["B"] + 1, M) if c["ragged"] else np.full(M, c["B"])
    out = dict(batch=[int(b) for b in batch], stale=_staleness(c, rs), tables=[])
    for t, (V, d, fields, per) in enumerate(_tables(c)):
        counts = np.repeat(batch[:, None], fields, 1)
        if per:
            counts = rs.poisson(counts * float(per))
        off = np.concatenate([[0], np.cumsum(counts.sum(1))])
        n = int(off[-1])
        g = _gen(seed, 2 + t)
        field = torch.repeat_interleave(torch.arange(fields, device="cuda").repeat(M),
                                        torch.as_tensor(counts.reshape(-1), device="cuda"), output_size=n)
        p = 1.0 - c["zipf"]
        u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
        lo, hi = 0.5 ** p, (V + 0.5) ** p
        rank = (lo + u * (hi - lo)).pow_(1.0 / p).round_().clamp_(1, V).to(torch.int64)
        del u
        mul = []
        for _ in range(fields):
            a = int(rs.randint(1, 1 << 30)) % V or 1
            while math.gcd(a, V) != 1:
                a += 1
            mul.append(a)
        mul = torch.as_tensor(np.asarray(mul, np.int64), device="cuda")
        add = torch.as_tensor(rs.randint(0, 1 << 30, fields).astype(np.int64), device="cuda")
        salt = torch.as_tensor(rs.randint(0, 1 << 62, fields, dtype=np.int64), device="cuda")
        ids = (mul[field] * (rank - 1) + add[field]) % V if c["ids"] == "direct" else _mix(rank ^ salt[field])
        del rank, field
        rows = torch.empty(n, d, device="cuda").normal_(0.0, 0.01, generator=g)
        out["tables"].append(dict(ids=ids, rows=rows, off=[int(v) for v in off]))
    if c["D"]:
        out["dense"] = torch.empty(M, (c["D"] + 3) & ~3, device="cuda").normal_(0.0, 0.01, generator=_gen(seed, 1))
    return out


def _fill_state(w, s0, s1, tag, adam, gen):
    """A trained state: weights, optimizer state, the rows' step tags."""
    w.uniform_(-0.0625, 0.0625, generator=gen)
    if adam:
        s0.normal_(0.0, 1e-3, generator=gen)
        s1.uniform_(1e-7, 1e-5, generator=gen)
    else:
        s0.uniform_(ACC0, 2 * ACC0, generator=gen)
    if tag is not None:
        tag.random_(0, START + 1, generator=gen)


# ---- the server ------------------------------------------------------------------------

class _Memory:
    """Memory that a handle owns; a tensor over it keeps the handle."""

    def __init__(self, owner, ptr, shape, kind):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": shape, "typestr": kind, "data": (ptr, False), "version": 3}


def _view(g, p, shape, kind="<f4"):
    return torch.as_tensor(_Memory(g, p.value, shape, kind), device="cuda") if p.value else None


_STREAM = []


def _server(c, batch):
    """A handle on this program's stream, START steps old, and views of its state."""
    def opt(name):
        return B.opt_desc(OPTS[name], LR[name], ACC0, B1, B2, EPS)
    tables = []
    for V, d, fields, per in _tables(c):
        n = c["B"] * fields * (per or 1)
        tables.append((V, d, MODES[c["ids"]], int(n + 8 * math.sqrt(n) + 64) if per else n, opt(c["opt"])))
    D = c["D"]
    g = B.GBA(tables, D, opt(c["dense_opt"]), sum(batch), 2 * c["M"], iota=c["iota"],
              row_staleness=c["row_staleness"], sparse_denominator=c["den"], seed=7, stream=_STREAM[0],
              decay=c["decay"], lam=LAMBDA if c["decay"] else 1.0, drop_latest=c["drop_latest"])
    L, p = g.L, [ctypes.c_void_p() for _ in range(4)]
    if c["eager"]:
        g.set_eager_dense(True)
    zero = torch.zeros((D + 3) & ~3, device="cuda")
    none = (B.gba_sparse_grad * max(1, len(tables)))()
    for k in range(START):  # steps of one message that holds nothing
        B.check(L.gba_push_ref(g.h, k, none, zero.data_ptr() if D else None, sum(batch)), g.h)
        B.check(L.gba_try_apply(g.h), g.h)
    g.sync()
    views = []
    for t, (V, d, _, _) in enumerate(_tables(c)):
        B.check(L.gba_get_table(g.h, t, *[ctypes.byref(q) for q in p]), g.h)
        views.append([_view(g, q, (V, d)) for q in p[:3]] + [_view(g, p[3], (V,), "<i4")])
    B.check(L.gba_get_dense(g.h, *[ctypes.byref(q) for q in p[:3]]), g.h)
    views.append([_view(g, q, (D,)) for q in p[:3]] if D else None)
    if c["overlap"]:
        g.set_overlap(True)
    return g, views


def prepare(case, seed):
    c = dict(BASE, **case)
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    torch.cuda.set_stream(_STREAM[0])
    x = _inputs(c, seed) if c["kind"] == "step" else _inputs(dict(c, D=0), seed)
    g, views = _server(c, x["batch"])
    hashed = c["ids"] == "hash"
    if not hashed:  # rows of a hash table start from their ids
        for t in range(len(views) - 1):
            _fill_state(*views[t], c["opt"] == "adam", _gen(seed, 100 + t))
    if c["D"]:
        _fill_state(*views[-1], None, c["dense_opt"] == "adam", _gen(seed, 99))
    st = dict(g=g, x=x, tokens=[int(s) for s in x["stale"]])
    pulls = []
    for m in range(c["pulls"]):
        for t, tb in enumerate(x["tables"]):
            pulls.append((t, tb["ids"][tb["off"][m]:tb["off"][m + 1]]))
    st["pulls"] = pulls
    if c["kind"] == "pull":
        torch.cuda.synchronize()
        return st
    # the messages as the ABI takes them
    src = x
    if c["push"] == "host":
        src = dict(x, tables=[dict(tb, ids=tb["ids"].cpu().pin_memory(), rows=tb["rows"].cpu().pin_memory())
                              for tb in x["tables"]])
        if c["D"]:
            src["dense"] = x["dense"].cpu().pin_memory()
        st["x"] = src
    st["push"] = g.L.gba_push_ref if c["push"] == "ref" else g.L.gba_push
    st["messages"] = []
    for m in range(c["M"]):
        grads = []
        for tb, (_, d, _, _) in zip(src["tables"], _tables(c)):
            a, b = tb["off"][m], tb["off"][m + 1]
            grads.append(B.gba_sparse_grad(tb["ids"].data_ptr() + 8 * a if b > a else None, b - a,
                                           tb["rows"].data_ptr() + 4 * d * a if b > a else None))
        dense = ctypes.c_void_p(src["dense"][m].data_ptr()) if c["D"] else None
        st["messages"].append(((B.gba_sparse_grad * len(grads))(*grads), dense, x["batch"][m]))
    out = {}
    if not hashed:
        for t, v in enumerate(views[:-1]):
            out["table%d" % t] = {k: a for k, a in zip(("w", "s0", "s1", "tag"), v) if a is not None}
    if c["D"]:
        out["dense"] = {k: a for k, a in zip(("w", "s0", "s1"), views[-1]) if a is not None}
    st["state"] = out
    torch.cuda.synchronize()
    return st


def run(state):
    g = state["g"]
    out = {}
    if "push" in state:
        k, push, h = g.version(), state["push"], g.h
        for s, (grads, dense, b) in zip(state["tokens"], state["messages"]):
            rc = push(h, max(0, k - s), grads, dense, b)
            if rc:
                B.check(rc, h, "push")
        if g.try_apply() != 1:
            raise RuntimeError("the messages did not make a step")
        out.update(state["state"])
    if state["pulls"]:  # pull responding: the current rows of the workers' ids
        out["pulled"] = [g.pull(t, ids) for t, ids in state["pulls"]]
    return out


# ---- what a pass cannot do without -----------------------------------------------------

def _distinct(V, fields, n, zipf):
    """Expected distinct rows among n ids of `fields` fields over V rows each."""
    p, per = 1.0 - zipf, n / max(1, fields)
    edge = np.unique(np.concatenate([np.arange(min(V, 4096) + 1), np.geomspace(1, V, 400).astype(np.int64), [V]]))
    edge = edge[(edge >= 0) & (edge <= V)].astype(np.float64)
    cdf = ((edge + 0.5) ** p - 0.5 ** p) / ((V + 0.5) ** p - 0.5 ** p)
    width, mass = np.diff(edge), np.diff(cdf)
    one = float(np.sum(width * -np.expm1(-per * mass / width)))
    return V * -math.expm1(fields * math.log1p(-min(one / V, 1 - 1e-12)))


def _kept(c):
    """Expected share of the messages that the rule keeps."""
    kind, *p = c["stale"].split(":")
    if kind == "fresh":
        f = 1.0
    elif kind == "geometric":
        late = float(p[1])
        f = (1 - late) * (1 - (float(p[0]) / (1 + float(p[0]))) ** (c["iota"] + 1))
        f += late * min(1.0, max(0, c["iota"] - 4) / 16.0)
    else:
        f = 1 - (c["iota"] + 2.0) ** -float(p[0])
    return f * max(0, c["M"] - c["drop_latest"]) / c["M"]


def work(case):
    """Ids read once; kept gradient rows and dense gradients read once (all of
    them where they are handed over to be copied); the state of the rows that
    move and of the dense parameters read and written, with the rows' tags.
    Pulls: ids and rows read, rows written."""
    c = dict(BASE, **case)
    nbytes = flops = 0.0
    f = _kept(c)
    for V, d, fields, per in _tables(c):
        n = _mean_ids(c, (V, d, fields, per))
        pulled = n * c["pulls"] / c["M"]
        nbytes += pulled * (8 + 8.0 * d)
        if c["kind"] == "step":
            moved = _distinct(V, fields, n * f, c["zipf"])
            state = 3 if c["opt"] == "adam" else 2
            nbytes += 8 * n + 4.0 * d * n * (f if c["push"] == "ref" else 1) + moved * (8.0 * d * state + 8)
            flops += d * (n * f + 12 * moved)
    if c["kind"] == "step" and c["D"]:
        state = 3 if c["dense_opt"] == "adam" else 2
        nbytes += 4.0 * c["D"] * (c["M"] * (f if c["push"] == "ref" else 1) + 2 * state)
        flops += c["D"] * (c["M"] * f + 12.0)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Pulled rows are copies.  A step's sums are formed in float32 with
    compensation and its updates are a handful of float32 operations: against
    64 bits, the state after a step was measured within 4.2e-8 (2-norm), most of
    it the rounding of the results themselves."""
    return "exact" if case.get("kind") == "pull" else {"rel": 1.7e-7, "max": 4e-6}


# ---- the same in 64 bits -----------------------------------------------------------------

def _adagrad(w, s0, s1, g, lr, t):
    s0 = s0 + g * g
    return w - lr * g / s0.sqrt(), s0, s1


def _adam(w, s0, s1, g, lr, t):
    b1, b2 = float(np.float32(B1)), float(np.float32(B2))
    s0 = b1 * s0 + (1 - b1) * g
    s1 = b2 * s1 + (1 - b2) * g * g
    return w - lr * (s0 / (1 - b1 ** t)) / ((s1 / (1 - b2 ** t)).sqrt() + float(np.float32(EPS))), s0, s1


def _update(name, *a):
    return (_adam if name == "adam" else _adagrad)(*a, float(np.float32(LR[name])), START + 1)


def _weight(c, s):
    """Weights of gradients of staleness s (float64 tensor)."""
    f = (s <= c["iota"]).double()
    return f * float(np.float32(LAMBDA)) ** s.double() if c["decay"] else f


def _hash_rows(ids, d, t):
    """Initial weights of 64-bit ids in table t of a server with seed 7."""
    e = ids[:, None] * d + torch.arange(d, device="cuda")
    return (((_mix(e ^ (7 ^ ((t + 1) << 48))) >> 40) & 0xFFFFFF) - (1 << 23)).double() * 2.0 ** -27


def exact(case, seed):
    c = dict(BASE, **case)
    x = _inputs(c if c["kind"] == "step" else dict(c, D=0), seed)
    M, step = c["M"], c["kind"] == "step"
    stale = torch.as_tensor(x["stale"], device="cuda")
    out, pulled = {}, {}
    late = torch.arange(M, device="cuda") >= M - c["drop_latest"]
    for t, (tb, (V, d, _, _)) in enumerate(zip(x["tables"], _tables(c))):
        hashed, adam = c["ids"] == "hash", c["opt"] == "adam"
        if c["ids"] == "modulo":  # the unsigned value modulo V
            row = (tb["ids"] % V + torch.where(tb["ids"] < 0, (1 << 64) % V, 0)) % V
        else:
            row = tb["ids"]
        u, at = torch.unique(row, return_inverse=True)
        del row
        if hashed:
            w = _hash_rows(u, d, t)
            s0 = torch.full_like(w, 0.0 if adam else float(np.float32(ACC0)))
            s1 = torch.zeros_like(w) if adam else None
            tag = torch.zeros(u.numel(), dtype=torch.int32, device="cuda")
            where = torch.arange(u.numel(), device="cuda")
        else:
            w, s0 = torch.empty(V, d, device="cuda"), torch.empty(V, d, device="cuda")
            s1 = torch.empty(V, d, device="cuda") if adam else None
            tag = torch.empty(V, dtype=torch.int32, device="cuda")
            _fill_state(w, s0, s1, tag, adam, _gen(seed, 100 + t))
            w, s0, s1 = w.double(), s0.double(), s1.double() if adam else None
            where = u
        if not step:
            for m in range(c["pulls"]):
                pulled[m, t] = w[where[at[tb["off"][m]:tb["off"][m + 1]]]]
            continue
        off = torch.as_tensor(tb["off"], device="cuda")
        msg = torch.repeat_interleave(torch.arange(M, device="cuda"), off.diff(), output_size=tb["off"][-1])
        token = START - stale[msg]
        ref = START if c["row_staleness"] else tag[where[at]].long()
        f = _weight(c, (ref - token).clamp_(min=0))
        f[late[msg]] = 0.0
        pair = torch.unique(at * (2 * M) + msg * 2 + (f > 0))  # (row, message, kept)
        rows_of, kept = pair // (2 * M), (pair & 1).double()
        zeros = torch.zeros(u.numel(), dtype=torch.float64, device="cuda")
        kept_pairs = zeros.index_add(0, rows_of, kept)
        del token, ref, msg
        den = zeros.index_add(0, rows_of, torch.ones_like(kept)) if c["den"] == 0 else (
            kept_pairs if c["den"] == 1 else torch.full_like(zeros, M))
        total = torch.zeros(u.numel(), d, dtype=torch.float64, device="cuda")
        chunk = max(1, (1 << 27) // d)
        for a in range(0, at.numel(), chunk):
            b = slice(a, a + chunk)
            total.index_add_(0, at[b], tb["rows"][b].double().mul_(f[b, None]))
        del tb["rows"], f, pair, rows_of, kept
        mv = torch.nonzero(kept_pairs > 0)[:, 0]
        i = where[mv]
        grad = total[mv] / den[mv, None]
        del total
        nw, n0, n1 = _update(c["opt"], w[i], s0[i], s1[i] if adam else None, grad)
        w[i], s0[i], tag[i] = nw, n0, START + 1
        if adam:
            s1[i] = n1
        del nw, n0, n1, grad
        for m in range(c["pulls"]):
            pulled[m, t] = w[where[at[tb["off"][m]:tb["off"][m + 1]]]]
        if not hashed:
            out["table%d" % t] = {k: v for k, v in zip(("w", "s0", "s1", "tag"), (w, s0, s1, tag)) if v is not None}
    if step and c["D"]:
        D = c["D"]
        dw, d0, d1 = torch.empty(D, device="cuda"), torch.empty(D, device="cuda"), None
        if c["dense_opt"] == "adam":
            d1 = torch.empty(D, device="cuda")
        _fill_state(dw, d0, d1, None, d1 is not None, _gen(seed, 99))
        f = _weight(c, stale)
        f[late] = 0.0
        grad = torch.zeros(D, dtype=torch.float64, device="cuda")
        for m in range(M):
            grad.add_(x["dense"][m, :D].double(), alpha=float(f[m]))
        new = _update(c["dense_opt"], dw.double(), d0.double(), d1.double() if d1 is not None else None, grad / M)
        out["dense"] = {k: v for k, v in zip(("w", "s0", "s1"), new) if v is not None}
    if c["pulls"]:
        out["pulled"] = [pulled[m, t] for m in range(c["pulls"]) for t in range(len(x["tables"]))]
    return out
