"""Cases that time the framework through its public entry points.

Three groups stand for what a program does with the library: it evaluates
concepts over a knowledge base (one at a time, or a batch of hypotheses
scored against examples), it ranks candidates with the surrogate (encode,
forward, top-k), and it trains the surrogate.  Every input is drawn on the
GPU from the seed: knowledge bases with Poisson or capped Zipf out-degrees,
Bernoulli concepts, value columns with missing entries, numeric and string
concrete roles; hypotheses as random expression trees over all constructors.
"""
import math
import random
import struct

import numpy as np
import torch

import paper_2412_00802_gb300 as H

DEV = "cuda"
ATOM, NOT, AND, OR, SOME, ALL, MIN, MAX, EXACTLY, GE, LE, EQ, SEQ, CONTAINS = 1, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16
VALUES = 1000.0            # values of columns and numeric roles are uniform in [0, VALUES)
MISSING = 0.1              # share of individuals without a column value
EXAMPLES = 0.01            # share of individuals that are positive, and that are negative examples
N_STRINGS, N_PATTERNS = 100_000, 64
D = 512                    # the surrogate's width
TARGET_MAP = (0.6, 0.4, 0.1, 0.15, 4.0)
ADAM_LR = 2e-5             # the tail of a half-cosine decay from 2e-3


def listed():
    return [
        # one concept on a knowledge base of 10,000 individuals: an interactive query, all latency
        dict(name="eval_10k", kind="eval", n=10_000, concepts=50, roles=8, degree=3.0, law="poisson", props=4),
        # a first look at many hypotheses on that knowledge base: counts and instance sets of 1,000 small ones
        dict(name="score_10k", kind="score", n=10_000, concepts=50, roles=8, degree=3.0, law="poisson", props=4,
             hyps=1000, length=15, depth=4, share=0.0, sets=True),
        # one concept of nested restrictions over 10^7 individuals with heavy-tailed role degrees
        dict(name="eval_10m", kind="eval", n=10_000_000, concepts=200, roles=8, degree=8.0, law="zipf", props=4),
        # the batched workload: 4,096 uneven hypotheses with shared sub-concepts over 10^6 individuals
        dict(name="score_1m", kind="score", n=1_000_000, concepts=100, roles=16, degree=6.0, law="poisson", props=8,
             hyps=4096, length=40, depth=8, share=0.3, sets=False),
        # one batch of a beam search's refinements of 64 hypotheses, 4 * 10^6 individuals, heavy-tailed degrees
        dict(name="refine_4m", kind="refine", n=4_000_000, concepts=300, roles=32, degree=10.0, law="zipf", props=32,
             hyps=2048, beam=64),
        # restrictions over numeric and string roles with several values per individual: 3 on each of 8 roles
        dict(name="concrete_10m", kind="concrete", n=10_000_000, num_roles=4, num_values=4.0, str_roles=4,
             str_values=2.0),
        # structural encodings of a ranking round's candidates
        dict(name="encode_65536", kind="encode", rows=65_536),
        # predictions for a ranking round's candidates
        dict(name="forward_65536", kind="forward", rows=65_536),
        # predictions for what is left of a small search step after duplicates are dropped: few rows, an odd number
        dict(name="forward_1999", kind="forward", rows=1_999),
        # exact scores of a round and its best 5 %
        dict(name="rank_65536", kind="rank", rows=65_536),
        # steps late in the training on a full training set, in its batches, then the weights
        dict(name="train_4096", kind="train", rows=4_096, steps=16),
        # a search's online training on fewer candidates than its batch: a ragged batch, then the weights
        dict(name="train_1000", kind="train", rows=1_000, steps=16),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["eval", "score", "score", "refine", "concrete", "encode", "forward", "forward", "rank", "train"])
    law = rng.choice(["poisson", "zipf"])
    if kind == "eval":
        return dict(kind=kind, n=size(1_000, 10_000_000), concepts=rng.randint(5, 200), roles=rng.randint(2, 8),
                    degree=round(rng.uniform(2.0, 8.0), 2), law=law, props=rng.randint(1, 8))
    if kind == "score":
        return dict(kind=kind, n=size(2_000, 1_000_000), concepts=rng.randint(20, 100), roles=rng.randint(2, 16),
                    degree=round(rng.uniform(2.0, 6.0), 2), law=law, props=rng.randint(1, 8), hyps=size(16, 4_096),
                    length=rng.randint(5, 40), depth=rng.randint(3, 8), share=round(rng.uniform(0.0, 0.3), 2),
                    sets=False)
    if kind == "refine":
        return dict(kind=kind, n=size(50_000, 4_000_000), concepts=rng.randint(50, 300), roles=rng.randint(4, 32),
                    degree=round(rng.uniform(3.0, 10.0), 2), law=law, props=rng.randint(2, 32), hyps=size(256, 2_048),
                    beam=rng.choice([16, 32, 64]))
    if kind == "concrete":
        return dict(kind=kind, n=size(5_000, 10_000_000), num_roles=rng.randint(1, 4),
                    num_values=round(rng.uniform(1.0, 4.0), 2), str_roles=rng.randint(1, 4),
                    str_values=round(rng.uniform(0.5, 2.0), 2))
    if kind == "train":
        return dict(kind=kind, rows=size(256, 4_096), steps=rng.randint(4, 16))
    return dict(kind=kind, rows=size(200, 65_536))


# ---------------------------------------------------------------------------- knowledge bases
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _degrees(g, n, mean, law):
    if law == "poisson":
        return torch.poisson(torch.full((n,), mean, device=DEV), generator=g).to(torch.int64)
    # P(d) proportional to (d + s)^-2.2 on {0..cap}, s by bisection so that the mean degree is as stated
    cap = min(10_000, n // 4)
    d = np.arange(cap + 1, dtype=np.float64)
    lo, hi = 1e-3, 1e3
    for _ in range(60):
        s = math.sqrt(lo * hi)
        w = (d + s) ** -2.2
        lo, hi = (s, hi) if (w * d).sum() / w.sum() < mean else (lo, s)
    cdf = torch.from_numpy(np.cumsum(w / w.sum())).to(DEV, torch.float32)
    return torch.searchsorted(cdf, torch.rand(n, device=DEV, generator=g)).clamp_(max=cap)


def _row_ptr(rows, n):
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(rows, minlength=n), 0, out=rp[1:])
    return rp.to(torch.int32)


def _role(g, n, mean, law):
    """(row_ptr, col) of a role and of its inverse: distinct uniform targets, rows sorted."""
    deg = _degrees(g, n, mean, law)
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), deg)
    key = torch.unique(rows * n + torch.randint(0, n, (rows.numel(),), device=DEV, generator=g))
    rows, cols = key // n, key % n
    back = torch.sort(cols * n + rows)[0]
    inv_rows, inv_cols = back // n, back % n
    return (_row_ptr(rows, n), cols.to(torch.int32)), (_row_ptr(inv_rows, n), inv_cols.to(torch.int32))


def _pack(member):
    """bool [k][words * 32] -> int32 [k][words], least significant bit first."""
    w = torch.tensor([1, 2, 4, 8, 16, 32, 64, 128], dtype=torch.uint8, device=DEV)
    b = (member.to(torch.uint8).view(member.shape[0], -1, 8) * w).sum(-1, dtype=torch.uint8)
    return b.contiguous().view(torch.int32)


def _concepts(g, n, count):
    wp = H.hedl_row_words(n)
    out = torch.empty((count, wp), dtype=torch.int32, device=DEV)
    p = 0.01 + 0.49 * torch.rand(count, device=DEV, generator=g)
    step = max(1, 100_000_000 // (wp * 32))
    for c in range(0, count, step):
        m = torch.rand((min(step, count - c), wp * 32), device=DEV, generator=g) < p[c:c + step, None]
        m[:, n:] = False
        out[c:c + step] = _pack(m)
    return out


def _values(g, shape):
    return VALUES * torch.rand(shape, device=DEV, generator=g)


def _load(case, seed):
    """The knowledge base of a case, on the GPU and registered with its examples."""
    g, n = _gen(seed), case["n"]
    concepts = _concepts(g, n, case.get("concepts", 8))
    pairs = [_role(g, n, case["degree"], case["law"]) for _ in range(case.get("roles", 0))]
    props = None
    if case.get("props"):
        props = _values(g, (case["props"], (n + 3) // 4 * 4))
        props[torch.rand(props.shape, device=DEV, generator=g) < MISSING] = float("nan")

    def owners(mean):
        return torch.repeat_interleave(torch.arange(n, device=DEV), _degrees(g, n, mean, "poisson"))

    nums, strs, table, patterns = [], [], None, []
    for _ in range(case.get("num_roles", 0)):
        rows = owners(case["num_values"])
        nums.append((_row_ptr(rows, n), _values(g, (rows.numel(),))))
    for _ in range(case.get("str_roles", 0)):
        rows = owners(case["str_values"])
        ids = torch.randint(0, N_STRINGS, (rows.numel(),), device=DEV, generator=g).to(torch.int32)
        strs.append((_row_ptr(rows, n), ids))
    if strs:   # distinct strings of 3 to 10 letters over a 6-letter alphabet: the index in base 6, then a random tail
        r = np.random.default_rng(seed)
        text = np.full((N_STRINGS, 10), 0, np.uint8)
        for k in range(7):
            text[:, k] = 97 + (np.arange(N_STRINGS) // 6 ** k) % 6
        text[:, 7:] = 97 + r.integers(0, 6, (N_STRINGS, 3))
        lens = 7 + r.integers(0, 4, N_STRINGS)
        off = np.zeros(N_STRINGS + 1, np.int32)
        np.cumsum(lens, out=off[1:])
        chars = text[np.arange(10)[None, :] < lens[:, None]]
        table = (torch.from_numpy(off).to(DEV), torch.from_numpy(chars).to(DEV), N_STRINGS, int(off[-1]))
        patterns = [b""] + [bytes(97 + r.integers(0, 6, r.integers(1, 5)).astype(np.uint8)) for _ in range(N_PATTERNS - 1)]
    kb = H.hedl_kb_load(n, concepts, [f for f, _ in pairs], [i for _, i in pairs], props, num_roles=nums,
                        str_roles=strs, str_table=table, patterns=patterns)
    e = torch.rand((1, H.hedl_row_words(n) * 32), device=DEV, generator=g)
    e[:, n:] = 0.5
    H.hedl_examples_set(kb, _pack(e < EXAMPLES)[0], _pack(e > 1.0 - EXAMPLES)[0])
    return kb


# ---------------------------------------------------------------------------- hypotheses
def _insn(op, a=0, b=0, inverse=False):
    return op | int(inverse) << 8 | a << 16 | b << 32


def _bits(x):
    return struct.unpack("<I", struct.pack("<f", x))[0]


class _Trees:
    """Random concepts as postfix programs over a case's symbols."""

    def __init__(self, case, rng, share=0.0):
        self.c, self.r, self.share, self.pool = case, rng, 0.0, []
        if share:
            self.pool = [self.uneven(9, 4) for _ in range(256)]
            self.share = share

    def atom(self):
        return [_insn(ATOM, self.r.randrange(self.c["concepts"]))]

    def data(self):
        return [_insn(self.r.choice((GE, LE)), self.r.randrange(self.c["props"]), _bits(self.r.uniform(0, VALUES)))]

    def role(self, filler, ops=(SOME, ALL, MIN, MAX), role=None):
        op = self.r.choice(ops)
        b = self.r.randint(1, 4) if op in (MIN, MAX, EXACTLY) else 0
        role = self.r.randrange(self.c["roles"]) if role is None else role
        return filler + [_insn(op, role, b, self.r.random() < 0.5)]

    def leaf(self):
        return self.atom() if self.r.random() < 0.8 else self.data()

    def tree(self, length, depth):
        """A tree of this many instructions and at most this depth (length < 2 ** depth)."""
        r, most = self.r, 2 ** (depth - 1) - 1   # the most instructions that a child can hold
        if length == 1:
            return self.leaf()
        if self.pool and length <= 9 and r.random() < self.share:
            return list(r.choice(self.pool))
        if length == 2 or (length - 1 <= most and r.random() < 5 / 7):
            kid = self.tree(length - 1, depth - 1)
            return kid + [_insn(NOT)] if r.random() < 0.2 else self.role(kid)
        k = r.randint(max(1, length - 1 - most), min(most, length - 2))
        return self.tree(k, depth - 1) + self.tree(length - 1 - k, depth - 1) + [_insn(r.choice((AND, OR)))]

    def uneven(self, length, depth):
        """A tree of uniform length in 1..length and depth limit in 1..depth, among those that exist."""
        while True:
            n, d = self.r.randint(1, length), self.r.randint(1, depth)
            if d <= n < 2 ** d:
                return self.tree(n, d)


def _flat(progs):
    offs = np.zeros(len(progs) + 1, np.uint32)
    np.cumsum([len(p) for p in progs], out=offs[1:])
    return np.array([w for p in progs for w in p], np.uint64), offs


def _hypotheses(case, rng):
    if case["kind"] == "concrete":
        progs = []
        for q in range(case["num_roles"]):   # the case has no one-value properties: property q is numeric role q
            progs += [[_insn(ATOM, rng.randrange(8)), _insn(op, q, _bits(rng.uniform(0, VALUES))), _insn(AND)]
                      for op in (GE, LE, EQ)]
        for q in range(case["str_roles"]):
            progs += [[_insn(ATOM, rng.randrange(8)), _insn(op, q, rng.randrange(most)), _insn(AND)]
                      for op, most in ((SEQ, N_STRINGS), (CONTAINS, N_PATTERNS), (CONTAINS, N_PATTERNS))]
        return progs
    t = _Trees(case, rng, case.get("share", 0.0))
    if case["kind"] == "eval":   # three nested restrictions beside a fourth, over different roles where there are four
        roles = rng.sample(range(case["roles"]), min(4, case["roles"])) * 2
        x = t.atom() + t.atom() + [_insn(AND)]
        for k in range(3):
            x = t.role(x, (SOME, MIN), roles[k])
        y = t.role(t.atom(), role=roles[3]) + t.data() + [_insn(OR)]
        return [x + y + [_insn(rng.choice((AND, OR)))]]
    if case["kind"] == "score":
        return [t.uneven(case["length"], case["depth"]) for _ in range(case["hyps"])]
    beam = [t.tree(rng.randint(3, 12), 5) for _ in range(case["beam"])]
    progs = []
    for k in range(case["hyps"]):   # add a conjunct or a disjunct, or wrap in a restriction
        p = beam[k % len(beam)]
        u = rng.random()
        if u < 0.6:
            x = rng.random()
            more = t.atom() if x < 0.5 else t.data() if x < 0.8 else t.role(t.atom(), (SOME,))
            progs.append(p + more + [_insn(AND if u < 0.3 else OR)])
        else:
            progs.append(t.role(p, (SOME, ALL, MIN)))
    return progs


# ---------------------------------------------------------------------------- the surrogate
def _params(seed):
    r = np.random.default_rng(seed)
    lim = 1.0 / math.sqrt(D)
    parts = [r.uniform(-lim, lim, n).astype(np.float32) if w else np.zeros(n, np.float32)
             for n, w in ((D * D, 1), (D, 0), (D * D, 1), (D, 0), (2 * D, 1), (2, 0))]
    return np.concatenate(parts)


def _encodings(g, rows):
    """Counts scaled by 1/4, mostly zero, some negative, as the encoder gives them."""
    x = 0.25 * torch.poisson(torch.full((rows, D), 0.25, device=DEV), generator=g)
    return (x * (1 - 2 * (torch.rand((rows, D), device=DEV, generator=g) < 0.2))).to(torch.bfloat16)


def _candidates(case, seed):
    """Programs of a ranking round on the device: 512 shapes, every symbol and threshold drawn anew."""
    rng, r, rows = random.Random(seed), np.random.default_rng(seed), case["rows"]
    t = _Trees(dict(concepts=200, roles=32, props=16), rng)
    flat, offs = _flat([t.uneven(24, 7) for _ in range(512)])
    pick = r.integers(0, 512, rows)
    lens = (offs[1:] - offs[:-1])[pick].astype(np.int64)
    out = np.zeros(rows + 1, np.int64)
    np.cumsum(lens, out=out[1:])
    p = flat[np.repeat(offs[pick].astype(np.int64) - out[:-1], lens) + np.arange(out[-1])]
    op, m = p & np.uint64(0xFF), p.size
    keep = (p & np.uint64(0xFF0000FFFF)).astype(np.uint64)   # op, inverse flag, a cardinality's n
    atom = op | r.integers(0, 200, m).astype(np.uint64) << np.uint64(16)
    role = keep | r.integers(0, 32, m).astype(np.uint64) << np.uint64(16)
    thr = r.uniform(0, VALUES, m).astype(np.float32).view(np.uint32).astype(np.uint64)
    data = op | r.integers(0, 16, m).astype(np.uint64) << np.uint64(16) | thr << np.uint64(32)
    p = np.where(op == ATOM, atom, np.where((op >= SOME) & (op <= EXACTLY), role, np.where(op >= GE, data, p)))
    grid = np.sort(r.uniform(0, VALUES, (16, 15)).astype(np.float32), axis=1)
    stats = r.integers(-8, 9, 200 + 16 * 32).astype(np.int32)
    prior = r.uniform(0.4, 0.9, (rows, 2)).astype(np.float32)
    return [torch.from_numpy(a).to(DEV) for a in (p.view(np.int64), out.astype(np.int32), grid, prior, stats)]


def _network(seed):
    m = H.hedl_mlp_create(_params(seed))
    H.hedl_mlp_set_target_map(m, TARGET_MAP)
    return m


def _training_set(case, seed):
    g = _gen(seed)
    X = _encodings(g, case["rows"] * case["steps"])
    w = torch.randn((D, 2), device=DEV, generator=g) * 0.05
    T = torch.sigmoid(X.float() @ w + 0.1 * torch.randn((X.shape[0], 2), device=DEV, generator=g))
    return X.view(case["steps"], case["rows"], D), T.view(case["steps"], case["rows"], 2)


def _counts(case, seed):
    """Coverage counts of a round: few distinct accuracies, so that ties are met."""
    g, rows = _gen(seed), case["rows"]
    tp = torch.randint(0, 200, (rows,), device=DEV, generator=g)
    fp = torch.randint(0, 200, (rows,), device=DEV, generator=g)
    return torch.stack([tp, fp, 200 - tp, 200 - fp], 1).to(torch.int32)


# ---------------------------------------------------------------------------- the entry points of this file
def prepare(case, seed):
    kind, g = case["kind"], _gen(seed)
    if kind in ("eval", "score", "refine", "concrete"):
        kb = _load(case, seed)
        progs, offs = _flat(_hypotheses(case, random.Random(seed)))
        s = dict(kb=kb, progs=progs, offs=offs, n=len(offs) - 1)
        ws = H.hedl_workspace_size(kb, progs, offs)
        s["ws"] = torch.empty(ws, dtype=torch.uint8, device=DEV)
        if kind == "eval":
            s["out"] = torch.zeros(H.hedl_row_words(case["n"]), dtype=torch.int32, device=DEV)
        else:
            s["counts"] = torch.zeros((s["n"], 4), dtype=torch.int32, device=DEV)
            s["sets"] = torch.zeros((s["n"], H.hedl_row_words(case["n"])), dtype=torch.int32, device=DEV) \
                if case.get("sets") else None
    elif kind == "encode":
        progs, offs, grid, prior, stats = _candidates(case, seed)
        s = dict(progs=progs, offs=offs, grid=grid, prior=prior, stats=stats,
                 X=torch.empty((case["rows"], D), dtype=torch.bfloat16, device=DEV))
    elif kind == "forward":
        s = dict(mlp=_network(seed), X=_encodings(g, case["rows"]),
                 Y=torch.empty((case["rows"], 2), device=DEV),
                 ws=torch.empty(H.hedl_mlp_workspace_size(case["rows"]), dtype=torch.uint8, device=DEV))
    elif kind == "rank":
        rows = case["rows"]
        s = dict(counts=_counts(case, seed), scores=torch.empty((rows, 2), device=DEV),
                 idx=torch.empty(max(1, rows // 20), dtype=torch.int32, device=DEV),
                 ws=torch.empty(H.hedl_select_workspace_size(rows), dtype=torch.uint8, device=DEV))
    else:
        X, T = _training_set(case, seed)
        s = dict(mlp=_network(seed), X=X, T=T, loss=torch.zeros(case["steps"], device=DEV),
                 ws=torch.empty(H.hedl_mlp_workspace_size(case["rows"]), dtype=torch.uint8, device=DEV))
        for k in range(4):   # a network in the middle of its training: Adam has moments
            H.hedl_mlp_train_step(s["mlp"], X[k], T[k], 0.0, s["ws"])
    s["kind"] = kind
    return s


def run(s):
    kind = s["kind"]
    if kind == "eval":
        H.hedl_eval_concept(s["kb"], s["progs"], s["out"], s["ws"])
        return s["out"]
    if kind in ("score", "refine", "concrete"):   # new hypotheses are planned, then executed
        plan = H.hedl_plan_batch(s["kb"], s["progs"], s["offs"])
        if s["ws"].numel() < H.hedl_plan_info_get(plan)["workspace_bytes"]:
            raise RuntimeError("the workspace is too small")
        H.hedl_plan_execute(s["kb"], plan, s["counts"], s["sets"], s["ws"])
        return [s["counts"]] if s["sets"] is None else [s["counts"], s["sets"]]
    if kind == "encode":
        H.hedl_encode(s["progs"], s["offs"], s["X"], s["grid"], s["prior"], s["stats"], 200)
        return s["X"]
    if kind == "forward":
        H.hedl_mlp_forward(s["mlp"], s["X"], s["Y"], s["ws"])
        return s["Y"]
    if kind == "rank":
        H.hedl_scores_from_counts(s["counts"], s["scores"])
        H.hedl_select_top(s["scores"], s["idx"].numel(), s["idx"], s["ws"])
        return [s["scores"], s["idx"]]
    for k in range(s["X"].shape[0]):
        H.hedl_mlp_train_step(s["mlp"], s["X"][k], s["T"][k], ADAM_LR, s["ws"], s["loss"][k:k + 1])
    return [s["loss"], H.hedl_mlp_get(s["mlp"])[0]]


def work(case):
    """Inputs read once and outputs written once; operations of the surrogate's matrix products."""
    kind = case["kind"]
    if kind in ("encode", "forward", "rank", "train"):
        rows, params = case["rows"], 2 * D * D + 4 * D + 2
        if kind == "encode":   # about 12 instructions a program
            return dict(bytes=rows * (12 * 8 + 4 + 8 + 2 * D), flops=0)
        if kind == "forward":
            return dict(bytes=rows * (2 * D + 8) + 2 * params, flops=2 * rows * (2 * D * D + 2 * D))
        if kind == "rank":
            return dict(bytes=rows * (16 + 8 + 8) + 4 * (rows // 20), flops=0)
        # forward, both weight gradients and one activation gradient; weights and moments read and written
        return dict(bytes=case["steps"] * (rows * (2 * D + 8) + 24 * params),
                    flops=case["steps"] * 2 * rows * (5 * D * D + 6 * D))
    n = case["n"]
    row = 4 * ((n + 31) // 32)
    if kind == "eval":   # four restrictions, three concepts, one column, the result
        return dict(bytes=4 * (4 * n + 4 * n * case["degree"]) + 4 * row + 4 * n, flops=0)
    if kind == "concrete":
        per = case["num_roles"] * (1 + case["num_values"]) + case["str_roles"] * (1 + case["str_values"])
        return dict(bytes=4 * n * per + 10 * row + 48 * (case["num_roles"] + case["str_roles"]), flops=0)
    # every symbol that a large enough batch names: roles both ways, columns, concepts, examples
    hyps = case["hyps"]
    length = case.get("length", 16) / 2
    roles = min(2 * case["roles"], hyps * length / 4)
    named = min(case["concepts"], hyps * length / 2)
    cols = min(case["props"], hyps * length / 10)
    out = hyps * (16 + (row if case.get("sets") else 0))
    return dict(bytes=roles * 4 * n * (1 + case["degree"]) + cols * 4 * n + (named + 2) * row + out, flops=0)


# ---------------------------------------------------------------------------- 64-bit values
def _split(p):
    out, o = [], 0
    for shape in ((D, D), (D,), (D, D), (D,), (2, D), (2,)):
        n = math.prod(shape)
        out.append(p[o:o + n].view(shape))
        o += n
    return out


def exact(case, seed):
    kind, g = case["kind"], _gen(seed)
    if kind == "rank":
        c = _counts(case, seed).double()
        acc, den = (c[:, 0] + c[:, 3]) / c.sum(1), 2 * c[:, 0] + c[:, 1] + c[:, 2]
        return [torch.stack([acc, torch.where(den > 0, 2 * c[:, 0] / den.clamp(min=1), torch.zeros_like(den))], 1), None]
    if kind not in ("forward", "train"):
        return None
    p = torch.from_numpy(_params(seed)).to(DEV).double()
    mean, scale = (torch.tensor(TARGET_MAP[k:k + 2], dtype=torch.float32, device=DEV).double() for k in (0, 2))

    def forward(w, x):   # products with weights rounded to bfloat16, as the network is defined
        w1, b1, w2, b2, w3, b3 = w
        w1, w2, w3 = (v.float().to(torch.bfloat16).double() for v in (w1, w2, w3))
        a1 = (x @ w1.T + b1).clamp(min=0)
        a2 = (a1 @ w2.T + b2).clamp(min=0)
        return a1, a2, a2 @ w3.T + b3, w2, w3

    if kind == "forward":
        return forward(_split(p), _encodings(g, case["rows"]).double())[2] * scale + mean
    X, T = _training_set(case, seed)
    rows, steps = case["rows"], case["steps"]
    m, v, losses = torch.zeros_like(p), torch.zeros_like(p), []
    b1, b2 = (float(np.float32(b)) for b in (0.9, 0.999))
    for t, k in enumerate(list(range(4)) + list(range(steps)), 1):
        x, y = X[k].double(), (T[k].double() - mean) / scale
        a1, a2, u, w2, w3 = forward(_split(p), x)
        weight = 1 + TARGET_MAP[4] * y[:, :1].clamp(min=0)
        du = 2 * weight * (u - y) / rows
        d2 = (du @ w3) * (a2 > 0)
        d1 = (d2 @ w2) * (a1 > 0)
        grad = torch.cat([z.reshape(-1) for z in (d1.T @ x, d1.sum(0), d2.T @ a1, d2.sum(0), du.T @ a2, du.sum(0))])
        m = b1 * m + (1 - b1) * grad
        v = b2 * v + (1 - b2) * grad * grad
        if t > 4:
            losses.append((weight * (u - y) ** 2).sum() / rows)
            p = p - ADAM_LR * (m / (1 - b1 ** t)) / ((v / (1 - b2 ** t)).sqrt() + 1e-8)
    return [torch.stack(losses), p]
