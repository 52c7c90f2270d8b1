"""The surrogate's kernels at the sizes where their tiles, chunks and registers end."""
import numpy as np
import pytest

from oracle import surrogate as S
from synth import programs as P
from tests import surrogate_bounds as SB

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2412_00802_gb300 import build
    build.build()
    import paper_2412_00802_gb300 as H
    from paper_2412_00802_gb300 import surrogate as sg
    return torch, H, sg


def _batch(B, seed):
    r = np.random.default_rng(seed)
    X = (0.25 * r.poisson(0.3, (B, 512)) * r.choice([-1, 1], (B, 512), p=[0.2, 0.8])).astype(np.float32)
    return X, r.uniform(size=(B, 2)).astype(np.float32)


# 64-row K blocks and grad_splits (64, 192), 128-row tiles, 32-row chunks of the output layer, one row
@pytest.mark.parametrize("B", [1, 31, 33, 64, 65, 127, 129, 192, 193, 1000])
def test_gradients_of_ragged_batches_on_tcgen05(env, B):
    """Every gradient element within the derived bound (tests/surrogate_bounds.py), from inputs that start
    16 bytes apart from an aligned address and from inputs that start 2 bytes after one."""
    torch, H, sg = env
    X, T = _batch(B, 100 + B)
    p = sg.init_params(3)
    ops = {}
    ref_loss, ref = S.backward(sg.split_params(p), X, T, rounding=True, operands=ops)
    tol = SB.gradient_tolerances(ops)
    Td = torch.from_numpy(T).to("cuda")
    for shift in (0, 1):   # bf16 elements
        raw = torch.zeros(B * 512 + 8, dtype=torch.bfloat16, device="cuda")
        Xd = raw[shift:shift + B * 512].view(B, 512)
        Xd.copy_(torch.from_numpy(X))
        s = sg.Surrogate(p)
        loss = torch.full((1,), 7.0, device="cuda")
        H.hedl_mlp_gradients(s.mlp, Xd, Td, s._workspace(B), loss)
        H.hedl_mlp_status(s.mlp)
        _, g, _ = H.hedl_mlp_get(s.mlp)
        bad = SB.gradient_violations(sg.split_params(g), ref, tol)
        assert not bad, (shift, bad)
        assert abs(float(loss.item()) - ref_loss) <= 1e-3 * abs(ref_loss)


# tiles of 64, 128 and 256 columns, their first and last sizes; a row tile that ends in its first or a later warp
@pytest.mark.parametrize("B", [1, 31, 33, 129, 3584, 3585, 7168, 7169, 7267, 20001])
def test_forward_of_every_tile_shape(env, B):
    """Predictions within test_gpu_surrogate.py's bf16 bounds of the oracle, also for a batch's last rows alone."""
    torch, H, sg = env
    X, _ = _batch(B, 7)
    p = sg.init_params(4)
    s = sg.Surrogate(p)
    Xd = torch.from_numpy(X).to("cuda").to(torch.bfloat16)
    Y = s.predict(Xd).cpu().numpy()
    H.hedl_mlp_status(s.mlp)
    ref, _ = S.forward(sg.split_params(p), X, rounding=True)
    scale = max(1.0, np.abs(ref).max())
    assert np.abs(Y - ref).max() <= 2e-2 * scale
    assert np.abs(Y - ref).mean() <= 2e-3 * max(1.0, np.abs(ref).mean())
    few = s.predict(Xd[-64:].contiguous()).cpu().numpy()
    assert np.abs(Y[-64:] - few).max() <= 2e-2 * scale


# one cluster block's share of 8,192 keys and its neighbours; several tiles a block; all, one and half wanted
@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 1023, 8192, 65535, 65536, 65537, 200001])
@pytest.mark.parametrize("kind", ["ties", "distinct", "equal", "wild"])
def test_select_top_at_the_edges(env, n, kind):
    torch, H, sg = env
    r = np.random.default_rng(n)
    if kind == "ties":
        Y = (r.integers(0, 7, (n, 2)) / 7).astype(np.float32)
    elif kind == "distinct":
        Y = r.uniform(-1, 1, (n, 2)).astype(np.float32)
    elif kind == "equal":
        Y = np.full((n, 2), 0.25, np.float32)
    else:   # every bit pattern class: both signs, infinities, NaN, denormals, zeros
        pool = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1e-42, -1e-42, 1.0, -1.0, 3e38], np.float32)
        Y = pool[r.integers(0, len(pool), (n, 2))]
    u = Y.view(np.uint32).astype(np.uint64)
    key = np.where(np.isnan(Y), np.uint64(0),
                   np.where(u >> np.uint64(31), ~u & np.uint64(0xFFFFFFFF), u | np.uint64(0x80000000)))
    order = np.lexsort((np.arange(n), ~key[:, 1], ~key[:, 0]))
    Yd = torch.from_numpy(Y).to("cuda")
    for k in sorted({1, (n + 1) // 2, max(1, n // 20), n}):
        got = sg.Surrogate().select(Yd, k).cpu().numpy().view(np.uint32)
        assert np.array_equal(got, np.sort(order[:k])), k


@pytest.mark.parametrize("scale", [1, 1 << 12, 1 << 23, (1 << 30) - 1])
def test_scores_of_small_and_large_counts(env, scale):
    """The float quotient below 2^24 and the double one above give the double quotient rounded to float."""
    torch, H, sg = env
    r = np.random.default_rng(scale)
    c = np.concatenate([r.integers(0, scale + 1, (4000, 4)), np.full((1, 4), scale), np.zeros((1, 4), np.int64),
                        [[0, 0, 0, scale]], [[scale, 0, 0, 0]]]).astype(np.uint32)
    got = torch.empty((len(c), 2), device="cuda")
    H.hedl_scores_from_counts(torch.from_numpy(c.view(np.int32)).to("cuda"), got)
    d = c.astype(np.float64)
    with np.errstate(invalid="ignore"):
        acc = np.where(d.sum(1) > 0, (d[:, 0] + d[:, 3]) / d.sum(1), 0)
        f1 = np.where(2 * d[:, 0] + d[:, 1] + d[:, 2] > 0, 2 * d[:, 0] / (2 * d[:, 0] + d[:, 1] + d[:, 2]), 0)
    assert np.array_equal(got.cpu().numpy(), np.stack([acc, f1], 1).astype(np.float32))


def _program(r, n):
    """A random program of n instructions, left, right and unary chains mixed."""
    prog = [P.insn(P.ATOM, 0, int(r.integers(0, 300)))]
    while len(prog) < n:
        u = r.random()
        leaf = P.insn(P.ATOM, 0, int(r.integers(0, 300))) if r.random() < 0.7 else \
            P.insn(int(r.choice([P.DGE, P.DLE, P.DEQ])), 0, int(r.integers(0, 6)), P.f32_bits(float(r.normal())))
        op = P.insn(int(r.choice([P.AND, P.OR])))
        if u < 0.3 and len(prog) + 2 <= n:
            prog = prog + [leaf, op]
        elif u < 0.6 and len(prog) + 2 <= n:
            prog = [leaf] + prog + [op]
        elif u < 0.75:
            prog.append(P.insn(P.NOT))
        else:
            prog.append(P.insn(int(r.choice([P.EXISTS, P.FORALL, P.ATLEAST, P.ATMOST, P.EXACTLY])), int(r.integers(0, 2)),
                               int(r.integers(0, 40)), int(r.integers(0, 9))))
    return np.array(prog, np.uint64)


def test_encoder_at_register_edges(env):
    """Lengths around 32 and 64 instructions (one and two registers a lane) and around the 256 that are encoded;
    rows that start 2 bytes after an aligned address; a program that leaves two operands."""
    torch, H, sg = env
    r = np.random.default_rng(5)
    progs = [_program(r, n) for n in (1, 2, 31, 32, 33, 63, 64, 65, 96, 255, 256, 257, 400) for _ in range(4)]
    grid = np.sort(r.normal(size=(6, 15)).astype(np.float32), axis=1)
    atoms, thr = r.integers(-9, 10, 300), r.integers(-9, 10, (6, 2, 16))
    want = S.encode_batch(progs, grid, None, (atoms, thr))
    # two programs in one: the second is encoded as such, the first one's single atom counts at depth 0
    two = np.concatenate([[np.uint64(P.insn(P.ATOM, 0, 5))], progs[8]])
    extra = S.encode(progs[8], grid, None, (atoms, thr)).astype(np.float64)
    for at, v in ((0, 1), (504, 1), (84 + 5, 1), (497, int(atoms[5])), (493 + min(len(two) - 1, 39) // 10, -1),
                  (493 + min(len(two), 39) // 10, 1)):
        extra[at] += 0.25 * v
    flat, offs = P.pack_batch(progs + [two])
    s = sg.Surrogate(grid=grid)
    s.stats = torch.from_numpy(np.concatenate([atoms, thr.reshape(-1)]).astype(np.int32)).to("cuda")
    s.n_stat_concepts = 300
    want = S.bf16(np.concatenate([want, extra.astype(np.float32)[None]]))   # what a bf16 row holds
    assert np.array_equal(s.encode(flat, offs).float().cpu().numpy(), want)
    raw = torch.zeros(len(want) * 512 + 8, dtype=torch.bfloat16, device="cuda")
    X = raw[1:1 + len(want) * 512].view(-1, 512)
    H.hedl_encode(torch.from_numpy(flat.view(np.int64)).to("cuda"), torch.from_numpy(offs.view(np.int32)).to("cuda"), X,
                  s.grid, None, s.stats, 300)
    assert np.array_equal(X.float().cpu().numpy(), want)
