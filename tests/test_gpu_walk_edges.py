"""The walks over CSR rows where their windows, rings and batches end, against the oracle."""
import numpy as np
import pytest

from synth import kb as K, programs as P
from synth.rng import Rng
from tests import oracle_pins as pins
from tests.gpu_util import H, compare_batch, device_kb

pytestmark = pytest.mark.gpu

# row lengths around a warp's 32, three entries at a time, 96 a step of a long row, the 256-edge windows, three windows,
# and the 4,096 edges whose masks a lone walk keeps
LENGTHS = [0, 1, 2, 3, 4, 7, 8, 31, 32, 33, 34, 63, 64, 65, 95, 96, 97, 255, 256, 257, 511, 512, 513, 767, 768, 769, 1025,
           4095, 4096, 4097, 5000]


def _kb(n, seed, spread):
    """Two roles and a numeric role whose rows take LENGTHS (at most n), `spread` short rows between long ones."""
    r = np.random.default_rng(seed)
    deg = r.poisson(2.0, n)
    long = [x for x in LENGTHS if x <= n]
    at = np.arange(0, n, spread)[:len(long)] + (seed % 5)
    deg[at[at < n]] = np.array(long)[:np.count_nonzero(at < n)]
    deg = np.minimum(deg, n)
    edges = [[(a, int(b)) for a in range(n) for b in r.choice(n, deg[a], replace=False)],
             [(int(a), int(b)) for a, b in r.integers(0, n, (3 * n, 2))]]
    concepts = [np.nonzero(r.random(n) < p)[0].tolist() for p in (0.02, 0.3, 0.5, 0.97)]
    values = [(a, float(v)) for a in range(n) for v in r.integers(0, 3000, deg[a])]
    return K.from_arrays(n, concepts, edges, [], list(range(0, n, 7)), list(range(1, n, 7)), num_roles=[values])


def _restrictions(r, count, big):
    """Counting restrictions over few thresholds (bit-sliced ones up to 6; with big, any)."""
    out = []
    for k in range(count):
        op = ("some", "all", "min", "max", "exactly")[r.randint(0, 4)]
        n = "" if op in ("some", "all") else f"{r.randint(0, 6) if not big or r.random() < 0.5 else r.randint(7, 4200)} "
        out.append(P.compile_text(f"({op} {n}r{r.randint(0, 1)}{'-' if r.random() < 0.3 else ''} "
                                  f"{('A0', 'A1', 'A2', 'A3', '(not A1)', 'TOP')[r.randint(0, 5)]})"))
    return out


@pytest.mark.parametrize("n,spread", [(1, 1), (33, 1), (129, 4), (1000, 1), (6200, 1), (6200, 40), (6200, 200)])
def test_rows_of_every_length(n, spread):
    """Lone walks, bit-sliced walks of one and two words an individual, and concrete-role walks."""
    kb = _kb(n, 3 * n + spread, spread)
    dkb = device_kb(kb)
    r = Rng(n, spread)
    compare_batch(kb, dkb, _restrictions(r, 60, True), H.HEDL_NO_SLICE)
    compare_batch(kb, dkb, _restrictions(r, 24, False), H.HEDL_SLICE_ALL)     # at most 32 slices a group
    compare_batch(kb, dkb, _restrictions(r, 300, False))                       # over 32 in some
    compare_batch(kb, dkb, [P.compile_text(f"({op} p0 {t})") for op in ("ge", "le", "eq") for t in (-1, 0, 1500, 2999, 4000)])
    for p in _restrictions(r, 12, True):                                       # one at a time: narrow tiles
        want, _ = compare_batch(kb, dkb, [p], 0)
        assert np.array_equal(want, compare_batch(kb, dkb, [p], H.HEDL_LEVELS)[0])


@pytest.mark.parametrize("skew", [1, 2, 3])
def test_rows_at_unaligned_addresses(skew):
    """Row pointers and successors that start 4, 8 and 12 bytes after a 16-byte boundary: the copies of 4 bytes."""
    import torch
    kb = _kb(2500, 11 + skew, 60)
    ref = device_kb(kb)
    keep = []

    def shifted(t):
        raw = torch.zeros(t.numel() + 4, dtype=t.dtype, device=t.device)
        keep.append(raw)
        raw[skew:skew + t.numel()] = t
        return raw[skew:skew + t.numel()]
    dkb = device_kb(kb)
    dkb.handle = H.hedl_kb_load(kb.n, ref.concepts, [(shifted(a), shifted(b)) for a, b in ref.roles],
                                [(shifted(a), shifted(b)) for a, b in ref.inv_roles], None,
                                num_roles=[(shifted(a), shifted(b)) for a, b in ref.num_roles])
    H.hedl_examples_set(dkb.handle, ref.pos, ref.neg)
    r = Rng(skew, 5)
    for flags in (0, H.HEDL_NO_SLICE, H.HEDL_SLICE_ALL):
        compare_batch(kb, dkb, _restrictions(r, 80, flags == H.HEDL_NO_SLICE), flags)
    compare_batch(kb, dkb, [P.compile_text("(and A2 (ge p0 2500))"), P.compile_text("(or A0 (eq p0 77))")])


@pytest.mark.parametrize("n", [40_000, 300_000])
def test_work_items_of_several_segments(n):
    """Batches large enough that a work item holds several segments (up to eight), with programs past the instructions
    and leaf rows that a work item keeps in shared memory; waiting restrictions in nested fillers."""
    kb = K.generate(K.CONFIGS["batch"].scaled(n, seed=5, n_concepts=30, n_roles=4, n_props=3, n_pos=900, n_neg=900))
    dkb = device_kb(kb)
    r = Rng(n, 1)
    progs = [np.array(pins.random_program(r, kb, r.randint(2, 6)).postfix(), np.uint64) for _ in range(700)]
    wide = "A0"
    for k in range(1, 24):
        wide = f"(or {wide} (and A{k} A{(k * 7) % 30}))"
    progs += [P.compile_text(wide), P.compile_text(f"(some r1 {wide})"), P.compile_text(f"(min 2 r1- (and (some r0 A3) {wide}))")]
    sample = list(range(0, len(progs), 40)) + list(range(700, 703))
    base, _ = compare_batch(kb, dkb, progs, 0, sample=sample)
    for flags in (H.HEDL_LEVELS, H.HEDL_NO_SLICE, H.HEDL_PLAIN):
        assert np.array_equal(base, dkb.score(*P.pack_batch(progs), flags)), flags


@pytest.mark.parametrize("stage", [0, 1])
@pytest.mark.parametrize("n,spread", [(33, 1), (1000, 1), (6200, 40)])
def test_lone_walks_in_blocks_of_eight_chunks(n, spread, stage):
    """Blocks of 256 edges: rows of every length, a batch of lone walks and one restriction at a time."""
    kb = _kb(n, 5 * n + spread, spread)
    dkb = device_kb(kb)
    H.hedl_tuning_set(dkb.handle, role_block=8, stage_fillers=stage)
    r = Rng(n, 3 + spread)
    compare_batch(kb, dkb, _restrictions(r, 60, True), H.HEDL_NO_SLICE)
    compare_batch(kb, dkb, _restrictions(r, 24, True))
    for p in _restrictions(r, 12, True):
        compare_batch(kb, dkb, [p], 0)
