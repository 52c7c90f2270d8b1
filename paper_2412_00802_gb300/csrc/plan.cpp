// Host planner: turns a batch of postfix hypothesis programs into the device
// work queue executed by the segment interpreter (exec.cu).
//
// The paper builds an evaluation plan (a query plan fixing the order of the
// DL operations and their inputs) for each hypothesis on the CPU before it
// runs (Section IV), multi-threaded across a batch (Section V).  Here the plan
// of a whole batch is one DAG:
//   1. every program is decoded and validated, and its nodes are hash-consed
//      into one DAG shared by the batch (common sub-concepts are evaluated
//      once; AND/OR operands are put in canonical order and NOT NOT X folds to
//      X, which changes no instance set);
//   2. a node is materialized as a full bitset ("slot") if it is the filler
//      of a role restriction (a role restriction reads its filler at
//      arbitrary individuals, so the filler must exist over all individuals
//      first) or if it is used twice or more and its inline expansion holds a
//      role restriction (so that work is done once);
//   3. every materialized node and every hypothesis root becomes a segment:
//      a role-free boolean program whose leaves are atoms, data ranges,
//      slots and role restrictions over slots or concept rows;
//   4. role restrictions that share a role, direction and stage (walk_stages)
//      with another one become bit-sliced role groups (up to 64 per group,
//      evaluated by one transposed-filler walk) instead of living inside a
//      segment;
//   5. tasks get levels (1 + the deepest producer of a slot they read) and
//      are grouped by (level, first role read); each group's work items are
//      (task, tile) pairs in tile-major order so that tasks sweeping the same
//      role stream the same CSR rows at about the same time;
//   6. the tile shape: 32 words per warp, or 16 / 8 / 4 with one round when a
//      level that walks a role holds too few tasks to fill the GPU.
#include <algorithm>
#include <cstring>
#include <utility>

#include "hedl_internal.h"

namespace hedl {

namespace {

struct PNode {
    uint8_t op;
    uint8_t inv;
    uint16_t pad;
    uint32_t a;
    uint32_t b;
    int32_t k0, k1;
};

// Hash-consing table: open addressing over node indices (no allocation a
// node; a batch of 4,096 hypotheses makes 50,000), keyed by the node's fields.
class NodeTable {
  public:
    explicit NodeTable(size_t n) {
        size_t cap = 64;
        while (cap < 2 * n) cap <<= 1;
        slots_.assign(cap, -1);
        mask_ = cap - 1;
    }
    // the index of a node equal to n, or -1 with *slot set to where insert puts it
    int32_t find(const PNode &n, const std::vector<PNode> &nodes, size_t *slot) const {
        for (size_t at = hash(n) & mask_;; at = (at + 1) & mask_) {
            const int32_t i = slots_[at];
            if (i < 0) {
                *slot = at;
                return -1;
            }
            const PNode &o = nodes[i];
            if (o.op == n.op && o.inv == n.inv && o.a == n.a && o.b == n.b && o.k0 == n.k0 && o.k1 == n.k1) return i;
        }
    }
    void insert(size_t slot, int32_t i) { slots_[slot] = i; }

  private:
    static size_t hash(const PNode &n) {
        const uint64_t x = (uint64_t)n.op | ((uint64_t)n.inv << 8) | ((uint64_t)n.a << 16) | ((uint64_t)n.b << 32);
        const uint64_t y = (uint64_t)(uint32_t)n.k0 | ((uint64_t)(uint32_t)n.k1 << 32);
        uint64_t h = x * 0x9E3779B97F4A7C15ull ^ (y + 0x632BE59BD9B4E019ull + (x << 6) + (x >> 2));
        h ^= h >> 31;
        h *= 0xBF58476D1CE4E5B9ull;
        return (size_t)(h ^ (h >> 29));
    }
    std::vector<int32_t> slots_;
    size_t mask_ = 0;
};

inline bool is_role(uint32_t op) { return op >= HEDL_OP_EXISTS && op <= HEDL_OP_EXACTLY; }
inline bool is_data(uint32_t op) { return op >= HEDL_OP_DGE && op <= HEDL_OP_DEQ; }
inline bool is_str(uint32_t op) { return op == HEDL_OP_SEQ || op == HEDL_OP_SCONTAINS; }
// Algorithmic bytes of a data restriction on property id a: a one-value
// column (4N), or a numeric role's row pointers and values (4(N+1) + 4M).
inline uint64_t data_bytes(const hedl_kb *kb, uint32_t a, uint64_t N) {
    if (a < kb->n_props) return 4 * N;
    return 4 * (N + 1) + 4ull * kb->num_host[a - kb->n_props].n_vals;
}
// ... and of a string restriction: the role's row pointers and ids, plus
// SCONTAINS's row of the containment bitmap.
inline uint64_t str_bytes(const hedl_kb *kb, uint32_t op, uint32_t a, uint64_t N) {
    return 4 * (N + 1) + 4ull * kb->str_host[a].n_vals + (op == HEDL_OP_SCONTAINS ? 4 * kb->contain_words : 0);
}

// operands of an op, -1 for an unknown one
struct Arity {
    int8_t of[256];
    constexpr Arity() : of() {
        for (int op = 0; op < 256; ++op) of[op] = -1;
        for (int op : {HEDL_OP_ATOM, HEDL_OP_TOP, HEDL_OP_BOT, HEDL_OP_DGE, HEDL_OP_DLE, HEDL_OP_DEQ, HEDL_OP_SEQ,
                       HEDL_OP_SCONTAINS})
            of[op] = 0;
        for (int op : {HEDL_OP_NOT, HEDL_OP_EXISTS, HEDL_OP_FORALL, HEDL_OP_ATLEAST, HEDL_OP_ATMOST, HEDL_OP_EXACTLY})
            of[op] = 1;
        of[HEDL_OP_AND] = of[HEDL_OP_OR] = 2;
    }
};
constexpr Arity ARITY;
inline int arity(uint32_t op) { return ARITY.of[op & 0xFF]; }

const char *op_name(uint32_t op) {
    static const char *names[] = {"?", "ATOM", "TOP", "BOT", "NOT", "AND", "OR", "EXISTS", "FORALL",
                                  "ATLEAST", "ATMOST", "EXACTLY", "DGE", "DLE", "DEQ", "SEQ", "SCONTAINS"};
    return op < 17 ? names[op] : "?";
}

}  // namespace

int validate_program(const hedl_kb *kb, const uint64_t *prog, uint32_t len, std::string *why) {
    if (len == 0) {
        *why = "empty program";
        return HEDL_ERR_BAD_PROGRAM;
    }
    int depth = 0;
    for (uint32_t k = 0; k < len; ++k) {
        uint64_t w = prog[k];
        uint32_t op = (uint32_t)(w & 0xFF);
        uint32_t a = (uint32_t)((w >> 16) & 0xFFFF);
        int ar = arity(op);
        char buf[160];
        if (ar < 0) {
            snprintf(buf, sizeof buf, "instruction %u: unknown op %u", k, op);
            *why = buf;
            return HEDL_ERR_BAD_PROGRAM;
        }
        if ((op == HEDL_OP_ATOM && a >= kb->n_concepts) || (is_role(op) && a >= kb->n_roles) ||
            (is_data(op) && a >= kb->n_props + kb->n_num) || (is_str(op) && a >= kb->n_str)) {
            snprintf(buf, sizeof buf, "instruction %u: %s names id %u, out of range", k, op_name(op), a);
            *why = buf;
            return HEDL_ERR_BAD_PROGRAM;
        }
        if (op == HEDL_OP_SCONTAINS && (uint32_t)(w >> 32) >= kb->n_patterns) {
            snprintf(buf, sizeof buf, "instruction %u: SCONTAINS names pattern %u, out of range", k,
                     (uint32_t)(w >> 32));
            *why = buf;
            return HEDL_ERR_BAD_PROGRAM;
        }
        if (depth < ar) {
            snprintf(buf, sizeof buf, "instruction %u: %s pops an empty stack", k, op_name(op));
            *why = buf;
            return HEDL_ERR_BAD_PROGRAM;
        }
        depth = depth - ar + 1;
        if (depth > HEDL_MAX_STACK) {
            snprintf(buf, sizeof buf, "instruction %u: more than %d operands on the stack", k, HEDL_MAX_STACK);
            *why = buf;
            return HEDL_ERR_BAD_PROGRAM;
        }
    }
    if (depth != 1) {
        *why = "program leaves " + std::to_string(depth) + " operands, not 1";
        return HEDL_ERR_BAD_PROGRAM;
    }
    return HEDL_OK;
}

uint64_t hash_programs(const uint64_t *progs, const uint32_t *offs, uint32_t H) {
    uint64_t h = 0xCBF29CE484222325ull ^ H;
    auto mix = [&](uint64_t v) {
        h ^= v + 0x9E3779B97F4A7C15ull + (h << 6) + (h >> 2);
        h *= 0x100000001B3ull;
    };
    for (uint32_t i = 0; i <= H; ++i) mix(offs[i]);
    for (uint32_t i = 0; i < offs[H]; ++i) mix(progs[i]);
    return h;
}

PlanImpl::~PlanImpl() = default;

namespace {

template <class T>
uint64_t put(std::vector<uint8_t> &img, const std::vector<T> &v) {
    uint64_t off = (img.size() + 255) & ~uint64_t(255);
    img.resize(off + v.size() * sizeof(T));
    if (!v.empty()) memcpy(img.data() + off, v.data(), v.size() * sizeof(T));
    return off;
}

// The stage (1, 2, ...) at which each bit-sliceable role restriction walks;
// 0 for every other node, and for all of them if none could share a walk (and
// all is false: lone ones are not sliced then).  A restriction may walk once
// those nested in its filler have (a stage later than all of them), and has to
// by the stage that leaves one stage for each restriction around it, in a plan
// of as many stages as the deepest nesting.  At each stage a role and direction
// walks if one of its ready restrictions cannot wait; then all its ready ones
// walk with it.  Otherwise only whole groups of SLICES * MAX_PARTS walk (waiting
// could not save their walk), the ones with the least time left first.  A role
// and direction of one or two restrictions does not wait: two lone walks over
// bitset fillers cost about as much as a shared one with its transpose.
// Walking every restriction as soon as it is ready (one group per role,
// direction and nesting depth) takes 231 walks for 2,048 refinements over 64
// roles and directions and 225 for a batch of 4,096 over 32; this takes 137
// and 177 (2,048 refinements at 4 * 10^6 individuals 57.3 -> 35.4 ms).  A plan
// may get more levels for it, without fewer walks in some batches of a few
// hypotheses.  Over 738 batches of 16 to 2,000 hypotheses on 10^4 to 4 * 10^6
// individuals waiting takes 0.85 to 0.93 of the time (geometric mean of each size
// and degree law), 0.90 also where it saves no walk and adds levels; one batch in
// nine gets more than 5 % slower, and neither the walks nor the levels tell which.
// key_of numbers the (stage, role, direction) triples 0, 1, ... by stage; key_size counts their restrictions.
//
// Each node is finished once, when its last operand is, and a role and
// direction is looked at only at the stages where a restriction of it becomes
// ready or due: the time grows with the batch, not with its depth or the KB's roles.
void walk_stages(const std::vector<PNode> &nodes, uint32_t n_roles, bool all, std::vector<uint32_t> &stage,
                 std::vector<uint32_t> &key_of, std::vector<uint32_t> &key_size) {
    constexpr uint32_t NONE = 0xFFFFFFFFu, WHOLE = SLICES * MAX_PARTS;
    const uint32_t NN = (uint32_t)nodes.size();
    // the nodes with a restriction in their expression, children first
    struct Inner {
        uint32_t node, role;       // role: key into roles; NONE: no sliceable restriction
        uint32_t kid[2];           // such nodes among the operands, or NONE
        uint32_t users, next[2];   // the nodes that read this one: 2 * reader + operand, linked through next
        uint16_t waits, step;      // operands that are not complete yet; 1 for a restriction
        uint32_t ready;            // the stage that completed the others, then this one
        uint32_t limit;            // the stage by which it has to be complete
        uint32_t link;             // the next of the restrictions that become ready with this one
    };
    struct Role {
        uint32_t total = 0, looked = 0, least = NONE;   // least: the smallest limit of the pending ones
        std::vector<uint32_t> pending;                  // ready restrictions that wait
    };
    // roles and directions by their number, unless the KB has far more than the batch can name
    const bool direct = 2ull * n_roles <= 4ull * NN + 64;
    std::vector<uint32_t> named;
    if (!direct) {
        for (const PNode &n : nodes)
            if (is_role(n.op)) named.push_back(2 * n.a + n.inv);
        std::sort(named.begin(), named.end());
        named.erase(std::unique(named.begin(), named.end()), named.end());
    }
    std::vector<Role> roles(direct ? 2 * (size_t)n_roles : named.size());
    std::vector<Inner> inner;
    std::vector<uint32_t> at(NN), depth;   // a node's place in inner or NONE; nesting depths by place
    inner.reserve(NN);
    depth.reserve(NN);
    uint32_t last = 0;
    bool shared = all;
    for (uint32_t i = 0; i < NN; ++i) {
        const PNode &n = nodes[i];
        const bool role = is_role(n.op);
        const uint32_t kid[2] = {n.k0 >= 0 ? at[n.k0] : NONE, n.k1 >= 0 ? at[n.k1] : NONE};
        at[i] = NONE;
        if (!role && kid[0] == NONE && kid[1] == NONE) continue;
        const uint32_t me = at[i] = (uint32_t)inner.size();
        Inner x{i, NONE, {kid[0], kid[1]}, NONE, {NONE, NONE}, 0, role, 0, 0, NONE};
        uint32_t d = 0;
        for (uint32_t k = 0; k < 2; ++k)
            if (kid[k] != NONE) {
                d = std::max(d, depth[kid[k]]);
                x.next[k] = std::exchange(inner[kid[k]].users, 2 * me + k);
                ++x.waits;
            }
        if (role && (n.op == HEDL_OP_EXISTS || n.op == HEDL_OP_FORALL || n.b <= SLICE_MAX_N)) {
            const uint32_t key = 2 * n.a + n.inv;
            x.role = direct ? key : (uint32_t)(std::lower_bound(named.begin(), named.end(), key) - named.begin());
            shared |= ++roles[x.role].total > 1;
        }
        depth.push_back(d + (role ? 1u : 0u));
        last = std::max(last, depth.back());
        inner.push_back(x);
    }
    if (!shared) return;
    for (Inner &x : inner) x.limit = last;
    for (size_t q = inner.size(); q-- > 0;) {
        const Inner &x = inner[q];
        const uint32_t l = x.limit - x.step;
        for (uint32_t k : x.kid)
            if (k != NONE) inner[k].limit = std::min(inner[k].limit, l);
    }
    std::vector<uint32_t> ready(last + 2, NONE);   // restrictions that become ready at a stage: the first one
    struct Due {
        uint32_t role, next;
    };
    std::vector<Due> dues;
    std::vector<uint32_t> due(last + 1, NONE);     // roles and directions of which a restriction is due: the first one
    std::vector<uint32_t> finished, looked;
    auto operands_done = [&](uint32_t q) {
        Inner &x = inner[q];
        if (x.role != NONE) x.link = std::exchange(ready[x.ready + 1], q);
        else x.ready += x.step, finished.push_back(q);
    };
    auto spread = [&]() {   // from the finished nodes to those that read them
        while (!finished.empty()) {
            const Inner &x = inner[finished.back()];
            finished.pop_back();
            for (uint32_t e = x.users; e != NONE; e = inner[e >> 1].next[e & 1]) {
                Inner &u = inner[e >> 1];
                u.ready = std::max(u.ready, x.ready);
                if (--u.waits == 0) operands_done(e >> 1);
            }
        }
    };
    for (uint32_t q = 0; q < inner.size(); ++q)
        if (inner[q].waits == 0) operands_done(q);
    spread();
    auto look = [&](uint32_t k, uint32_t s) {
        if (std::exchange(roles[k].looked, s) != s) looked.push_back(k);
    };
    auto when_due = [&](uint32_t k, uint32_t limit) {   // limit: the new least one
        roles[k].least = limit;
        dues.push_back({k, due[limit]});
        due[limit] = (uint32_t)dues.size() - 1;
    };
    for (uint32_t s = 1; s <= last; ++s) {
        for (uint32_t e = due[s]; e != NONE; e = dues[e].next) look(dues[e].role, s);
        for (uint32_t q = ready[s]; q != NONE; q = inner[q].link) {
            Role &r = roles[inner[q].role];
            r.pending.push_back(q);
            if (inner[q].limit < r.least) when_due(inner[q].role, std::max(inner[q].limit, s));
            if (r.total < 3 || r.least <= s || r.pending.size() >= WHOLE) look(inner[q].role, s);
        }
        for (uint32_t k : looked) {
            Role &r = roles[k];
            size_t n = r.pending.size();   // how many walk now
            if (r.total >= 3 && r.least > s) {
                n = n / WHOLE * WHOLE;
                if (n && n < r.pending.size())
                    std::nth_element(r.pending.begin(), r.pending.begin() + (ptrdiff_t)n, r.pending.end(),
                                     [&](uint32_t x, uint32_t y) {
                                         return inner[x].limit != inner[y].limit ? inner[x].limit < inner[y].limit : x < y;
                                     });
            }
            if (n == 0) continue;
            for (size_t q = 0; q < n; ++q) {
                Inner &x = inner[r.pending[q]];
                x.ready = stage[x.node] = s, key_of[x.node] = (uint32_t)key_size.size();
                finished.push_back(r.pending[q]);
            }
            key_size.push_back((uint32_t)n);
            r.pending.erase(r.pending.begin(), r.pending.begin() + (ptrdiff_t)n);
            r.least = NONE;
            if (!r.pending.empty()) when_due(k, inner[r.pending[0]].limit);   // the first of the rest is the least
        }
        looked.clear();
        spread();
    }
}

}  // namespace

int build_plan(const hedl_kb *kb, const uint64_t *progs, const uint32_t *offs, uint32_t H, unsigned flags,
               PlanImpl **out) {
    *out = nullptr;
    if (H == 0) return fail(HEDL_ERR_INVALID_ARG, "empty batch (H = 0)");
    if (offs[0] != 0) return fail(HEDL_ERR_INVALID_ARG, "offs[0] must be 0");
    for (uint32_t h = 0; h < H; ++h) {
        if (offs[h + 1] < offs[h]) return fail(HEDL_ERR_INVALID_ARG, "offs must be non-decreasing");
        std::string why;
        int e = validate_program(kb, progs + offs[h], offs[h + 1] - offs[h], &why);
        if (e) return fail(e, "program " + std::to_string(h) + ": " + why);
    }
    auto *p = new PlanImpl();
    p->flags = flags;
    p->n_hyps = H;
    p->tuning = kb->tuning;
    const uint64_t N = kb->n, B = 4ull * kb->wp;
    p->info.n_hyps = H;
    p->info.total_insns = offs[H];

    if (flags & HEDL_PLAIN) {
        // One launch per operation: keep the programs; the stack of the
        // deepest program sizes the workspace.
        p->progs.assign(progs, progs + offs[H]);
        p->offs.assign(offs, offs + H + 1);
        uint32_t maxd = 1;
        uint64_t mb = 0;
        for (uint32_t h = 0; h < H; ++h) {
            int d = 0;
            for (uint32_t k = offs[h]; k < offs[h + 1]; ++k) {
                uint32_t op = (uint32_t)(progs[k] & 0xFF);
                uint32_t a = (uint32_t)((progs[k] >> 16) & 0xFFFF);
                d = d - arity(op) + 1;
                maxd = std::max<uint32_t>(maxd, (uint32_t)d);
                if (op == HEDL_OP_ATOM) mb += B, p->info.n_atom_loads++;
                else if (is_data(op)) mb += data_bytes(kb, a, N), p->info.n_data_ops++;
                else if (is_str(op)) mb += str_bytes(kb, op, a, N), p->info.n_data_ops++;
                else if (is_role(op)) mb += 4 * (N + 1) + 4ull * kb->role_edges[a] + 2 * B, p->info.n_role_ops++;
            }
            mb += 2 * B + 16;  // scoring
        }
        p->plain_depth = maxd;
        p->info.model_bytes = mb;
        // workspace: header page, accumulators [H][2], stack rows
        uint64_t acc_off = 256;
        uint64_t rows_off = (acc_off + 8ull * H + 255) & ~uint64_t(255);
        p->ws_bytes = rows_off + (uint64_t)(maxd + 1) * B;
        p->info.workspace_bytes = p->ws_bytes;
        p->info.n_levels = 0;
        *out = p;
        return HEDL_OK;
    }

    const bool cse = !(flags & HEDL_NO_CSE);
    std::vector<PNode> nodes;
    nodes.reserve(offs[H] + 16);
    NodeTable memo(cse ? offs[H] : 0);   // at most one node an instruction
    auto make = [&](PNode n) -> int32_t {
        // canonical form: ignored fields zeroed, commutative operands ordered
        if (!is_role(n.op)) n.inv = 0;
        if (!(n.op == HEDL_OP_ATOM || is_role(n.op) || is_data(n.op) || is_str(n.op))) n.a = 0;
        if (!(n.op == HEDL_OP_ATLEAST || n.op == HEDL_OP_ATMOST || n.op == HEDL_OP_EXACTLY || is_data(n.op) ||
              is_str(n.op)))
            n.b = 0;
        if (cse) {
            if ((n.op == HEDL_OP_AND || n.op == HEDL_OP_OR) && n.k0 > n.k1) std::swap(n.k0, n.k1);
            if (n.op == HEDL_OP_NOT && nodes[n.k0].op == HEDL_OP_NOT) return nodes[n.k0].k0;
            size_t slot;
            const int32_t same = memo.find(n, nodes, &slot);
            if (same >= 0) return same;
            memo.insert(slot, (int32_t)nodes.size());
        }
        nodes.push_back(n);
        return (int32_t)nodes.size() - 1;
    };

    std::vector<int32_t> roots(H);
    int32_t st[HEDL_MAX_STACK];   // validated: no program holds more
    for (uint32_t h = 0; h < H; ++h) {
        int sp = 0;
        for (uint32_t k = offs[h]; k < offs[h + 1]; ++k) {
            uint64_t w = progs[k];
            PNode n{};
            n.op = (uint8_t)(w & 0xFF);
            n.inv = (uint8_t)((w >> 8) & 1);
            n.a = (uint32_t)((w >> 16) & 0xFFFF);
            n.b = (uint32_t)(w >> 32);
            n.k0 = n.k1 = -1;
            const int ar = arity(n.op);
            sp -= ar;
            if (ar > 0) n.k0 = st[sp];
            if (ar > 1) n.k1 = st[sp + 1];
            st[sp++] = make(n);
        }
        roots[h] = st[0];
    }
    const uint32_t NN = (uint32_t)nodes.size();
    p->info.n_nodes = NN;

    // reference counts (parents + hypothesis roots)
    std::vector<uint32_t> refc(NN, 0);
    for (uint32_t i = 0; i < NN; ++i) {
        if (nodes[i].k0 >= 0) refc[nodes[i].k0]++;
        if (nodes[i].k1 >= 0) refc[nodes[i].k1]++;
    }
    for (uint32_t h = 0; h < H; ++h) refc[roots[h]]++;

    // materialization (children are created before parents, so index order
    // is a topological order)
    std::vector<uint8_t> mat(NN, 0);
    for (uint32_t i = 0; i < NN; ++i)
        if (is_role(nodes[i].op) && nodes[nodes[i].k0].op != HEDL_OP_ATOM) mat[nodes[i].k0] = 1;
    // Bit-sliced role restrictions: each is materialized and evaluated by its
    // role group's shared walk (counting ones need n <= SLICE_MAX_N).  A walk
    // costs its edges' gathers, whatever the number of slices up to
    // SLICES * MAX_PARTS, so restrictions of one role and direction wait for
    // each other: walk_stages gives every eligible restriction the stage it
    // walks at.  A walk of one restriction only costs a transpose and a
    // 32-times larger filler, so by default a restriction is sliced only when
    // another one has the same role, direction and stage.
    const bool sliced = !(flags & HEDL_NO_SLICE);
    std::vector<uint8_t> sl(NN, 0);
    std::vector<uint32_t> stage(NN, 0), key_of(NN, 0), key_size;
    if (sliced) {
        walk_stages(nodes, kb->n_roles, (flags & HEDL_SLICE_ALL) != 0, stage, key_of, key_size);
        for (uint32_t i = 0; i < NN; ++i)
            if (stage[i] && ((flags & HEDL_SLICE_ALL) || key_size[key_of[i]] >= 2)) sl[i] = mat[i] = 1;
    }
    std::vector<uint8_t> role_inline(NN, 0);
    std::vector<uint32_t> need(NN, 1);
    for (uint32_t i = 0; i < NN; ++i) {
        const PNode &n = nodes[i];
        auto ri = [&](int32_t c) { return c >= 0 && !mat[c] && role_inline[c]; };
        role_inline[i] = is_role(n.op) || ri(n.k0) || ri(n.k1);
        if (!mat[i] && refc[i] >= 2 && role_inline[i] && n.op != HEDL_OP_ATOM) mat[i] = 1;
        // stack need (Sethi-Ullman), materialized children count as leaves
        auto nd = [&](int32_t c) -> uint32_t { return mat[c] ? 1u : need[c]; };
        if (n.op == HEDL_OP_NOT) need[i] = nd(n.k0);
        else if (n.op == HEDL_OP_AND || n.op == HEDL_OP_OR) {
            uint32_t a = nd(n.k0), b = nd(n.k1);
            uint32_t v = a == b ? a + 1 : std::max(a, b);
            if (v > (uint32_t)STACK_MAX - 1) {   // keep every segment within the device stack
                mat[a >= b ? n.k0 : n.k1] = 1;
                a = nd(n.k0);
                b = nd(n.k1);
                v = a == b ? a + 1 : std::max(a, b);
            }
            need[i] = v;
        } else need[i] = 1;
    }

    // With staged fillers each segment may read one role restriction (its
    // filler is copied to shared memory once per work item): any further role
    // restriction in a segment's inline expansion becomes its own segment.
    const bool staged = use_staging(kb, kb->tuning);
    p->staged = staged;
    if (staged) {
        std::vector<int32_t> seg_roots;
        for (uint32_t i = 0; i < NN; ++i)
            if (mat[i]) seg_roots.push_back((int32_t)i);
        for (uint32_t h = 0; h < H; ++h)
            if (!mat[roots[h]]) seg_roots.push_back(roots[h]);
        std::vector<int32_t> dfs;
        for (int32_t r : seg_roots) {
            bool kept = false;
            dfs.clear();
            dfs.push_back(r);
            while (!dfs.empty()) {
                int32_t i = dfs.back();
                dfs.pop_back();
                if (i != r && mat[i]) continue;
                const PNode &n = nodes[i];
                if (is_role(n.op)) {
                    if (kept && i != r) mat[i] = 1;
                    kept = true;
                    continue;   // its filler is a slot or a concept row, not inline
                }
                if (n.k1 >= 0) dfs.push_back(n.k1);
                if (n.k0 >= 0) dfs.push_back(n.k0);
            }
        }
    }

    // slots and segments
    std::vector<uint32_t> slot_of(NN, NO_SLOT);
    uint32_t n_slots = 0;
    for (uint32_t i = 0; i < NN; ++i)
        if (mat[i]) slot_of[i] = n_slots++;
    if (n_slots > REF_ID) {
        delete p;
        return fail(HEDL_ERR_INVALID_ARG, "batch too large: more than 2^30 materialized intermediate sets");
    }
    std::vector<Seg> segs;
    std::vector<DInsn> code;
    std::vector<uint32_t> read_list, read_off{0};   // the slots segment s reads: read_list[read_off[s] .. read_off[s + 1])
    std::vector<uint32_t> seg_of_slot(n_slots, 0);
    std::vector<uint32_t> role_key;  // first role read, for grouping
    // Algorithmic bytes, the per-operation model (no credit for sharing a CSR
    // walk or for caches): an atom read B (a role restriction's filler concept
    // included), a data range 4N, a role restriction 4(N+1) + 4E + 2B (row
    // pointers, columns, filler written and read), a hypothesis score
    // 2B + 16, over the operations left after common sub-concepts are shared.
    uint64_t model = 0;

    struct Frame { int32_t n; int state; };
    std::vector<Frame> fr;
    std::vector<uint32_t> reads;
    auto keep_reads = [&](std::vector<uint32_t> &v) {   // sorted, each once
        if (v.size() > 1) {
            std::sort(v.begin(), v.end());
            v.erase(std::unique(v.begin(), v.end()), v.end());
        }
        read_list.insert(read_list.end(), v.begin(), v.end());
        read_off.push_back((uint32_t)read_list.size());
    };
    auto emit_segment = [&](int32_t root, uint32_t out_slot, uint32_t hyp) {
        Seg s{};
        s.code_off = (uint32_t)code.size();
        s.out_slot = out_slot;
        s.hyp = hyp;
        s.filler = NO_FILLER;
        reads.clear();
        uint32_t rk = 0xFFFFFFFFu;
        // iterative post-order emission, larger stack need first
        fr.clear();
        fr.push_back({root, 0});
        int depth = 0, maxdepth = 0;
        while (!fr.empty()) {
            Frame &f = fr.back();
            int32_t i = f.n;
            const PNode &n = nodes[i];
            bool leafish = (i != root && mat[i]) || arity(n.op) == 0 || is_role(n.op);
            if (leafish) {
                DInsn d{};
                if (i != root && mat[i]) {
                    d.op = D_SLOT;
                    d.ref = slot_of[i];
                    reads.push_back(slot_of[i]);   // bytes counted with the restriction that made it
                } else if (n.op == HEDL_OP_ATOM) {
                    d.op = D_ATOM;
                    d.a = n.a;
                    model += B;
                    p->info.n_atom_loads++;
                } else if (n.op == HEDL_OP_TOP || n.op == HEDL_OP_BOT) {
                    d.op = n.op;
                } else if (is_data(n.op)) {
                    const bool num = n.a >= kb->n_props;   // a numeric concrete role
                    d.op = D_DATA | (n.op << 16) | (num ? 1u << 8 : 0u);
                    d.a = num ? n.a - kb->n_props : n.a;
                    d.b = n.b;
                    model += data_bytes(kb, n.a, N);
                    p->info.n_data_ops++;
                } else if (is_str(n.op)) {   // a string concrete role
                    d.op = D_DATA | (n.op << 16) | (1u << 9);
                    d.a = n.a;
                    d.b = n.b;
                    model += str_bytes(kb, n.op, n.a, N);
                    p->info.n_data_ops++;
                } else {  // role restriction
                    int32_t c = n.k0;
                    d.op = D_ROLE | ((uint32_t)n.inv << 8) | ((uint32_t)n.op << 16);
                    d.a = n.a;
                    d.b = n.b;
                    if (nodes[c].op == HEDL_OP_ATOM && !mat[c]) {
                        d.ref = nodes[c].a;
                        model += B;   // the filler concept's row: an atom leaf of the plain method
                    } else {
                        d.ref = REF_SLOT | slot_of[c];
                        reads.push_back(slot_of[c]);
                    }
                    if (rk == 0xFFFFFFFFu) rk = n.a * 2 + n.inv;
                    if (s.filler == NO_FILLER) s.filler = d.ref | (n.op == HEDL_OP_FORALL ? REF_NEG : 0u);
                    const DevCSR &g = kb->csr_host[2 * n.a + n.inv];
                    model += 4 * (N + 1) + 4ull * g.n_edges + 2 * B;
                    p->info.n_role_ops++;
                }
                code.push_back(d);
                depth++;
                maxdepth = std::max(maxdepth, depth);
                fr.pop_back();
                continue;
            }
            if (n.op == HEDL_OP_NOT) {
                if (f.state == 0) {
                    f.state = 1;
                    fr.push_back({n.k0, 0});
                } else {
                    DInsn d{};
                    d.op = D_NOT;
                    code.push_back(d);
                    fr.pop_back();
                }
                continue;
            }
            // AND / OR
            auto nd = [&](int32_t c) -> uint32_t { return mat[c] ? 1u : need[c]; };
            int32_t first = nd(n.k0) >= nd(n.k1) ? n.k0 : n.k1;
            int32_t second = first == n.k0 ? n.k1 : n.k0;
            if (f.state == 0) {
                f.state = 1;
                fr.push_back({first, 0});
            } else if (f.state == 1) {
                f.state = 2;
                fr.push_back({second, 0});
            } else {
                DInsn d{};
                d.op = n.op;
                code.push_back(d);
                depth--;
                fr.pop_back();
            }
        }
        s.code_len = (uint32_t)code.size() - s.code_off;
        p->max_stack = std::max(p->max_stack, (uint32_t)maxdepth);
        if (hyp != NO_HYP) model += 2 * B + 16;
        keep_reads(reads);
        role_key.push_back(rk);
        segs.push_back(s);
    };
    for (uint32_t i = 0; i < NN; ++i)
        if (mat[i] && !sl[i]) {
            seg_of_slot[slot_of[i]] = (uint32_t)segs.size();
            emit_segment((int32_t)i, slot_of[i], NO_HYP);
        }
    for (uint32_t h = 0; h < H; ++h) {
        if (mat[roots[h]]) {  // the root is already a slot: the segment reads it
            Seg s{};
            s.code_off = (uint32_t)code.size();
            s.code_len = 1;
            s.out_slot = NO_SLOT;
            s.hyp = h;
            s.filler = NO_FILLER;
            DInsn d{};
            d.op = D_SLOT;
            d.ref = slot_of[roots[h]];
            code.push_back(d);
            model += 2 * B + 16;
            reads.assign(1, slot_of[roots[h]]);
            keep_reads(reads);
            role_key.push_back(0xFFFFFFFFu);
            segs.push_back(s);
            p->max_stack = std::max(p->max_stack, 1u);
        } else {
            emit_segment(roots[h], NO_SLOT, h);
        }
    }
    if (p->max_stack > (uint32_t)STACK_MAX) {
        delete p;
        return fail(HEDL_ERR_BAD_PROGRAM, "internal: segment stack exceeds the device limit");
    }
    const uint32_t NSEG = (uint32_t)segs.size();
    const uint64_t FT_PART = 4ull * 32ull * kb->wp;   // one FT word per individual (>= 4 N bytes)

    uint32_t max_stage = 0;   // of the sliced restrictions, grouped by key (stage, role, direction)
    for (uint32_t i = 0; i < NN; ++i)
        if (sl[i]) max_stage = std::max(max_stage, stage[i]);

    // Production level of every slot and level of every segment.  A segment
    // reading nothing is at level 0 and otherwise one level above the slots it
    // reads.  A sliced role restriction is ready one level above its filler's
    // transpose, which runs one level above the filler's producer (level 0 for
    // a concept row); all restrictions of a group key walk together, at the
    // level of the group's last-ready one.  A filler holds only sliced
    // restrictions of earlier stages, so materialized nodes are taken by the
    // last stage in their expression, children first: the sliced restrictions
    // of a stage (their fillers belong to earlier ones), then its segments.
    std::vector<uint32_t> slot_level(n_slots, 0), seg_level(NSEG, 0);
    std::vector<uint32_t> group_level(key_size.size(), 0);
    auto seg_lvl = [&](uint32_t sidx) {
        uint32_t lvl = 0;
        for (uint32_t q = read_off[sidx]; q < read_off[sidx + 1]; ++q) lvl = std::max(lvl, slot_level[read_list[q]] + 1);
        return lvl;
    };
    {
        std::vector<uint32_t> last_stage(NN, 0), first(max_stage + 2, 0), by_stage;
        for (uint32_t i = 0; i < NN; ++i) {
            const PNode &n = nodes[i];
            uint32_t d = std::max(n.k0 >= 0 ? last_stage[n.k0] : 0u, n.k1 >= 0 ? last_stage[n.k1] : 0u);
            if (sl[i]) d = stage[i];
            last_stage[i] = d;
            if (mat[i]) first[d + 1]++;
        }
        for (uint32_t d = 1; d < first.size(); ++d) first[d] += first[d - 1];
        by_stage.resize(first.back());
        std::vector<uint32_t> at(first.begin(), first.end() - 1);
        for (uint32_t i = 0; i < NN; ++i)
            if (mat[i]) by_stage[at[last_stage[i]]++] = i;
        for (uint32_t d = 0; d <= max_stage; ++d) {
            for (uint32_t q = first[d]; q < first[d + 1]; ++q) {
                const uint32_t i = by_stage[q];
                if (!sl[i]) continue;
                const int32_t f = nodes[i].k0;
                const bool concept_filler = nodes[f].op == HEDL_OP_ATOM && !mat[f];
                uint32_t &lvl = group_level[key_of[i]];
                lvl = std::max(lvl, concept_filler ? 1u : slot_level[slot_of[f]] + 2u);
            }
            for (uint32_t q = first[d]; q < first[d + 1]; ++q)
                if (sl[by_stage[q]]) slot_level[slot_of[by_stage[q]]] = group_level[key_of[by_stage[q]]];
            for (uint32_t q = first[d]; q < first[d + 1]; ++q) {
                const uint32_t i = by_stage[q];
                if (sl[i]) continue;
                const uint32_t sidx = seg_of_slot[slot_of[i]];
                slot_level[slot_of[i]] = seg_level[sidx] = seg_lvl(sidx);
            }
        }
    }
    for (uint32_t sidx = 0; sidx < NSEG; ++sidx)
        if (segs[sidx].hyp != NO_HYP) seg_level[sidx] = seg_lvl(sidx);

    // role groups: sliced restrictions keyed by (level, role, direction), up to
    // SLICES * MAX_PARTS at a time (one FT word per 32 of them); those of
    // a (stage, role, direction) share a level, and stages that come out on one level share groups
    std::vector<RGroup> rgroups;
    std::vector<uint32_t> task_level(seg_level);
    std::vector<uint32_t> task_key(role_key);
    uint64_t ft_bytes = 0;
    {
        std::vector<std::pair<uint64_t, uint32_t>> keyed;   // ((level << 32) | role2, node)
        for (uint32_t i = 0; i < NN; ++i)
            if (sl[i]) keyed.push_back({((uint64_t)slot_level[slot_of[i]] << 32) | (nodes[i].a * 2 + nodes[i].inv), i});
        std::stable_sort(keyed.begin(), keyed.end(),
                         [](const std::pair<uint64_t, uint32_t> &x, const std::pair<uint64_t, uint32_t> &y) {
                             return x.first < y.first;
                         });
        for (size_t k = 0; k < keyed.size();) {
            size_t k2 = k;
            while (k2 < keyed.size() && keyed[k2].first == keyed[k].first && k2 - k < SLICES * MAX_PARTS) ++k2;
            RGroup g{};
            g.role2 = (uint32_t)(keyed[k].first & 0xFFFFFFFFu);
            g.n = (uint32_t)(k2 - k);
            g.parts = g.n > SLICES ? MAX_PARTS : 1u;
            reads.clear();
            for (size_t q = k; q < k2; ++q) {
                const uint32_t i = keyed[q].second;
                const PNode &n = nodes[i];
                const int32_t f = n.k0;
                const uint32_t s_ = (uint32_t)(q - k);
                if (nodes[f].op == HEDL_OP_ATOM && !mat[f]) {
                    g.filler[s_] = nodes[f].a;
                    model += B;   // the filler concept's row
                } else {
                    g.filler[s_] = REF_SLOT | slot_of[f];
                    reads.push_back(slot_of[f]);
                }
                if (n.op == HEDL_OP_FORALL) g.filler[s_] |= REF_NEG;
                g.out[s_] = slot_of[i];
                // the counts 0 .. 7 (7: or more) at which the restriction holds
                const uint32_t le = n.b >= 7 ? 0xFFu : (2u << n.b) - 1u, lt = n.b == 0 ? 0u : le >> 1;
                uint32_t holds = n.op == HEDL_OP_EXISTS    ? 0xFEu
                                 : n.op == HEDL_OP_FORALL  ? 0x01u   // successors outside C
                                 : n.op == HEDL_OP_ATLEAST ? 0xFFu & ~lt
                                 : n.op == HEDL_OP_ATMOST  ? le
                                                           : le & ~lt;
                for (; holds; holds &= holds - 1) g.want[s_ / SLICES][__builtin_ctz(holds)] |= 1u << (s_ % SLICES);
                p->info.n_role_ops++;
            }
            keep_reads(reads);                              // of the transpose
            read_off.push_back((uint32_t)read_list.size());   // the walk reads no slot
            const uint32_t gi = (uint32_t)rgroups.size();
            const uint32_t wl = (uint32_t)(keyed[k].first >> 32);
            // transpose task, then walk task
            Seg t{};
            t.code_off = gi;
            t.out_slot = NO_SLOT;
            t.hyp = NO_HYP;
            t.filler = NO_FILLER;
            t.kind = TASK_TRANSPOSE;
            segs.push_back(t);
            task_level.push_back(wl - 1);
            task_key.push_back(g.role2 | 0x80000000u);
            Seg w = t;
            w.kind = TASK_WALK;
            const uint32_t walk_task = (uint32_t)segs.size();
            segs.push_back(w);
            task_level.push_back(wl);
            task_key.push_back(g.role2);
            for (uint32_t s_ = 0; s_ < g.n; ++s_) seg_of_slot[g.out[s_]] = walk_task;
            const DevCSR &csr = kb->csr_host[g.role2];
            model += (uint64_t)g.n * (4 * (N + 1) + 4ull * csr.n_edges + 2 * B);
            g.ft_off = ft_bytes;   // relative to the FT region until the slots are placed
            ft_bytes += g.parts * FT_PART;
            rgroups.push_back(g);
            k = k2;
        }
    }
    const uint32_t NS = (uint32_t)segs.size();

    // dependencies (the producer task of every slot read; a walk waits for its transpose)
    std::vector<uint32_t> deps;
    uint32_t n_levels = 0;
    for (uint32_t s_ = 0; s_ < NS; ++s_) {
        segs[s_].dep_off = (uint32_t)deps.size();
        if (segs[s_].kind == TASK_WALK) {
            deps.push_back((s_ - 1) | DEP_FINE);
        } else {
            for (uint32_t q = read_off[s_]; q < read_off[s_ + 1]; ++q) {
                const uint32_t by = seg_of_slot[read_list[q]];
                deps.push_back(by | (segs[by].kind == TASK_SEGMENT ? 0u : DEP_FINE));
            }
        }
        segs[s_].dep_cnt = (uint32_t)deps.size() - segs[s_].dep_off;
        n_levels = std::max(n_levels, task_level[s_] + 1);
    }
    if (flags & HEDL_TEST_UNSAT_DEP) {
        // the last segment additionally waits on a counter past the real
        // ones, which nothing ever increments
        segs[NSEG - 1].dep_off = (uint32_t)deps.size();
        segs[NSEG - 1].dep_cnt = 1;
        deps.push_back(NS);
    }

    // Tile shape.  A warp covers 32 words a round by default.  When some level
    // that walks a role holds only a few segments (a small batch, a single
    // hypothesis), its tiles would keep only a fraction of the resident warps
    // busy, each walking 32 words in sequence: then a warp covers fewer words
    // (down to 4, one round per item) so that the level spreads over about
    // four times as many warp-rounds as there are resident warps (32 per SM at
    // 64 registers), which also balances rows of very different degree.  Plans
    // with role groups keep the default shape for their segments.
    const Tuning &t = p->tuning;
    uint32_t WW = 32, rounds = t.rounds;
    if (rgroups.empty() && kb->n_sms > 0) {
        std::vector<uint32_t> segs_at(n_levels, 0);
        std::vector<uint8_t> walks_at(n_levels, 0);
        for (uint32_t s_ = 0; s_ < NS; ++s_) {
            const uint32_t L = task_level[s_];
            segs_at[L]++;
            for (uint32_t pc = 0; pc < segs[s_].code_len; ++pc)
                if ((code[segs[s_].code_off + pc].op & 0xFFu) == D_ROLE) walks_at[L] = 1;
        }
        uint64_t smin = UINT64_MAX;
        for (uint32_t L = 0; L < n_levels; ++L)
            if (walks_at[L]) smin = std::min<uint64_t>(smin, segs_at[L]);
        const uint64_t resident = 32ull * (uint64_t)kb->n_sms;
        if (smin != UINT64_MAX)
            while (WW > 4 && smin * kb->wp < 4ull * resident * WW * t.wpl) WW >>= 1;
        if (WW < 32) rounds = 1;
    }
    const uint32_t TW = t.warps * WW * t.wpl * rounds;
    const uint32_t n_tiles = (kb->wp + TW - 1) / TW;
    // Transposes and walks have tiles of their own, FW words a warp: 32, or
    // fewer while the walks of an average level that has some would give the
    // resident warps (24 an SM at 80 registers) less than four items each to
    // even out.  (Large batches: 16 items a warp, 8 to 16 words, was no faster.)
    uint32_t FW = 0, n_fine = 0;
    if (!rgroups.empty()) {
        std::vector<uint8_t> walks_at(n_levels, 0);
        for (uint32_t s_ = NSEG; s_ < NS; ++s_)
            if (segs[s_].kind == TASK_WALK) walks_at[task_level[s_]] = 1;
        const uint64_t levels = std::count(walks_at.begin(), walks_at.end(), (uint8_t)1);
        const uint64_t resident = 24ull * (uint64_t)std::max(kb->n_sms, 1);
        FW = 32;
        while (FW > 4 && rgroups.size() * kb->wp < 4 * resident * FW * levels) FW >>= 1;
        n_fine = (kb->wp + t.warps * FW - 1) / (t.warps * FW);
    }
    auto fine = [&](uint32_t task) { return segs[task].kind != TASK_SEGMENT; };
    // Segments of a work item: as many (up to SEG_BATCH) as leave an average
    // level two items a resident CTA; a staged filler belongs to one segment.
    uint32_t SB = 1;
    if (!rgroups.empty() && !staged) {
        const uint64_t ctas = std::max<uint64_t>(1, 24ull * (uint64_t)std::max(kb->n_sms, 1) / t.warps);
        SB = (uint32_t)std::min<uint64_t>(SEG_BATCH, std::max<uint64_t>(1, (uint64_t)NSEG * n_tiles / (2 * ctas * n_levels)));
    }
    std::vector<uint32_t> order(NS);
    for (uint32_t s = 0; s < NS; ++s) order[s] = s;
    std::stable_sort(order.begin(), order.end(), [&](uint32_t x, uint32_t y) {
        if (task_level[x] != task_level[y]) return task_level[x] < task_level[y];
        if (task_key[x] != task_key[y]) return task_key[x] < task_key[y];
        return fine(x) < fine(y);
    });
    std::vector<Group> groups;
    std::vector<uint32_t> gsegs;
    std::vector<uint32_t> level_items(n_levels + 1, 0);
    uint64_t items = 0;
    for (uint32_t k = 0; k < NS;) {
        uint32_t s0 = order[k];
        Group g{};
        g.item_begin = (uint32_t)items;
        g.seg_begin = (uint32_t)gsegs.size();
        g.level = task_level[s0];
        uint32_t k2 = k;
        while (k2 < NS && task_level[order[k2]] == g.level && task_key[order[k2]] == task_key[s0] &&
               fine(order[k2]) == fine(s0)) {
            gsegs.push_back(order[k2]);
            ++k2;
        }
        g.n_segs = k2 - k;
        items += fine(s0) ? (uint64_t)g.n_segs * n_fine : (uint64_t)((g.n_segs + SB - 1) / SB) * n_tiles;
        level_items[g.level + 1] = (uint32_t)items;
        if (fine(s0)) g.level |= GROUP_FINE;
        groups.push_back(g);
        k = k2;
    }
    for (uint32_t l = 1; l <= n_levels; ++l) level_items[l] = std::max(level_items[l], level_items[l - 1]);
    // the (task, tile) pairs that the plan reports, and the items made of them
    if (items >= 0xFFFFFFFFull || (uint64_t)NS * n_tiles >= 0xFFFFFFFFull) {
        delete p;
        return fail(HEDL_ERR_INVALID_ARG, "batch too large: more than 2^32 work items");
    }

    // image: header, tables, counters; then the slots
    std::vector<uint8_t> &img = p->image;
    img.reserve(sizeof(PlanHeader) + segs.size() * sizeof(Seg) + groups.size() * sizeof(Group) + 4 * gsegs.size() +
                4 * deps.size() + code.size() * sizeof(DInsn) + 4 * level_items.size() + 4 * (NS + 5 + 2ull * H) +
                rgroups.size() * sizeof(RGroup) + 10 * 256);
    img.resize(sizeof(PlanHeader));
    PlanHeader hd{};
    hd.n_items = (uint32_t)items;
    hd.n_segs = NS;
    hd.n_groups = (uint32_t)groups.size();
    hd.n_hyps = H;
    hd.n_tiles = n_tiles;
    hd.tile_words = TW;
    hd.warp_words = WW | FW << 8 | (FW ? SB << 16 : 0u);
    hd.n_slots = n_slots;
    hd.flags = flags;
    hd.n_levels = n_levels;
    hd.n_deps = (uint32_t)deps.size();
    hd.off_segs = put(img, segs);
    hd.off_groups = put(img, groups);
    hd.off_gsegs = put(img, gsegs);
    hd.off_deps = put(img, deps);
    hd.off_code = put(img, code);
    hd.off_level_items = put(img, level_items);
    hd.n_rgroups = (uint32_t)rgroups.size();
    // counters: Counters + done[NS + 1] + acc[H][2]
    std::vector<uint32_t> zeros(4 + (NS + 1) + 2ull * H, 0);
    hd.off_ctr = put(img, zeros);
    p->ctr_off = hd.off_ctr;
    p->ctr_bytes = zeros.size() * 4;
    hd.off_rgroups = put(img, rgroups);   // FT offsets patched below, once the slots are placed
    img.resize((img.size() + 255) & ~size_t(255));
    hd.off_slots = img.size();
    hd.off_ft = (hd.off_slots + (uint64_t)n_slots * B + 255) & ~uint64_t(255);
    for (size_t g = 0; g < rgroups.size(); ++g) rgroups[g].ft_off += hd.off_ft;
    if (!rgroups.empty()) memcpy(img.data() + hd.off_rgroups, rgroups.data(), rgroups.size() * sizeof(RGroup));
    hd.timeout_ns = (uint64_t)t.timeout_ms * 1000000ull;
    memcpy(img.data(), &hd, sizeof hd);
    p->image_bytes = img.size();
    p->slots_off = hd.off_slots;
    p->ws_bytes = hd.off_ft + ft_bytes;
    p->n_rgroups = (uint32_t)rgroups.size();
    p->info.n_role_groups = (uint32_t)rgroups.size();
    p->level_items = level_items;

    p->info.n_segments = NS;
    p->info.n_slots = n_slots;
    p->info.n_levels = n_levels;
    p->n_items = (uint32_t)items;
    p->info.n_items = NS * n_tiles;
    p->info.tile_words = TW;
    p->info.warp_words = WW;
    p->info.workspace_bytes = p->ws_bytes;
    p->info.image_bytes = p->image_bytes;
    p->info.model_bytes = model;
    *out = p;
    return HEDL_OK;
}

}  // namespace hedl
