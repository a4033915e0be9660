// S5 Barnes (1990) grouped interaction lists (Sec. 2.2 steps 3 and 5; Sec. 3.1.2).
//
// One warp per group (a team of 2 or 4 when groups are few) walks its box's tree from the
// root with a stack.  Every
// node the recursive walk visits is tested, in this order:
//   prune  -- the node's cell is farther than r_cut from the group's particle box (the
//             box of finest-level cells that holds the group's particles; periodic
//             box-to-box distance), so none of its particles can act (Eq. 2 is 0);
//   accept -- level >= l_min and the opening criterion holds: cell side l and the
//             distance d from the node's cell centre to the nearest point of the group
//             cell satisfy l < theta d; the node enters the list as one particle at its
//             centre of mass (Sec. 3.1.2);
//   leaf   -- an opened leaf puts its particles into the list, each but those whose
//             finest cell passes the prune test (the same integer test at level 21);
//   open   -- the node's children are tested next.
// No node inside a pruned or accepted subtree is tested.  The entries are the same set
// as the recursive walk's; their order within a list is the order of the steps (the
// debug dump sorts each list back into preorder, i.e. by first particle).
// Every test is done in integer units u = L/2^22 against thresholds the host derives
// from the FP64 comparisons (double)S*u*u > r_cut*r_cut and (double)l*l < theta*theta*S,
// so the lists are exact and bit-identical to a sequential FP64 walk.
//
// Entries are written as float4 (x, y, z, m) relative to the group's cell centre in
// r_cut units (Sec. 3.1.1: positions passed relative to the group centre): the cell
// offset (an exact integer in u, wrapped to the nearest image) times u/r_cut, plus the
// particle's FP32 offset from its own leaf centre (or the node's COM offset from its
// cell centre).  The group's own particles get the same float4 in irel[], so a
// particle and its own list entry are bit-identical and the self pair has r = 0.
//
// Lists are contiguous per group inside pages handed out by an atomic counter; a list
// that does not fit the warp's current page is walked again into fresh pages.  A second
// walk costs as much as the first, so a warp takes fresh pages for a mean list before the walk
// when the room left is below its mean list length so far (and a page before its first
// group: a warp of a small call walks one or two groups in all).  It leaves at most half as
// much room behind that way as its lists take (the bound on the pool is in grow_caps); past
// that it walks into the room there is.  List stage before and after, one
// GB300: 4 k particles 0.096 -> 0.053 ms, 100 k 0.197 -> 0.107, 300 k 0.287 -> 0.176, 128^3
// halo mix 1.200 -> 1.177.  With a single page whatever the mean, 20000 lists of 6200 entries
// took 8.20 ms and three pages each; 5.11 ms and two.
//
// The walk may start below the root.  Let K be a level at or above the first level at
// which any node can be accepted: with the group's particle box inside its cell, a node of
// half side h that passes the prune test lies at squared distance at most
// (sqrt(T_prune) + sqrt(3) h)^2 from the group cell, so no node of a level k with that
// bound <= A[k] (or k < l_min) is ever accepted, and every node above level K that the
// recursive walk reaches is opened or, for a leaf, emptied.  A node below the root that
// passes the prune test has every ancestor passing it too, as long as no ancestor's nearest
// image differs from the image that holds the node; for an ancestor of half side <= L/4
// that holds when L/4 > sqrt(T_prune) + the particle box's half side + its offset from
// the cell centre, on every axis.  Under those two conditions the walk's entries are the
// level-K nodes that pass their tests (and the leaves above level K that pass the prune
// test) taken as the first step, which k_start_table makes a lookup: the level-K cells
// within r_cut of the group's particle box are enumerated, each names its node (or the
// leaf above it, taken once), and the children of the root down to level K are never
// tested.  A group that fails a condition, or whose cells are too many, walks from the
// root.
#include <algorithm>

#include "common.cuh"

namespace greem {

__device__ __forceinline__ int wrap_delta(int d, int &sh)
{
    sh = 0;
    if (d >= kHalfPeriod) {
        d -= kPeriod;
        sh = -1;
    } else if (d < -kHalfPeriod) {
        d += kPeriod;
        sh = 1;
    }
    return d;
}

__device__ __forceinline__ unsigned shift_code(int sx, int sy, int sz)
{
    auto c = [](int s) -> unsigned { return s == 0 ? 0u : (s > 0 ? 1u : 2u); };
    return c(sx) | (c(sy) << 2) | (c(sz) << 4);
}

__device__ __forceinline__ Node load_node(const Node *p)
{
    const uint4 *q = reinterpret_cast<const uint4 *>(p);
    uint4 a = __ldg(q), b = __ldg(q + 1);
    Node n;
    n.ix = a.x; n.iy = a.y; n.iz = a.z; n.lvl = a.w;
    n.begin = b.x; n.end = b.y; n.skip = b.z; n.parent = b.w;
    return n;
}

// Geometry of a cell against the group: the offset of its centre from the group's cell
// centre (u, wrapped to the nearest image; with SHIFT also the image's shift code, which
// only index entries record), the squared gap to the group's particle box, and the
// squared distance from its centre to the group cell (both in u^2).  cell_gap computes
// what the prune test needs; the accept distance follows only for cells that pass it.
struct CellTest {
    int dx, dy, dz;
    unsigned shc;
    long long Sg;
};

// rx, ry, rz: the cell centre minus the group's cell centre (u), before wrapping; h: the
// cell's half side (u).
template <bool SHIFT>
__device__ __forceinline__ CellTest cell_gap(int rx, int ry, int rz, int h, const int4 tb, const int4 th)
{
    CellTest c;
    int sx, sy, sz;
    c.dx = wrap_delta(rx, sx);
    c.dy = wrap_delta(ry, sy);
    c.dz = wrap_delta(rz, sz);
    c.shc = SHIFT ? shift_code(sx, sy, sz) : 0u;
    const int gx = max(0, abs(c.dx - tb.x) - h - th.x), gy = max(0, abs(c.dy - tb.y) - h - th.y),
              gz = max(0, abs(c.dz - tb.z) - h - th.z);
    c.Sg = (long long)gx * gx + (long long)gy * gy + (long long)gz * gz;
    return c;
}

__device__ __forceinline__ long long cell_dist2(const CellTest &c, int hg)
{
    const int ex = max(0, abs(c.dx) - hg), ey = max(0, abs(c.dy) - hg), ez = max(0, abs(c.dz) - hg);
    return (long long)ex * ex + (long long)ey * ey + (long long)ez * ez;
}

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// The items of a warp's sources, 32 at a time.  Source lanes (those with items) leave what
// their items need in shared memory in the order of the lanes, and the lane of item t finds
// its source's place from the sources that begin in the window [t0, t0 + 32): one warp OR,
// one ballot and two population counts, where a search over the lanes' offsets and a shuffle
// per value took 11 to 14 dependent shuffles.  List stage, 128^3 halo mix / 256^3 / 64 boxes:
// 1.167 / 3.355 / 6.07 -> 1.120 / 3.204 / 5.94 ms.
__device__ __forceinline__ uint32_t source_place(bool source, uint32_t off, uint32_t t0, unsigned le)
{
    const unsigned FULL = 0xffffffffu;
    const uint32_t d = off - t0;
    const unsigned heads = __reduce_or_sync(FULL, source && d < 32u ? 1u << d : 0u);
    const unsigned before = __ballot_sync(FULL, source && off < t0);
    return __popc(before) + __popc(heads & le) - 1;
}

// ---------------------------------------------------------------- start tables
constexpr uint32_t kCoarseLeaf = 0x80000000u;  // table entry: a leaf above level K
constexpr uint32_t kMaxStartCells = 512;       // more candidate cells: walk from the root

// A list warp's counters, kept in shared memory by its lane 0 and added to the status
// word once, when the warp runs out of groups.
enum { kTallyPadded, kTallyLen, kTallyInter, kTallyStart, kTallyGroups, kTallyLeft, kTallyN };

// A 10-bit integer's bits spread to every third bit (Morton interleave).
__device__ __forceinline__ uint32_t spread_bits3(uint32_t v)
{
    v = (v | (v << 16)) & 0x030000FFu;
    v = (v | (v << 8)) & 0x0300F00Fu;
    v = (v | (v << 4)) & 0x030C30C3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

__device__ __forceinline__ uint32_t cell_morton(uint32_t x, uint32_t y, uint32_t z)
{
    return (spread_bits3(x) << 2) | (spread_bits3(y) << 1) | spread_bits3(z);
}

// One thread per level-(K-1) cell of a box: the descent from the root to the node of
// that cell gives the entries of its 8 level-K children, written as two 16-byte stores.
__global__ void __launch_bounds__(256) k_start_table(const Node *__restrict__ nodes, const uint32_t *__restrict__ kids,
                                                     const uint32_t *__restrict__ base,
                                                     const BoxPar *__restrict__ bps, int nbox,
                                                     uint32_t *__restrict__ tbl, const DevStatus *__restrict__ st)
{
    // the tree is incomplete, or there is none after a wait that gave up: no list is walked
    if (st->flags & (ST_NODE_CAP | ST_TIMEOUT)) return;
    for (int b = blockIdx.y; b < nbox; b += gridDim.y) {
        const BoxPar &bp = bps[b];
        const int K = bp.kstart;
        if (K < 2) continue;
        const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
        if (c >= (1u << (3 * (K - 1)))) continue;
        uint32_t r = base[bp.p_begin];  // the box's root
        bool empty = false;
        for (int d = 1; d < K; d++) {
            const uint32_t lv = nodes[r].lvl;
            if (lv & 256u) break;  // a leaf above level K-1 holds the cell
            const uint32_t oct = (c >> (3 * (K - 1 - d))) & 7u;
            const uint32_t mask = (lv >> 16) & 255u;
            if (!(mask & (1u << oct))) {
                empty = true;
                break;
            }
            r = kids[(size_t)r * 8 + __popc(mask & ((1u << oct) - 1u))];
        }
        uint32_t e[8];
        const uint32_t lv = nodes[r].lvl;
#pragma unroll
        for (int o = 0; o < 8; o++) {
            if (empty) e[o] = kNone;
            else if (lv & 256u) e[o] = r | kCoarseLeaf;
            else {
                const uint32_t mask = (lv >> 16) & 255u;
                e[o] = (mask & (1u << o)) ? kids[(size_t)r * 8 + __popc(mask & ((1u << o) - 1u))] : kNone;
            }
        }
        uint4 *dst = reinterpret_cast<uint4 *>(tbl + bp.tbl_off + (size_t)c * 8);
        dst[0] = make_uint4(e[0], e[1], e[2], e[3]);
        dst[1] = make_uint4(e[4], e[5], e[6], e[7]);
    }
}

void launch_start_table(const Node *nodes, const uint32_t *kids, const uint32_t *base, const BoxPar *bps, int nbox,
                        int kmax, uint32_t *tbl, const DevStatus *st, cudaStream_t s)
{
    if (kmax < 2 || nbox < 1) return;
    const uint32_t cells = 1u << (3 * (kmax - 1));
    const dim3 grid((cells + 255) / 256, (unsigned)std::min(nbox, 65535));
    k_start_table<<<grid, 256, 0, s>>>(nodes, kids, base, bps, nbox, tbl, st);
    g_launches++;
}

// The warps that walk one group together (W consecutive warps of a block; each chunk of 32
// cells or particles goes to the next warp, and every warp keeps the walk's state).  A
// chunk's entries and pushes go where one warp alone would put them: `mine` counts this
// warp's, `before` those of the lower warps, `total` all of the team's.
template <int W>
struct Team {
    uint32_t *slots = nullptr;  // two rows of W counts, used in turn: one barrier per exchange
    uint32_t row = 0;
    int wid = 0, bar = 0;       // warp within the team; the team's barrier
    __device__ __forceinline__ void sync() const
    {
        if constexpr (W == 1) __syncwarp();
        else asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(32 * W) : "memory");
    }
    __device__ __forceinline__ void place(uint32_t mine, int lane, uint32_t &before, uint32_t &total)
    {
        if constexpr (W == 1) {
            before = 0;
            total = mine;
        } else {
            const unsigned FULL = 0xffffffffu;
            if (lane == 0) slots[row * W + wid] = mine;
            sync();
            const uint32_t v = lane < W ? slots[row * W + lane] : 0u;
            row ^= 1u;
            total = __reduce_add_sync(FULL, v);
            before = __reduce_add_sync(FULL, lane < wid ? v : 0u);
        }
    }
};

// One tested cell per lane: an accepted node becomes one entry at its centre of mass
// (acc), a node to open or a leaf to empty goes onto the stack (push).  Returns false
// when the stack would overflow (the status is set; the call is retried).
template <bool INDEX, int W>
__device__ __forceinline__ bool take_cells(const ListArgs &a, Team<W> &team, bool acc, bool push, uint32_t child,
                                           const CellTest &ct, float kf, unsigned long long pos0, uint32_t room,
                                           int lane, unsigned lt, uint32_t &cnt, uint32_t &nacc,
                                           uint32_t *__restrict__ stk, uint32_t &sp, uint32_t cap)
{
    const unsigned FULL = 0xffffffffu;
    const unsigned ab = __ballot_sync(FULL, acc);
    uint32_t na = __popc(ab), np = 0, a0 = 0, p0 = 0;
    unsigned pb = 0;
    if constexpr (W > 1) {
        pb = __ballot_sync(FULL, push);
        uint32_t before, total;
        team.place(na | ((uint32_t)__popc(pb) << 16), lane, before, total);
        a0 = before & 0xffffu;
        p0 = before >> 16;
        na = total & 0xffffu;
        np = total >> 16;
    }
    if (acc) {
        const uint32_t p = cnt + a0 + __popc(ab & lt);
        const float4 v = __ldg(a.noff + child);
        const float4 e = make_float4(__fadd_rn(__fmul_rn((float)ct.dx, kf), v.x),
                                     __fadd_rn(__fmul_rn((float)ct.dy, kf), v.y),
                                     __fadd_rn(__fmul_rn((float)ct.dz, kf), v.z), v.w);
        if (p < room) {
            a.flist[pos0 + p] = e;
            if (INDEX) a.ilist[pos0 + p] = (unsigned long long)child | (1ull << 32) | ((unsigned long long)ct.shc << 33);
        }
    }
    cnt += na;
    nacc += na;
    if constexpr (W == 1) {
        pb = __ballot_sync(FULL, push);
        np = __popc(pb);
    }
    if (sp + np > cap) {
        if (lt == 0u) atomicOr(&a.st->flags, ST_STACK);
        return false;
    }
    if (push) stk[sp + p0 + __popc(pb & lt)] = child;
    sp += np;
    return true;
}

// What a walk needs of its group, in shared memory: 64 bytes per warp, read by broadcast
// where a test needs them (the memory clobber keeps the loads behind the stores of the next
// group's words).  Held in registers they would spill others: the walker keeps 32
// warps per SM at 64 registers (spill stores 268 -> 80 bytes before the teams, 184 with them;
// with the one scan per step and the
// one copy of the walk: 1.120 / 3.204 / 5.94 -> 1.034 / 3.045 / 5.46 ms).
//   0: cell centre and half side (u)        1: particle box centre minus cell centre; first particle
//   2: its half sides; end of the particles 3: T_prune (two words), k_f, l_min
__device__ __forceinline__ int4 group_word(uint32_t gsm, int k)
{
    int4 v;
    asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(gsm + 16u * k) : "memory");
    return v;
}
__device__ __forceinline__ long long word_tprune(const int4 w)
{
    return (long long)(((unsigned long long)(uint32_t)w.y << 32) | (uint32_t)w.x);
}

// The first step of a walk that starts at level K = bp.kstart (see the header): the
// level-K cells within r_cut of the group's particle box, tested like the children of an
// opened node.  Returns false if the group must walk from the root instead (sp is then
// untouched); sets overflow on a stack overflow.
template <bool INDEX, int W>
__device__ __forceinline__ bool start_cells(const ListArgs &a, Team<W> &team, uint32_t gsm, const BoxPar &bp, uint32_t *__restrict__ stk, unsigned long long pos0,
                                            uint32_t room, int lane, unsigned lt, uint32_t &cnt,
                                            uint32_t &nacc, uint32_t &sp, bool &overflow)
{
    const int K = bp.kstart;
    if (K < 2) return false;
    const int4 gc = group_word(gsm, 0), tb = group_word(gsm, 1), th = group_word(gsm, 2);
    const int R = bp.rprune;
    const int quarter = kPeriod / 4;
    if (quarter - th.x - abs(tb.x) <= R || quarter - th.y - abs(tb.y) <= R || quarter - th.z - abs(tb.z) <= R)
        return false;
    const int sh = 22 - K, nK = 1 << K;
    const uint32_t mK = (uint32_t)nK - 1u;
    // per axis: the level-K cells whose gap to the particle box is at most R (unwrapped
    // indices from c0, n of them; the whole axis once if that many reach around)
    auto range = [&](int gc, int t0, int t1, int &c0, int &n) {
        const int lo = gc + t0 - t1 - R, hi = gc + t0 + t1 + R;
        c0 = (lo - 1) >> sh;
        n = (hi >> sh) - c0 + 1;
        if (n >= nK) {
            c0 = 0;
            n = nK;
        }
    };
    int cx0, nx, cy0, ny, cz0, nz;
    range(gc.x, tb.x, th.x, cx0, nx);
    range(gc.y, tb.y, th.y, cy0, ny);
    range(gc.z, tb.z, th.z, cz0, nz);
    const uint32_t ncand = (uint32_t)(nx * ny * nz);
    if (ncand > kMaxStartCells) return false;
    const uint32_t *tb_k = a.tbl + bp.tbl_off;
    const long long Tp = bp.T_prune;
    const int hK = 1 << (kMaxLevel - K);  // half side of a level-K cell (u)
    const bool acc_level = K >= bp.lmin;
    const long long AK = bp.A[K];
    const float kf = bp.k_f;
    // lane's candidate t = (ix ny + iy) nz + iz, advanced by the team's chunks
    const int l0 = 32 * team.wid + lane;
    int iz = l0 % nz, iy = (l0 / nz) % ny, ix = l0 / (nz * ny);
    const int sz = (32 * W) % nz, qz = (32 * W) / nz, sy = qz % ny, sx = qz / ny;
    for (uint32_t c0 = 0; c0 < ncand; c0 += 32 * W) {
        const uint32_t t = c0 + (uint32_t)l0;
        bool acc = false, push = false, node_coarse = false;
        uint32_t node = 0;
        CellTest ct;
        ct.dx = ct.dy = ct.dz = 0;
        ct.shc = 0;
        if (t < ncand) {
            const uint32_t wx = (uint32_t)(cx0 + ix) & mK, wy = (uint32_t)(cy0 + iy) & mK,
                           wz = (uint32_t)(cz0 + iz) & mK;
            const uint32_t e = __ldg(tb_k + cell_morton(wx, wy, wz));
            if (e != kNone) {
                if (e & kCoarseLeaf) {
                    // a leaf above level K: tested once, from the first of its cells among
                    // the candidates (per axis, the first index whose cell is in its block)
                    node = e & ~kCoarseLeaf;
                    node_coarse = true;
                    const Node nd = load_node(a.nodes + node);
                    const int kl = (int)(nd.lvl & 255u);
                    const uint32_t bs = 1u << (K - kl);
                    auto first = [&](uint32_t a0, int c0a) -> int {
                        const uint32_t w = (uint32_t)c0a & mK;
                        return ((w - a0) & mK) < bs ? 0 : (int)((a0 - w) & mK);
                    };
                    const int fsh = kMaxLevel - K;
                    if (ix == first(nd.ix >> fsh, cx0) && iy == first(nd.iy >> fsh, cy0) &&
                        iz == first(nd.iz >> fsh, cz0)) {
                        const int hl = 1 << (kMaxLevel - kl);
                        ct = cell_gap<INDEX>(2 * (int)nd.ix + hl - gc.x, 2 * (int)nd.iy + hl - gc.y,
                                             2 * (int)nd.iz + hl - gc.z, hl, tb, th);
                        push = ct.Sg <= Tp;
                    }
                } else {
                    node = e;
                    ct = cell_gap<INDEX>((int)(wx << sh) + hK - gc.x, (int)(wy << sh) + hK - gc.y,
                                         (int)(wz << sh) + hK - gc.z, hK, tb, th);
                    if (ct.Sg <= Tp) {
                        acc = acc_level && cell_dist2(ct, gc.w) > AK;
                        push = !acc;
                    }
                }
            }
        }
        if (!take_cells<INDEX, W>(a, team, acc, push, node, ct, kf, pos0, room, lane, lt, cnt, nacc, stk, sp, a.stack_cap)) {
            overflow = true;
            break;
        }
        if (INDEX) {
            // a count for tests (each walk of a group counts: the rare walk into fresh
            // pages counts twice)
            const unsigned cb = __ballot_sync(0xffffffffu, push && node_coarse);
            if (cb && lt == 0u) atomicAdd(&a.st->sum_coarse, (unsigned long long)__popc(cb));
        }
        iz += sz;
        const int cz = iz >= nz;
        iz -= cz ? nz : 0;
        iy += sy + cz;
        const int cy = iy >= ny;
        iy -= cy ? ny : 0;
        ix += sx + cy;
    }
    return true;
}

// Walks one group's list; writes entries [pos0, pos0+total), the first `room` of them;
// returns total.  stk is this warp's stack (a.stack_cap entries); an overflow sets the status.
//
// The stack holds nodes that passed the prune test and failed the accept test: leaves,
// whose particles are emitted, and nodes to open.  Each step pops up to 32 of them, one
// per lane.  The children of the opened nodes are then spread over the lanes, 32 at a
// time: a child's cell follows from its parent's cell and its octant (the parent's
// child-octant mask), so prune and accept are decided without loading the child; an
// accepted child is written as one entry at its centre of mass, and the others are
// pushed.  Last, the particles of the popped leaves are spread over the lanes and each
// goes through the per-particle r_cut test unless its whole leaf lies within r_cut.
// INDEX: the index entries are written too (a.ilist).
template <bool INDEX, int W>
__device__ __forceinline__ uint32_t walk_group(const ListArgs &a, Team<W> &team, uint32_t gsm, const BoxPar &bp,
                               uint32_t root, uint32_t *__restrict__ stk, const uint8_t *__restrict__ octq,
                               uint4 *__restrict__ src,
                               unsigned long long pos0, uint32_t room, int lane, uint32_t &nacc,
                               bool &from_table)
{
    const unsigned FULL = 0xffffffffu;
    const unsigned lt = (1u << lane) - 1u, le = lt | (1u << lane);
    nacc = 0;
    const uint32_t cap = a.stack_cap;
    uint32_t cnt = 0;
    uint32_t sp = 0;
    bool overflow = false;
    from_table = start_cells<INDEX, W>(a, team, gsm, bp, stk, pos0, room, lane, lt, cnt, nacc, sp, overflow);
    if (!from_table) {
        if (team.wid == 0 && lane == 0) stk[0] = root;
        sp = 1;
    }
    team.sync();
    while (sp > 0 && !overflow) {
        const uint32_t nb = min(sp, 32u);
        const uint32_t sbase = sp - nb;
        const bool valid = (uint32_t)lane < nb;
        const uint32_t m = valid ? stk[sbase + lane] : 0u;
        __syncwarp();  // (a team's pushes come after its first exchange)
        sp = sbase;
        Node nd;
        unsigned long long lb = 0;
        if (valid) {
            nd = load_node(a.nodes + m);
            lb = __ldg(a.lbox + m);  // of leaves only; loaded beside the node
        } else {
            nd.ix = nd.iy = nd.iz = 0; nd.lvl = 0; nd.begin = nd.end = nd.skip = 0; nd.parent = 0;
        }
        const int k = nd.lvl & 255u;
        const bool leaf = valid && (nd.lvl & 256u) != 0;
        const uint32_t mask = valid && !leaf ? (nd.lvl >> 16) & 255u : 0u;
        // the popped node's centre minus the group's cell centre (u, before wrapping)
        const int hn = 1 << (kMaxLevel - k);
        const int4 gc = group_word(gsm, 0);
        const int ncx = 2 * (int)nd.ix + hn - gc.x, ncy = 2 * (int)nd.iy + hn - gc.y, ncz = 2 * (int)nd.iz + hn - gc.z;

        // ---- the popped leaves: which particles, and what their entries take from the leaf
        uint32_t ne = 0;
        float bx = 0.f, by = 0.f, bz = 0.f;
        unsigned shc = 0;   // test flag in bit 6, own in bit 7; INDEX: the leaf's shift code in bits 0-5
        int ox = 0, oy = 0, oz = 0;
        if (leaf) {
            const int4 tb = group_word(gsm, 1), th = group_word(gsm, 2), pw = group_word(gsm, 3);
            const long long Tp = word_tprune(pw);
            const float kf = __int_as_float(pw.z);
            const int h = hn;
            const CellTest lc = cell_gap<INDEX>(ncx, ncy, ncz, h, tb, th);
            // the box of the leaf's particles (finest cells, in slots of q; k_leaf_boxes),
            // its centre relative to the group's cell centre in the leaf's image and its
            // half sides (u): beyond r_cut of the group's particle box, no particle is
            // kept; within it, every particle is (each particle's finest cell is inside)
            const int q = h > 256 ? (h >> 8) : 1;
            const int lx = (int)(lb & 255u), ly = (int)((lb >> 16) & 255u), lz = (int)((lb >> 32) & 255u);
            const int ux = (int)((lb >> 8) & 255u), uy = (int)((lb >> 24) & 255u), uz = (int)((lb >> 40) & 255u);
            const int bcx = lc.dx - h + (lx + ux + 1) * q - tb.x, bcy = lc.dy - h + (ly + uy + 1) * q - tb.y,
                      bcz = lc.dz - h + (lz + uz + 1) * q - tb.z;
            const int bhx = (ux + 1 - lx) * q, bhy = (uy + 1 - ly) * q, bhz = (uz + 1 - lz) * q;
            const int gx = max(0, abs(bcx) - bhx - th.x), gy = max(0, abs(bcy) - bhy - th.y),
                      gz = max(0, abs(bcz) - bhz - th.z);
            const bool none = (long long)gx * gx + (long long)gy * gy + (long long)gz * gz > Tp;
            const int fx = max(0, abs(bcx) + bhx - th.x), fy = max(0, abs(bcy) + bhy - th.y),
                      fz = max(0, abs(bcz) + bhz - th.z);
            const bool test_each = (long long)fx * fx + (long long)fy * fy + (long long)fz * fz > Tp;
            ne = none ? 0u : nd.end - nd.begin;
            bx = __fmul_rn((float)lc.dx, kf);
            by = __fmul_rn((float)lc.dy, kf);
            bz = __fmul_rn((float)lc.dz, kf);
            // the group's own particles leave their positions in irel; a leaf lies in the group
            // whole or not at all
            const bool own = nd.begin >= (uint32_t)tb.w && nd.begin < (uint32_t)th.w;
            shc = lc.shc | (test_each ? 64u : 0u) | (own ? 128u : 0u);
            // a particle in finest cell c of this leaf sits at 2c + o (u) from the centre of
            // the group's particle box, in the leaf's image
            ox = lc.dx - ncx - gc.x + 1 - tb.x;
            oy = lc.dy - ncy - gc.y + 1 - tb.y;
            oz = lc.dz - ncz - gc.z + 1 - tb.z;
        }
        // ---- the sources of both loops below, in shared memory
        const uint32_t nch = __popc(mask);
        uint32_t o, ctot, tot;  // the lane's first child or particle, and how many there are
        if (!__any_sync(FULL, ne >> 18)) {  // a node has children or particles: one scan for both
            const uint32_t v = nch | (ne << 9), x = warp_incl_scan(v, lane), last = __shfl_sync(FULL, x, 31);
            o = mask ? (x - v) & 511u : (x - v) >> 9;
            ctot = last & 511u;
            tot = last >> 9;
        } else {  // leaves of the finest level can hold any number of particles
            const uint32_t x = warp_incl_scan(nch, lane), y = warp_incl_scan(ne, lane);
            o = mask ? x - nch : y - ne;
            ctot = __shfl_sync(FULL, x, 31);
            tot = __shfl_sync(FULL, y, 31);
        }
        const unsigned inner = __ballot_sync(FULL, mask != 0), full = __ballot_sync(FULL, ne != 0);
        const uint32_t n_inner = __popc(inner);  // the particles' sources come after the children's
        if (mask) {
            uint4 *d = src + 2 * __popc(inner & lt);
            d[0] = make_uint4(o, m, nd.lvl, (uint32_t)ncx);
            d[1] = make_uint4((uint32_t)ncy, (uint32_t)ncz, 0u, 0u);
        }
        if (ne) {
            uint4 *d = src + 2 * (n_inner + __popc(full & lt));
            d[0] = make_uint4(nd.begin - o, shc, (uint32_t)ox, (uint32_t)oy);
            d[1] = make_uint4((uint32_t)oz, __float_as_uint(bx), __float_as_uint(by), __float_as_uint(bz));
        }
        const bool is_inner = mask != 0, is_full = ne != 0;
        __syncwarp();

        // ---- children of the opened nodes: prune, accept (one entry), or push
        for (uint32_t c0 = 32 * team.wid; c0 < ctot + 32 * team.wid; c0 += 32 * W) {
            const uint32_t t = c0 + lane;
            const uint4 *sp_ = src + 2 * source_place(is_inner, o, c0, le);
            const uint4 u = sp_[0];
            const uint2 v = *reinterpret_cast<const uint2 *>(sp_ + 1);
            const uint32_t o_s = u.x, pm = u.y, plvl = u.z;
            const int pcx = (int)u.w, pcy = (int)v.x, pcz = (int)v.y;
            const int4 pw = group_word(gsm, 3);
            bool acc = false, push = false;
            uint32_t child = 0;
            CellTest ct;
            if (t < ctot) {
                const int4 tb = group_word(gsm, 1), th = group_word(gsm, 2);
                const uint32_t q = t - o_s;
                const uint32_t oct = octq[((plvl >> 13) & (255u << 3)) | q];
                const int kc = (int)(plvl & 255u) + 1;
                const int hc = 1 << (kMaxLevel - kc);
                // a child's centre is its parent's shifted by +-hc per axis
                ct = cell_gap<INDEX>(pcx + ((oct & 4u) ? hc : -hc), pcy + ((oct & 2u) ? hc : -hc),
                                     pcz + ((oct & 1u) ? hc : -hc), hc, tb, th);
                if (ct.Sg <= word_tprune(pw)) {
                    child = __ldg(a.kids + (size_t)pm * 8 + q);
                    acc = kc >= pw.w && cell_dist2(ct, group_word(gsm, 0).w) > bp.A[kc];
                    push = !acc;
                }
            }
            if (!take_cells<INDEX, W>(a, team, acc, push, child, ct, __int_as_float(pw.z), pos0, room, lane, lt, cnt, nacc, stk, sp, cap)) {
                overflow = true;  // the caller's list is incomplete; the call is retried with a larger stack
                break;
            }
        }
        __syncwarp();
        if (overflow) break;

        // ---- particles of the popped leaves
        for (uint32_t t0 = 32 * team.wid; t0 < tot + 32 * team.wid; t0 += 32 * W) {
            const uint32_t t = t0 + lane;
            const uint4 *sp_ = src + 2 * (n_inner + source_place(is_full, o, t0, le));
            const uint4 u = sp_[0], v4 = sp_[1];
            const unsigned sh_s = u.y;
            const int ox_s = (int)u.z, oy_s = (int)u.w, oz_s = (int)v4.x;
            const float bx_s = __uint_as_float(v4.y), by_s = __uint_as_float(v4.z), bz_s = __uint_as_float(v4.w);
            bool keep = false;
            float4 e;
            uint32_t j = kNone;
            if (t < tot) {
                j = u.x + t;
                const float4 v = __ldg(a.poff + j);
                keep = true;
                if (sh_s & 64u) {
                    // the particle's finest cell, in its leaf's image, against the particle box
                    const int4 th = group_word(gsm, 2);
                    const long long Tp = word_tprune(group_word(gsm, 3));
                    const unsigned long long c = __ldg(a.pcell + j);
                    const int px = 2 * (int)((uint32_t)c & 0x1fffffu) + ox_s;
                    const int py = 2 * (int)((uint32_t)(c >> 21) & 0x1fffffu) + oy_s;
                    const int pz = 2 * (int)(uint32_t)(c >> 42) + oz_s;
                    const int qx = max(0, abs(px) - 1 - th.x), qy = max(0, abs(py) - 1 - th.y),
                              qz = max(0, abs(pz) - 1 - th.z);
                    keep = (long long)qx * qx + (long long)qy * qy + (long long)qz * qz <= Tp;
                }
                e = make_float4(__fadd_rn(bx_s, v.x), __fadd_rn(by_s, v.y), __fadd_rn(bz_s, v.z), v.w);
                if (sh_s & 128u) a.irel[j] = e;
            }
            const unsigned kb = __ballot_sync(FULL, keep);
            uint32_t before, total;
            team.place(__popc(kb), lane, before, total);
            if (keep) {
                const uint32_t p = cnt + before + __popc(kb & lt);
                if (p < room) {
                    a.flist[pos0 + p] = e;
                    if (INDEX) a.ilist[pos0 + p] = (unsigned long long)j | ((unsigned long long)(sh_s & 63u) << 33);
                }
            }
            cnt += total;
        }
        team.sync();  // the sources are read, the pushes made
    }
    team.sync();
    return cnt;
}

// A block's shared memory.
struct ListShared {
    uint8_t octq[256 * 8];  // octq[8 mask + q]: the octant of the (q+1)-th set bit of an 8-bit child mask
    unsigned long long tallies[kListWarps][kTallyN];
    uint4 sources[kListWarps][64];  // walk_group's sources, two words of 16 bytes each
    int4 gconst[kListWarps][4];     // group_word
    uint32_t slots[2 * kListWarps];
    unsigned long long word[kListWarps];
};

// The lists of all groups, W warps per group.
template <bool INDEX, int W>
__device__ __forceinline__ void build_lists(const ListArgs &a, ListShared &sm, uint32_t G)
{
    constexpr int BT = kListWarps / W;  // teams per block
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tm = warp / W;  // team within the block
    const uint8_t *octq = sm.octq;
    uint4 *src = sm.sources[warp];
    const uint32_t gsm = (uint32_t)__cvta_generic_to_shared(sm.gconst[tm]);
    Team<W> team;
    if constexpr (W > 1) {
        team.slots = sm.slots + 2 * W * tm;
        team.wid = warp % W;
        team.bar = 1 + tm;
    }
    const bool first = team.wid == 0 && lane == 0;  // the team's first thread
    // the first thread's value, for every thread of the team
    auto share = [&](unsigned long long v) -> unsigned long long {
        if constexpr (W == 1) return __shfl_sync(FULL, v, 0);
        if (first) sm.word[tm] = v;
        team.sync();
        v = sm.word[tm];
        team.sync();
        return v;
    };
    unsigned long long *tally = sm.tallies[tm];
    uint32_t *stk = a.stack + (size_t)(blockIdx.x * BT + tm) * a.stack_cap;
    unsigned long long page_cur = 0, page_end = 0;
    bool exhausted = false;  // the pool ran out: only count what the lists need
    // np fresh pages become the warp's current ones; false (and the status) past the pool
    auto take_pages = [&](unsigned long long np) -> bool {
        unsigned long long page0 = 0;
        if (first) page0 = atomicAdd(&a.st->list_pages, np);
        page0 = share(page0);
        if ((page0 + np) * a.page > a.cap) {
            if (first) atomicOr(&a.st->flags, ST_LIST_CAP);
            page_cur = page_end = 0;
            exhausted = true;
            return false;
        }
        page_cur = page0 * a.page;
        page_end = (page0 + np) * a.page;
        return true;
    };
    for (;;) {
        unsigned long long gi = 0;
        if (first) gi = atomicAdd(&a.st->work[0], 1ull);
        gi = share(gi);
        if (gi >= G) break;
        const uint32_t g = (uint32_t)gi;
        if constexpr (W == 1) __syncwarp();  // the last group's constants are read, the tallies written
        const Group gr = a.groups[g];
        const BoxPar &bp = a.bps[gr.box];
        if (first) {
            int4 *w = sm.gconst[tm];
            const int4 tb = a.gbox[2 * (size_t)g], th = a.gbox[2 * (size_t)g + 1];
            const unsigned long long Tp = (unsigned long long)bp.T_prune;
            w[0] = make_int4(gr.cx, gr.cy, gr.cz, gr.hg);
            w[1] = make_int4(tb.x, tb.y, tb.z, (int)gr.begin);
            w[2] = make_int4(th.x, th.y, th.z, (int)(gr.begin + gr.count));
            w[3] = make_int4((int)(uint32_t)Tp, (int)(uint32_t)(Tp >> 32), __float_as_int(bp.k_f), bp.lmin);
        }
        const uint32_t root = a.base[bp.p_begin];
        const uint32_t left = (uint32_t)(page_end - page_cur);
        const float sum = (float)tally[kTallyPadded], ng = (float)tally[kTallyGroups];
        if (!exhausted && (left == 0 || ((float)left * ng < sum && 2.0f * (float)(tally[kTallyLeft] + left) <= sum))) {
            // one page more than the whole pages of a mean list
            take_pages(1u + (uint32_t)__fdividef(sum, fmaxf(ng, 1.0f) * (float)a.page));
            if (first) tally[kTallyLeft] += left;
        }
        team.sync();
        uint32_t nacc = 0, len = 0, padded = 0;
        bool placed = false;
        for (bool again = false;; again = true) {
            bool from_table = false;
            len = walk_group<INDEX, W>(a, team, gsm, bp, root, stk, octq, src, page_cur, (uint32_t)(page_end - page_cur), lane,
                                    nacc, from_table);
            padded = (len + 7u) & ~7u;
            if (!again && first) {
                tally[kTallyStart] += from_table ? 1u : 0u;
                tally[kTallyPadded] += padded;
                tally[kTallyGroups]++;
            }
            if (exhausted) break;
            placed = page_cur + padded <= page_end;
            if (placed || !take_pages((padded + a.page - 1) / a.page)) break;
        }
        if (!placed) {
            if (first) {
                a.loff[g] = 0;
                a.llen[g] = 0;
                a.lraw[g] = 0;
                if (a.qcnt) a.qcnt[g] = 0;
            }
            continue;
        }
        for (uint32_t t = len + lane; t < padded && team.wid == 0; t += 32) {
            a.flist[page_cur + t] = make_float4(16.f, 16.f, 16.f, 0.f);
            if (INDEX) a.ilist[page_cur + t] = ~0ull;
        }
        if (first) {
            a.loff[g] = page_cur;
            a.llen[g] = padded;
            a.lraw[g] = len;
            if (a.qcnt) a.qcnt[g] = nacc;
            tally[kTallyLen] += len;
            tally[kTallyInter] += (unsigned long long)len * a.groups[g].count;
        }
        page_cur += padded;
    }
    if (first) {
        DevStatus *st = a.st;
        if (tally[kTallyPadded]) atomicAdd(&st->sum_padded, tally[kTallyPadded]);
        if (tally[kTallyLen]) atomicAdd(&st->sum_len, tally[kTallyLen]);
        if (tally[kTallyInter]) atomicAdd(&st->sum_inter, tally[kTallyInter]);
        if (tally[kTallyStart]) atomicAdd(&st->sum_start, tally[kTallyStart]);
    }
}

template <bool INDEX>
__global__ void __launch_bounds__(kListWarps * 32, kListBlocksPerSM) k_lists(ListArgs a)
{
    __shared__ ListShared sm;
    for (uint32_t m = threadIdx.x; m < 256; m += blockDim.x) {
        uint32_t q = 0;
        for (uint32_t o = 0; o < 8; o++)
            if (m & (1u << o)) sm.octq[8 * m + q++] = (uint8_t)o;
        for (; q < 8; q++) sm.octq[8 * m + q] = 0;
    }
    if (threadIdx.x < kListWarps * kTallyN) (&sm.tallies[0][0])[threadIdx.x] = 0;
    __syncthreads();
    if (a.st->flags & ST_NODE_CAP) return;  // the tree was truncated: the call is retried
    const uint32_t G = *a.n_groups, warps = gridDim.x * kListWarps;
    // Few groups: several warps walk one together, as a walk is a chain of dependent round
    // trips and most of the warps would have none.  A team's warps all pop and scan, so with
    // enough groups for the warps one each is faster.  List stage with 1 / 2 / 4 warps per
    // group, on 4864 warps (us): 512 groups 34.8 / 32.4 / 28.4, 963 57 / 47 / 41, 1630 67 /
    // 53 / 57, 2657 73.5 / 67.3 / 77.5, 4096 71.4 / 75.8 / 104, 9923 146 / 199 / 252.
    if (4 * (unsigned long long)G <= warps) build_lists<INDEX, 4>(a, sm, G);
    else if (3 * (unsigned long long)G <= 2 * (unsigned long long)warps) build_lists<INDEX, 2>(a, sm, G);
    else build_lists<INDEX, 1>(a, sm, G);
}

void launch_lists(const ListArgs &a, cudaStream_t s, int nsm)
{
    if (a.ilist) k_lists<true><<<nsm * kListBlocksPerSM, kListWarps * 32, 0, s>>>(a);
    else k_lists<false><<<nsm * kListBlocksPerSM, kListWarps * 32, 0, s>>>(a);
    g_launches++;
}

}  // namespace greem
