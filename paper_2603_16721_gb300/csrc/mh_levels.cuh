// Greedy rounds by bands of score levels, and their counters by cover rounds (included by
// mh_kernels.cu, inside its anonymous namespace).
//
// The loop of Algorithm 1 picks one combination per round.  U only shrinks, so a
// combination's TP, and with it its score, only falls, and the rounds visit scores in
// descending order.  So with every combination of a score of at least tau at hand (the
// band's members, with their tumors), the rounds down to tau need no further search: the
// best member by key is picked, the members' scores follow from their tumors still in U,
// and so on until the best is below tau, which is where the next band starts.  A band is one
// pass over the kept leaf parents whose bound reaches tau and one grid barrier; its picks are
// made by every block alike.  A solve has 1 to 12 bands where it has 12 to 740 rounds (15 to
// 23 bands with rows too dense to list), and each round used to cost a chain of about 10 us
// (scan, re-evaluation, grid barrier, slot reduction, winner rows).  tau is chosen so that at
// most 64 bounds per block reach it; where a single level already has more (the last ones:
// thousands of combinations of two or three tumors), the band is that level.  Its rounds are
// then the lexicographically first set of pairwise disjoint intersections among the members,
// since a member that meets a pick has fallen below the level for good.  A level with more
// members than are worth a list (see members_worth) is picked one member a step.
//
// The counters of every round (visited and pruned nodes per depth) do not depend on
// how the winners were found, only on the round cr(s) in which each tumor is covered:
// a node whose intersection over all tumors is y holds |y_r| = #{s in y : cr(s) >= r}
// of them in round r, so with the sums of "Counting by per-sample sums"
//     max(|y_r| - 1, 0) = #{s in y without its last-covered tumor : cr(s) >= r},
// and one pass over the kept nodes after the last level adds each node's weight at
// cr(s) of every tumor but the last; suffix sums over the rounds finish every counter.
//
// Bounds: ub[i] of leaf parent i is at least the best score + 1 of its leaves with
// TP >= 2 in the current U (scores only fall).  It is brought down only when the level
// reaches it: first to a_num |y| + a_den Nn of its uncovered tumors, then by evaluating
// the leaves.  TP = 1 leaves are the champions (see phase_champions).  Champions need no
// update: one whose combination covers two uncovered tumors is outscored by that leaf.

// Per-block scratch of the levels.  The builds with several blocks per SM keep it small.
template <bool kBig>
struct LevelSh {
    static constexpr int kIlp = kBig ? 4 : 1;        // bounds a lane reads at once
    static constexpr int kQ = kBig ? 2048 : 256;     // records queued per scan segment: 32 kIlp per warp
    static constexpr int kWin = kBig ? 64 : 16;      // records evaluated together
    static constexpr int kHist = kBig ? 6144 : 1;    // (round, counter) bins kept on chip
    u32 q[kQ];
    Rec rec[kWin];                                    // window: the record, its samples in U
    u32 ri[kWin];                                     // its index
    int tasks[kWin];                                  // tasks of 32 column words
    u64 nb[kWin];                                     // its best leaf below the level
    int emit[kWin];                                   // whether it has members of the level
    static constexpr int kEm = kBig ? 256 : 32;
    u64 em[kEm];                                      // the window's members: gene, TP << 16, FP << 32, record << 48
    u32 tally[kTally];                                // bounds below the band by distance
    u64 wmax[kMaxWarpsPerBlock];
    u64 cov[kMaxWords];
    u32 hlo[kHist], hhi[kHist];
    u16 cr[kBig ? kMaxSamples : 1];                   // the round that covers each tumor
    u16 ord[kMaxSamples];                             // the tumors by that round, last first
    int qn, en, ec, nd, alive, k, more;
    int full;                                         // enough members were counted
};
constexpr u32 kDenseBit = 0x80000000u;  // queue entry: an unlisted (dense) record
// A bound word is a score + 1 (below 2^44) and a flag: the record has members in the band
// being resolved, its leaves are looked at again in the next one.
constexpr u64 kEmitted = 1ull << 63;

// The members go to out while there is room (cap) and are counted up to `limit`: the block that
// passes it raises its flag `full` and counts no more, so that neither the counter nor the time
// spent on it grows with a level that has no list anyway.
struct LevelOut {
    Member *out;
    u32 *count;
    u32 cap, limit;
    int *full;
    __device__ __forceinline__ u32 take() const { return *(volatile int *)full ? 0xffffffffu : atomicAdd(count, 1u); }
    __device__ __forceinline__ bool room(u32 i) const  // of what take returned (its latency ends here)
    {
        if (i < cap) return true;
        if (i >= limit) *(volatile int *)full = 1;
        return false;
    }
};

// Ascending original indices of a prefix of L genes.
__device__ __forceinline__ void prefix_po(const Cohort &c, const Prefix &p, int L, int *po)
{
#pragma unroll
    for (int q = 0; q < kMaxH - 1; ++q) po[q] = 0;
    for (int q = 0; q < L; ++q) {
        const int v = c.orig[prefix_gene(p, q)];
        int k = q - 1;
        while (k >= 0 && po[k] > v) {
            po[k + 1] = po[k];
            --k;
        }
        po[k + 1] = v;
    }
}

// (t2 also takes TP and FP, below the tuple's bits.)
__device__ __forceinline__ Member *new_member(const LevelOut &o, const Key &k, int tp, int fp)
{
    const u32 i = o.take();
    if (!o.room(i)) return nullptr;
    Member *m = o.out + i;
    m->t0 = k.t0;
    m->t1 = k.t1;
    m->t2 = k.t2 | (u64)fp << 16 | (u64)tp;
    m->k = (u16)tp;
    return m;
}

// The member of record r's leaf gene g, by a whole warp: a lane per gene of the tuple
// (its place among the original indices by counting), a lane per listed tumor or row word.
__device__ __noinline__ void emit_warp(const Cohort &c, const LevelOut &o, const Rec &r, bool dense, const u64 *Ush, int L,
                                       int g, int tp, int fp)
{
    const int lane = threadIdx.x & 31;
    u32 at = 0;
    if (lane == 0) at = o.take();
    const int mine = lane < L ? prefix_gene(r.p, lane) : g;
    const int v = lane <= L ? (int)__ldg(c.orig + mine) : 0x10000;
    u64 y = 0;
    bool has = false;
    if (dense) {
        if (lane < c.Wt) {
            y = Ush[lane] & __ldg(c.T + (size_t)g * c.WTp + lane);
#pragma unroll
            for (int q = 0; q < kMaxH - 1; ++q)
                if (q < L) y &= __ldg(c.T + (size_t)prefix_gene(r.p, q) * c.WTp + lane);
        }
    } else if (lane < (int)r.ky) {
        has = (__ldg(c.CT + (size_t)r.ids[lane] * c.GW + (g >> 6)) >> (g & 63)) & 1ull;
    }
    int place = 0;
    for (int q = 0; q <= L; ++q) place += __shfl_sync(kFull, v, q) < v ? 1 : 0;
    const u64 x = lane <= L ? (u64)v << (16 * (3 - (place & 3))) : 0ull;
    u64 t[3];
#pragma unroll
    for (int w = 0; w < 3; ++w) {
        const u64 xw = place >> 2 == w ? x : 0ull;
        t[w] = (u64)__reduce_or_sync(kFull, (unsigned)(xw >> 32)) << 32 | __reduce_or_sync(kFull, (unsigned)xw);
    }
    at = __shfl_sync(kFull, at, 0);
    if (!o.room(at)) return;
    Member *m = o.out + at;
    if (lane == 0) {
        m->t0 = t[0];
        m->t1 = t[1];
        m->t2 = t[2] | (u64)fp << 16 | (u64)tp;
        m->k = (u16)tp;
    }
    if (tp > kMemIds) return;
    if (dense) {
        int n = warp_incl_scan(__popcll(y), lane) - __popcll(y);
        for (; y; y &= y - 1) m->ids[n++] = (u16)(lane * 64 + __ffsll((long long)y) - 1);
    } else {
        const unsigned b = __ballot_sync(kFull, has);
        if (has) m->ids[__popc(b & ((1u << lane) - 1u))] = r.ids[lane];
    }
}

// A leaf of listed record r (its samples those in U) at column word wi, bit bt.
__device__ __noinline__ void emit_listed(const Cohort &c, const LevelOut &o, const Rec &r, int L, int wi, int bt, int tp,
                                         int fp)
{
    int po[kMaxH - 1];
    prefix_po(c, r.p, L, po);
    Member *m = new_member(o, leaf_key(0, po, L, c.orig[wi * 64 + bt]), tp, fp);
    if (!m || tp > kMemIds) return;
    int n = 0;
    for (int q = 0; q < (int)r.ky; ++q)
        if ((__ldg(c.CT + (size_t)r.ids[q] * c.GW + wi) >> bt) & 1ull) m->ids[n++] = r.ids[q];
}

// A leaf of a dense record, y in ys.
__device__ __noinline__ void emit_dense(const Cohort &c, const LevelOut &o, const Prefix &p, const u64 *ys, int L, int g,
                                        int tp, int fp)
{
    int po[kMaxH - 1];
    prefix_po(c, p, L, po);
    Member *m = new_member(o, leaf_key(0, po, L, c.orig[g]), tp, fp);
    if (!m || tp > kMemIds) return;
    int n = 0;
    for (int w = 0; w < c.Wt; ++w)
        for (u64 y = ys[w] & __ldg(c.T + (size_t)g * c.WTp + w); y; y &= y - 1)
            m->ids[n++] = (u16)(w * 64 + __ffsll((long long)y) - 1);
}

// A record's first 64 bytes (prefix, sizes, tumors) and its other samples.
static_assert(offsetof(Rec, ids) + sizeof(u16) * kListT <= 64, "tumors in the first four 16-byte words");
__device__ __forceinline__ void load_rec_tumors(Rec *dst, const Rec *src)
{
#pragma unroll
    for (int i = 0; i < 4; ++i) reinterpret_cast<uint4 *>(dst)[i] = __ldcg(reinterpret_cast<const uint4 *>(src) + i);
}
__device__ __forceinline__ void load_rec_normals(Rec *dst, const Rec *src)
{
    const u16 *s = src->ids + kListT;
    for (int i = 0; i < (int)dst->kn && i < kListN; ++i) dst->ids[kListT + i] = __ldcg(s + i);
}

// Where the evaluation of a window leaves the members it finds: in the block's list, for
// emit_warp, or beyond its room straight to the level; with `least` only the smallest original
// index of a record's leaf genes is kept, in least[2 j] (with the record's prefix the smallest
// tuple: a smaller gene more makes a smaller tuple).
struct EmitList {
    u64 *em;
    int *n;
    int cap, j;  // j: the record's place in the window
    u32 *least;
};

// One (record, column word) item of a listed record in a band: its leaves of scores from
// tau on are emitted, the best one below goes to nb.
__device__ __forceinline__ void leaf_item_level(const Cohort &c, const Solve &s, const LevelOut &o, const EmitList &el,
                                                const Rec &r, int L, int wi, u64 rw, u64 tau, u64 &nb, bool &emitted)
{
    const int ky = r.ky, kn = r.kn;
    const int pt = bit_length(ky), pn = kn ? bit_length(kn) : 0;
    u64 tpl[kPlanesT] = {0, 0, 0, 0, 0};
    u64 m = 0, m2 = 0;
    for (int q = 0; q < ky; q += kEvalLoads) {
        u64 x[kEvalLoads];
#pragma unroll
        for (int k = 0; k < kEvalLoads; ++k)
            x[k] = q + k < ky ? __ldg(c.CT + (size_t)r.ids[q + k] * c.GW + wi) & rw : 0ull;
#pragma unroll
        for (int k = 0; k < kEvalLoads; ++k) {
            m2 |= m & x[k];
            m |= x[k];
            planes_add(tpl, x[k], pt);
        }
    }
    if (!m2) return;
    u64 fpl[kPlanesN] = {0, 0, 0, 0};
    for (int q = 0; q < kn; q += kEvalLoads) {
        u64 x[kEvalLoads];
#pragma unroll
        for (int k = 0; k < kEvalLoads; ++k)
            x[k] = q + k < kn ? __ldg(c.CN + (size_t)r.ids[kListT + q + k] * c.GW + wi) : 0ull;
#pragma unroll
        for (int k = 0; k < kEvalLoads; ++k) planes_add(fpl, x[k], pn);
    }
    const u64 top = s.a_den * (u64)c.Nn + 1;
    while (m2) {
        const int bt = __ffsll((long long)m2) - 1;
        m2 &= m2 - 1;
        const int tp = planes_get(tpl, bt, pt);
        const u64 b1 = s.a_num * (u64)tp + top;
        if (b1 <= nb) continue;  // no better than what is known below the band
        const int fp = planes_get(fpl, bt, pn);
        const u64 s1 = b1 - s.a_den * (u64)fp;
        if (s1 >= tau) {
            emitted = true;
            if (__builtin_expect(el.least != nullptr, 0)) {
                atomicMin(el.least + 2 * el.j, (u32)__ldg(c.orig + wi * 64 + bt));
                continue;
            }
            const int p = atomicAdd(el.n, 1);
            if (p < el.cap) el.em[p] = (u64)(wi * 64 + bt) | (u64)tp << 16 | (u64)fp << 32 | (u64)el.j << 48;
            else emit_listed(c, o, r, L, wi, bt, tp, fp);
        } else if (s1 > nb) {
            nb = s1;
        }
    }
}

// Bit-sliced counts of many columns: eight columns at a time through carry-save adders
// (about 64 logic operations per eight columns instead of eight ripple additions).
constexpr int kWide = 12;  // counts <= 2048
__device__ __forceinline__ void csa(u64 &h, u64 &l, u64 a, u64 b, u64 x)
{
    const u64 u = a ^ b;
    h = (a & b) | (u & x);
    l = u ^ x;
}
__device__ __forceinline__ void wide_add8(u64 (&p)[kWide], const u64 (&x)[8], int used)
{
    u64 ta, tb, fa, fb, e;
    csa(ta, p[0], p[0], x[0], x[1]);
    csa(tb, p[0], p[0], x[2], x[3]);
    csa(fa, p[1], p[1], ta, tb);
    csa(ta, p[0], p[0], x[4], x[5]);
    csa(tb, p[0], p[0], x[6], x[7]);
    csa(fb, p[1], p[1], ta, tb);
    csa(e, p[2], p[2], fa, fb);
#pragma unroll
    for (int i = 3; i < kWide; ++i)
        if (i < used) {
            const u64 t = p[i] & e;
            p[i] ^= e;
            e = t;
        }
}

// Adds the column words wi of the samples set in the words ys (non-zero words: bits) to
// the lanes' counters p: the warp's lanes form cg groups of 32 / cg words, group `grp` takes
// every cg-th sample (listed in ids, 1536 at a time; 16 loads in flight), and the groups'
// counters are added up in the end, so that every lane of a word holds its counts.
constexpr int kIdWords = 24;
__device__ void wide_columns(const u64 *C, int GW, const u64 *ys, unsigned bits, int wi, bool in, int cg, int grp,
                             u16 *ids, u64 (&p)[kWide], int used)
{
    const int lane = threadIdx.x & 31;
    for (int w0 = 0; w0 < kMaxWords; w0 += kIdWords) {
        const unsigned part = w0 == 0 ? bits & ((1u << kIdWords) - 1u) : bits & ~((1u << kIdWords) - 1u);
        if (!part) continue;
        u64 y = (part >> lane) & 1u ? ys[lane] : 0ull;
        const int pc = __popcll(y), inc = warp_incl_scan(pc, lane), cnt = __shfl_sync(kFull, inc, 31);
        __syncwarp();
        for (int n = inc - pc; y; y &= y - 1) ids[n++] = (u16)(lane * 64 + __ffsll((long long)y) - 1);
        __syncwarp();
        for (int q0 = 0; q0 < cnt; q0 += 16 * cg) {
            u64 x[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) {
                const int q = q0 + cg * u + grp;
                x[u] = in && q < cnt ? __ldg(C + (size_t)ids[q] * GW + wi) : 0ull;
            }
#pragma unroll
            for (int v = 0; v < 16; v += 8) {
                const u64 z[8] = {x[v], x[v + 1], x[v + 2], x[v + 3], x[v + 4], x[v + 5], x[v + 6], x[v + 7]};
                wide_add8(p, z, used);
            }
        }
    }
    for (int off = 16; off >= 32 / cg; off >>= 1) {  // group sums: bit-sliced additions over the lanes of a word
        u64 carry = 0;
#pragma unroll
        for (int i = 0; i < kWide; ++i)
            if (i < used) {
                const u64 o = __shfl_xor_sync(kFull, p[i], off);
                const u64 u = p[i] ^ o, nc = (p[i] & o) | (u & carry);
                p[i] = u ^ carry;
                carry = nc;
            }
    }
}

// y (over U) and n of a prefix of L genes as words in the warp scratch, lane w forming
// word w; by / bn: the non-zero ones.  Returns |y|; kn = |n|.
__device__ __forceinline__ int dense_words(const Cohort &c, const u64 *Ush, const Prefix &p, int L, Batch &b, unsigned &by,
                                           unsigned &bn, int &kn, int lane)
{
    u64 y = 0, n = 0;
    if (lane < c.Wt) y = Ush[lane];
    if (lane < c.Wn) n = ~0ull;
#pragma unroll
    for (int i = 0; i < kMaxH - 1; ++i) {
        if (i >= L) break;
        const int g = prefix_gene(p, i);
        if (lane < c.Wt) y &= __ldg(c.T + (size_t)g * c.WTp + lane);
        if (lane < c.Wn) n &= __ldg(c.N + (size_t)g * c.WNp + lane);
    }
    __syncwarp();
    b.ys[lane] = y;
    b.ns[lane] = n;
    by = __ballot_sync(kFull, y != 0);
    bn = __ballot_sync(kFull, n != 0);
    __syncwarp();
    kn = (int)__reduce_add_sync(kFull, (unsigned)__popcll(n));
    return (int)__reduce_add_sync(kFull, (unsigned)__popcll(y));
}

// 32 / cg column words of a dense record (its y / n words in the warp scratch, k = |y|):
// leaves of scores from tau on are emitted, the best below goes to nb.  By columns, 64 leaves a lane
// at a time: |y| + |n| coalesced loads per word where the rows of the leaf genes would take
// 64 (Wt + Wn) scattered ones.  With cg > 1 the samples of a word, and then its leaves, are
// shared by cg lanes: one record is spread over all warps of the block.
__device__ __noinline__ void dense_item_level(const Cohort &c, const Solve &s, const LevelOut &o, const EmitList &el, Batch &b,
                                              const Prefix &p, unsigned by, unsigned bn, int k, int kn, int L, int lo,
                                              int wi, int cg, u64 tau, u64 &nb, bool &emitted)
{
    const int lane = threadIdx.x & 31, grp = lane / (32 / cg), last = (c.G - 1) >> 6;
    const bool in = wi <= last;
    u16 *ids = reinterpret_cast<u16 *>(b.r);
    static_assert(sizeof(b.r) >= kIdWords * 64 * sizeof(u16), "the samples of kIdWords words in the records' place");
    u64 tp[kWide], fp[kWide];
#pragma unroll
    for (int i = 0; i < kWide; ++i) tp[i] = fp[i] = 0;
    const int pt = max(bit_length(k), 3), pn = kn ? max(bit_length(kn), 3) : 0;
    wide_columns(c.CT, c.GW, b.ys, by, wi, in, cg, grp, ids, tp, pt);
    u64 m2 = 0;
#pragma unroll
    for (int i = 1; i < kWide; ++i) m2 |= tp[i];
    if (in) m2 &= range_word(wi, lo, c.G - 1);
    else m2 = 0;
    if (!__any_sync(kFull, m2 != 0)) return;
    wide_columns(c.CN, c.GW, b.ns, bn, wi, in, cg, grp, ids, fp, pn);
    const u64 top = s.a_den * (u64)c.Nn + 1;
    if (cg > 1) {  // the lane's share of the word's leaves
        const int span = 64 / cg;
        m2 &= ((1ull << span) - 1ull) << (span * grp);
    }
    while (m2) {
        const int bt = __ffsll((long long)m2) - 1;
        m2 &= m2 - 1;
        const int t = planes_get(tp, bt, pt);
        const u64 b1 = s.a_num * (u64)t + top;
        if (b1 <= nb) continue;
        const int f = planes_get(fp, bt, pn);
        const u64 s1 = b1 - s.a_den * (u64)f;
        if (s1 >= tau) {
            emitted = true;
            if (__builtin_expect(el.least != nullptr, 0)) {
                atomicMin(el.least + 2 * el.j, (u32)__ldg(c.orig + wi * 64 + bt));
                continue;
            }
            const int q = atomicAdd(el.n, 1);
            if (q < el.cap) el.em[q] = (u64)(wi * 64 + bt) | (u64)t << 16 | (u64)f << 32 | (u64)el.j << 48;
            else emit_dense(c, o, p, b.ys, L, wi * 64 + bt, t, f);
        } else if (s1 > nb) {
            nb = s1;
        }
    }
}

__device__ __forceinline__ Prefix load_prefix(const Rec *r)
{
    Prefix p;
    p.w0 = __ldcg(&r->p.w0);
    p.w1 = __ldcg(&r->p.w1);
    return p;
}

// The kept frontiers' shard offsets and sizes, read once per launch.
struct FrontTab {
    int soff[kMaxH][kShards + 1];
    long long n[kMaxH];
};

// Reads the kept frontiers' sizes; returns false (for every thread) if one overflowed.
__device__ bool front_table(const Frontiers &f, const u32 *counts, int h, FrontTab &ft, Batch &b)
{
    __shared__ int overflow;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) overflow = 0;
    __syncthreads();
    if (warp == 0) {
        for (int l = h == 2 ? 1 : 2; l <= h - 1; ++l) {
            const long long nl = front_open(counts, l, f.cap[l], b.soff, lane);
            if (nl < 0 && lane == 0) overflow = 1;
            for (int i = lane; i <= kShards; i += 32) ft.soff[l][i] = b.soff[i];
            if (lane == 0) ft.n[l] = nl;
            __syncwarp();
        }
    }
    __syncthreads();
    return overflow == 0;
}

// The records are cut into groups of R <= 32 neighbours, R the smallest power of two that
// gives every warp of the team at most one group while it can; group j belongs to block
// j mod B and, there, to warp (j / B) mod W.  A warp reads its groups' bounds together,
// records appended together spread out, and few records still reach every warp.
struct Share {
    u32 n, B, W, r, R;
    __device__ Share(u32 n_, u32 B_, u32 W_, u32 r_) : n(n_), B(B_), W(W_), r(r_), R(32)
    {
        while (R > 1 && (u64)(R / 2) * B * W >= n) R /= 2;
    }
    // the record of a lane in the warp's k-th group (>= n: none)
    __device__ u32 at(u32 k, u32 warp, u32 lane) const
    {
        return lane < R ? R * (r + B * (warp + W * k)) + lane : 0xffffffffu;
    }
    __device__ u32 steps() const  // the most groups a warp of the block has
    {
        const u32 groups = (n + R - 1) / R;
        const u32 mine = groups > r ? (groups - r + B - 1) / B : 0u;
        return (mine + W - 1) / W;
    }
};

__device__ __forceinline__ void block_level_max(u64 v, u64 *wmax, u64 *out)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = warp_max_u64(v);
    if (lane == 0) wmax[warp] = v;
    __syncthreads();
    if (warp == 0) {
        const u64 m = warp_max_u64(lane < (int)(blockDim.x >> 5) ? wmax[lane] : 0ull);
        if (lane == 0 && m) atomicMax(out, m);
    }
}

// Window entry j of the block: the column words of its leaves.
template <bool kBig>
__device__ __forceinline__ void window_tasks(const Cohort &c, LevelSh<kBig> &sh, int j, const Prefix &p, int L, bool dense)
{
    const int lo = prefix_gene(p, L - 1) + 1;
    sh.tasks[j] = lo > c.G - 1 ? 0 : ((c.G - 1) >> 6) - (lo >> 6) + 1;
    sh.nb[j] = 0;
    sh.emit[j] = 0;
    if (dense) atomicAdd(&sh.nd, 1);
}

// The block's window of nw records spread over its warps: listed records in tasks of 32
// column words, dense ones in tasks of 32 / cg words, cg the smallest that gives every
// warp two tasks (a single dense record of 19,000 genes: 38 tasks of 8 words), and no more
// words than there are (300 genes: 5 of them, and the samples of a word shared by 4 lanes).  Then the
// members found, a warp each; or (one) of each record its best leaf of score tau, see
// EmitList, and the record's |y| beside it.
template <bool kBig>
__device__ void window_eval(const Cohort &c, const Solve &s, const LevelOut &o, LevelSh<kBig> &sh, Batch &b, const u64 *Ush,
                            int nw, int L, u64 tau, bool one = false)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int words = ((c.G - 1) >> 6) + 1;
    int cg = 1;
    while (cg < 16 && (16 / cg >= words || sh.nd * ((((c.G - 1) >> 6) + 32 / cg) / (32 / cg)) < 2 * nwarps)) cg *= 2;
    const int dw = 32 / cg;
    auto ntasks = [&](int j) {
        const int per = sh.ri[j] & kDenseBit ? dw : 32;
        return (sh.tasks[j] + per - 1) / per;
    };
    const int i0 = lane < nw ? ntasks(lane) : 0;
    const int i1 = LevelSh<kBig>::kWin > 32 && lane + 32 < nw ? ntasks((lane + 32) % LevelSh<kBig>::kWin) : 0;
    const int inc0 = warp_incl_scan(i0, lane);
    const int inc1 = __shfl_sync(kFull, inc0, 31) + warp_incl_scan(i1, lane);
    const int T = __shfl_sync(kFull, inc1, 31);
    u32 *least = one ? reinterpret_cast<u32 *>(sh.em) : nullptr;
    EmitList el{sh.em, &sh.ec, LevelSh<kBig>::kEm, 0, least};
    static_assert(LevelSh<kBig>::kEm >= LevelSh<kBig>::kWin, "two words per record of the window");
    for (int x = warp; x < T; x += nwarps) {
        // its record: the number of records whose tasks end at or before x
        const int j = __popc(__ballot_sync(kFull, lane < nw && inc0 <= x)) +
                      __popc(__ballot_sync(kFull, lane + 32 < nw && inc1 <= x));
        const int e0 = __shfl_sync(kFull, inc0, (j - 1) & 31), e1 = __shfl_sync(kFull, inc1, (j - 33) & 31);
        const int first = j == 0 ? 0 : (j <= 32 ? e0 : e1);
        const Rec &r = sh.rec[j];
        const int lo = prefix_gene(r.p, L - 1) + 1;
        u64 nb = 0;
        bool emitted = false;
        el.j = j;
        if (sh.ri[j] & kDenseBit) {
            unsigned by, bn;
            int kn;
            const int k = dense_words(c, Ush, r.p, L, b, by, bn, kn, lane);
            if (one && lane == 0) least[2 * j + 1] = (u32)k;
            const int wi = (lo >> 6) + (x - first) * dw + (lane & (dw - 1));
            dense_item_level(c, s, o, el, b, r.p, by, bn, k, kn, L, lo, wi, cg, tau, nb, emitted);
            __syncwarp();
        } else {
            const int wi = (lo >> 6) + (x - first) * 32 + lane;
            if (wi <= (c.G - 1) >> 6) leaf_item_level(c, s, o, el, r, L, wi, range_word(wi, lo, c.G - 1), tau, nb, emitted);
        }
        nb = warp_max_u64(nb);
        const bool em = __any_sync(kFull, emitted);
        if (lane == 0 && nb) atomicMax(&sh.nb[j], nb);
        if (lane == 0 && em) sh.emit[j] = 1;
    }
    __syncthreads();
    if (one) return;
    const int ne = sh.ec < LevelSh<kBig>::kEm ? sh.ec : LevelSh<kBig>::kEm;
    for (int e = warp; e < ne; e += nwarps) {
        const u64 m = sh.em[e];
        const int j = (int)(m >> 48);
        emit_warp(c, o, sh.rec[j], (sh.ri[j] & kDenseBit) != 0, Ush, L, (int)(m & 0xffffull), (int)((m >> 16) & 0xffffull),
                  (int)((m >> 32) & 0xffffull));
    }
}

// Round 0 of a solve by levels, after the build: every leaf parent's best leaf with
// TP >= 2 (its bound ub, and for a listed record the leaf's key lb and the sum of TP - 1
// over those leaves, lc) and the champions give the first level.
template <bool kBig>
__device__ void level_first(const Cohort &c, const Solve &s, const Frontiers &f, LevelSh<kBig> &sh, Batch &b, const Team &t,
                            const FrontTab &ft, const u64 *Ush)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int l = s.h - 1;
    u64 *ub = f.ub[l];
    u64 best = 0;
    for (int smp = t.rank * (int)blockDim.x + (int)threadIdx.x; smp < c.Nt; smp += t.size * (int)blockDim.x) {
        const u64 v = __ldcg(&s.champ[smp].s);
        best = v > best ? v : best;
    }
    const Share sr((u32)ft.n[l], (u32)t.size, (u32)nwarps, (u32)t.rank);
    const u32 steps = sr.steps();
    if (threadIdx.x == 0) sh.qn = 0;
    __syncthreads();
    for (u32 k = 0; k < steps; ++k) {
        // listed records 32 at a time; dense ones queue up for the whole block
        const u32 i = sr.at(k, (u32)warp, (u32)lane);
        const bool in = i < sr.n;
        bool dense = false, here = false;
        if (in) {
            load_rec(&b.r[lane], f.F[l] + front_slot(f.cap[l], ft.soff[l], i));
            dense = is_dense(b.r[lane].ky, b.r[lane].kn);
        }
        if (dense) {
            const int p = atomicAdd(&sh.qn, 1);
            if (p < LevelSh<kBig>::kQ) sh.q[p] = i;
            else here = true;
        }
        leaf_parents_eval(c, s, b, in && !dense, l, lane);
        if (in && !dense) {
            Key kb = key_empty();
            if (b.pb[lane]) {
                int po[kMaxH - 1];
#pragma unroll
                for (int q = 0; q < kMaxH - 1; ++q) po[q] = q < l ? b.po[lane][q] : 0;
                kb = unpack_leaf(b.pb[lane], po, l);
            }
            ub[i] = kb.s;
            f.lb[l][i] = kb;
            f.lc[l][i] = b.rc[lane];
            best = kb.s > best ? kb.s : best;
        }
        __syncwarp();
        unsigned hm = __ballot_sync(kFull, here);
        while (hm) {  // the queue is full: by this warp alone
            const int j = __ffs(hm) - 1;
            hm &= hm - 1;
            unsigned by, bn;
            int kn;
            const u32 ij = __shfl_sync(kFull, i, j);
            const Prefix p = load_prefix(f.F[l] + front_slot(f.cap[l], ft.soff[l], ij));
            const int ky = dense_words(c, Ush, p, l, b, by, bn, kn, lane);
            const int lo = prefix_gene(p, l - 1) + 1;
            u64 nb = 0;
            bool em = false;
            for (int w0 = lo >> 6; w0 <= (c.G - 1) >> 6; w0 += 32)
                dense_item_level(c, s, LevelOut{}, EmitList{}, b, p, by, bn, ky, kn, l, lo, w0 + lane, 1, ~0ull, nb, em);
            nb = warp_max_u64(nb);
            if (lane == j) {
                ub[i] = nb;
                f.lb[l][i].s = 0;
                best = nb > best ? nb : best;
            }
            __syncwarp();
        }
    }
    __syncthreads();
    const int nq = sh.qn < LevelSh<kBig>::kQ ? sh.qn : LevelSh<kBig>::kQ;
    for (int w0 = 0; w0 < nq; w0 += LevelSh<kBig>::kWin) {
        const int nw = nq - w0 < LevelSh<kBig>::kWin ? nq - w0 : LevelSh<kBig>::kWin;
        const int j = (int)threadIdx.x;
        if (threadIdx.x == 0) sh.nd = sh.ec = 0;
        __syncthreads();
        if (j < nw) {
            const u32 i = sh.q[w0 + j];
            load_rec(&sh.rec[j], f.F[l] + front_slot(f.cap[l], ft.soff[l], i));
            sh.ri[j] = i | kDenseBit;
            window_tasks<kBig>(c, sh, j, sh.rec[j].p, l, true);
        }
        __syncthreads();
        window_eval<kBig>(c, s, LevelOut{}, sh, b, Ush, nw, l, ~0ull);
        __syncthreads();
        if (j < nw) {
            const u64 v = sh.nb[j];
            ub[sh.ri[j] & ~kDenseBit] = v;
            f.lb[l][sh.ri[j] & ~kDenseBit].s = 0;
            best = v > best ? v : best;
        }
        __syncthreads();
    }
    block_level_max(best, sh.wmax, &s.lev->lmax[0]);
}

// Bounds below Lk by distance, in units of a_num: tally j counts those at most tally_width(j)
// (and more than the next smaller one) below Lk.  16 bits each per thread, added up per block.
__device__ __forceinline__ u32 tally_width(int j) { return j & 1 ? 2u << (j >> 1) : (j == 0 ? 1u : 3u << ((j >> 1) - 1)); }
struct Tally {
    u64 n[kTally / 4] = {};
    __device__ __forceinline__ void add(u64 Lk, u64 a_num, u64 v)
    {
        const u64 d = Lk - v;
        if (d > a_num * tally_width(kTally - 1)) return;
        int j = 0;
#pragma unroll
        for (int q = 0; q < kTally - 1; ++q) j += a_num * tally_width(q) < d ? 1 : 0;
#pragma unroll
        for (int w = 0; w < kTally / 4; ++w) n[w] += j >> 2 == w ? 1ull << (16 * (j & 3)) : 0ull;
    }
    __device__ __forceinline__ void flush(u32 *out)
    {
        const int lane = threadIdx.x & 31;
        u64 any = 0;
#pragma unroll
        for (int w = 0; w < kTally / 4; ++w) any |= n[w];
        if (!__any_sync(kFull, any != 0)) return;
#pragma unroll
        for (int w = 0; w < kTally / 4; ++w) {
            const u64 v = warp_sum_u64(n[w]);
            if (lane < 4) {
                const u32 x = (u32)((v >> (16 * lane)) & 0xffffull);
                if (x) atomicAdd(out + 4 * w + lane, x);
            }
            n[w] = 0;
        }
    }
};

// The bounds' tally of the first band (the later ones are counted during the search).
template <bool kBig>
__device__ void level_tally(const Solve &s, const Frontiers &f, LevelSh<kBig> &sh, const Team &t, const FrontTab &ft, u64 Lk,
                            int step)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const u64 *ub = f.ub[s.h - 1];
    const Share sr((u32)ft.n[s.h - 1], (u32)t.size, (u32)nwarps, (u32)t.rank);
    if (threadIdx.x < kTally) sh.tally[threadIdx.x] = 0;
    __syncthreads();
    Tally ty;
    for (u32 k = 0; k < sr.steps(); ++k) {
        const u32 i = sr.at(k, (u32)warp, (u32)lane);
        const u64 v = i < sr.n ? __ldcg(ub + i) : 0ull;
        if (v) ty.add(Lk, s.a_num, v);  // (0: no leaf left)
        if ((k & 63u) == 63u) ty.flush(sh.tally);
    }
    ty.flush(sh.tally);
    __syncthreads();
    if (threadIdx.x < kTally && sh.tally[threadIdx.x]) atomicAdd(&s.lev->tally[step & 3][threadIdx.x], sh.tally[threadIdx.x]);
}

// The step after the next starts from zero (rank 0).
__device__ __forceinline__ void level_clear(const Solve &s, const Team &t, int step)
{
    if (t.rank != 0) return;
    if (threadIdx.x == 0) {
        s.lev->lmax[(step + 2) & 3] = 0;
        s.lev->mcnt[(step + 2) & 3] = 0;
    }
    if (threadIdx.x < kTally) s.lev->tally[(step + 2) & 3][threadIdx.x] = 0;
}

// The band of step `step`, scores + 1 from tau to Lk: the block's share of the leaf parents
// and champions whose scores reach tau leaves its members (counted up to `limit`), and the
// largest bound below it counts for the next band.  Every thread of the block calls it; a grid
// barrier follows.
template <bool kBig>
__device__ void level_search(const Cohort &c, const Solve &s, const Frontiers &f, LevelSh<kBig> &sh, Batch &b, const Team &t,
                             const FrontTab &ft, const u64 *Ush, u64 Lk, u64 tau, int step, u32 limit)
{
    constexpr int kIlpS = LevelSh<kBig>::kIlp, kWin = LevelSh<kBig>::kWin, kQ = LevelSh<kBig>::kQ;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int l = s.h - 1;
    u64 *ub = f.ub[l];
    level_clear(s, t, step);
    const LevelOut o{s.mem + (size_t)(step & 1) * s.mcap, &s.lev->mcnt[step & 3], s.mcap, limit, &sh.full};
    if (threadIdx.x == 0) {
        sh.full = 0;
        sh.qn = sh.en = sh.ec = sh.nd = sh.more = 0;
    }
    if (threadIdx.x < kTally) sh.tally[threadIdx.x] = 0;
    __syncthreads();
    const u64 top = s.a_den * (u64)c.Nn + 1, unit = s.a_num < s.a_den ? s.a_num : s.a_den;
    u64 next = 0;
    // with a_num = 0 a score does not depend on TP: a champion is the best of all the
    // combinations of its tumor, and one combination is picked per step
    const bool flat = s.a_num == 0;
    for (int s0 = t.rank * (int)blockDim.x; s0 < c.Nt; s0 += t.size * (int)blockDim.x) {
        const int smp = s0 + (int)threadIdx.x;
        Key k = key_empty();
        if (smp < c.Nt && in_mask(Ush, smp)) {
            const u64 v = __ldcg(&s.champ[smp].s);
            if (v >= tau) {
                k.s = v;
                k.t0 = __ldcg(&s.champ[smp].t0);
                k.t1 = __ldcg(&s.champ[smp].t1);
                k.t2 = __ldcg(&s.champ[smp].t2);
            }
            if ((v < tau || flat) && v > next) next = v;
        }
        if (flat) {
            const Key m = warp_max_key(k);
            k.s = lane == 0 ? m.s : 0;
            k.t0 = m.t0;
            k.t1 = m.t1;
            k.t2 = m.t2;
        }
        if (k.s) {
            Member *m = new_member(o, k, 1, c.Nn - (int)((k.s - 1 - s.a_num) / s.a_den));
            if (m) m->ids[0] = (u16)smp;
        }
    }
    const Share sr((u32)ft.n[l], (u32)t.size, (u32)nwarps, (u32)t.rank);
    const u32 steps = flat ? 0u : sr.steps();
    Tally ty;
    for (int pass = 0; steps > 0; ++pass) {
        // the block's bounds; those that reach tau are queued (what does not fit is found by
        // another scan after the queue is done: its bounds still reach tau)
        if (pass > 0) {
            if (threadIdx.x == 0) sh.qn = sh.en = sh.ec = sh.nd = sh.more = 0;
            __syncthreads();
        }
        for (u32 k0 = 0; k0 < steps; k0 += kIlpS) {
            u64 v[kIlpS];
#pragma unroll
            for (int u = 0; u < kIlpS; ++u) {
                const u32 i = sr.at(k0 + u, (u32)warp, (u32)lane);
                v[u] = k0 + u < steps && i < sr.n ? __ldcg(ub + i) : 0ull;
            }
#pragma unroll
            for (int u = 0; u < kIlpS; ++u) {
                const u32 i = sr.at(k0 + u, (u32)warp, (u32)lane);
                u64 w = v[u];
                if (w & kEmitted) {
                    if (pass > 0) continue;  // done in this band
                    w &= ~kEmitted;          // members of the last band
                    ub[i] = w;
                }
                if (w >= tau) {
                    const int p = atomicAdd(&sh.qn, 1);
                    if (p < kQ) sh.q[p] = i;
                    else sh.more = 1;
                } else if (w && pass == 0) {
                    next = w > next ? w : next;
                    ty.add(Lk, s.a_num, w);
                }
            }
            if ((k0 & 63u) + kIlpS >= 64u) ty.flush(sh.tally);
        }
        __syncthreads();
        const int nq = sh.qn < kQ ? sh.qn : kQ;
        const bool more = sh.more != 0;
        auto lowered = [&](u32 i, u64 v) {
            ub[i] = v;
            next = v > next ? v : next;
            if (v) ty.add(Lk, s.a_num, v);
        };
        // the queued records: their samples still in U; what the cheaper bound lowers is done,
        // an untouched listed record whose best leaf takes all its samples at FP = 0 gives its
        // cached leaf (if no other can reach tau), the others are evaluated (queue entries reused)
        for (int q0 = 0; q0 < nq; q0 += (int)blockDim.x) {
            const int qi = q0 + lane * nwarps + warp;  // few entries: one per warp
            const bool act = qi < nq;
            const u32 i = act ? sh.q[qi] : 0u;
            __syncthreads();  // entries of this pass are read before evaluations overwrite them
            Rec &r = b.r[lane];
            bool dense = false, eval = false;
            int k = 0, k0y = 0;
            const Rec *src = nullptr;
            if (act) {
                src = f.F[l] + front_slot(f.cap[l], ft.soff[l], i);
                load_rec_tumors(&r, src);
                dense = is_dense(r.ky, r.kn);
                k0y = r.ky;
                if (!dense) {
                    for (int q = 0; q < k0y; ++q) {
                        const int smp = r.ids[q];
                        if (in_mask(Ush, smp)) r.ids[k++] = (u16)smp;
                    }
                    r.ky = (u16)k;
                }
            }
            __syncwarp();
            unsigned dm = __ballot_sync(kFull, dense);
            while (dm) {  // dense: |y| from the rows, the whole warp
                const int j = __ffs(dm) - 1;
                dm &= dm - 1;
                u64 y = 0;
                if (lane < c.Wt) {
                    y = Ush[lane];
#pragma unroll
                    for (int q = 0; q < kMaxH - 1; ++q)
                        if (q < l) y &= __ldg(c.T + (size_t)prefix_gene(b.r[j].p, q) * c.WTp + lane);
                }
                const int ky = (int)__reduce_add_sync(kFull, (unsigned)__popcll(y));
                if (lane == j) k = ky;
            }
            if (act) {
                const u64 bound = k >= 2 ? s.a_num * (u64)k + top : 0ull;
                if (bound < tau) {
                    lowered(i, bound);
                } else if (!dense && k == k0y && bound - unit < tau && __ldcg(&f.lb[l][i].s) == bound) {
                    Key kc;  // (of all the record's tumors: no count in t2)
                    kc.t0 = __ldcg(&f.lb[l][i].t0);
                    kc.t1 = __ldcg(&f.lb[l][i].t1);
                    kc.t2 = __ldcg(&f.lb[l][i].t2);
                    Member *m = new_member(o, kc, k, 0);
                    if (m && k <= kMemIds)
                        for (int q = 0; q < k; ++q) m->ids[q] = r.ids[q];
                    ub[i] = bound | kEmitted;
                } else {
                    eval = true;
                }
            }
            if (eval) {
                const int p = atomicAdd(&sh.en, 1);
                if (p < kWin) {  // the first window is filled here
                    load_rec_normals(&r, src);
                    copy_rec(&sh.rec[p], &r);
                    sh.ri[p] = i | (dense ? kDenseBit : 0u);
                    window_tasks<kBig>(c, sh, p, r.p, l, dense);
                } else {
                    sh.q[p] = i;  // p < the entries read so far
                }
            }
            __syncthreads();
        }
        const int ne = sh.en;
        for (int w0 = 0; w0 < ne; w0 += kWin) {
            const int nw = ne - w0 < kWin ? ne - w0 : kWin;
            const int j = (int)threadIdx.x;
            if (w0 > 0) {
                if (threadIdx.x == 0) sh.nd = sh.ec = 0;
                __syncthreads();
                if (j < nw) {
                    const u32 i = sh.q[w0 + j];
                    Rec &r = sh.rec[j];
                    load_rec(&r, f.F[l] + front_slot(f.cap[l], ft.soff[l], i));
                    const bool dense = is_dense(r.ky, r.kn);
                    if (!dense) {
                        int k = 0;
                        for (int q = 0; q < (int)r.ky; ++q) {
                            const int smp = r.ids[q];
                            if (in_mask(Ush, smp)) r.ids[k++] = (u16)smp;
                        }
                        r.ky = (u16)k;
                    }
                    sh.ri[j] = i | (dense ? kDenseBit : 0u);
                    window_tasks<kBig>(c, sh, j, r.p, l, dense);
                }
                __syncthreads();
            }
            window_eval<kBig>(c, s, o, sh, b, Ush, nw, l, tau);
            __syncthreads();
            if (j < nw) {
                // the best leaf below the band; with members, the record is looked at again
                const u32 i = sh.ri[j] & ~kDenseBit;
                if (sh.emit[j]) {
                    ub[i] = Lk | kEmitted;
                    next = sh.nb[j] > next ? sh.nb[j] : next;
                } else {
                    lowered(i, sh.nb[j]);
                }
            }
            __syncthreads();
        }
        if (!more) break;
    }
    ty.flush(sh.tally);
    block_level_max(next, sh.wmax, &s.lev->lmax[(step + 1) & 3]);
    if (threadIdx.x < kTally && sh.tally[threadIdx.x])
        atomicAdd(&s.lev->tally[(step + 1) & 3][threadIdx.x], sh.tally[threadIdx.x]);
}

// The most members of level Lk that are worth a list, with `left` tumors uncovered: every
// pick covers at least tp of them (more normals take more tumors to the same score), so
// there are at most left / tp picks to come.  A list costs every block some passes over it,
// 0.02 us a member (0.8 us with more tumors than it lists, their rows are read), a pick
// without a list one step of about 15 us: 700 or 20 members a pick.
__device__ __forceinline__ u32 members_worth(u32 left, u32 tp, bool big)
{
    const u32 picks = max(left / max(tp, 1u), 1u);
    return big ? max(20u * picks, 64u) : max(700u * picks, 4096u);
}
__device__ __forceinline__ u32 level_worth(const Cohort &c, const Solve &s, u64 Lk, u32 left)
{
    const u64 base = s.a_den * (u64)c.Nn + 1;
    u64 tp = Lk > base && s.a_num ? (Lk - base + s.a_num - 1) / s.a_num : 1ull;
    tp = tp < 2048 ? tp : 2048;
    return min(s.mlimit, members_worth(left, (u32)tp, tp > kMemIds));
}

// (Both sides, ms of a solve, by lists of any length / as here: 60 groups of 14 tumors that
// share 100 genes, three hits, 9.7 million members 204 / 5.1; 20 groups of 30 tumors, 3.2 million
// of unlisted tumors 1666 / 4.7; 60 genes in all of 64 tumors, four hits, 0.5 million 403 / 2.4;
// 95 pairs sharing 200 genes, two hits 24 / 1.9, 17 us a pick.)

// A step of a level with more members than are worth a list: the best member of the block's
// share (score Lk, the smallest tuple) goes to the block's slot.  A record's best leaf is kept
// in lb with the number of the record's tumors in U, and is valid while that many are left (U
// only shrinks), so a step evaluates only the records that the last picks touched; the others
// are read from lb.  Every thread of the block calls it; a grid barrier follows.
template <bool kBig>
__device__ __noinline__ void level_search_one(const Cohort &c, const Solve &s, const Rec *F, u32 cap, u64 *ub, Key *lb,
                                              LevelSh<kBig> &sh, Batch &b, const Team &t, const FrontTab &ft,
                                              const u64 *Ush, u64 Lk, int step)
{
    constexpr int kWin = LevelSh<kBig>::kWin, kQ = LevelSh<kBig>::kQ;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int l = s.h - 1;
    level_clear(s, t, step);
    const u64 top = s.a_den * (u64)c.Nn + 1;
    u64 next = 0;
    u32 *least = reinterpret_cast<u32 *>(sh.em);
    Key *wb = warp_keys();  // the warp's best member so far
    if (lane == 0) wb[warp] = key_empty();
    __syncwarp();
    auto offer = [&](Key k) {  // by the whole warp; an empty key: none
        if (!__any_sync(kFull, k.s != 0)) return;
        k.t2 &= ~0xffffffffull;
        k = warp_max_key(k);
        if (lane == 0 && key_better(k, wb[warp])) wb[warp] = k;
    };
    auto load_key = [](const Key *p) {
        Key k;
        k.s = __ldcg(&p->s);
        k.t0 = __ldcg(&p->t0);
        k.t1 = __ldcg(&p->t1);
        k.t2 = __ldcg(&p->t2);
        return k;
    };
    for (int s0 = t.rank * (int)blockDim.x; s0 < c.Nt; s0 += t.size * (int)blockDim.x) {
        const int smp = s0 + (int)threadIdx.x;
        Key k = key_empty();
        if (smp < c.Nt && in_mask(Ush, smp)) {
            const u64 v = __ldcg(&s.champ[smp].s);
            if (v == Lk) k = load_key(s.champ + smp);
            else if (v < Lk && v > next) next = v;
        }
        offer(k);
    }
    const Share sr((u32)ft.n[l], (u32)t.size, (u32)nwarps, (u32)t.rank);
    const u32 steps = sr.steps();
    auto lowered = [&](u32 i, u64 v) {
        ub[i] = v;
        next = v > next ? v : next;
    };
    for (int pass = 0; steps > 0; ++pass) {  // as in level_search: what does not fit the queue is found by another scan
        if (threadIdx.x == 0) sh.qn = sh.en = sh.more = 0;
        __syncthreads();
        for (u32 k0 = 0; k0 < steps; ++k0) {
            const u32 i = sr.at(k0, (u32)warp, (u32)lane);
            u64 w = i < sr.n ? __ldcg(ub + i) : 0ull;
            if (w & kEmitted) {
                if (pass > 0) continue;  // done in this step
                w &= ~kEmitted;
                ub[i] = w;
            }
            if (w >= Lk) {
                const int p = atomicAdd(&sh.qn, 1);
                if (p < kQ) sh.q[p] = i;
                else sh.more = 1;
            } else if (w && pass == 0) {
                next = w > next ? w : next;
            }
        }
        __syncthreads();
        const int nq = sh.qn < kQ ? sh.qn : kQ;
        const bool more = sh.more != 0;
        for (int q0 = 0; q0 < nq; q0 += (int)blockDim.x) {
            const int qi = q0 + lane * nwarps + warp;
            const bool act = qi < nq;
            const u32 i = act ? sh.q[qi] : 0u;
            __syncthreads();  // entries of this pass are read before the records to evaluate overwrite them
            Rec &r = b.r[lane];
            bool dense = false;
            int k = 0, k0y = 0;
            if (act) {
                load_rec_tumors(&r, F + front_slot(cap, ft.soff[l], i));
                dense = is_dense(r.ky, r.kn);
                k0y = r.ky;
                if (!dense)
                    for (int q = 0; q < k0y; ++q) k += in_mask(Ush, r.ids[q]) ? 1 : 0;
            }
            __syncwarp();
            unsigned dm = __ballot_sync(kFull, dense);
            while (dm) {
                const int j = __ffs(dm) - 1;
                dm &= dm - 1;
                u64 y = 0;
                if (lane < c.Wt) {
                    y = Ush[lane];
#pragma unroll
                    for (int q = 0; q < kMaxH - 1; ++q)
                        if (q < l) y &= __ldg(c.T + (size_t)prefix_gene(b.r[j].p, q) * c.WTp + lane);
                }
                const int ky = (int)__reduce_add_sync(kFull, (unsigned)__popcll(y));
                if (lane == j) k = ky;
            }
            Key best = key_empty();
            if (act) {
                const u64 bound = k >= 2 ? s.a_num * (u64)k + top : 0ull;
                if (bound < Lk) {
                    lowered(i, bound);
                } else {
                    const Key kb = load_key(lb + i);
                    const int of = (int)(kb.t2 & 0xffffull);
                    if (kb.s && kb.s <= Lk && (of ? of : k0y) == k) {
                        if (kb.s == Lk) {
                            best = kb;
                            ub[i] = Lk | kEmitted;
                        } else {
                            lowered(i, kb.s);
                        }
                    } else {
                        sh.q[atomicAdd(&sh.en, 1)] = i;  // at most the entries read so far
                    }
                }
            }
            offer(best);
            __syncthreads();
        }
        const int ne = sh.en;
        for (int w0 = 0; w0 < ne; w0 += kWin) {
            const int nw = ne - w0 < kWin ? ne - w0 : kWin;
            const int j = (int)threadIdx.x;
            if (threadIdx.x == 0) sh.nd = sh.ec = 0;
            __syncthreads();
            if (j < nw) {
                const u32 i = sh.q[w0 + j];
                Rec &r = sh.rec[j];
                load_rec(&r, F + front_slot(cap, ft.soff[l], i));
                const bool dense = is_dense(r.ky, r.kn);
                int k = 0;
                if (!dense) {
                    for (int q = 0; q < (int)r.ky; ++q) {
                        const int smp = r.ids[q];
                        if (in_mask(Ush, smp)) r.ids[k++] = (u16)smp;
                    }
                    r.ky = (u16)k;
                }
                sh.ri[j] = i | (dense ? kDenseBit : 0u);
                least[2 * j] = ~0u;
                least[2 * j + 1] = (u32)k;
                window_tasks<kBig>(c, sh, j, r.p, l, dense);
            }
            __syncthreads();
            window_eval<kBig>(c, s, LevelOut{}, sh, b, Ush, nw, l, Lk, true);
            Key best = key_empty();
            if (j < nw) {
                const u32 i = sh.ri[j] & ~kDenseBit;
                if (sh.emit[j]) {
                    int po[kMaxH - 1];
                    prefix_po(c, sh.rec[j].p, l, po);
                    best = leaf_key(Lk, po, l, (int)least[2 * j]);
                    lb[i] = Key{Lk, best.t0, best.t1, best.t2 | (u64)least[2 * j + 1]};
                    ub[i] = Lk | kEmitted;
                    next = sh.nb[j] > next ? sh.nb[j] : next;
                } else {
                    lowered(i, sh.nb[j]);
                }
            }
            offer(best);
            __syncthreads();
        }
        if (!more) break;
    }
    block_level_max(next, sh.wmax, &s.lev->lmax[(step + 1) & 3]);
    if (warp == 0) {
        const Key k = warp_max_key(lane < nwarps ? wb[lane] : key_empty());
        if (lane == 0) s.slots[(size_t)(step & 1) * s.nslots + t.rank] = k;
    }
}

// Row words of the tumors that carry all genes of k, lane w: word w.
__device__ __forceinline__ u64 key_rows(const Cohort &c, const Key &k, int h, int lane)
{
    u64 y = lane < c.Wt ? ~0ull : 0ull;
#pragma unroll
    for (int q = 0; q < kMaxH; ++q)
        if (q < h && lane < c.Wt) y &= __ldg(c.TO + (size_t)key_get(k, q) * c.WTp + lane);
    return y;
}
__device__ __forceinline__ Key member_key(const Member *m)
{
    Key k;
    k.t0 = __ldcg(&m->t0);
    k.t1 = __ldcg(&m->t1);
    k.t2 = __ldcg(&m->t2);
    k.s = 0;
    return k;
}
// Score + 1 of a member with tp tumors (FP beside the tuple in t2).
__device__ __forceinline__ u64 member_score(const Cohort &c, const Solve &s, u64 t2, int tp)
{
    return s.a_num * (u64)tp + s.a_den * (u64)(c.Nn - (int)((t2 >> 16) & 0xffffull)) + 1;
}
constexpr u64 kTupleBits = ~0xffffffffull;  // of t2
// A pick: its key, TP in the low bits of t2.
__device__ __forceinline__ void record_pick(const Solve &s, const Key &k, u64 score, int pos, int tp)
{
    s.sel[pos] = Key{score, k.t0, k.t1, (k.t2 & kTupleBits) | (u64)tp};
}

// One pick: the best of the threads' keys k (score Lk or empty), with every uncovered tumor
// it covers.  sh.k is the number of picks.
template <bool kBig>
__device__ int pick_best(const Cohort &c, const Solve &s, LevelSh<kBig> &sh, u64 *Ush, Key k, u64 Lk, int K, bool lead)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    Key *wk = warp_keys();
    k = warp_max_key(k);
    if (lane == 0) wk[warp] = k;
    __syncthreads();
    if (warp == 0) {
        k = warp_max_key(lane < nwarps ? wk[lane] : key_empty());
        if (k.s) {
            const u64 y = key_rows(c, k, s.h, lane) & (lane < c.Wt ? Ush[lane] : 0ull);
            const int tp = (int)__reduce_add_sync(kFull, (unsigned)__popcll(y));
            if (lane < c.Wt) Ush[lane] &= ~y;
            if (lead)
                for (u64 x = y; x; x &= x - 1) s.covsel[lane * 64 + __ffsll((long long)x) - 1] = K;
            if (lane == 0) {
                sh.k = 1;
                if (lead) record_pick(s, k, Lk, K, tp);
            }
        }
    }
    __syncthreads();
    return sh.k;
}

// a_num = 0: one pick of the members.
template <bool kBig>
__device__ int select_flat(const Cohort &c, const Solve &s, LevelSh<kBig> &sh, u64 *Ush, const Member *mem, int n, u64 Lk,
                           int K, bool lead)
{
    Key k = key_empty();
    for (int i = (int)threadIdx.x; i < n; i += (int)blockDim.x) {
        Key m = member_key(mem + i);
        m.s = Lk;
        if (key_better(m, k)) k = m;
    }
    return pick_best<kBig>(c, s, sh, Ush, k, Lk, K, lead);
}

// One pick from the blocks' slots of level_search_one.
template <bool kBig>
__device__ int select_one(const Cohort &c, const Solve &s, LevelSh<kBig> &sh, u64 *Ush, int step, int blocks, u64 Lk, int K,
                          bool lead)
{
    const Key *slots = s.slots + (size_t)(step & 1) * s.nslots;
    Key k = key_empty();
    for (int i = (int)threadIdx.x; i < blocks; i += (int)blockDim.x) {
        Key m;
        m.s = __ldcg(&slots[i].s);
        m.t0 = __ldcg(&slots[i].t0);
        m.t1 = __ldcg(&slots[i].t1);
        m.t2 = __ldcg(&slots[i].t2);
        if (key_better(m, k)) k = m;
    }
    if (threadIdx.x == 0) sh.k = 0;
    const int got = pick_best<kBig>(c, s, sh, Ush, k, Lk, K, lead);
    if (lead && (int)threadIdx.x < c.WTp) s.U[threadIdx.x] = Ush[threadIdx.x];
    __syncthreads();  // sh.k is free again
    return got;
}

// A pool of members (list: their indexes): their tumors as row words on chip (word-major, so
// that neighbouring threads read neighbouring words), a member per thread.  A member's place
// in the tuple order is found once, so that its key is one word (score above tau, then place)
// and the best one is found by one or two 32-bit warp maxima; every warp then takes the pick's
// tumors out of its own copy of U.  Only the warps that hold members take part (up to 32
// members: one warp, no barrier).  Whole keys and a block barrier took 1.15 us per pick.  Ends
// when the best is below tau, or picks all that are left at once when each has one tumor.
// (Scores above tau fit 24 bits, see the choice of tau.)
constexpr int kPoolMax = 256;
struct PoolSh {
    u64 U[kPoolMax / 32][kMaxWords];
    u32 w[2][kPoolMax / 32];
    u32 pr[2][kPoolMax / 32];
    u64 left;
    int got;
    u32 one[kMaxSamples];  // best key of a tumor
    Key key[kPoolMax];
    u32 list[kPoolMax];
    u16 ord[kPoolMax];  // by place: the member
    u64 y[1];           // Wt x n
};
template <bool kBig>
__device__ int select_pool(const Cohort &c, const Solve &s, LevelSh<kBig> &sh, PoolSh &ps, u64 *Ush, const Member *mem, int n,
                           u64 tau, int K, bool lead, u64 &fallen)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    for (int i = warp; i < n; i += nwarps) {
        const Member *src = mem + ps.list[i];
        const Key k = member_key(src);
        const int m = (int)__ldcg(&src->k);
        const int id = lane < kMemIds ? (int)__ldcg(&src->ids[lane]) : 0;
        u64 y = 0;
        if (m <= kMemIds) {
            for (int q = 0; q < m; ++q) {
                const int x = __shfl_sync(kFull, id, q);
                if ((x >> 6) == lane) y |= 1ull << (x & 63);
            }
        } else {
            y = key_rows(c, k, s.h, lane) & (lane < c.Wt ? Ush[lane] : 0ull);
        }
        if (lane < c.Wt) ps.y[(size_t)lane * n + i] = y;
        if (lane == 0) ps.key[i] = k;
    }
    const int aw = (n + 31) / 32;
    if (warp < aw) ps.U[warp][lane] = Ush[lane];
    for (int x = (int)threadIdx.x; x < c.Nt; x += (int)blockDim.x) ps.one[x] = 0;
    if (threadIdx.x == 0) ps.left = 0;
    __syncthreads();
    if (warp < aw) {
        const auto meet = [&]() {
            if (aw > 1) asm volatile("bar.sync 1, %0;" ::"r"(32 * aw) : "memory");
            else __syncwarp();
        };
        u64 *U = ps.U[warp];
        const int i = (int)threadIdx.x;
        const bool in = i < n;
        const Key mine = in ? ps.key[i] : key_empty();
        int place = 0;
        if (in) {
            for (int j = 0; j < n; ++j) {  // (equal tuples: a champion and the leaf it is, the same pick)
                const u64 t0 = ps.key[j].t0;
                if (t0 < mine.t0) ++place;
                else if (t0 == mine.t0 && j != i) {
                    const u64 a1 = ps.key[j].t1, a2 = ps.key[j].t2 & kTupleBits, b2 = mine.t2 & kTupleBits;
                    if (a1 < mine.t1 || (a1 == mine.t1 && (a2 < b2 || (a2 == b2 && j < i)))) ++place;
                }
            }
            ps.ord[place] = (u16)i;
        }
        const u64 base = s.a_den * (u64)(c.Nn - (int)((mine.t2 >> 16) & 0xffffull)) + 1;
        auto tumors = [&]() {
            int tp = 0;
            if (in)
                for (int w = 0; w < c.Wt; ++w) tp += __popcll(ps.y[(size_t)w * n + i] & U[w]);
            return tp;
        };
        auto cover = [&](u64 y, int pos) {
            for (u64 b = y; b; b &= b - 1) s.covsel[lane * 64 + __ffsll((long long)b) - 1] = pos;
        };
        int got = 0, tp = 0;
        u32 key = 0;
        bool ones = false;
        for (int it = 0;; ++it) {
            tp = tumors();
            const u64 sc = base + s.a_num * (u64)tp;
            key = tp && sc >= tau ? (u32)(sc - tau + 1) << 8 | (u32)(255 - place) : 0u;
            u32 best = __reduce_max_sync(kFull, key);
            bool pairs = __any_sync(kFull, key != 0 && tp > 1);
            if (aw > 1) {  // (two copies: one is read while the next iteration writes the other)
                if (lane == 0) {
                    ps.w[it & 1][warp] = best;
                    ps.pr[it & 1][warp] = pairs;
                }
                meet();
                best = __reduce_max_sync(kFull, lane < aw ? ps.w[it & 1][lane] : 0u);
                pairs = __any_sync(kFull, lane < aw && ps.pr[it & 1][lane]);
            } else {
                __syncwarp();
            }
            if (best == 0) break;
            if (!pairs) {  // a tumor each
                ones = true;
                break;
            }
            const int win = ps.ord[255 - (best & 255u)];
            const u64 y = lane < c.Wt ? ps.y[(size_t)lane * n + win] & U[lane] : 0ull;
            if (lead && warp == aw - 1) {
                const int t = (int)__reduce_add_sync(kFull, (unsigned)__popcll(y));
                if (lane == 0) record_pick(s, ps.key[win], (u64)(best >> 8) - 1 + tau, K + got, t);
                cover(y, K + got);
            }
            ++got;
            __syncwarp();
            if (lane < c.Wt) U[lane] &= ~y;
            __syncwarp();
        }
        if (ones) {  // the best member of each tumor
            if (threadIdx.x == 0) ps.got = got;
            int smp = 0;
            if (key)
                for (int w = 0; w < c.Wt; ++w) {
                    const u64 y = ps.y[(size_t)w * n + i] & U[w];
                    if (y) smp = w * 64 + __ffsll((long long)y) - 1;
                }
            if (key) atomicMax(&ps.one[smp], key);
            meet();
            const bool pick = key && ps.one[smp] == key;
            int pos = 0;
            if (pick) {
                pos = atomicAdd(&ps.got, 1);
                if (lead) {
                    record_pick(s, mine, (u64)(key >> 8) - 1 + tau, K + pos, 1);
                    s.covsel[smp] = K + pos;
                }
                for (int w = 0; w < aw; ++w) atomicAnd((unsigned long long *)&ps.U[w][smp >> 6], ~(1ull << (smp & 63)));
            }
            meet();
            got = ps.got;
        }
        // what the members left over still have (TP = 1 is the champions')
        tp = tumors();
        const u64 left = warp_max_u64(in && tp >= 2 ? base + s.a_num * (u64)tp : 0ull);
        if (lane == 0 && left) atomicMax(&ps.left, left);
        if (warp == 0) {
            Ush[lane] = U[lane];
            if (lane == 0) ps.got = got;
        }
    }
    __syncthreads();
    fallen = max(fallen, ps.left);
    return ps.got;
}

// A level of many members (those of score Lk), most of them pairs: repeatedly, a member none
// of whose tumors has a better member is picked, and what meets the picks drops out (the
// lexicographically first set of disjoint ones, whatever the order of the list, in a few
// repetitions).  Members of up to four tumors and one tuple word (h <= 4)
// are worked on in shared memory, the smallest tuple per tumor as two 32-bit minima (native
// atomics; a 64-bit minimum is a loop of exchanges).
constexpr int kMany = 4096;
struct ManySh {
    u64 t[kMany];    // tuple (~0: dropped)
    u64 id[kMany];   // tumors, 16 bits each, 0xffff: none
    u32 hi[kMaxSamples], lo[kMaxSamples];
};
template <bool kBig>
__device__ int select_many(const Cohort &c, const Solve &s, LevelSh<kBig> &sh, ManySh &ms, u64 *Ush, const Member *mem, int n,
                           u64 Lk, int K, bool lead, u64 &fallen)
{
    u32 *cov32 = reinterpret_cast<u32 *>(sh.cov);
    const int T = (int)blockDim.x;
    for (int i = (int)threadIdx.x; i < n; i += T) {
        const uint4 *p = reinterpret_cast<const uint4 *>(mem + i);
        const uint4 a = __ldcg(p), d = __ldcg(p + 1);
        const int k = (int)(d.z & 0xffffu);
        const u64 raw = (u64)(d.z >> 16) | (u64)d.w << 16;          // ids 0 .. 2
        const u64 id3 = k > 3 ? (u64)__ldcg(&mem[i].ids[3]) : 0xffffull;
        u64 id = raw | id3 << 48;
        if (k < 4) id |= ~0ull << (16 * k);
        const bool in = member_score(c, s, (u64)d.y << 32 | d.x, k) == Lk;
        ms.t[i] = in ? (u64)a.y << 32 | a.x : ~0ull;
        ms.id[i] = id;
    }
    auto each = [&](u64 id, auto &&fn) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int x = (int)((id >> (16 * q)) & 0xffffull);
            if (x != 0xffff) fn(x);
        }
    };
    int picked = 0;
    for (;;) {
        for (int i = (int)threadIdx.x; i < c.Nt; i += T) ms.hi[i] = ms.lo[i] = ~0u;
        if (threadIdx.x < kMaxWords) sh.cov[threadIdx.x] = 0;
        if (threadIdx.x == 0) sh.alive = 0;
        __syncthreads();
        int live = 0;
        for (int i = (int)threadIdx.x; i < n; i += T) {
            const u64 t = ms.t[i], id = ms.id[i];
            if (t == ~0ull) continue;
            bool alive = true;
            each(id, [&](int x) { alive = alive && in_mask(Ush, x); });
            if (!alive) {
                ms.t[i] = ~0ull;
                continue;
            }
            ++live;
            each(id, [&](int x) { atomicMin(&ms.hi[x], (u32)(t >> 32)); });
        }
        live = (int)__reduce_add_sync(kFull, (unsigned)live);
        if ((threadIdx.x & 31) == 0 && live) atomicAdd(&sh.alive, live);
        __syncthreads();
        if (sh.alive == 0) break;
        for (int i = (int)threadIdx.x; i < n; i += T) {
            const u64 t = ms.t[i], id = ms.id[i];
            if (t == ~0ull) continue;
            each(id, [&](int x) { if (ms.hi[x] == (u32)(t >> 32)) atomicMin(&ms.lo[x], (u32)t); });
        }
        __syncthreads();
        for (int i = (int)threadIdx.x; i < n; i += T) {
            const u64 t = ms.t[i], id = ms.id[i];
            if (t == ~0ull) continue;
            bool top = true;
            each(id, [&](int x) { top = top && ms.hi[x] == (u32)(t >> 32) && ms.lo[x] == (u32)t; });
            if (!top) continue;
            const int pos = atomicAdd(&sh.k, 1);
            int k = 0;
            each(id, [&](int x) {
                ++k;
                atomicOr(&cov32[x >> 5], 1u << (x & 31));
                if (lead) s.covsel[x] = K + pos;
            });
            if (lead) record_pick(s, Key{Lk, t, 0ull, 0ull}, Lk, K + pos, k);
        }
        __syncthreads();
        const int alive = sh.alive, now = sh.k;
        if (threadIdx.x < kMaxWords) Ush[threadIdx.x] &= ~sh.cov[threadIdx.x];
        __syncthreads();
        if (alive == now - picked) break;  // every live member was picked
        picked = now;
    }
    const int got = sh.k;
    if (got < n) {
        u64 left = 0;
        for (int i = (int)threadIdx.x; i < n; i += T) {
            int kl = 0;
            each(ms.id[i], [&](int x) { kl += in_mask(Ush, x) ? 1 : 0; });
            if (kl) left = max(left, member_score(c, s, __ldcg(&mem[i].t2), kl));
        }
        left = warp_max_u64(left);
        if ((threadIdx.x & 31) == 0) sh.wmax[threadIdx.x >> 5] = left;
        __syncthreads();
        for (int w = 0; w < T / 32; ++w) fallen = max(fallen, sh.wmax[w]);
    }
    return got;
}

// The same for members of any size and any h, read from memory in every pass; members of
// more than kMemIds tumors from their rows, a word per lane.
// Per tumor the smallest tuple of a live member: words 0 and 1 (h <= 8: no third), and the one
// gene of word 2 that h = 9 has (the top of it, in 32 bits, so that the most tumors fit beside
// the scratch of 8 warps: every build takes every solve by levels, and a solve that a
// batch stops in one build goes on in any other).
struct BestSh {
    u64 w[2][kMaxSamples];
    u32 last[kMaxSamples];
};
static_assert(kMaxH <= 9 && sizeof(BestSh) <= kWarpsPerBlock * sizeof(Batch), "in the batch scratch of the smallest build");
template <bool kBig>
__device__ int select_any(const Cohort &c, const Solve &s, LevelSh<kBig> &sh, BestSh &best, u64 *Ush, const Member *mem,
                          int n, u64 Lk, int K, bool lead, u64 &fallen)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int h = s.h, nk = (h + 3) / 4, Nt = c.Nt;
    u32 *cov32 = reinterpret_cast<u32 *>(sh.cov);
    int picked = 0;
    for (;;) {
        for (int i = (int)threadIdx.x; i < Nt; i += (int)blockDim.x) {
            best.w[0][i] = best.w[1][i] = ~0ull;
            best.last[i] = ~0u;
        }
        if (threadIdx.x < kMaxWords) sh.cov[threadIdx.x] = 0;
        if (threadIdx.x == 0) sh.alive = 0;
        __syncthreads();
        // passes 0 .. nk - 1: per tumor the smallest tuple of a live member, 64 bits at a
        // time; the last pass picks
        for (int pass = 0; pass <= nk; ++pass) {
            for (int base = warp * 32; base < n; base += nwarps * 32) {
                const int i = base + lane;
                int k = 0;
                bool alive = false;
                uint4 v[4];
                if (i < n) {
                    const uint4 *p = reinterpret_cast<const uint4 *>(mem + i);
#pragma unroll
                    for (int q = 0; q < 4; ++q) v[q] = __ldcg(p + q);
                }
                Key key = key_empty();
                key.s = Lk;
                u32 idw[kMemIds / 2];
                bool in = false;  // a member of the level
                if (i < n) {
                    key.t0 = (u64)v[0].y << 32 | v[0].x;
                    key.t1 = (u64)v[0].w << 32 | v[0].z;
                    key.t2 = (u64)v[1].y << 32 | v[1].x;
                    k = (int)(v[1].z & 0xffffu);
                    in = member_score(c, s, key.t2, k) == Lk;
                    key.t2 &= kTupleBits;
                    const u32 w[9] = {(v[1].z >> 16) | (v[1].w << 16), (v[1].w >> 16) | (v[2].x << 16),
                                      (v[2].x >> 16) | (v[2].y << 16), (v[2].y >> 16) | (v[2].z << 16),
                                      (v[2].z >> 16) | (v[2].w << 16), (v[2].w >> 16) | (v[3].x << 16),
                                      (v[3].x >> 16) | (v[3].y << 16), (v[3].y >> 16) | (v[3].z << 16),
                                      (v[3].z >> 16) | (v[3].w << 16)};
#pragma unroll
                    for (int q = 0; q < 9; ++q) idw[q] = w[q];
                }
                const bool listed = in && k <= kMemIds;
                auto visit = [&](auto &&f) {  // f(tumor) for the listed member's tumors
#pragma unroll
                    for (int q = 0; q < kMemIds; ++q)
                        if (q < k) f((int)((idw[q / 2] >> (16 * (q & 1))) & 0xffffu));
                };
                // whether the member's tuple is the best at tumor smp as far as words < p
                auto tied = [&](const Key &kk, int smp, int p) {
                    bool e = p < 1 || best.w[0][smp] == kk.t0;
                    e = e && (p < 2 || best.w[1][smp] == kk.t1);
                    return e && (p < 3 || best.last[smp] == (u32)(kk.t2 >> 32));
                };
                auto lower = [&](const Key &kk, int smp, int p) {
                    const u64 x = p == 0 ? kk.t0 : kk.t1;
                    if (p == 2) atomicMin(&best.last[smp], (u32)(kk.t2 >> 32));
                    else if (x < best.w[p][smp]) atomicMin(&best.w[p][smp], x);
                };
                auto cover = [&](int smp, int pos) {
                    atomicOr(&cov32[smp >> 5], 1u << (smp & 31));
                    if (lead) s.covsel[smp] = K + pos;
                };
                if (listed) {
                    alive = true;
                    visit([&](int smp) { alive = alive && in_mask(Ush, smp); });
                    if (alive && pass < nk) {
                        visit([&](int smp) { if (tied(key, smp, pass)) lower(key, smp, pass); });
                    } else if (alive) {
                        bool top = true;
                        visit([&](int smp) { top = top && tied(key, smp, nk); });
                        if (top) {
                            const int pos = atomicAdd(&sh.k, 1);
                            if (lead) record_pick(s, key, Lk, K + pos, k);
                            visit([&](int smp) { cover(smp, pos); });
                        }
                    }
                }
                unsigned big = __ballot_sync(kFull, in && !listed), lives = __ballot_sync(kFull, alive);
                while (big) {  // many tumors: from the rows, a word per lane
                    const int src = __ffs(big) - 1;
                    big &= big - 1;
                    Key kk = key;
                    kk.t0 = __shfl_sync(kFull, key.t0, src);
                    kk.t1 = __shfl_sync(kFull, key.t1, src);
                    kk.t2 = __shfl_sync(kFull, key.t2, src);
                    const int kb = __shfl_sync(kFull, k, src);
                    const u64 y = key_rows(c, kk, h, lane) & (lane < c.Wt ? Ush[lane] : 0ull);
                    if ((int)__reduce_add_sync(kFull, (unsigned)__popcll(y)) != kb) continue;
                    lives |= 1u << src;
                    if (pass < nk) {
                        for (u64 x = y; x; x &= x - 1) {
                            const int smp = lane * 64 + __ffsll((long long)x) - 1;
                            if (tied(kk, smp, pass)) lower(kk, smp, pass);
                        }
                    } else {
                        bool top = true;
                        for (u64 x = y; x && top; x &= x - 1) top = tied(kk, lane * 64 + __ffsll((long long)x) - 1, nk);
                        if (!__all_sync(kFull, top)) continue;
                        int pos = 0;
                        if (lane == 0) pos = atomicAdd(&sh.k, 1);
                        pos = __shfl_sync(kFull, pos, 0);
                        if (lead && lane == 0) record_pick(s, kk, Lk, K + pos, kb);
                        for (u64 x = y; x; x &= x - 1) cover(lane * 64 + __ffsll((long long)x) - 1, pos);
                    }
                }
                if (pass == 0 && lane == 0 && lives) atomicAdd(&sh.alive, __popc(lives));
            }
            __syncthreads();
            if (pass == 0 && sh.alive == 0) break;
        }
        const int live = sh.alive, now = sh.k;
        if (threadIdx.x < kMaxWords) Ush[threadIdx.x] &= ~sh.cov[threadIdx.x];
        __syncthreads();
        // done when every live member was picked (none is left when none was alive)
        if (live == now - picked) break;
        picked = now;
    }
    const int K1 = sh.k;
    if (K1 < n) {  // what the members left over still have (the champions among them too)
        u64 left = 0;
        for (int base = warp * 32; base < n; base += nwarps * 32) {
            const int i = base + lane;
            const int k = i < n ? (int)__ldcg(&mem[i].k) : 0;
            int kl = 0;
            if (k <= kMemIds)
                for (int q = 0; q < k; ++q) kl += in_mask(Ush, (int)__ldcg(&mem[i].ids[q])) ? 1 : 0;
            if (kl) left = max(left, member_score(c, s, __ldcg(&mem[i].t2), kl));
            unsigned big = __ballot_sync(kFull, k > kMemIds);
            while (big) {
                const int src = __ffs(big) - 1;
                big &= big - 1;
                const Key ks = member_key(mem + base + src);
                const u64 y = key_rows(c, ks, h, lane) & (lane < c.Wt ? Ush[lane] : 0ull);
                const int kb = (int)__reduce_add_sync(kFull, (unsigned)__popcll(y));
                if (kb) left = max(left, member_score(c, s, ks.t2, kb));
            }
        }
        left = warp_max_u64(left);
        if (lane == 0) sh.wmax[warp] = left;
        __syncthreads();
        for (int w = 0; w < nwarps; ++w) fallen = max(fallen, sh.wmax[w]);
    }
    return K1;
}

// The picks of a band from its n members, by every block on the same input.  U of the block
// is brought up to date; the lead block (rank 0) records the picks from position K on.
// Returns their number, or -1 (nothing done) when the top level alone has more than a pool
// takes and the list is not worth its passes (open: uncovered tumors); fallen: the largest score + 1 that a member
// left over still has (a listed record's cached leaf takes all its tumors at FP = 0, so that
// score bounds the record).  Every thread of the block calls it.
template <bool kBig>
__device__ int level_select(const Cohort &c, const Solve &s, LevelSh<kBig> &sh, Batch *scratch, u64 *Ush, int n, u64 Lk,
                            u64 tau, int step, int K, bool lead, u64 &fallen, u32 open)
{
    const Member *mem = s.mem + (size_t)(step & 1) * s.mcap;
    fallen = 0;
    if (n == 0) return 0;
    static_assert(sizeof(ManySh) <= 16 * sizeof(Batch), "in the batch scratch");
    PoolSh &ps = *reinterpret_cast<PoolSh *>(scratch);
    const int room = (int)((sizeof(Batch) * (blockDim.x >> 5) - sizeof(PoolSh)) / (8 * (size_t)c.Wt));
    const int pool = min(min(kPoolMax, (int)blockDim.x), room), T = (int)blockDim.x;
    int got = 0, take = n;
    if (threadIdx.x == 0) sh.k = 0;
    if (s.a_num == 0) {
        got = select_flat<kBig>(c, s, sh, Ush, mem, n, Lk, K, lead);
    } else {
        if (n > pool && tau < Lk) {
            // the best members that the pool takes: a histogram by distance to the top, in units
            // of a_num; the others' best score goes on to the next band
            constexpr int kBins = kTallyMost + 2;
            static_assert(kBins <= kMaxSamples, "the histogram in the place of PoolSh::one");
            u32 *hist = ps.one;
            for (int i = (int)threadIdx.x; i < kBins; i += T) hist[i] = 0;
            __syncthreads();
            auto bin = [&](int i) {
                const u64 sc = member_score(c, s, __ldcg(&mem[i].t2), (int)__ldcg(&mem[i].k));
                return (int)((Lk - sc + s.a_num - 1) / s.a_num);  // <= tally_width(kTally - 1) < kBins
            };
            for (int i = (int)threadIdx.x; i < n; i += T) atomicAdd(&hist[bin(i)], 1u);
            __syncthreads();
            int q = 0;
            u32 sum = hist[0];
            take = 0;
            while (sum <= (u32)pool) {
                take = (int)sum;
                if (++q >= kBins) break;
                sum += hist[q];
            }
            --q;  // bins 0 .. q are in the pool
            if (q >= 0) tau = max(tau, Lk - s.a_num * (u64)q);
            __syncthreads();
            u64 out = 0;
            for (int i = (int)threadIdx.x; i < n; i += T) {
                if (q >= 0 && bin(i) <= q) {
                    const int p = atomicAdd(&sh.k, 1);
                    ps.list[p] = (u32)i;
                } else {
                    out = max(out, member_score(c, s, __ldcg(&mem[i].t2), (int)__ldcg(&mem[i].k)));
                }
            }
            out = warp_max_u64(out);
            if ((threadIdx.x & 31) == 0) sh.wmax[threadIdx.x >> 5] = out;
            __syncthreads();
            if (q >= 0)
                for (int w = 0; w < T / 32; ++w) fallen = max(fallen, sh.wmax[w]);
            if (threadIdx.x == 0) sh.k = 0;
            __syncthreads();
            if (q < 0) take = n;  // the top level alone is more
        } else if (n <= pool && (tau < Lk || n <= 32)) {
            for (int i = (int)threadIdx.x; i < n; i += T) ps.list[i] = (u32)i;
            __syncthreads();
        }
        if (take <= pool && (tau < Lk || take <= 32)) {
            got = take ? select_pool<kBig>(c, s, sh, ps, Ush, mem, take, tau, K, lead, fallen) : 0;
        } else {  // the top level alone (if there are others, their records are looked at again)
            // the fewest and the most tumors of a member: the same answers in every block
            u32 *few = reinterpret_cast<u32 *>(sh.wmax), *most = few + 1;
            u32 kmin = ~0u, kmax = 0;
            if (threadIdx.x == 0) {
                *few = ~0u;
                *most = 0;
            }
            __syncthreads();
            for (int i = (int)threadIdx.x; i < n; i += T) {
                const u32 k = __ldcg(&mem[i].k);
                kmin = min(kmin, k);
                kmax = max(kmax, k);
            }
            kmin = __reduce_min_sync(kFull, kmin);
            kmax = __reduce_max_sync(kFull, kmax);
            if ((threadIdx.x & 31) == 0) {
                atomicMin(few, kmin);
                atomicMax(most, kmax);
            }
            __syncthreads();
            kmin = *few;
            kmax = *most;
            if ((u32)n > min(s.mlimit, members_worth(open, kmin, kmax > (u32)kMemIds))) {
                __syncthreads();
                return -1;
            }
            if (kBig && s.h <= 4 && n <= kMany && kmax <= 4) got = select_many<kBig>(c, s, sh, *reinterpret_cast<ManySh *>(scratch), Ush, mem, n, Lk, K, lead, fallen);
            else got = select_any<kBig>(c, s, sh, *reinterpret_cast<BestSh *>(scratch), Ush, mem, n, Lk, K, lead, fallen);
        }
    }
    if (lead && (int)threadIdx.x < c.WTp) s.U[threadIdx.x] = Ush[threadIdx.x];
    __syncthreads();  // the scratch and sh.k are free again
    return got;
}

// The rounds of a finished solve: the K picks in key order (score, then tuple), the first
// maxr of them recorded as the rounds' selections, and the round cr that covers each tumor
// (R - 1, the last one searched, for the others: they are uncovered in every round).
__device__ void level_rounds(const Cohort &c, const Solve &s, const Team &t, int K, int R, int maxr)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5, h = s.h;
    for (int smp = t.rank * (int)blockDim.x + (int)threadIdx.x; smp < c.Nt; smp += t.size * (int)blockDim.x)
        if (__ldcg(s.covsel + smp) < 0) s.cr[smp] = (u16)(R - 1);
    for (int i = t.rank * nwarps + warp; i < K; i += t.size * nwarps) {
        Key k;
        k.s = __ldcg(&s.sel[i].s);
        k.t0 = __ldcg(&s.sel[i].t0);
        k.t1 = __ldcg(&s.sel[i].t1);
        k.t2 = __ldcg(&s.sel[i].t2);
        int better = 0;
        for (int j = lane; j < K; j += 32) {
            Key o;
            o.s = __ldcg(&s.sel[j].s);
            o.t0 = __ldcg(&s.sel[j].t0);
            o.t1 = __ldcg(&s.sel[j].t1);
            o.t2 = __ldcg(&s.sel[j].t2);
            better += key_better(o, k) ? 1 : 0;
        }
        const int r = (int)__reduce_add_sync(kFull, (unsigned)better);
        if (r < maxr) {
            const int tp = (int)(k.t2 & 0xffffull);
            const int fp = c.Nn - (int)((k.s - 1 - s.a_num * (u64)tp) / s.a_den);
            if (lane < h) s.res[(size_t)r * (h + 2) + lane] = key_get(k, lane);
            if (lane == 0) {
                s.res[(size_t)r * (h + 2) + h] = tp;
                s.res[(size_t)r * (h + 2) + h + 1] = fp;
            }
        }
        for (int smp = lane; smp < c.Nt; smp += 32)
            if (__ldcg(s.covsel + smp) == i) s.cr[smp] = (u16)(r < R ? r : R - 1);
    }
}

// Adds v at (round r, counter e), e = 2 (depth - 1) + 0 for visited, + 1 for surviving
// nodes: on chip (a 32-bit word and its carries), or as the change of the counter itself.
struct CountOut {
    u32 *lo, *hi;  // nullptr: straight to cnt
    u64 *cnt;
    int h2;
    __device__ __forceinline__ void add(int r, int e, u32 v) const
    {
        const int b = r * h2 + e;
        if (lo) {
            const u32 old = atomicAdd(lo + b, v);
            if (old + v < v) atomicAdd(hi + b, 1u);
        } else {
            atomicAdd(cnt + b, e == 1 ? (u64)v : 0ull - (u64)v);
        }
    }
};

// Calls add(round, times) for the tumors of y (lane w: word w) but the last-covered one, each at
// its cover round, equal rounds of a step together (with few rounds most tumors share one: a
// lane each on one counter is served one after another).  Returns the last cover round (-1: y
// is empty).
template <class F>
__device__ __forceinline__ int cover_rounds(const u16 *cr, u64 y, int lane, F &&add)
{
    int mx = -1;
    auto put = [&](int v) {
        const unsigned peers = __match_any_sync(kFull, v);
        if (v >= 0 && lane == __ffs(peers) - 1) add(v, (u32)__popc(peers));
    };
    for (u64 x = y; __any_sync(kFull, x != 0); x &= x - 1) {
        int v = -1;
        if (x) {
            const int q = cr[lane * 64 + __ffsll((long long)x) - 1];
            if (mx >= 0) v = q < mx ? q : mx;
            mx = q > mx ? q : mx;
        }
        put(v);
    }
    const int top = (int)__reduce_max_sync(kFull, (unsigned)(mx + 1)) - 1;
    const int last = __ffs(__ballot_sync(kFull, mx == top)) - 1;
    put(lane == last ? -1 : mx);
    return top;
}

// Chunk `ch` (32 column words) of a dense leaf parent's leaves: its tumors' columns in
// cover order (ord), 16 loads in flight; the sum of a tumor is added by its lane, or one sum of
// 16 tumors when they share a round.  The tumors are listed first, 128 places of the order at a
// time (1536 fit the warp's records; the rest of a longer list follows).  Bound by latency: a
// warp takes 1.4 us a group of 16 (the column words from L2) and 0.7 us to list 128 places.  All
// counters of 1000 genes, 500 tumors at 0.1, two hits, one round: 282 us with tumors shifted
// into place 16 at a time, depth 1 by 32 genes a warp and the order by counting predecessors, 58
// now; 200 genes, 2000 tumors at 0.2, three hits 927 -> 376.
__device__ __noinline__ void dense_counts(const Cohort &c, const CountOut &out, const u16 *cr, const u16 *ord, Batch &b,
                                          const Prefix &p, int l, int ch)
{
    const int lane = threadIdx.x & 31;
    const int lo = prefix_gene(p, l - 1) + 1, wi = ch * 32 + lane;
    if (lo > c.G - 1 || ch * 32 + 31 < (lo >> 6)) return;
    u64 y = lane < c.Wt ? ~0ull : 0ull;
#pragma unroll
    for (int q = 0; q < kMaxH - 1; ++q)
        if (q < l && lane < c.Wt) y &= __ldg(c.T + (size_t)prefix_gene(p, q) * c.WTp + lane);
    u16 *ids = reinterpret_cast<u16 *>(b.r);
    constexpr int kIds = (int)(sizeof(b.r) / sizeof(u16)) & ~15;
    __syncwarp();
    b.ys[lane] = y;
    __syncwarp();
    const bool on = wi <= (c.G - 1) >> 6 && wi >= (lo >> 6);
    const u64 rw = on ? range_word(wi, lo, c.G - 1) : 0ull;
    // (loads without conditions: a lane beyond the words reads the last one and drops it)
    const u64 *col = c.CT + min(wi, (c.G - 1) >> 6);
    const int GW = c.GW;
    u64 m = 0;
    int n = 0;  // tumors listed
    const int Nt = c.Nt;
    for (int q0 = 0; q0 < Nt;) {
        for (; q0 < Nt && n <= kIds - 128; q0 += 128) {
            int smp[4];
            bool in[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) smp[u] = ord[min(q0 + 32 * u + lane, Nt - 1)];
#pragma unroll
            for (int u = 0; u < 4; ++u) in[u] = q0 + 32 * u + lane < Nt && in_mask(b.ys, smp[u]);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned hit = __ballot_sync(kFull, in[u]);
                if (in[u]) ids[n + __popc(hit & ((1u << lane) - 1u))] = (u16)smp[u];
                n += __popc(hit);
            }
        }
        __syncwarp();
        const int end = q0 < Nt ? n & ~15 : n;  // whole groups of 16 while more are to come
        for (int i0 = 0; i0 < end; i0 += 16) {
            const int k = end - i0 < 16 ? end - i0 : 16;
            u64 x[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) x[q] = __ldg(col + (size_t)ids[i0 + (q < k ? q : 0)] * GW);
#pragma unroll
            for (int q = 0; q < 16; ++q) x[q] &= q < k ? rw : 0ull;
            const int first = cr[ids[i0]], last = cr[ids[i0 + k - 1]];
            if (first == last) {
                u32 sum = 0;
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    sum += (u32)__popcll(x[q] & m);
                    m |= x[q];
                }
                sum = __reduce_add_sync(kFull, sum);
                if (lane == 0 && sum) out.add(first, 2 * l + 1, sum);
            } else {
                u32 mine = 0;
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const u32 v = __reduce_add_sync(kFull, (u32)__popcll(x[q] & m));
                    m |= x[q];
                    if (lane == q) mine = v;
                }
                if (lane < k && mine) out.add(cr[ids[i0 + lane]], 2 * l + 1, mine);
            }
        }
        __syncwarp();
        const u16 rest = end + lane < n ? ids[end + lane] : (u16)0;  // fewer than 16
        __syncwarp();
        if (end + lane < n) ids[lane] = rest;
        n -= end;
    }
}

// The counters of all R rounds from cr: see the head of this file.  Every block adds its
// share of the genes (depth 1), the tumors' per-sample sums and the kept nodes into the
// rounds' counter words; level_counts_end finishes them after a grid barrier.
template <bool kBig>
__device__ void level_counts(const Cohort &c, const Solve &s, const Frontiers &f, LevelSh<kBig> &sh, Batch &b, const Team &t,
                             const FrontTab &ft, int R)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5, h = s.h, h2 = 2 * h;
    const u16 *cr = s.cr;  // written before the last grid barrier, first read after it
    const bool chip = kBig && R * h2 <= LevelSh<kBig>::kHist;
    const CountOut out{chip ? sh.hlo : nullptr, sh.hhi, s.cnt, h2};
    if (kBig) {
        for (int i = (int)threadIdx.x; i < c.Nt; i += (int)blockDim.x) sh.cr[i] = __ldcg(s.cr + i);
        cr = sh.cr;
        if (chip)
            for (int i = (int)threadIdx.x; i < R * h2; i += (int)blockDim.x) sh.hlo[i] = sh.hhi[i] = 0;
    }
    if (threadIdx.x == 0) sh.qn = 0;
    __syncthreads();
    // per-sample sums of depths 2 .. h: a tumor counts in the rounds up to its cover round
    {
        const int per = h2 - 2;
        for (int x = t.rank * (int)blockDim.x + (int)threadIdx.x; x < c.Nt * per; x += t.size * (int)blockDim.x) {
            const int smp = x / per, e = x % per;  // e: 0 .. h - 2 surviving, then visited, of depth e % (h - 1) + 2
            const int d = e % (h - 1) + 1;
            const bool vis = e >= h - 1;
            const u64 v = __ldcg(s.ssum + (size_t)smp * h2 + (vis ? h + d : d));
            if (v) atomicAdd(s.cnt + (size_t)cr[smp] * h2 + 2 * d + (vis ? 0 : 1), v);
        }
    }
    // depth 1: gene g survives up to the cover round of its last tumor; the others weigh
    // hi(2) - g each in depth 2's correction
    {
        const int last1 = c.G - h, hi2 = c.G - h + 1;
        const Share sg((u32)(last1 < 0 ? 0 : last1 + 1), (u32)t.size, (u32)nwarps, (u32)t.rank);
        for (u32 k0 = 0; k0 < sg.steps(); ++k0) {
            const u32 gi = sg.at(k0, (u32)warp, (u32)lane);
            const int g = gi < sg.n ? (int)gi : 0;
            const int k = gi < sg.n ? (int)__ldg(&c.GR[g].ky) : 0;
            if (k >= 1 && k <= kListT) {
                int mx = -1;
                for (int q = 0; q < k; ++q) {
                    const int r = cr[__ldg(&c.GR[g].ids[q])];
                    if (mx >= 0) out.add(r < mx ? r : mx, 2, (u32)(hi2 - g));
                    mx = r > mx ? r : mx;
                }
                out.add(mx, 1, 1u);
            }
            unsigned many = __ballot_sync(kFull, k > kListT);
            while (many) {
                const int gd = __shfl_sync(kFull, g, __ffs(many) - 1);
                many &= many - 1;
                const u64 y = lane < c.Wt ? __ldg(c.T + (size_t)gd * c.WTp + lane) : 0ull;
                const int top = cover_rounds(cr, y, lane, [&](int r, u32 times) { out.add(r, 2, times * (u32)(hi2 - gd)); });
                if (lane == 0) out.add(top, 1, 1u);
            }
        }
    }
    // kept nodes: depths 2 .. h - 1, and the leaves of the leaf parents
    for (int l = h == 2 ? 1 : 2; l <= h - 1; ++l) {
        const bool leafp = l == h - 1;
        const int hiN = c.G - h + l;  // hi(l + 1), 0-based
        const Share sr((u32)ft.n[l], (u32)t.size, (u32)nwarps, (u32)t.rank);
        const u32 steps = sr.steps();
        for (u32 k0 = 0; k0 < steps; ++k0) {
            const u32 i = sr.at(k0, (u32)warp, (u32)lane);
            const bool in = i < sr.n;
            Rec &r = b.r[lane];
            bool dense = false;
            int k = 0;
            __syncwarp();
            if (in) {
                load_rec(&r, f.F[l] + front_slot(f.cap[l], ft.soff[l], i));
                dense = is_dense(r.ky, r.kn);
            }
            if (in && !dense) {
                k = r.ky;
                if (k == 2) {  // a lane each: the tumor covered first
                    const int x = min((int)cr[r.ids[0]], (int)cr[r.ids[1]]);
                    if (l >= 2) {
                        out.add(x, 2 * (l - 1) + 1, 1u);
                        out.add(x, 2 * l, (u32)(hiN - prefix_gene(r.p, l - 1)));
                    }
                    if (leafp) {  // every leaf of both
                        const u64 lc = __ldcg(f.lc[l] + i);
                        if (lc) out.add(x, h2 - 1, (u32)lc);
                    }
                }
            }
            __syncwarp();
            unsigned dm = __ballot_sync(kFull, dense);
            if (l >= 2)
                while (dm) {
                    const int j = __ffs(dm) - 1;
                    dm &= dm - 1;
                    const Prefix p = b.r[j].p;
                    const u32 wt = (u32)(hiN - prefix_gene(p, l - 1));
                    u64 y = lane < c.Wt ? ~0ull : 0ull;
#pragma unroll
                    for (int q = 0; q < kMaxH - 1; ++q)
                        if (q < l && lane < c.Wt) y &= __ldg(c.T + (size_t)prefix_gene(p, q) * c.WTp + lane);
                    cover_rounds(cr, y, lane, [&](int r, u32 times) {
                        out.add(r, 2 * (l - 1) + 1, times);
                        out.add(r, 2 * l, times * wt);
                    });
                }
            if (leafp && dense) {
                const int p = atomicAdd(&sh.qn, 1);
                if (p < LevelSh<kBig>::kQ) sh.q[p] = i;  // more of them: a second scan below
            }
            // listed nodes of three tumors or more, the warp on one at a time: a lane per tumor
            // finds its place in the cover order (last first) by counting; all but the first add
            // the node's weight; then the leaves of a leaf parent, by the tumors' columns in that
            // order: a leaf seen before (it holds a later-covered tumor) counts at the cover
            // round of each further one
            unsigned todo = __ballot_sync(kFull, in && !dense && k >= 3);
            while (todo) {
                const int j = __ffs(todo) - 1;
                todo &= todo - 1;
                Rec &rj = b.r[j];
                const int kj = rj.ky, lo = prefix_gene(rj.p, l - 1) + 1;
                const int id = lane < kj ? (int)rj.ids[lane] : 0, x = lane < kj ? (int)cr[id] : -1;
                int place = 0;
                for (int q = 0; q < kj; ++q) {
                    const int o = __shfl_sync(kFull, x, q);
                    place += o > x || (o == x && q < lane) ? 1 : 0;
                }
                if (l >= 2 && lane < kj && place > 0) {
                    out.add(x, 2 * (l - 1) + 1, 1u);
                    out.add(x, 2 * l, (u32)(hiN - lo + 1));
                }
                if (!leafp || lo > c.G - 1) continue;
                __syncwarp();
                if (lane < kj) rj.ids[place] = (u16)id;
                __syncwarp();
                u32 mine = 0;  // lane q: the sum of the q-th tumor
                const int w1 = (c.G - 1) >> 6;
                if (kj <= 4) {  // four words a lane at once
                    u32 acc[4] = {0, 0, 0, 0};
                    for (int w0 = lo >> 6; w0 <= w1; w0 += 128) {
                        u64 v[4][4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int wi = w0 + 32 * u + lane;
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                v[u][q] = wi <= w1 && q < kj ? __ldg(c.CT + (size_t)rj.ids[q] * c.GW + wi) : 0ull;
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int wi = w0 + 32 * u + lane;
                            u64 m = 0;
                            const u64 rw = wi <= w1 ? range_word(wi, lo, c.G - 1) : 0ull;
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const u64 z = v[u][q] & rw;
                                acc[q] += (u32)__popcll(z & m);
                                m |= z;
                            }
                        }
                    }
#pragma unroll
                    for (int q = 1; q < 4; ++q) {
                        const u32 v = __reduce_add_sync(kFull, acc[q]);
                        if (lane == q) mine = v;
                    }
                } else {
                    u32 acc[kListT];
#pragma unroll
                    for (int q = 0; q < kListT; ++q) acc[q] = 0;
                    for (int w0 = lo >> 6; w0 <= w1; w0 += 32) {
                        const int wi = w0 + lane;
                        u64 m = 0;
                        const u64 rw = wi <= w1 ? range_word(wi, lo, c.G - 1) : 0ull;
#pragma unroll
                        for (int q0 = 0; q0 < kListT; q0 += 10) {
                            if (q0 >= kj) break;
                            u64 v[10];
#pragma unroll
                            for (int q = 0; q < 10; ++q)
                                v[q] = wi <= w1 && q0 + q < kj ? __ldg(c.CT + (size_t)rj.ids[q0 + q] * c.GW + wi) & rw : 0ull;
#pragma unroll
                            for (int q = 0; q < 10; ++q) {
                                acc[q0 + q] += (u32)__popcll(v[q] & m);
                                m |= v[q];
                            }
                        }
                    }
#pragma unroll
                    for (int q = 1; q < kListT; ++q) {
                        if (q >= kj) break;
                        const u32 v = __reduce_add_sync(kFull, acc[q]);
                        if (lane == q) mine = v;
                    }
                }
                if (mine) out.add(cr[rj.ids[lane]], h2 - 1, mine);
                __syncwarp();
            }
        }
    }
    // leaves of the dense leaf parents: the same over all tumors in cover order, in tasks
    // of 32 column words
    __syncthreads();
    const int nq = sh.qn;
    if (nq > 0) {
        // (a counting sort; the order within a round does not matter.  Counting the tumors before
        // each one took 160 us for 2000.)
        u32 *bin = reinterpret_cast<u32 *>(&b - warp);  // rounds, in the block's scratch
        static_assert((kMaxSamples + 1) * sizeof(u32) <= kWarpsPerBlock * sizeof(Batch), "a word per round");
        for (int r = (int)threadIdx.x; r < R; r += (int)blockDim.x) bin[r] = 0;
        __syncthreads();
        for (int i = (int)threadIdx.x; i < c.Nt; i += (int)blockDim.x) atomicAdd(&bin[cr[i]], 1u);
        __syncthreads();
        if (warp == 0) {
            u32 later = 0;  // tumors of the later rounds
            for (int top = R; top > 0; top -= 32) {
                const int r = top - 1 - lane;
                const u32 x = r >= 0 ? bin[r] : 0u;
                const u32 inc = (u32)warp_incl_scan((int)x, lane);
                if (r >= 0) bin[r] = later + inc - x;
                later += __shfl_sync(kFull, inc, 31);
            }
        }
        __syncthreads();
        for (int i = (int)threadIdx.x; i < c.Nt; i += (int)blockDim.x) sh.ord[atomicAdd(&bin[cr[i]], 1u)] = (u16)i;
        __syncthreads();
        const int l = h - 1, nchunk = (((c.G - 1) >> 6) + 1 + 31) >> 5;
        if (nq <= LevelSh<kBig>::kQ) {
            for (int x = warp; x < nq * nchunk; x += nwarps) {
                const Rec *src = f.F[l] + front_slot(f.cap[l], ft.soff[l], sh.q[x / nchunk]);
                dense_counts(c, out, cr, sh.ord, b, load_prefix(src), l, x % nchunk);
            }
        } else {
            const Share sr((u32)ft.n[l], (u32)t.size, (u32)nwarps, (u32)t.rank);
            for (u32 k0 = 0; k0 < sr.steps(); ++k0) {
                const u32 i = sr.at(k0, (u32)warp, (u32)lane);
                const Rec *src = i < sr.n ? f.F[l] + front_slot(f.cap[l], ft.soff[l], i) : f.F[l];
                unsigned dm = __ballot_sync(kFull, i < sr.n && is_dense(__ldcg(&src->ky), __ldcg(&src->kn)));
                while (dm) {
                    const int j = __ffs(dm) - 1;
                    dm &= dm - 1;
                    const Rec *sj = (const Rec *)__shfl_sync(kFull, (u64)src, j);
                    for (int ch = 0; ch < nchunk; ++ch) dense_counts(c, out, cr, sh.ord, b, load_prefix(sj), l, ch);
                }
            }
        }
    }
    __syncthreads();
    if (chip)
        for (int i = (int)threadIdx.x; i < R * h2; i += (int)blockDim.x) {
            const u64 v = (u64)sh.hhi[i] << 32 | sh.hlo[i];
            if (v) atomicAdd(s.cnt + i, i % h2 == 1 ? v : 0ull - v);
        }
}

// Suffix sums over the rounds, by the lead block: visited and pruned of every round.
__device__ void level_counts_end(const Cohort &c, const Solve &s, int R)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5, h = s.h;
    for (int l = warp + 1; l <= h; l += nwarps) {
        u64 cv = 0, ca = 0;  // sums over the later rounds
        for (int top = R; top > 0; top -= 128) {
            u64 v[4], a[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {  // lane 0 the latest round of its 32
                const int r = top - 1 - 32 * u - lane;
                v[u] = r >= 0 ? __ldcg(s.cnt + ((size_t)r * h + l - 1) * 2) : 0ull;
                a[u] = r >= 0 ? __ldcg(s.cnt + ((size_t)r * h + l - 1) * 2 + 1) : 0ull;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = top - 1 - 32 * u - lane;
                for (int off = 1; off < 32; off <<= 1) {
                    const u64 pv = __shfl_up_sync(kFull, v[u], off), pa = __shfl_up_sync(kFull, a[u], off);
                    if (lane >= off) {
                        v[u] += pv;
                        a[u] += pa;
                    }
                }
                v[u] += cv;
                a[u] += ca;
                cv = __shfl_sync(kFull, v[u], 31);
                ca = __shfl_sync(kFull, a[u], 31);
                if (r >= 0) {
                    const u64 vis = l == 1 ? (c.G >= h ? (u64)(c.G - h + 1) : 0ull) : v[u];
                    s.cnt[((size_t)r * h + l - 1) * 2] = vis;
                    s.cnt[((size_t)r * h + l - 1) * 2 + 1] = vis - a[u];
                }
            }
        }
    }
}
