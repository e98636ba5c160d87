// Greedy rounds by score levels, and their counters by cover rounds (included by
// mh_kernels.cu, inside its anonymous namespace).
//
// The loop of Algorithm 1 picks one combination per round.  U only shrinks, so a
// combination's TP, and with it its score, only falls, and the rounds visit scores in
// descending order: while the best score is L, the rounds take combinations of score
// L in ascending tuple order, each unless a tumor of its intersection has been covered
// since (its score then is below L for good).  So the rounds of one level are the
// lexicographically first set of pairwise disjoint intersections among the level's
// combinations, and a whole level is resolved at once: a combination that no better one
// of the level meets is picked, what it meets drops out, and so on.  The search of a
// level is one pass over the kept leaf parents whose cached bound reaches it.  A solve
// has 10 to 40 levels where it has 50 to 700 rounds, and each used to cost a chain of
// about 10 us (scan, re-evaluation, grid barrier, slot reduction, winner rows).
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
    u64 wmax[kMaxWarpsPerBlock];
    u64 cov[kMaxWords];
    u32 hlo[kHist], hhi[kHist];
    u16 cr[kBig ? kMaxSamples : 1];                   // the round that covers each tumor
    u16 ord[kMaxSamples];                             // the tumors by that round, last first
    int qn, en, alive, k;
};
constexpr u32 kDenseBit = 0x80000000u;  // queue entry: an unlisted (dense) record
constexpr u64 kEmitted = 1ull << 63;    // ub flag: emitted at the level being resolved

struct LevelOut {
    Member *out;
    u32 *count;
    u32 cap;
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

__device__ __forceinline__ Member *new_member(const LevelOut &o, const Key &k, int tp)
{
    const u32 i = atomicAdd(o.count, 1u);
    if (i >= o.cap) return nullptr;
    Member *m = o.out + i;
    m->t0 = k.t0;
    m->t1 = k.t1;
    m->t2 = k.t2;
    m->k = (u16)tp;
    return m;
}

// A leaf of listed record r (its samples those in U) at column word wi, bit bt.
__device__ __noinline__ void emit_listed(const Cohort &c, const LevelOut &o, const Rec &r, int L, int wi, int bt, int tp)
{
    int po[kMaxH - 1];
    prefix_po(c, r.p, L, po);
    Member *m = new_member(o, leaf_key(0, po, L, c.orig[wi * 64 + bt]), tp);
    if (!m || tp > kMemIds) return;
    int n = 0;
    for (int q = 0; q < (int)r.ky; ++q)
        if ((__ldg(c.CT + (size_t)r.ids[q] * c.GW + wi) >> bt) & 1ull) m->ids[n++] = r.ids[q];
}

// A leaf of a dense record, y in ys.
__device__ __noinline__ void emit_dense(const Cohort &c, const LevelOut &o, const Prefix &p, const u64 *ys, int L, int g,
                                        int tp)
{
    int po[kMaxH - 1];
    prefix_po(c, p, L, po);
    Member *m = new_member(o, leaf_key(0, po, L, c.orig[g]), tp);
    if (!m || tp > kMemIds) return;
    int n = 0;
    for (int w = 0; w < c.Wt; ++w)
        for (u64 y = ys[w] & __ldg(c.T + (size_t)g * c.WTp + w); y; y &= y - 1)
            m->ids[n++] = (u16)(w * 64 + __ffsll((long long)y) - 1);
}

// One (record, column word) item of a listed record at level Lk: its leaves of that
// score are emitted, the best one below it goes to nb.
__device__ __forceinline__ void leaf_item_level(const Cohort &c, const Solve &s, const LevelOut &o, const Rec &r, int L,
                                                int wi, u64 rw, u64 Lk, u64 &nb, bool &emitted)
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
        if (b1 <= nb) continue;  // no better than what is known below the level
        const u64 s1 = b1 - s.a_den * (u64)planes_get(fpl, bt, pn);
        if (s1 == Lk) {
            emit_listed(c, o, r, L, wi, bt, tp);
            emitted = true;
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

// Adds column word wi of every sample set in the words ys (nonzero words: bits) to p.
__device__ __forceinline__ void wide_columns(const u64 *C, int GW, const u64 *ys, unsigned bits, int wi, bool in,
                                             u64 (&p)[kWide], int used)
{
    u64 cur = 0;
    int w = 0;
    for (;;) {
        u64 x[8];
        bool more = false;
#pragma unroll
        for (int k = 0; k < 8; ++k) {  // the same sample for every lane of the warp
            while (!cur && bits) {
                w = __ffs(bits) - 1;
                bits &= bits - 1;
                cur = ys[w];
            }
            x[k] = 0;
            if (cur) {
                const int smp = w * 64 + __ffsll((long long)cur) - 1;
                cur &= cur - 1;
                if (in) x[k] = __ldg(C + (size_t)smp * GW + wi);
                more = true;
            }
        }
        if (!more) break;
        wide_add8(p, x, used);
        if (!cur && !bits) break;
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

// 32 column words of a dense record (its y / n words in the warp scratch, k = |y|):
// leaves of score Lk are emitted, the best below goes to nb.  By columns, 64 leaves a
// lane at a time: |y| + |n| coalesced loads per word where the rows of the leaf genes
// would take 64 (Wt + Wn) scattered ones.
__device__ __noinline__ void dense_item_level(const Cohort &c, const Solve &s, const LevelOut &o, Batch &b, const Prefix &p,
                                              unsigned by, unsigned bn, int k, int kn, int L, int lo, int wi, u64 Lk,
                                              u64 &nb, bool &emitted)
{
    const int last = (c.G - 1) >> 6;
    const bool in = wi <= last;
    u64 tp[kWide], fp[kWide];
#pragma unroll
    for (int i = 0; i < kWide; ++i) tp[i] = fp[i] = 0;
    const int pt = bit_length(k), pn = kn ? bit_length(kn) : 0;
    wide_columns(c.CT, c.GW, b.ys, by, wi, in, tp, pt);
    u64 m2 = 0;
#pragma unroll
    for (int i = 1; i < kWide; ++i) m2 |= tp[i];
    if (in) m2 &= range_word(wi, lo, c.G - 1);
    else m2 = 0;
    if (!__any_sync(kFull, m2 != 0)) return;
    wide_columns(c.CN, c.GW, b.ns, bn, wi, in, fp, pn);
    const u64 top = s.a_den * (u64)c.Nn + 1;
    while (m2) {
        const int bt = __ffsll((long long)m2) - 1;
        m2 &= m2 - 1;
        const int t = planes_get(tp, bt, pt);
        const u64 b1 = s.a_num * (u64)t + top;
        if (b1 <= nb) continue;
        const u64 s1 = b1 - s.a_den * (u64)planes_get(fp, bt, pn);
        if (s1 == Lk) {
            emit_dense(c, o, p, b.ys, L, wi * 64 + bt, t);
            emitted = true;
        } else if (s1 > nb) {
            nb = s1;
        }
    }
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

// Sets up window entry j of the block from queue entry e.
template <bool kBig>
__device__ __forceinline__ void window_tasks(const Cohort &c, LevelSh<kBig> &sh, int j, const Prefix &p, int L)
{
    const int lo = prefix_gene(p, L - 1) + 1;
    sh.tasks[j] = lo > c.G - 1 ? 0 : ((((c.G - 1) >> 6) - (lo >> 6) + 1 + 31) >> 5);
    sh.nb[j] = 0;
    sh.emit[j] = 0;
}

// The block's window of nw records, in tasks of 32 column words spread over its warps.
template <bool kBig>
__device__ void window_eval(const Cohort &c, const Solve &s, const LevelOut &o, LevelSh<kBig> &sh, Batch &b, const u64 *Ush,
                            int nw, int L, u64 Lk)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int i0 = lane < nw ? sh.tasks[lane] : 0;
    const int i1 = LevelSh<kBig>::kWin > 32 && lane + 32 < nw ? sh.tasks[(lane + 32) % LevelSh<kBig>::kWin] : 0;
    const int inc0 = warp_incl_scan(i0, lane);
    const int inc1 = __shfl_sync(kFull, inc0, 31) + warp_incl_scan(i1, lane);
    const int T = __shfl_sync(kFull, inc1, 31);
    for (int tau = warp; tau < T; tau += nwarps) {
        // its record: the number of records whose tasks end at or before tau
        const int j = __popc(__ballot_sync(kFull, lane < nw && inc0 <= tau)) +
                      __popc(__ballot_sync(kFull, lane + 32 < nw && inc1 <= tau));
        const int e0 = __shfl_sync(kFull, inc0, (j - 1) & 31), e1 = __shfl_sync(kFull, inc1, (j - 33) & 31);
        const int first = j == 0 ? 0 : (j <= 32 ? e0 : e1);
        const Rec &r = sh.rec[j];
        const int lo = prefix_gene(r.p, L - 1) + 1;
        const int wi = (lo >> 6) + (tau - first) * 32 + lane;
        u64 nb = 0;
        bool emitted = false;
        if (sh.ri[j] & kDenseBit) {
            unsigned by, bn;
            int kn;
            const int k = dense_words(c, Ush, r.p, L, b, by, bn, kn, lane);
            dense_item_level(c, s, o, b, r.p, by, bn, k, kn, L, lo, wi, Lk, nb, emitted);
            __syncwarp();
        } else if (wi <= (c.G - 1) >> 6) {
            leaf_item_level(c, s, o, r, L, wi, range_word(wi, lo, c.G - 1), Lk, nb, emitted);
        }
        nb = warp_max_u64(nb);
        const bool em = __any_sync(kFull, emitted);
        if (lane == 0 && nb) atomicMax(&sh.nb[j], nb);
        if (lane == 0 && em) sh.emit[j] = 1;
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
            const Prefix p = b.r[j].p;
            const int ky = dense_words(c, Ush, p, l, b, by, bn, kn, lane);
            const int lo = prefix_gene(p, l - 1) + 1;
            u64 nb = 0;
            bool em = false;
            for (int w0 = lo >> 6; w0 <= (c.G - 1) >> 6; w0 += 32)
                dense_item_level(c, s, LevelOut{nullptr, nullptr, 0u}, b, p, by, bn, ky, kn, l, lo, w0 + lane, ~0ull, nb,
                                 em);
            nb = warp_max_u64(nb);
            if (lane == j) {
                ub[i] = nb;
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
        if (j < nw) {
            const u32 i = sh.q[w0 + j];
            load_rec(&sh.rec[j], f.F[l] + front_slot(f.cap[l], ft.soff[l], i));
            sh.ri[j] = i | kDenseBit;
            window_tasks<kBig>(c, sh, j, sh.rec[j].p, l);
        }
        __syncthreads();
        window_eval<kBig>(c, s, LevelOut{nullptr, nullptr, 0u}, sh, b, Ush, nw, l, ~0ull);
        __syncthreads();
        if (j < nw) {
            const u64 v = sh.nb[j];
            ub[sh.ri[j] & ~kDenseBit] = v;
            best = v > best ? v : best;
        }
        __syncthreads();
    }
    block_level_max(best, sh.wmax, &s.lev->lmax[0]);
}

// One level Lk (score + 1) of step `step`: the block's share of the leaf parents and
// champions of that score go to the level's members, and the largest bound below it to
// the next step's level.  Every thread of the block calls it; a grid barrier follows.
template <bool kBig>
__device__ void level_search(const Cohort &c, const Solve &s, const Frontiers &f, LevelSh<kBig> &sh, Batch &b, const Team &t,
                             const FrontTab &ft, const u64 *Ush, u64 Lk, int step, bool rerun)
{
    constexpr int kIlpS = LevelSh<kBig>::kIlp;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int l = s.h - 1;
    u64 *ub = f.ub[l];
    if (t.rank == 0 && threadIdx.x == 0) {  // the step after the next starts from zero
        s.lev->lmax[(step + 2) & 3] = 0;
        s.lev->mcnt[(step + 2) & 3] = 0;
    }
    const LevelOut o{s.mem + (size_t)(step & 1) * s.mcap, &s.lev->mcnt[step & 3], s.mcap};
    const u64 top = s.a_den * (u64)c.Nn + 1;
    // what a record can still hold after a level it had members in: they fall by a_num at
    // least (level_select finds to what), its other leaves are below the level already
    const u64 fall = Lk - s.a_num;
    u64 next = 0;
    // with a_num = 0 a score does not depend on TP: a champion is the best of all the
    // combinations of its tumor, and one combination is picked per step
    const bool flat = s.a_num == 0;
    for (int s0 = t.rank * (int)blockDim.x; s0 < c.Nt; s0 += t.size * (int)blockDim.x) {
        const int smp = s0 + (int)threadIdx.x;
        Key k = key_empty();
        if (smp < c.Nt && in_mask(Ush, smp)) {
            const u64 v = __ldcg(&s.champ[smp].s);
            if (v == Lk) {
                k.s = v;
                k.t0 = __ldcg(&s.champ[smp].t0);
                k.t1 = __ldcg(&s.champ[smp].t1);
                k.t2 = __ldcg(&s.champ[smp].t2);
            }
            if ((v < Lk || flat) && v > next) next = v;
        }
        if (flat) {
            const Key m = warp_max_key(k);
            k.s = lane == 0 ? m.s : 0;
            k.t0 = m.t0;
            k.t1 = m.t1;
            k.t2 = m.t2;
        }
        if (k.s) {
            Member *m = new_member(o, k, 1);
            if (m) m->ids[0] = (u16)smp;
        }
    }
    const Share sr((u32)ft.n[l], (u32)t.size, (u32)nwarps, (u32)t.rank);
    const u32 steps = flat ? 0u : sr.steps();
    for (u32 k0 = 0; k0 < steps; k0 += kIlpS) {
        // a segment of the scan: as many records as the queue takes
        if (threadIdx.x == 0) sh.qn = sh.en = 0;
        __syncthreads();
        u64 v[kIlpS];
#pragma unroll
        for (int u = 0; u < kIlpS; ++u) {
            const u32 i = sr.at(k0 + u, (u32)warp, (u32)lane);
            v[u] = k0 + u < steps && i < sr.n ? __ldcg(ub + i) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < kIlpS; ++u) {
            const u32 i = sr.at(k0 + u, (u32)warp, (u32)lane);
            if (v[u] & kEmitted) {  // emitted at the level before, or at this one if it is run again
                v[u] = rerun ? Lk : v[u] & ~kEmitted;
                if (!rerun) ub[i] = v[u];
            }
            if (v[u] >= Lk) sh.q[atomicAdd(&sh.qn, 1)] = i;
            else if (v[u] > next) next = v[u];
        }
        __syncthreads();
        const int nq = sh.qn;
        if (nq == 0) {
            __syncthreads();
            continue;
        }
        // the queued records: their samples still in U; what the cheaper bound lowers is
        // done, an untouched listed record whose best leaf takes all its samples at FP = 0
        // gives its cached leaf, the others are evaluated (queue entries reused)
        for (int q0 = 0; q0 < nq; q0 += (int)blockDim.x) {
            const int qi = q0 + (int)threadIdx.x;
            const bool act = qi < nq;
            const u32 i = act ? sh.q[qi] : 0u;
            __syncthreads();  // entries of this pass are read before evaluations overwrite them
            Rec &r = b.r[lane];
            bool dense = false, eval = false;
            int k = 0;
            if (act) {
                load_rec(&r, f.F[l] + front_slot(f.cap[l], ft.soff[l], i));
                dense = is_dense(r.ky, r.kn);
                if (!dense) {
                    const int k0y = r.ky;
                    for (int q = 0; q < k0y; ++q) {
                        const int smp = r.ids[q];
                        if (in_mask(Ush, smp)) r.ids[k++] = (u16)smp;
                    }
                    r.ky = (u16)k;
                    const u64 bound = k >= 2 ? s.a_num * (u64)k + top : 0ull;
                    if (bound < Lk) {
                        ub[i] = bound;
                        next = bound > next ? bound : next;
                    } else if (k == k0y && bound == Lk) {
                        Key kc;
                        kc.t0 = __ldcg(&f.lb[l][i].t0);
                        kc.t1 = __ldcg(&f.lb[l][i].t1);
                        kc.t2 = __ldcg(&f.lb[l][i].t2);
                        Member *m = new_member(o, kc, k);
                        if (m && k <= kMemIds)
                            for (int q = 0; q < k; ++q) m->ids[q] = r.ids[q];
                        // (looked at again at the next level: what is left of it is known then)
                        ub[i] = (Lk - (s.a_num < s.a_den ? s.a_num : s.a_den)) | kEmitted;
                    } else {
                        eval = true;
                    }
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
                if (lane == j) {
                    const u64 bound = ky >= 2 ? s.a_num * (u64)ky + top : 0ull;
                    if (bound < Lk) {
                        ub[i] = bound;
                        next = bound > next ? bound : next;
                    } else {
                        eval = true;
                    }
                }
            }
            if (eval) {
                const int p = atomicAdd(&sh.en, 1);
                if (p < LevelSh<kBig>::kWin) {  // the first window is filled here
                    copy_rec(&sh.rec[p], &r);
                    sh.ri[p] = i | (dense ? kDenseBit : 0u);
                    window_tasks<kBig>(c, sh, p, r.p, l);
                } else {
                    sh.q[p] = i;  // p <= the entries read so far
                }
            }
            __syncthreads();
        }
        const int ne = sh.en;
        for (int w0 = 0; w0 < ne; w0 += LevelSh<kBig>::kWin) {
            const int nw = ne - w0 < LevelSh<kBig>::kWin ? ne - w0 : LevelSh<kBig>::kWin;
            const int j = (int)threadIdx.x;
            if (w0 > 0) {
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
                    window_tasks<kBig>(c, sh, j, r.p, l);
                }
                __syncthreads();
            }
            window_eval<kBig>(c, s, o, sh, b, Ush, nw, l, Lk);
            __syncthreads();
            if (j < nw) {
                // the best leaf below the level, or what its members fall to
                const u64 v = sh.nb[j];
                ub[sh.ri[j] & ~kDenseBit] = sh.emit[j] ? (fall > v ? fall : v) | kEmitted : v;
                next = v > next ? v : next;
            }
            __syncthreads();
        }
    }
    block_level_max(next, sh.wmax, &s.lev->lmax[(step + 1) & 3]);
}

// The picks of a level from its n members, by every block on the same input: repeatedly,
// a member none of whose tumors has a better member is picked (the lexicographically
// first set, whatever the order of the list), and members that meet what was picked drop
// out.  U of the block is brought up to date; the lead block (rank 0) records the picks
// from position K on.  Returns their number; fallen: the largest score + 1 that a member
// left over still has (a listed record's cached leaf takes all its tumors at FP = 0, so
// that score bounds the record).  Every thread of the block calls it.
template <bool kBig>
__device__ int level_select(const Cohort &c, const Solve &s, LevelSh<kBig> &sh, u64 *best, u64 *Ush, int n, u64 Lk, int step,
                            int K, bool lead, u64 &fallen)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int h = s.h, nk = (h + 3) / 4, Nt = c.Nt;
    const Member *mem = s.mem + (size_t)(step & 1) * s.mcap;
    u32 *cov32 = reinterpret_cast<u32 *>(sh.cov);
    auto key_word = [](const Key &k, int p) { return p == 0 ? k.t0 : (p == 1 ? k.t1 : k.t2); };
    auto load_key = [&](int i) {
        Key k;
        k.s = Lk;
        k.t0 = __ldcg(&mem[i].t0);
        k.t1 = __ldcg(&mem[i].t1);
        k.t2 = __ldcg(&mem[i].t2);
        return k;
    };
    // lane w: word w of the tumors that carry all genes of k
    auto key_rows = [&](const Key &k) {
        u64 y = lane < c.Wt ? ~0ull : 0ull;
#pragma unroll
        for (int q = 0; q < kMaxH; ++q)
            if (q < h && lane < c.Wt) y &= __ldg(c.TO + (size_t)key_get(k, q) * c.WTp + lane);
        return y;
    };
    auto record = [&](const Key &k, int pos, int tp) {
        Key r = k;
        r.t2 |= (u64)tp;  // below the tuple's bits
        s.sel[K + pos] = r;
    };
    fallen = 0;
    if (threadIdx.x == 0) sh.k = 0;
    if (s.a_num == 0) {  // one pick: the best member, with every uncovered tumor it covers
        Key k = key_empty();
        for (int i = (int)threadIdx.x; i < n; i += (int)blockDim.x) {
            const Key m = load_key(i);
            if (key_better(m, k)) k = m;
        }
        Key *wk = warp_keys();
        k = warp_max_key(k);
        if (lane == 0) wk[warp] = k;
        __syncthreads();
        if (warp == 0) {
            k = warp_max_key(lane < nwarps ? wk[lane] : key_empty());
            if (k.s) {
                const u64 y = key_rows(k) & (lane < c.Wt ? Ush[lane] : 0ull);
                const int tp = (int)__reduce_add_sync(kFull, (unsigned)__popcll(y));
                if (lane < c.Wt) Ush[lane] &= ~y;
                if (lead)
                    for (u64 x = y; x; x &= x - 1) s.covsel[lane * 64 + __ffsll((long long)x) - 1] = K;
                if (lane == 0) {
                    sh.k = 1;
                    if (lead) record(k, 0, tp);
                }
            }
        }
        __syncthreads();
        if (lead && (int)threadIdx.x < c.WTp) s.U[threadIdx.x] = Ush[threadIdx.x];
        return sh.k;
    }
    int picked = 0;
    for (;;) {
        for (int i = (int)threadIdx.x; i < nk * Nt; i += (int)blockDim.x) best[i] = ~0ull;
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
                if (i < n) {
                    key.t0 = (u64)v[0].y << 32 | v[0].x;
                    key.t1 = (u64)v[0].w << 32 | v[0].z;
                    key.t2 = (u64)v[1].y << 32 | v[1].x;
                    k = (int)(v[1].z & 0xffffu);
                    const u32 w[9] = {(v[1].z >> 16) | (v[1].w << 16), (v[1].w >> 16) | (v[2].x << 16),
                                      (v[2].x >> 16) | (v[2].y << 16), (v[2].y >> 16) | (v[2].z << 16),
                                      (v[2].z >> 16) | (v[2].w << 16), (v[2].w >> 16) | (v[3].x << 16),
                                      (v[3].x >> 16) | (v[3].y << 16), (v[3].y >> 16) | (v[3].z << 16),
                                      (v[3].z >> 16) | (v[3].w << 16)};
#pragma unroll
                    for (int q = 0; q < 9; ++q) idw[q] = w[q];
                }
                const bool listed = i < n && k <= kMemIds;
                auto visit = [&](auto &&f) {  // f(tumor) for the listed member's tumors
#pragma unroll
                    for (int q = 0; q < kMemIds; ++q)
                        if (q < k) f((int)((idw[q / 2] >> (16 * (q & 1))) & 0xffffu));
                };
                // whether the member's tuple is the best at tumor smp as far as words < p
                auto tied = [&](const Key &kk, int smp, int p) {
                    bool e = true;
                    for (int a = 0; a < p; ++a) e = e && best[a * Nt + smp] == key_word(kk, a);
                    return e;
                };
                auto lower = [&](const Key &kk, int smp, int p) {
                    const u64 x = key_word(kk, p);
                    if (x < best[p * Nt + smp]) atomicMin(&best[p * Nt + smp], x);
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
                            if (lead) record(key, pos, k);
                            visit([&](int smp) { cover(smp, pos); });
                        }
                    }
                }
                unsigned big = __ballot_sync(kFull, i < n && !listed), lives = __ballot_sync(kFull, alive);
                while (big) {  // many tumors: from the rows, a word per lane
                    const int src = __ffs(big) - 1;
                    big &= big - 1;
                    Key kk = key;
                    kk.t0 = __shfl_sync(kFull, key.t0, src);
                    kk.t1 = __shfl_sync(kFull, key.t1, src);
                    kk.t2 = __shfl_sync(kFull, key.t2, src);
                    const int kb = __shfl_sync(kFull, k, src);
                    const u64 y = key_rows(kk) & (lane < c.Wt ? Ush[lane] : 0ull);
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
                        if (lead && lane == 0) record(kk, pos, kb);
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
    if (lead && (int)threadIdx.x < c.WTp) s.U[threadIdx.x] = Ush[threadIdx.x];
    const int K1 = sh.k;
    if (K1 < n) {  // what the members left over fall to (TP = 1 is the champions')
        u64 left = 0;
        for (int base = warp * 32; base < n; base += nwarps * 32) {
            const int i = base + lane;
            const int k = i < n ? (int)__ldcg(&mem[i].k) : 0;
            int kl = 0;
            if (k <= kMemIds)
                for (int q = 0; q < k; ++q) kl += in_mask(Ush, (int)__ldcg(&mem[i].ids[q])) ? 1 : 0;
            if (kl >= 2) left = max(left, Lk - s.a_num * (u64)(k - kl));
            unsigned big = __ballot_sync(kFull, k > kMemIds);
            while (big) {
                const int src = __ffs(big) - 1;
                big &= big - 1;
                const u64 y = key_rows(load_key(base + src)) & (lane < c.Wt ? Ush[lane] : 0ull);
                const int kb = (int)__reduce_add_sync(kFull, (unsigned)__popcll(y)), k0 = __shfl_sync(kFull, k, src);
                if (kb >= 2) left = max(left, Lk - s.a_num * (u64)(k0 - kb));
            }
        }
        left = warp_max_u64(left);
        if (lane == 0) sh.wmax[warp] = left;
        __syncthreads();
        for (int w = 0; w < nwarps; ++w) fallen = max(fallen, sh.wmax[w]);
    }
    return K1;
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

// Chunk `ch` (32 column words) of a dense leaf parent's leaves: its tumors' columns in
// cover order (ord), eight loads in flight.
__device__ __noinline__ void dense_counts(const Cohort &c, const CountOut &out, const u16 *cr, const u16 *ord, Batch &b,
                                          const Rec *src, int l, int ch)
{
    const int lane = threadIdx.x & 31;
    Prefix p;
    p.w0 = __ldcg(&src->p.w0);
    p.w1 = __ldcg(&src->p.w1);
    const int lo = prefix_gene(p, l - 1) + 1, wi = ch * 32 + lane;
    if (lo > c.G - 1 || ch * 32 + 31 < (lo >> 6)) return;
    u64 y = lane < c.Wt ? ~0ull : 0ull;
#pragma unroll
    for (int q = 0; q < kMaxH - 1; ++q)
        if (q < l && lane < c.Wt) y &= __ldg(c.T + (size_t)prefix_gene(p, q) * c.WTp + lane);
    __syncwarp();
    b.ys[lane] = y;
    __syncwarp();
    const bool on = wi <= (c.G - 1) >> 6 && wi >= (lo >> 6);
    const u64 rw = on ? range_word(wi, lo, c.G - 1) : 0ull;
    u64 m = 0;
    for (int q0 = 0; q0 < c.Nt; q0 += 32) {
        const int s0 = q0 + lane < c.Nt ? (int)ord[q0 + lane] : 0;
        unsigned hit = __ballot_sync(kFull, q0 + lane < c.Nt && in_mask(b.ys, s0));
        while (hit) {
            int id[8], n = 0;
            u64 x[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                id[q] = 0;
                if (hit) {
                    id[q] = __shfl_sync(kFull, s0, __ffs(hit) - 1);
                    hit &= hit - 1;
                    n = q + 1;
                }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) x[q] = on && q < n ? __ldg(c.CT + (size_t)id[q] * c.GW + wi) & rw : 0ull;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                if (q >= n) break;
                const u32 v = __reduce_add_sync(kFull, (u32)__popcll(x[q] & m));
                m |= x[q];
                if (lane == 0 && v) out.add(cr[id[q]], 2 * l + 1, v);
            }
        }
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
        for (int g0 = (t.rank * nwarps + warp) * 32; g0 <= last1; g0 += t.size * nwarps * 32) {
            const int g = g0 + lane;
            const int k = g <= last1 ? (int)__ldg(&c.GR[g].ky) : 0;
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
                const int gd = g0 + __ffs(many) - 1;
                many &= many - 1;
                const u64 y = lane < c.Wt ? __ldg(c.T + (size_t)gd * c.WTp + lane) : 0ull;
                int mx = -1;
                for (u64 x = y; x; x &= x - 1) {
                    const int r = cr[lane * 64 + __ffsll((long long)x) - 1];
                    if (mx >= 0) out.add(r < mx ? r : mx, 2, (u32)(hi2 - gd));
                    mx = r > mx ? r : mx;
                }
                const int top = (int)__reduce_max_sync(kFull, (unsigned)(mx + 1)) - 1;
                const int lead = __ffs(__ballot_sync(kFull, mx == top)) - 1;
                if (lane == lead) out.add(top, 1, 1u);
                else if (mx >= 0) out.add(mx, 2, (u32)(hi2 - gd));
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
                const u32 wt = (u32)(hiN - prefix_gene(r.p, l - 1));
                // its tumors by cover round, last first
                for (int q = 1; q < k; ++q) {
                    const u16 id = r.ids[q];
                    const int x = cr[id];
                    int p = q - 1;
                    while (p >= 0 && (int)cr[r.ids[p]] < x) {
                        r.ids[p + 1] = r.ids[p];
                        --p;
                    }
                    r.ids[p + 1] = id;
                }
                if (l >= 2)
                    for (int q = 1; q < k; ++q) {
                        const int x = cr[r.ids[q]];
                        out.add(x, 2 * (l - 1) + 1, 1u);
                        out.add(x, 2 * l, wt);
                    }
                if (leafp && k == 2) {  // both tumors: every leaf with TP = 2
                    const u64 lc = __ldcg(f.lc[l] + i);
                    if (lc) out.add(cr[r.ids[1]], h2 - 1, (u32)lc);
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
                    int mx = -1;
                    auto put = [&](int x) {
                        out.add(x, 2 * (l - 1) + 1, 1u);
                        out.add(x, 2 * l, wt);
                    };
                    for (u64 x = y; x; x &= x - 1) {
                        const int q = cr[lane * 64 + __ffsll((long long)x) - 1];
                        if (mx >= 0) put(q < mx ? q : mx);
                        mx = q > mx ? q : mx;
                    }
                    const int top = (int)__reduce_max_sync(kFull, (unsigned)(mx + 1)) - 1;
                    const int lead = __ffs(__ballot_sync(kFull, mx == top)) - 1;
                    if (lane != lead && mx >= 0) put(mx);
                }
            if (!leafp) continue;
            if (dense) {
                const int p = atomicAdd(&sh.qn, 1);
                if (p < LevelSh<kBig>::kQ) sh.q[p] = i;  // more of them: a second scan below
            }
            // leaves of the listed leaf parents with three tumors or more: the tumors'
            // columns in that order; a leaf seen before (it holds a later-covered tumor)
            // counts at the cover round of each further one
            unsigned todo = __ballot_sync(kFull, in && !dense && k >= 3);
            while (todo) {
                const int j = __ffs(todo) - 1;
                todo &= todo - 1;
                const Rec &rj = b.r[j];
                const int kj = rj.ky, lo = prefix_gene(rj.p, l - 1) + 1;
                u32 acc[kListT];
#pragma unroll
                for (int q = 0; q < kListT; ++q) acc[q] = 0;
                for (int w0 = lo >> 6; w0 <= (c.G - 1) >> 6; w0 += 32) {
                    const int wi = w0 + lane;
                    const bool on = wi <= (c.G - 1) >> 6;
                    u64 m = 0;
                    const u64 rw = on && lo <= c.G - 1 ? range_word(wi, lo, c.G - 1) : 0ull;
#pragma unroll
                    for (int q0 = 0; q0 < kListT; q0 += 4) {
                        if (q0 >= kj) break;
                        u64 x[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            x[q] = on && q0 + q < kj ? __ldg(c.CT + (size_t)rj.ids[q0 + q] * c.GW + wi) & rw : 0ull;
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            acc[q0 + q] += (u32)__popcll(x[q] & m);
                            m |= x[q];
                        }
                    }
                }
#pragma unroll
                for (int q = 1; q < kListT; ++q) {
                    if (q >= kj) break;
                    const u32 v = __reduce_add_sync(kFull, acc[q]);
                    if (lane == 0 && v) out.add(cr[rj.ids[q]], h2 - 1, v);
                }
            }
        }
    }
    // leaves of the dense leaf parents: the same over all tumors in cover order, in tasks
    // of 32 column words
    __syncthreads();
    const int nq = sh.qn;
    if (nq > 0) {
        for (int i = (int)threadIdx.x; i < c.Nt; i += (int)blockDim.x) {
            const int x = cr[i];
            int pos = 0;
            for (int j = 0; j < c.Nt; ++j) {
                const int y = cr[j];
                pos += (y > x || (y == x && j < i)) ? 1 : 0;
            }
            sh.ord[pos] = (u16)i;
        }
        __syncthreads();
        const int l = h - 1, nchunk = (((c.G - 1) >> 6) + 1 + 31) >> 5;
        if (nq <= LevelSh<kBig>::kQ) {
            for (int tau = warp; tau < nq * nchunk; tau += nwarps) {
                const Rec *src = f.F[l] + front_slot(f.cap[l], ft.soff[l], sh.q[tau / nchunk]);
                dense_counts(c, out, cr, sh.ord, b, src, l, tau % nchunk);
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
                    for (int ch = 0; ch < nchunk; ++ch) dense_counts(c, out, cr, sh.ord, b, sj, l, ch);
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
