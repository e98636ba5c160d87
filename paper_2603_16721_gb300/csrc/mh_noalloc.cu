// mh_solve_noalloc: the greedy solve of mh_solve for callers that cannot
// allocate device memory.
//
// Some callers cannot call cudaMalloc: code that runs while another component
// owns every byte of device memory through its own pool, plug-ins that are handed
// fixed buffers by a host framework, or callers that must not add allocator
// traffic (and its implicit synchronisation) to a latency-critical stream.  For
// them this entry point keeps every piece of scratch -- the sorted cohort store,
// its sample-major copies and lists, the uncovered-tumor mask, the search frontiers, the
// members and picks of the score levels, the counters and the round state -- in one
// file-scope __device__ array of fixed size.  The caller passes the packed rows
// and the output buffers, both in device memory.  Nothing here calls cudaMalloc,
// cudaFree or any allocating library routine, and the success path touches no
// host heap either.
//
// Every GPU that loads this library keeps the array (kScratchBytes) until the
// process exits.  The solve is the persistent one (by score levels, as mh_solve's), in the
// fixed pieces; where one of them is too small for it -- more than kNaLists mutations, a
// frontier of shared nodes beyond its region, no room for the cooperative launch -- the rounds
// run one kernel per phase instead, which needs none of these pieces.  Any other error of the
// persistent solve is returned.  Every call shares the array: calls whose work overlaps on the GPU
// (different streams, different host threads) race on it and must be
// serialised by the caller.  What must start at zero is cleared by each call.
#include <cstdarg>
#include <cstdio>
#include <cstring>

#include "mh.h"
#include "mh_internal.h"

namespace mh {

namespace {

// Limits of the no-allocation solve.
constexpr int kNaMaxG = 8192;
constexpr int kNaMaxNt = 1024;
constexpr int kNaMaxNn = 1024;
constexpr int kNaMaxH = 4;
constexpr u32 kNaFrontierCap = 1u << 17;  // entries per intermediate depth
constexpr int kNaMaxSlots = 4096;

constexpr int kNaWTp = kNaMaxNt / 64;  // 16 words
constexpr int kNaWNp = kNaMaxNn / 64;
constexpr int kNaGW = kNaMaxG / 64;    // 128 words
constexpr int kNaRounds = kNaMaxNt + 2;

constexpr size_t kNaLists = 1u << 20;        // tumor mutations listed (SL, SLo)
constexpr u32 kNaMembers = 1u << 16;         // members listed of a band of score levels

constexpr size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

// Byte offsets of the pieces inside the scratch array.
constexpr size_t kOffT = 0;
constexpr size_t kOffN = kOffT + align256(sizeof(u64) * kNaMaxG * kNaWTp);
constexpr size_t kOffTO = kOffN + align256(sizeof(u64) * kNaMaxG * kNaWNp);
constexpr size_t kOffNO = kOffTO + align256(sizeof(u64) * kNaMaxG * kNaWTp);
constexpr size_t kOffCT = kOffNO + align256(sizeof(u64) * kNaMaxG * kNaWNp);
constexpr size_t kOffCN = kOffCT + align256(sizeof(u64) * kNaMaxNt * kNaGW);
constexpr size_t kOffCTo = kOffCN + align256(sizeof(u64) * kNaMaxNn * kNaGW);
constexpr size_t kOffCC = kOffCTo + align256(sizeof(u64) * kNaMaxNt * kNaGW);
constexpr size_t kOffSL = kOffCC + align256(sizeof(u16) * kNaMaxNt * (kNaGW + 1));
constexpr size_t kOffSLo = kOffSL + align256(sizeof(u16) * kNaLists);
constexpr size_t kOffSO = kOffSLo + align256(sizeof(u16) * kNaLists);
constexpr size_t kOffGR = kOffSO + align256(sizeof(u32) * (kNaMaxNt + 1));
constexpr size_t kOffOrig = kOffGR + align256(sizeof(Rec) * kNaMaxG);
constexpr size_t kOffInv = kOffOrig + align256(sizeof(u16) * kNaMaxG);
constexpr size_t kOffKeys = kOffInv + align256(sizeof(u32) * kNaMaxG);
constexpr size_t kOffOrder = kOffKeys + align256(sizeof(u32) * kNaMaxG);
constexpr size_t kOffU = kOffOrder + align256(sizeof(u32) * kNaMaxG);
// one block, read back in one copy: the state, the store build's words, the frontier counts
constexpr size_t kOffState = kOffU + align256(sizeof(u64) * kNaWTp);
constexpr size_t kOffPrep = kOffState + 64;
constexpr size_t kOffCounts = kOffState + 256;
constexpr size_t kOffMs = kOffCounts + align256(sizeof(u32) * kCountSets * kCountWords);
constexpr size_t kOffWork = kOffMs + align256(sizeof(u32) * kNaMaxNt);
constexpr size_t kOffSync = kOffWork + align256(sizeof(u64) * (kWorkCount + kCountSets));
constexpr size_t kOffRes = kOffSync + align256(sizeof(GridSync));
constexpr size_t kOffCnt = kOffRes + align256(sizeof(int) * kNaRounds * (kNaMaxH + 2));
constexpr size_t kOffSlots = kOffCnt + align256(sizeof(u64) * 2 * kNaRounds * kNaMaxH);
constexpr size_t kOffCand = kOffSlots + align256(sizeof(Key) * kCountSets * kNaMaxSlots);
constexpr size_t kOffChamp = kOffCand + align256(sizeof(Key) * kCandidates);
constexpr size_t kOffChampOk = kOffChamp + align256(sizeof(Key) * kNaMaxNt);
constexpr size_t kOffSsum = kOffChampOk + align256(sizeof(int) * kNaMaxNt);
constexpr size_t kOffLevel = kOffSsum + align256(sizeof(u64) * kNaMaxNt * 2 * kNaMaxH);
constexpr size_t kOffSel = kOffLevel + align256(kLevelBytes);
constexpr size_t kOffCovsel = kOffSel + align256(sizeof(Key) * kNaMaxNt);
constexpr size_t kOffCr = kOffCovsel + align256(sizeof(int) * kNaMaxNt);
constexpr size_t kOffMem = kOffCr + align256(sizeof(u16) * kNaMaxNt);
constexpr size_t kOffF1 = kOffMem + align256(sizeof(Member) * 2 * kNaMembers);
constexpr size_t kOffF2 = kOffF1 + align256(sizeof(Rec) * kNaMaxG);
constexpr size_t kOffF3 = kOffF2 + align256(sizeof(Rec) * kNaFrontierCap);
// per leaf parent (of one depth): lb, ub, lc
constexpr size_t kOffLb = kOffF3 + align256(sizeof(Rec) * kNaFrontierCap);
constexpr size_t kOffUb = kOffLb + align256(sizeof(Key) * kNaFrontierCap);
constexpr size_t kOffLc = kOffUb + align256(sizeof(u64) * kNaFrontierCap);
constexpr size_t kScratchBytes = kOffLc + align256(sizeof(u64) * kNaFrontierCap);  // about 54 MB
static_assert(sizeof(int) * kStateWords <= 64, "the store build's words follow the state");
static_assert(kNaMaxG <= kNaLists, "one tumor's list always has room");

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

// Words at kOffPrep (cleared before the build): padding bits found; tumor mutations.
enum { kPrepBad = 0, kPrepMutations = 1, kPrepWords = 2 };

// Sort key of every gene, 12-bit tumor count above its 16-bit index (keys are unique, so their
// order is the stable "most sparse first, ties by index"), and every tumor's mutated genes (m).
// A thread per gene; counts in shared memory first.  Flags padding bits that are set.
constexpr int kNaKeyThreads = 128;
__global__ void __launch_bounds__(kNaKeyThreads) k_na_keys(const u64 *bm, int G, int Nt, int Nn, u32 *keys, u32 *m, int *prep)
{
    __shared__ u32 hist[kNaMaxNt];
    const int Wt = (Nt + 63) / 64, Wn = (Nn + 63) / 64;
    for (int i = threadIdx.x; i < Nt; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < G) {
        const u64 *row = bm + (size_t)g * (Wt + Wn);
        bool bad = Wn && (Nn & 63) && (row[Wt + Wn - 1] >> (Nn & 63));
        int pc = 0;
        for (int w = 0; w < Wt; ++w) {
            u64 x = row[w];
            pc += __popcll(x);
            if (w == Wt - 1 && (Nt & 63)) {
                if (x >> (Nt & 63)) bad = true;
                x &= (1ull << (Nt & 63)) - 1;
            }
            for (; x; x &= x - 1) atomicAdd(&hist[w * 64 + __ffsll((long long)x) - 1], 1u);
        }
        keys[g] = ((u32)pc << 16) | (u32)g;
        if (bad) atomicOr(prep + kPrepBad, 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < Nt; i += blockDim.x)
        if (hist[i]) atomicAdd(&m[i], hist[i]);
}

// order = the genes by key, each placed by the number of smaller keys: a warp per gene, all
// keys in shared memory (G^2 comparisons spread over the chip, 5 us at G = 8192, where a sort in
// one block took 90 steps between barriers).  The last block adds up the tumors' list offsets
// instead; lists too long for their pieces all start at 0 (they fit one by one, and the caller
// sees the total).
constexpr int kNaRankGenes = 64;  // per block
__global__ void __launch_bounds__(1024) k_na_rank(const u32 *keys, int G, u32 *order, const u32 *m, int Nt, u32 *SO, int *prep)
{
    __shared__ u32 sh[kNaMaxG];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (blockIdx.x == gridDim.x - 1) {
        const u32 mine = (int)threadIdx.x < Nt ? m[threadIdx.x] : 0;
        u32 v = mine;
        sh[threadIdx.x] = v;
        __syncthreads();
        for (int off = 1; off < 1024; off <<= 1) {
            const u32 o = (int)threadIdx.x >= off ? sh[threadIdx.x - off] : 0;
            __syncthreads();
            sh[threadIdx.x] = v += o;
            __syncthreads();
        }
        const u32 total = sh[1023];
        const bool fits = total <= kNaLists;
        if ((int)threadIdx.x < Nt) SO[threadIdx.x] = fits ? v - mine : 0;
        if (threadIdx.x == 0) {
            SO[Nt] = fits ? total : 0;
            prep[kPrepMutations] = (int)total;
        }
        return;
    }
    for (int i = threadIdx.x; i < G; i += blockDim.x) sh[i] = keys[i];
    __syncthreads();
    for (int k = warp; k < kNaRankGenes; k += 32) {
        const int g = blockIdx.x * kNaRankGenes + k;
        if (g >= G) break;
        const u32 key = sh[g];
        int n = 0;
        for (int i = lane; i < G; i += 32) n += sh[i] < key;
        n = __reduce_add_sync(0xffffffffu, n);
        if (lane == 0) order[n] = (u32)g;
    }
}

__global__ void k_na_unpack(const int *res, const int *state, int h, int capacity, int32_t *genes, int32_t *tp,
                            int32_t *fp, bool finished)
{
    if (finished && !state[1]) return;  // stopped early: the rounds run again
    const int k = state[0] < capacity ? state[0] : capacity;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < k; i += gridDim.x * blockDim.x) {
        const int *r = res + (size_t)i * (h + 2);
        for (int j = 0; j < h; ++j) genes[(size_t)i * h + j] = r[j];
        tp[i] = r[h];
        fp[i] = r[h + 1];
    }
}

int na_fail(int code, const char *fmt, ...)
{
    char buf[384];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    set_error_text(buf);
    return code;
}

#define NA_CUDA(call)                                                                                  \
    do {                                                                                               \
        cudaError_t e_ = (call);                                                                       \
        if (e_ != cudaSuccess) return na_fail(MH_ECUDA, "%s: %s", #call, cudaGetErrorString(e_));      \
    } while (0)

// Device address of the scratch array on the current device, looked up on every
// call: an address kept from an earlier call would be stale after a device reset
// or with a new primary context, and the lookup costs little next to a solve.
int scratch_for_current_device(unsigned char **ptr, int *num_sms)
{
    int dev = 0;
    NA_CUDA(cudaGetDevice(&dev));
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p)
        return na_fail(MH_ECUDA, "cudaGetSymbolAddress of the scratch array failed: %s", cudaGetErrorString(e));
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return na_fail(MH_ECUDA, "cudaDeviceGetAttribute: %s", cudaGetErrorString(e));
    *ptr = (unsigned char *)p;
    *num_sms = sms;
    return MH_OK;
}

}  // namespace

}  // namespace mh

using namespace mh;

extern "C" MH_API int mh_solve_noalloc(const uint64_t *d_bitmaps, int32_t G, int32_t Nt, int32_t Nn, int32_t h,
                                       mh_rational alpha, void *stream, int32_t *d_genes, int32_t *d_tp,
                                       int32_t *d_fp, int32_t capacity, int32_t *k_out, int32_t *rounds_out)
{
    if (!d_bitmaps || !d_genes || !d_tp || !d_fp || !k_out)
        return na_fail(MH_EINVAL, "mh_solve_noalloc: NULL input or output pointer");
    if (G < 1 || G > kNaMaxG || Nt < 0 || Nt > kNaMaxNt || Nn < 0 || Nn > kNaMaxNn)
        return na_fail(MH_EINVAL,
                       "mh_solve_noalloc: G=%d Nt=%d Nn=%d exceed the fixed scratch (G <= %d, Nt <= %d, Nn <= %d)",
                       G, Nt, Nn, kNaMaxG, kNaMaxNt, kNaMaxNn);
    if (h < 1 || h > kNaMaxH) return na_fail(MH_EINVAL, "mh_solve_noalloc: h=%d outside [1, %d]", h, kNaMaxH);
    if (alpha.num < 0 || alpha.den <= 0)
        return na_fail(MH_EINVAL, "mh_solve_noalloc: alpha=%d/%d needs num >= 0, den > 0", alpha.num, alpha.den);
    if (capacity < Nt) return na_fail(MH_EINVAL, "mh_solve_noalloc: capacity %d < Nt=%d", capacity, Nt);
    unsigned char *base = nullptr;
    int num_sms = 0;
    int rc = scratch_for_current_device(&base, &num_sms);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;

    Cohort c;
    c.G = G; c.Nt = Nt; c.Nn = Nn;
    c.Wt = (Nt + 63) / 64; c.Wn = (Nn + 63) / 64;
    c.WTp = (c.Wt + 1) & ~1;
    if (c.WTp < 2) c.WTp = 2;
    c.WNp = (c.Wn + 1) & ~1;
    if (c.WNp < 2) c.WNp = 2;
    c.GW = (((G + 63) / 64) + 1) & ~1;
    if (c.GW < 2) c.GW = 2;
    u64 *T = (u64 *)(base + kOffT), *N = (u64 *)(base + kOffN);
    u64 *TO = (u64 *)(base + kOffTO), *NO = (u64 *)(base + kOffNO);
    u64 *CT = (u64 *)(base + kOffCT), *CN = (u64 *)(base + kOffCN);
    u16 *CC = (u16 *)(base + kOffCC), *SL = (u16 *)(base + kOffSL), *SLo = (u16 *)(base + kOffSLo);
    u32 *SO = (u32 *)(base + kOffSO);
    u16 *orig = (u16 *)(base + kOffOrig);
    u32 *inv = (u32 *)(base + kOffInv);
    Rec *GR = (Rec *)(base + kOffGR);
    c.T = T; c.N = N; c.CT = CT; c.CN = CN; c.orig = orig; c.inv = inv;
    c.CC = nullptr;  // one kernel per phase: no running-count table, every subtree is searched
    c.SL = nullptr;
    c.SO = nullptr;
    c.SLo = nullptr;
    c.GR = nullptr;
    c.TO = nullptr;
    c.NO = nullptr;
    Cohort cl = c;  // by levels: the whole store
    cl.CC = Nt ? CC : nullptr;
    cl.SL = SL; cl.SO = SO; cl.SLo = SLo; cl.GR = GR; cl.TO = TO; cl.NO = NO;

    Solve s;
    s.h = h;
    s.prune = MH_PRUNE_PAPER;
    s.a_num = (u64)alpha.num;
    s.a_den = (u64)alpha.den;
    s.U = (u64 *)(base + kOffU);
    s.state = (int *)(base + kOffState);
    s.res = (int *)(base + kOffRes);
    s.cnt = (u64 *)(base + kOffCnt);
    s.slots = (Key *)(base + kOffSlots);
    s.work = (u64 *)(base + kOffWork);
    s.best_hint = s.work + kWorkCount;
    s.cand = (Key *)(base + kOffCand);
    s.champ = nullptr;  // one kernel per phase: no per-sample champions
    s.champ_ok = nullptr;
    s.ssum = nullptr;
    s.lev = nullptr;
    s.mem = nullptr;
    s.mcap = s.mlimit = 0;
    s.sel = nullptr;
    s.covsel = nullptr;
    s.cr = nullptr;
    s.cut = nullptr;
    s.shard = 0;
    s.nshards = 1;
    s.xbest = nullptr;
    const int leaf_blocks = num_sms * 4;
    s.nslots = level1_grid(c) > leaf_blocks ? level1_grid(c) : leaf_blocks;
    if (s.nslots > kNaMaxSlots) return na_fail(MH_EINVAL, "mh_solve_noalloc: %d SMs exceed the slot array", num_sms);
    u32 *counts = (u32 *)(base + kOffCounts);
    // each frontier is split into kShards equal regions (the region is the cap)
    Frontiers fr;
    for (int l = 0; l < kMaxH; ++l) {
        fr.F[l] = nullptr;
        fr.cap[l] = 0;
        fr.ub[l] = nullptr;
        fr.lb[l] = nullptr;
        fr.lc[l] = nullptr;
    }
    fr.F[1] = (Rec *)(base + kOffF1);
    fr.cap[1] = kNaMaxG / kShards;
    fr.F[2] = (Rec *)(base + kOffF2);
    fr.cap[2] = kNaFrontierCap / kShards;
    fr.F[3] = (Rec *)(base + kOffF3);
    fr.cap[3] = kNaFrontierCap / kShards;
    // by levels: champions, sums, members and picks; lb, ub, lc of the leaf parents (depth h - 1)
    Solve sl = s;
    sl.champ = (Key *)(base + kOffChamp);
    sl.champ_ok = (int *)(base + kOffChampOk);
    sl.ssum = (u64 *)(base + kOffSsum);
    sl.lev = (Level *)(base + kOffLevel);
    sl.mem = (Member *)(base + kOffMem);
    sl.mcap = sl.mlimit = kNaMembers;  // a level of more is picked one by one
    sl.sel = (Key *)(base + kOffSel);
    sl.covsel = (int *)(base + kOffCovsel);
    sl.cr = (u16 *)(base + kOffCr);
    Frontiers fl = fr;
    fl.lb[h - 1] = (Key *)(base + kOffLb);
    fl.ub[h - 1] = (u64 *)(base + kOffUb);
    fl.lc[h - 1] = (u64 *)(base + kOffLc);
    GridSync *gsync = (GridSync *)(base + kOffSync);

    // the store: sort keys and tumor counts, the order, then every piece
    u32 *keys = (u32 *)(base + kOffKeys), *order = (u32 *)(base + kOffOrder), *ms = (u32 *)(base + kOffMs);
    int *prep = (int *)(base + kOffPrep);
    NA_CUDA(cudaMemsetAsync(prep, 0, sizeof(int) * kPrepWords, st));
    NA_CUDA(cudaMemsetAsync(ms, 0, sizeof(u32) * kNaMaxNt, st));
    k_na_keys<<<(G + kNaKeyThreads - 1) / kNaKeyThreads, kNaKeyThreads, 0, st>>>((const u64 *)d_bitmaps, G, Nt, Nn, keys,
                                                                                 ms, prep);
    k_na_rank<<<(G + kNaRankGenes - 1) / kNaRankGenes + 1, 1024, 0, st>>>(keys, G, order, ms, Nt, SO, prep);
    StoreBuild sb;
    sb.c = cl;
    sb.bm = (const u64 *)d_bitmaps;
    sb.order = order;
    sb.SO = SO;
    sb.T = T; sb.N = N; sb.TO = TO; sb.NO = NO; sb.CT = CT; sb.CN = CN;
    sb.CTo = (u64 *)(base + kOffCTo);
    sb.CC = CC; sb.SL = SL; sb.SLo = SLo; sb.orig = orig; sb.inv = inv;
    sb.GR = GR;
    NA_CUDA(launch_store_build(sb, st));
    // the first round's frontiers decide whether the solve fits (U only shrinks: later
    // ones are smaller)
    launch_solve_init(c, s, Nt + 2, Nt + 1, counts, 1, st);
    if (Nt && h >= 2) {
        launch_level1(c, s, fr, counts, st);
        for (int l = 2; l <= h - 1; ++l) launch_expand(c, s, l, fr, counts, leaf_blocks, st);
    }
    NA_CUDA(cudaGetLastError());
    constexpr size_t kHead = kOffCounts - kOffState + sizeof(u32) * kNaMaxH * kShards * kShardStride;
    alignas(8) unsigned char head[kHead];
    NA_CUDA(cudaMemcpyAsync(head, base + kOffState, kHead, cudaMemcpyDeviceToHost, st));
    NA_CUDA(cudaStreamSynchronize(st));
    const int *hp = (const int *)(head + (kOffPrep - kOffState));
    const u32 *hc = (const u32 *)(head + (kOffCounts - kOffState));
    if (hp[kPrepBad]) return na_fail(MH_EINVAL, "mh_solve_noalloc: padding bits past Nt or Nn are set");
    auto too_large = [] {
        return na_fail(MH_ENOMEM, "mh_solve_noalloc: a search frontier exceeds the fixed scratch (%u prefixes per depth)",
                       kNaFrontierCap);
    };
    if (Nt)
        for (int l = 1; l < h; ++l)
            for (int i = 0; i < kShards; ++i)
                if (hc[shard_slot(l, i)] > fr.cap[l]) return too_large();

    int rounds = 0;
    bool done = Nt == 0;
    int st8[kStateWords] = {};
    const int pgrid = persistent_grid(num_sms, false);
    if (!done && pgrid > 0 && pgrid <= s.nslots && (size_t)hp[kPrepMutations] <= kNaLists) {
        launch_solve_init(cl, sl, Nt + 2, Nt + 1, counts, kCountSets, st, gsync);
        const cudaError_t le = launch_solve_persistent(cl, sl, fl, gsync, counts, pgrid, false, st);
        if (le == cudaSuccess) {
            k_na_unpack<<<4, 256, 0, st>>>(s.res, s.state, h, capacity, d_genes, d_tp, d_fp, true);
            NA_CUDA(cudaGetLastError());
            NA_CUDA(cudaMemcpyAsync(st8, s.state, sizeof st8, cudaMemcpyDeviceToHost, st));
            NA_CUDA(cudaStreamSynchronize(st));
            if (injected_timeout()) return na_fail(MH_ETIMEOUT, "injected timeout (mh_set_fault)");
            if (st8[2]) return solve_error(st8[2], "mh_solve_noalloc: a grid barrier timed out");
            if (st8[1] && !st8[3]) {
                *k_out = st8[0];
                if (rounds_out) *rounds_out = st8[4];
                return MH_OK;
            }
        } else if (le == cudaErrorCooperativeLaunchTooLarge || le == cudaErrorLaunchOutOfResources ||
                   le == cudaErrorMemoryAllocation) {
            cudaGetLastError();  // no room for the grid: one kernel per phase
        } else {
            return na_fail(MH_ECUDA, "mh_solve_noalloc: the launch of the solve failed: %s", cudaGetErrorString(le));
        }
    }
    // (over: what ran so far left its state and counts)
    launch_solve_init(c, s, Nt + 2, Nt + 1, counts, 1, st);
    const int grid = leaf_blocks;
    // rounds run on the device; the host enqueues them in growing batches
    int batch = 4;
    while (!done) {
        const int n = batch < Nt + 1 - rounds ? batch : Nt + 1 - rounds;
        for (int b = 0; b < n; ++b) {
            launch_level1(c, s, fr, counts, st);
            for (int l = 2; l <= h - 1; ++l) launch_expand(c, s, l, fr, counts, grid, st);
            if (h >= 2) launch_leaf(c, s, fr, counts, grid, st);
            launch_finalize(c, s, counts, st);
        }
        NA_CUDA(cudaGetLastError());
        NA_CUDA(cudaMemcpyAsync(st8, s.state, sizeof st8, cudaMemcpyDeviceToHost, st));
        NA_CUDA(cudaStreamSynchronize(st));
        rounds = st8[4];
        if (st8[3]) return too_large();
        done = st8[1] != 0 || rounds >= Nt + 1;
        batch = batch * 2 < 64 ? batch * 2 : 64;
    }
    k_na_unpack<<<4, 256, 0, st>>>(s.res, s.state, h, capacity, d_genes, d_tp, d_fp, false);
    NA_CUDA(cudaGetLastError());
    NA_CUDA(cudaMemcpyAsync(st8, s.state, sizeof st8, cudaMemcpyDeviceToHost, st));
    NA_CUDA(cudaStreamSynchronize(st));
    *k_out = st8[0];
    if (rounds_out) *rounds_out = rounds;
    return MH_OK;
}
