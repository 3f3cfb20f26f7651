// Box-operator products on the 5th-generation tensor cores (tcgen05, TMEM
// accumulators): M2M, L2L and the check -> equivalent solves; and the pair
// lists of the tree passes (the M2L itself: m2l_f16.cu).
//
// All pairs of an item share one operator (FP64-built, FP32-stored).  A CTA
// owns one item and one part of the operator: a block of its output rows
// times a block of its inner columns (two row halves up to p = 6; 4 x 2
// parts at p = 8, 4 x 4 at p = 10), so that the part fits in shared memory:
//   * the operator part, split into TF32 hi + lo parts and pre-swizzled in
//     global memory (128B swizzle, K-major), is copied into shared memory
//     once with cp.async.bulk and stays resident;
//   * 128-pair row tiles stream through: the producer threads gather the
//     source rows (the part's columns), split them into TF32 hi + lo and
//     write them swizzled into a ring of A stages;
//   * one thread issues tcgen05.mma kind::tf32 (M = 128 pairs, N = the
//     part's rows, K = 8 per instruction), three products per k-step
//     (hi*hi + hi*lo + lo*hi: FP32-level accuracy), accumulating in TMEM;
//   * the epilogue reads the accumulator with tcgen05.ld and adds each row
//     into the target row with red.global.add.v4.f32 (targets of one item
//     are distinct; items and inner parts overlap, hence the reduction).
// TF32 and not scaled halves: the factors of the check -> equivalent solves
// span 14 decades, more than a common scale per row can hold.
// Every wait is bounded (~1 s); on a timeout the kernel records an error
// code, drains its own MMAs, frees TMEM and returns.
#include "fmm.cuh"
#include "tc_ptx.cuh"
#include <cub/cub.cuh>
#include <algorithm>
#include <atomic>
#include <cstdio>

namespace pbfmm {

void radix_sort_pairs(const unsigned* keys_in, const int* vals_in, unsigned* keys_out, int* vals_out, long long n,
                      int bits, cudaStream_t st);

constexpr int kTcRows = 128;           // pairs per row tile (MMA M)
constexpr int kM2LSegBoxes = 8192;     // target boxes of one segment of the M2L pair list
constexpr int kTcItemPairs = 2048;     // pairs per self-test item
constexpr int kTcSmallItemPairs = 512; // M2M / L2L / check->equivalent items: few pairs per operator, many CTAs

// Operator split per padded size: NS parts of the output rows (MMA N =
// npad / NS) times KS parts of the inner dimension (npad / KS columns,
// whole 32-column blocks), so that one part (TF32 hi + lo) stays resident
// in shared memory beside a ring of STAGES A stages.  Each CTA owns one
// part; the KS parts of a row add into the target with the reduction.
template <int NPAD> struct TcCfg { static constexpr int NS = 2, KS = 1, STAGES = 3; };
template <> struct TcCfg<320> { static constexpr int NS = 4, KS = 2, STAGES = 3; };   // p = 8
template <> struct TcCfg<512> { static constexpr int NS = 4, KS = 4, STAGES = 2; };   // p = 10
static bool tc_split(int npad, int& ns, int& ks) {
    switch (npad) {
        case 32: case 64: case 128: case 160: ns = 2; ks = 1; return true;
        case 320: ns = TcCfg<320>::NS; ks = TcCfg<320>::KS; return true;
        case 512: ns = TcCfg<512>::NS; ks = TcCfg<512>::KS; return true;
        default: return false;
    }
}

// TF32 part of x, rounded to nearest (ties away from zero); x - hi is exact in FP32
__device__ __forceinline__ float tf32_hi(float x) {
    return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
}

// ---------------------------------------------------------------------------
// operator packing: [matrix][part = ns * KS + ks][hi|lo][kb][nh rows][32]
// swizzled (nh = npad / NS output rows, KB = npad / KS / 32 blocks of 32
// inner columns); the part a CTA owns is one contiguous block
// ---------------------------------------------------------------------------
__global__ void k_pack_box_ops(int npad, int NS, int KS, long long nmat, const float* __restrict__ m2l,
                              float* __restrict__ out) {
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long m2 = (long long)npad * npad;
    if (idx >= nmat * m2) return;
    long long mat = idx / m2;
    int n = (int)((idx % m2) / npad), k = (int)(idx % npad);
    const int nh = npad / NS, kc = npad / KS, kb_n = kc / 32;
    int ns = n / nh, nr = n % nh, ks = k / kc, kk = k % kc, kb = kk / 32, kq = kk % 32;
    float x = m2l[idx];
    float hi = tf32_hi(x), lo = x - hi;
    const long long part_bytes = 2LL * kb_n * nh * 128;
    char* base = (char*)out + (mat * NS * KS + ns * KS + ks) * part_bytes;
    uint32_t off = (uint32_t)kb * nh * 128 + sw128_off(nr, kq);
    *(float*)(base + off) = hi;
    *(float*)(base + (long long)kb_n * nh * 128 + off) = lo;
}

static void pack_tc(int npad, long long nmat, const float* src, DBuf<float>& dst, cudaStream_t st) {
    int ns = 0, ks = 0;
    if (!tc_split(npad, ns, ks)) throw Error(PB_EINVAL, "no tensor-core split for this operator size");
    const long long m2 = (long long)npad * npad;
    dst.alloc(nmat * m2 * 2, st);
    k_pack_box_ops<<<div_up(nmat * m2, 256), 256, 0, st>>>(npad, ns, ks, nmat, src, dst.p);
    PB_CHECK_LAUNCH();
}

void pack_box_ops_tc(Operators& O, cudaStream_t st) {
    int ns = 0, ks = 0;
    if (!tc_split(O.npad, ns, ks)) { O.have_tc = false; return; }
    if (O.m2m.p) pack_tc(O.npad, (long long)O.nlev * 8, O.m2m.p, O.m2m_tc, st);
    if (O.l2l.p) pack_tc(O.npad, (long long)O.nlev * 8, O.l2l.p, O.l2l_tc, st);
    if (O.uc2ue_w1.p) {
        pack_tc(O.npad, O.nlev, O.uc2ue_w1.p, O.uc2ue_w1_tc, st);
        pack_tc(O.npad, O.nlev, O.uc2ue_w2.p, O.uc2ue_w2_tc, st);
        pack_tc(O.npad, O.nlev, O.dc2de_w1.p, O.dc2de_w1_tc, st);
        pack_tc(O.npad, O.nlev, O.dc2de_w2.p, O.dc2de_w2_tc, st);
    }
    O.have_tc = true;
}

// ---------------------------------------------------------------------------
// V-list pairs grouped by (level, offset)
// ---------------------------------------------------------------------------
__global__ void k_pairs_emit(int nbox, const int* V, const int* V_n, const int* V_off, const int4* anchor,
                             int* key, int* tgt, int* src, int* idx) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nbox) return;
    int4 ab = anchor[b];
    for (int i = 0; i < V_n[b]; ++i) {
        int s = V[(long long)b * kVCap + i];
        int4 as = anchor[s];
        const int ox = as.x - ab.x, oy = as.y - ab.y, oz = as.z - ab.z;
        const int slot = abs(ox) * 16 + abs(oy) * 4 + abs(oz);
        const int sign = (ox < 0 ? 4 : 0) | (oy < 0 ? 2 : 0) | (oz < 0 ? 1 : 0);
        int e = V_off[b] + i;
        key[e] = (((b / kM2LSegBoxes) * 64 + slot) * 32 + ab.w) * 8 + sign;   // segment, |offset|, level (< 22), signs
        tgt[e] = b;
        src[e] = s;
        idx[e] = e;
    }
}

// first pair and key of every run of equal keys
__global__ void k_pair_runs(int n, const int* key, int cap, int2* runs, int* count) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || (i > 0 && key[i] == key[i - 1])) return;
    const int k = atomicAdd(count, 1);
    if (k < cap) runs[k] = make_int2(i, key[i]);
}

__global__ void k_pairs_gather(int n, const int* idx, const int* key, const int* t, const int* s, int* tgt, int* src,
                               int* srcx) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int k = idx[i], sb = s[k];
    tgt[i] = t[k];
    src[i] = sb;
    srcx[i] = sb | (key[i] & 7) << 28;
}

void build_m2l_pairs(fmm_tree* T) {
    cudaStream_t st = T->ctx->stream;
    const int nb = T->nbox;
    const long long np = T->n_v;
    auto& P = T->m2l_pairs;
    P.npairs = np;
    P.nitems32 = P.ntile_even = P.ntile_odd = P.nseg = 0;
    if (np == 0) return;
    PB_REQUIRE(nb < (1 << 28), PB_EINVAL, "octree has too many boxes for the interaction pair lists");
    DBuf<int> voff, key, tgt, src, idx, key_s, idx_s;
    voff.alloc(nb + 1, st);
    {
        size_t tmp = 0;
        cub::DeviceScan::ExclusiveSum(nullptr, tmp, T->V_n.p, voff.p, nb, st);
        DBuf<char> t;
        t.alloc(std::max<size_t>(tmp, 1), st);
        cub::DeviceScan::ExclusiveSum(t.p, tmp, T->V_n.p, voff.p, nb, st);
    }
    key.alloc(np, st); tgt.alloc(np, st); src.alloc(np, st);
    idx.alloc(np, st); key_s.alloc(np, st); idx_s.alloc(np, st);
    k_pairs_emit<<<div_up(nb, 128), 128, 0, st>>>(nb, T->V.p, T->V_n.p, voff.p, T->anchor.p, key.p, tgt.p, src.p,
                                                  idx.p);
    PB_CHECK_LAUNCH();
    // stable: each group keeps the box order
    int bits = 14;
    while ((nb - 1) / kM2LSegBoxes >> (bits - 14)) ++bits;
    radix_sort_pairs((const unsigned*)key.p, idx.p, (unsigned*)key_s.p, idx_s.p, np, bits, st);
    P.tgt.alloc(np, st);
    P.src.alloc(np, st);
    P.srcx.alloc(np, st);
    k_pairs_gather<<<div_up(np, 256), 256, 0, st>>>((int)np, idx_s.p, key_s.p, tgt.p, src.p, P.tgt.p, P.src.p,
                                                     P.srcx.p);
    PB_CHECK_LAUNCH();
    // the runs of equal keys: (first pair, key), in any order, then sorted
    DBuf<int2> druns;
    DBuf<int> dn;
    int cap = 8192, nrun = 0;
    std::vector<int2> runs;
    for (;;) {
        druns.alloc(cap, st);
        dn.alloc(1, st);
        dn.zero(st);
        k_pair_runs<<<div_up(np, 256), 256, 0, st>>>((int)np, key_s.p, cap, druns.p, dn.p);
        PB_CHECK_LAUNCH();
        runs.resize(cap);
        PB_CUDA(cudaMemcpyAsync(&nrun, dn.p, sizeof(int), cudaMemcpyDeviceToHost, st));
        PB_CUDA(cudaMemcpyAsync(runs.data(), druns.p, cap * sizeof(int2), cudaMemcpyDeviceToHost, st));
        PB_CUDA(cudaStreamSynchronize(st));
        if (nrun <= cap) break;
        cap = nrun;
    }
    runs.resize(nrun);
    std::sort(runs.begin(), runs.end(), [](const int2& x, const int2& y) { return x.x < y.x; });
    runs.push_back(make_int2((int)np, -1));
    std::vector<int4> even, odd, items32;
    std::vector<int> seg_even, seg_odd;
    auto cut = [](std::vector<int4>& v, long long a, long long b, int step, int z) {
        for (; a < b; a += step) v.push_back(make_int4((int)a, (int)std::min<long long>(step, b - a), z, 0));
    };
    for (int i = 0; i < nrun;) {
        // one (segment, |offset|, level): the runs of its signs, then the whole group
        const int k = runs[i].y;
        if (i == 0 || k >> 14 != runs[i - 1].y >> 14) {
            seg_even.push_back((int)even.size());
            seg_odd.push_back((int)odd.size());
        }
        int j = i;
        for (; j < nrun && runs[j].y >> 3 == k >> 3; ++j) {
            const int kj = runs[j].y, slot = (kj >> 8) & 63, lev = (kj >> 3) & 31, sg = kj & 7;
            const int o[3] = {slot >> 4, (slot >> 2) & 3, slot & 3};
            const int off = ((sg & 4 ? -o[0] : o[0]) + 3) * 49 + ((sg & 2 ? -o[1] : o[1]) + 3) * 7 +
                            ((sg & 1 ? -o[2] : o[2]) + 3);
            cut(odd, runs[j].x, runs[j + 1].x, 128, off * 32 + lev);
            cut(items32, runs[j].x, runs[j + 1].x, 32, lev * kNumOffsets + off);
        }
        cut(even, runs[i].x, runs[j].x, 128, (k >> 3) & 2047);
        i = j;
    }
    P.nseg = (int)seg_even.size();
    seg_even.push_back((int)even.size());
    seg_odd.push_back((int)odd.size());
    P.seg_even.alloc(seg_even.size(), st);
    P.seg_odd.alloc(seg_odd.size(), st);
    PB_CUDA(cudaMemcpyAsync(P.seg_even.p, seg_even.data(), seg_even.size() * sizeof(int), cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaMemcpyAsync(P.seg_odd.p, seg_odd.data(), seg_odd.size() * sizeof(int), cudaMemcpyHostToDevice, st));
    auto up = [&](const std::vector<int4>& v, DBuf<int4>& d, int& n) {
        n = (int)v.size();
        d.alloc(v.size(), st);
        PB_CUDA(cudaMemcpyAsync(d.p, v.data(), v.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
    };
    up(even, P.tiles_even, P.ntile_even);
    up(odd, P.tiles_odd, P.ntile_odd);
    up(items32, P.items32, P.nitems32);
    PB_CUDA(cudaStreamSynchronize(st));
}

// Items of the check -> equivalent solves on the tensor cores: the boxes of
// each level (one row each) in chunks of at most kTcSmallItemPairs.
static void level_items(const std::vector<int>& lvl_off, int nlev, DBuf<int4>& items, int& n, cudaStream_t st) {
    std::vector<int4> h;
    for (int l = 0; l < nlev; ++l)
        for (int a = lvl_off[l]; a < lvl_off[l + 1]; a += kTcSmallItemPairs)
            h.push_back(make_int4(a, std::min(kTcSmallItemPairs, lvl_off[l + 1] - a), l, 0));
    n = (int)h.size();
    if (h.empty()) return;
    items.alloc(h.size(), st);
    PB_CUDA(cudaMemcpyAsync(items.p, h.data(), h.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaStreamSynchronize(st));
}

void build_c2e_items(fmm_tree* T) {
    cudaStream_t st = T->ctx->stream;
    if ((int)T->sleaf_lvl_off.size() == T->nlev + 1)
        level_items(T->sleaf_lvl_off, T->nlev, T->c2e_items_up, T->n_c2e_up, st);
    if ((int)T->xbox_lvl_off.size() == T->nlev + 1)
        level_items(T->xbox_lvl_off, T->nlev, T->c2e_items_dn, T->n_c2e_dn, st);
}

// Parent-child pairs for M2M / L2L on the tensor cores: children of level
// >= 3 grouped by (level, octant), ascending box order inside a group.
void build_pc_pairs(fmm_tree* T) {
    cudaStream_t st = T->ctx->stream;
    auto& P = T->pc_pairs;
    const int nb = T->nbox;
    std::vector<int> par(nb);
    std::vector<int4> anc(nb);
    PB_CUDA(cudaMemcpyAsync(par.data(), T->parent.p, nb * sizeof(int), cudaMemcpyDeviceToHost, st));
    PB_CUDA(cudaMemcpyAsync(anc.data(), T->anchor.p, nb * sizeof(int4), cudaMemcpyDeviceToHost, st));
    PB_CUDA(cudaStreamSynchronize(st));
    std::vector<std::vector<int>> bucket((size_t)T->nlev * 8);
    for (int c = 0; c < nb; ++c) {
        if (anc[c].w < 3) continue;
        int oct = ((anc[c].x & 1) << 2) | ((anc[c].y & 1) << 1) | (anc[c].z & 1);
        bucket[(size_t)anc[c].w * 8 + oct].push_back(c);
    }
    std::vector<int> hp, hc;
    std::vector<int4> items;
    P.level_item_off.assign(T->nlev + 1, 0);
    for (int l = 0; l < T->nlev; ++l) {
        P.level_item_off[l] = (int)items.size();
        for (int o = 0; o < 8; ++o) {
            auto& v = bucket[(size_t)l * 8 + o];
            for (size_t a = 0; a < v.size(); a += kTcSmallItemPairs) {
                int cnt = (int)std::min<size_t>(kTcSmallItemPairs, v.size() - a);
                items.push_back(make_int4((int)hc.size(), cnt, l * 8 + o, 0));
                for (int k = 0; k < cnt; ++k) { hc.push_back(v[a + k]); hp.push_back(par[v[a + k]]); }
            }
        }
    }
    P.level_item_off[T->nlev] = (int)items.size();
    P.nitems = (int)items.size();
    if (items.empty()) return;
    P.parent.alloc(hp.size(), st);
    P.child.alloc(hc.size(), st);
    P.items.alloc(items.size(), st);
    PB_CUDA(cudaMemcpyAsync(P.parent.p, hp.data(), hp.size() * sizeof(int), cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaMemcpyAsync(P.child.p, hc.data(), hc.size() * sizeof(int), cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaMemcpyAsync(P.items.p, items.data(), items.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaStreamSynchronize(st));
}

// ---------------------------------------------------------------------------
// the kernel: warp-specialised pipeline
//   warps 0-7   producers: two threads per pair row gather the source box's
//               Qu row, split it into TF32 hi + lo and write it swizzled
//               into a ring of A stages (one K block each);
//   warps 8-11  epilogue: one TMEM lane quarter each; read the finished
//               accumulator and add every row into its target's Qd row;
//   warp 12     one thread issues the MMAs and the commits.
// Two TMEM accumulators alternate between tiles, so the epilogue of a tile
// overlaps the MMAs of the next and the gathers of the one after.
// ---------------------------------------------------------------------------
constexpr int kTcProdWarps = 8;
constexpr int kTcEpiWarps = 4;
constexpr int kTcThreads = 32 * (kTcProdWarps + kTcEpiWarps + 1);

constexpr int kTcEpiLd = 16;                    // accumulator columns per epilogue TMEM load
constexpr int kTcEpiStride = 20;                // padded row of the epilogue transpose buffer (floats)

template <int STAGES>
struct TcSmem {
    // per epilogue warp: 32 rows x kTcEpiLd columns, transposed through shared
    // memory so that each reduction instruction covers 8 rows x 64 B
    alignas(16) float epi[kTcEpiWarps][32][kTcEpiStride];
    uint64_t barB, full[STAGES], empty[STAGES], accf[2], acce[2];
    uint32_t tmem_slot;
    int failed;
};

// bounded wait that gives up as soon as another role of the CTA has failed;
// a timeout marks the CTA failed
__device__ __forceinline__ bool mbar_wait_cta(uint64_t* bar, uint32_t parity, volatile int* failed,
                                              long long limit) {
    long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (*failed) return false;
        if (clock64() - t0 > limit) {
            *failed = 1;
            return false;
        }
    }
    return true;
}

// Operator set and box vectors of one launch; blockIdx.z selects the set, so
// one launch serves the Laplace and the Yukawa half of the paired apply
// (their pair lists and operator indices coincide).
struct TcSets {
    const float* ops[2];
    const float* X[2];
    float* Y[2];
    long long wait_limit;    // cycles a role waits on a barrier before giving up (set at launch)
    int store;               // 1: every target row has one product and one inner part: store, do not add
    int sub, chunk;          // an item's pairs are cut into `sub` pieces of `chunk` pairs, one CTA (and part) each (0: by the launch)
};

template <int NPAD>
__global__ void __launch_bounds__(kTcThreads, 1) k_box_ops_tc(const int4* __restrict__ items, const int* __restrict__ ptgt,
                                                          const int* __restrict__ psrc, const TcSets sets,
                                                          int* __restrict__ err) {
    // Generic tensor-core box-operator product: for every pair p of the
    // item, Y[tgt[p]] += Op(item) X[src[p]] (Op resident for the CTA).
    // Used for M2M / L2L (operator per child level and octant) and for the factored
    // check -> equivalent solves (operator per level).
    const float* __restrict__ ops = sets.ops[blockIdx.z];
    const float* __restrict__ Qu = sets.X[blockIdx.z];
    float* __restrict__ Qd = sets.Y[blockIdx.z];
    const long long wl = sets.wait_limit;
    constexpr int NS = TcCfg<NPAD>::NS, KS = TcCfg<NPAD>::KS, kTcStages = TcCfg<NPAD>::STAGES;
    constexpr int NH = NPAD / NS;                    // output rows of this CTA (MMA N)
    constexpr int KC = NPAD / KS;                    // inner columns of this CTA
    constexpr int KB = KC / 32;                      // K blocks of 32 tf32 (128 B)
    static_assert(NH % 16 == 0 && NH <= 256 && KC % 32 == 0, "tensor-core split");
    constexpr uint32_t B_SPLIT = KB * NH * 128;      // bytes of one of hi / lo
    constexpr uint32_t A_SPLIT = kTcRows * 128;      // 16 KB
    constexpr uint32_t ACOLS = NH <= 32 ? 32 : (NH <= 64 ? 64 : (NH <= 128 ? 128 : 256));   // one accumulator
    constexpr uint32_t TCOLS = 2 * ACOLS;
    constexpr uint32_t IDESC = idesc_tf32(NH);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* sB = smem;                               // [hi|lo][KB][NH][128]
    uint8_t* sA = smem + 2 * B_SPLIT;                 // [stage][hi|lo][128][128]
    TcSmem<kTcStages>* S = (TcSmem<kTcStages>*)(sA + kTcStages * 2 * A_SPLIT);
    volatile int* failed = &S->failed;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int4 it = items[blockIdx.x / sets.sub];
    const int skip = (blockIdx.x % sets.sub) * sets.chunk;
    it.x += skip;
    it.y = min(it.y - skip, sets.chunk);
    if (it.y <= 0) return;
    const int part = blockIdx.y;                     // operator part: rows half, inner columns kpart
    const int half = part / KS, kpart = part % KS;
    const int first = it.x, npairs = it.y;
    const int opi = it.z;
    const int ntile = (npairs + kTcRows - 1) / kTcRows;

    if (tid == 0) {
        mbar_init(&S->barB, 1);
        for (int q = 0; q < kTcStages; ++q) {
            mbar_init(&S->full[q], kTcProdWarps * 32);
            mbar_init(&S->empty[q], 1);
        }
        for (int q = 0; q < 2; ++q) {
            mbar_init(&S->accf[q], 1);
            mbar_init(&S->acce[q], kTcEpiWarps * 32);
        }
        S->failed = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(&S->tmem_slot, TCOLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = S->tmem_slot;

    // resident operator part: hi and lo, one bulk copy each
    if (tid == 0) {
        const uint8_t* gB = (const uint8_t*)ops + ((long long)opi * (NS * KS) + part) * (2LL * B_SPLIT);
        mbar_arrive_expect_tx(&S->barB, 2 * B_SPLIT);
        bulk_g2s(sB, gB, B_SPLIT, &S->barB);
        bulk_g2s(sB + B_SPLIT, gB + B_SPLIT, B_SPLIT, &S->barB);
    }

    if (warp < kTcProdWarps) {
        // ---- producers: lane l8 = lane % 8 carries 16 B of a 128-B K-block row;
        // a warp instruction covers 4 whole rows (coalesced). Thread rows:
        // i * 32 + warp * 4 + lane / 8, i = 0..3.
        const int l8 = lane & 7, rbase = warp * 4 + (lane >> 3);
        auto src_of = [&](int tile, int i) -> int {
            const int r = tile * kTcRows + i * 32 + rbase;
            return (tile < ntile && r < npairs) ? psrc[first + r] : -1;
        };
        // Register rotation: once K block kb of a tile is in its stage, the
        // same registers load block kb of the next tile, so each gather has a
        // whole tile of MMA time to arrive.
        float4 v[KB][4];
        int sn[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int s0 = src_of(0, i);
            const float4* q4 = s0 >= 0 ? (const float4*)(Qu + (size_t)s0 * NPAD + kpart * KC) : nullptr;
#pragma unroll
            for (int kb = 0; kb < KB; ++kb) v[kb][i] = q4 ? q4[kb * 8 + l8] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) sn[i] = src_of(1, i);
        int g = 0;
        for (int tile = 0; tile < ntile; ++tile) {
#pragma unroll
            for (int kb = 0; kb < KB; ++kb, ++g) {
                const int s = g % kTcStages, n = g / kTcStages;
                if (n > 0 && !mbar_wait_cta(&S->empty[s], (n - 1) & 1, failed, wl)) goto prod_done;
                uint8_t* aHi = sA + (size_t)s * 2 * A_SPLIT;
                uint8_t* aLo = aHi + A_SPLIT;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 x = v[kb][i];
                    float4 h = make_float4(tf32_hi(x.x), tf32_hi(x.y), tf32_hi(x.z), tf32_hi(x.w));
                    float4 l = make_float4(x.x - h.x, x.y - h.y, x.z - h.z, x.w - h.w);
                    uint32_t off = sw128_off(i * 32 + rbase, l8 * 4);
                    *(float4*)(aHi + off) = h;
                    *(float4*)(aLo + off) = l;
                }
                fence_proxy_async();
                mbar_arrive(&S->full[s]);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4* qn = sn[i] >= 0 ? (const float4*)(Qu + (size_t)sn[i] * NPAD + kpart * KC) : nullptr;
                    v[kb][i] = qn ? qn[kb * 8 + l8] : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) sn[i] = src_of(tile + 2, i);
        }
    prod_done:
        __syncwarp();
    } else if (warp < kTcProdWarps + kTcEpiWarps) {
        // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) ... + 31
        const int q = warp & 3;
        const int erow = q * 32 + lane;
        for (int tile = 0; tile < ntile; ++tile) {
            const int a = tile & 1, u = tile >> 1;
            const int r = tile * kTcRows + erow;
            const int t = r < npairs ? ptgt[first + r] : -1;
            bool ok = mbar_wait_cta(&S->accf[a], u & 1, failed, wl);
            if (!__all_sync(0xffffffffu, ok)) break;
            tc_fence_after();
            float (*buf)[kTcEpiStride] = S->epi[q];
#pragma unroll 1
            for (int c0 = 0; c0 < NH; c0 += kTcEpiLd) {
                float v[kTcEpiLd];
                tmem_ld16(taddr + ((uint32_t)(q * 32) << 16) + a * ACOLS + c0, v);
#pragma unroll
                for (int c = 0; c < kTcEpiLd; c += 4)
                    *(float4*)&buf[lane][c] = make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]);
                __syncwarp();
                // lane: row j * 8 + lane / 4 of the warp's 32, columns 4 (lane % 4) .. + 3
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int rr = j * 8 + (lane >> 2), cc = (lane & 3) * 4;
                    const float4 x = *(const float4*)&buf[rr][cc];
                    const int tr = __shfl_sync(0xffffffffu, t, rr);
                    float* y = Qd + (size_t)tr * NPAD + half * NH + c0 + cc;
                    if (tr < 0) continue;
                    if (KS == 1 && sets.store) *(float4*)y = x;
                    else red_add_v4(y, x.x, x.y, x.z, x.w);
                }
                __syncwarp();
            }
            tc_fence_before();
            mbar_arrive(&S->acce[a]);
        }
        __syncwarp();
    } else {
        // ---- MMA issuer
        if (lane == 0) {
            uint64_t* last = nullptr;      // barrier of the last commit, and its phase parity
            uint32_t last_par = 0;
            int g = 0;
            bool ok = mbar_wait_cta(&S->barB, 0, failed, wl);
            for (int tile = 0; ok && tile < ntile; ++tile) {
                const int a = tile & 1, u = tile >> 1;
                if (u > 0 && !(ok = mbar_wait_cta(&S->acce[a], (u - 1) & 1, failed, wl))) break;
                const uint32_t dacc = taddr + a * ACOLS;
                for (int kb = 0; kb < KB; ++kb, ++g) {
                    const int s = g % kTcStages, n = g / kTcStages;
                    if (!(ok = mbar_wait_cta(&S->full[s], n & 1, failed, wl))) break;
                    tc_fence_after();
                    const uint32_t aH = smem_u32(sA + (size_t)s * 2 * A_SPLIT), aL = aH + A_SPLIT;
                    const uint32_t bH = smem_u32(sB) + kb * NH * 128, bL = bH + B_SPLIT;
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) {
                        const uint32_t acc0 = (kb > 0 || ks > 0) ? 1u : 0u;
                        mma_tf32(dacc, sw128_desc(aH + ks * 32), sw128_desc(bH + ks * 32), IDESC, acc0);
                        mma_tf32(dacc, sw128_desc(aH + ks * 32), sw128_desc(bL + ks * 32), IDESC, 1u);
                        mma_tf32(dacc, sw128_desc(aL + ks * 32), sw128_desc(bH + ks * 32), IDESC, 1u);
                    }
                    mma_commit(&S->empty[s]);
                    last = &S->empty[s];
                    last_par = n & 1;
                }
                if (!ok) break;
                mma_commit(&S->accf[a]);
                last = &S->accf[a];
                last_par = u & 1;
            }
            // every MMA issued here has completed before TMEM is freed and the
            // CTA's shared memory given up, whichever role gave up waiting: an
            // epilogue that timed out leaves the last ones in flight
            if (last) mbar_wait(last, last_par);
        }
        __syncwarp();
    }

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0 && S->failed) {
        atomicExch(err, 1);
        mbar_wait(&S->barB, 0);         // the operator copy has landed before shared memory is released
    }
    if (warp == 0) tmem_dealloc(taddr, TCOLS);
}

template <int NPAD>
static constexpr size_t tc_smem_bytes() {
    using C = TcCfg<NPAD>;
    return 1024 + 2 * (size_t)(NPAD / C::KS / 32) * (NPAD / C::NS) * 128 + C::STAGES * 2 * (size_t)kTcRows * 128 +
           sizeof(TcSmem<C::STAGES>);
}
static_assert(tc_smem_bytes<160>() <= 232448 && tc_smem_bytes<320>() <= 232448 && tc_smem_bytes<512>() <= 232448,
              "shared memory per CTA");
// opt in to the large shared-memory carve-out once per process, kernel and
// device (not a stream operation, so it stays out of captured graphs)
template <typename F>
static void smem_optin(F* kernel, size_t bytes, bool* done) {
    int dev = 0;
    PB_CUDA(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64 && !done[dev]) {
        PB_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
        done[dev] = true;
    }
}

static int tc_sm_count() {
    static std::atomic<int> n{0};
    if (n.load() == 0) {
        int dev = 0, v = 0;
        PB_CUDA(cudaGetDevice(&dev));
        PB_CUDA(cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev));
        n.store(v);
    }
    return n.load();
}

template <int NPAD>
static void launch_tc_items(const int4* items, int nitems, const int* tgt, const int* src, const TcSets& sets,
                            int nsets, int* err, cudaStream_t st) {
    if (nitems <= 0) return;
    TcSets s2 = sets;
    s2.wait_limit = g_wait_limit.load();
    if (s2.sub == 0) {
        // pieces of an item: whole (512 pairs, four row tiles, 17 to 21 us, mostly
        // latency), or down to one row tile (9 us) where SMs would else have no CTA
        int sub = 1;
        while (sub < kTcSmallItemPairs / kTcRows &&
               (long long)nitems * sub * TcCfg<NPAD>::NS * TcCfg<NPAD>::KS * nsets < tc_sm_count())
            sub *= 2;
        s2.sub = sub;
        s2.chunk = kTcSmallItemPairs / sub;
    }
    dim3 grid(nitems * s2.sub, TcCfg<NPAD>::NS * TcCfg<NPAD>::KS, nsets);
    static bool done[64] = {false};
    const size_t sm = tc_smem_bytes<NPAD>();
    smem_optin(k_box_ops_tc<NPAD>, sm, done);
    k_box_ops_tc<NPAD><<<grid, kTcThreads, sm, st>>>(items, tgt, src, s2, err);
    PB_CHECK_LAUNCH();
}

static bool tc_dispatch(int npad, const int4* items, int nitems, const int* tgt, const int* src, const TcSets& sets,
                        int nsets, int* err, cudaStream_t st) {
    switch (npad) {
        case 32: launch_tc_items<32>(items, nitems, tgt, src, sets, nsets, err, st); return true;
        case 64: launch_tc_items<64>(items, nitems, tgt, src, sets, nsets, err, st); return true;
        case 128: launch_tc_items<128>(items, nitems, tgt, src, sets, nsets, err, st); return true;
        case 160: launch_tc_items<160>(items, nitems, tgt, src, sets, nsets, err, st); return true;
        case 320: launch_tc_items<320>(items, nitems, tgt, src, sets, nsets, err, st); return true;
        case 512: launch_tc_items<512>(items, nitems, tgt, src, sets, nsets, err, st); return true;
        default: return false;
    }
}

static bool tc_ok(const Operators& O) {
    int ns, ks;
    return O.have_tc && tc_split(O.npad, ns, ks);
}

// M2M (up = true: parents at level l - 1 += M2M children at level l) or L2L
// (children at level l += L2L parents at level l - 1) on the tensor cores,
// for one operator set (O2 == nullptr) or for two in one launch; false when
// the tensor-core path does not apply
bool pc_tc_launch2(const fmm_tree* T, const Operators& O, const Operators* O2, int child_level, bool up, float* Q,
                   float* Q2, int* err, cudaStream_t st) {
    if (!tc_ok(O) || !O.m2m_tc.p || !O.l2l_tc.p) return false;
    if (O2 && (!tc_ok(*O2) || !O2->m2m_tc.p || !O2->l2l_tc.p || O2->npad != O.npad)) return false;
    const auto& P = T->pc_pairs;
    if (child_level < 3 || child_level >= T->nlev || (int)P.level_item_off.size() != T->nlev + 1) return false;
    const int i0 = P.level_item_off[child_level], i1 = P.level_item_off[child_level + 1];
    if (i1 <= i0) return true;
    const int* tgt = up ? P.parent.p : P.child.p;
    const int* src = up ? P.child.p : P.parent.p;
    TcSets sets{{up ? O.m2m_tc.p : O.l2l_tc.p, O2 ? (up ? O2->m2m_tc.p : O2->l2l_tc.p) : nullptr},
                {Q, Q2}, {Q, Q2}};
    return tc_dispatch(O.npad, P.items.p + i0, i1 - i0, tgt, src, sets, O2 ? 2 : 1, err, st);
}

bool pc_tc_launch(const fmm_tree* T, const Operators& O, int child_level, bool up, float* Q, int* err,
                  cudaStream_t st) {
    return pc_tc_launch2(T, O, nullptr, child_level, up, Q, nullptr, err, st);
}

// Check -> equivalent solve Y = W2 (W1 X) at the upward (sleaf) or downward
// (X-list) boxes on the tensor cores: two passes through `tmp`.  Every row of
// a pass receives exactly one product; up to p = 6 it is stored, at p = 8 and
// 10 the operator's inner parts add into tmp (zeroed first) and into Y, whose
// rows of those boxes must be zero on entry. One operator set, or two (O2, X2, Y2, tmp2)
// in the same launches. False when the tensor-core path does not apply.
// In the fixed-order mode not with more than two inner parts (p = 10): two
// added to zero give the same bits in either order, four do not.
bool c2e_tc_ok(const fmm_tree* T, const Operators& O) {
    int parts = 0, ks = 0;
    return tc_ok(O) && O.uc2ue_w1_tc.p && tc_split(O.npad, parts, ks) && !(T->ctx->deterministic && ks > 2);
}

// The X-list boxes that keep P2L at a direct-list threshold (see the
// field comment in fmm_tree), with their check -> equivalent items; once per
// tree and threshold, on the host (the first apply runs uncaptured).
const XFar* build_xbox_far(fmm_tree* T, int thrX) {
    auto& slot = T->xfar[thrX];
    if (slot) return slot.get();
    auto X = std::make_unique<XFar>();
    cudaStream_t st = T->ctx->stream;
    const int nb = T->nbox, nx = T->n_xbox;
    std::vector<int> ids(std::max(nx, 1)), nch(nb), b0(nb), b1(nb);
    if (nx) PB_CUDA(cudaMemcpyAsync(ids.data(), T->xbox_ids.p, nx * sizeof(int), cudaMemcpyDeviceToHost, st));
    PB_CUDA(cudaMemcpyAsync(nch.data(), T->nchild.p, nb * sizeof(int), cudaMemcpyDeviceToHost, st));
    PB_CUDA(cudaMemcpyAsync(b0.data(), T->same ? T->sb.p : T->tb.p, nb * sizeof(int), cudaMemcpyDeviceToHost, st));
    PB_CUDA(cudaMemcpyAsync(b1.data(), T->same ? T->se.p : T->te.p, nb * sizeof(int), cudaMemcpyDeviceToHost, st));
    PB_CUDA(cudaStreamSynchronize(st));
    std::vector<int> far;
    far.reserve(nx);
    for (int i = 0; i < nx; ++i) {
        const int b = ids[i];
        if (!(nch[b] == 0 && b1[b] - b0[b] <= thrX)) far.push_back(b);
    }
    std::vector<int> lvl(T->nlev + 1, 0);
    for (int l = 0; l <= T->nlev; ++l)
        lvl[l] = (int)(std::lower_bound(far.begin(), far.end(), T->lvl_off[l]) - far.begin());
    X->ids.alloc(std::max<size_t>(far.size(), 1), st);
    if (!far.empty())
        PB_CUDA(cudaMemcpyAsync(X->ids.p, far.data(), far.size() * sizeof(int), cudaMemcpyHostToDevice, st));
    X->n = (int)far.size();
    level_items(lvl, T->nlev, X->items, X->nitems, st);
    slot = std::move(X);
    return slot.get();
}

bool c2e_tc_launch2(const fmm_tree* T, const Operators& O, const Operators* O2, bool up, const float* X, float* Y,
                    float* tmp, const float* X2, float* Y2, float* tmp2, int* err, cudaStream_t st,
                    const XFar* far) {
    if (!c2e_tc_ok(T, O)) return false;
    if (O2 && (!c2e_tc_ok(T, *O2) || O2->npad != O.npad)) return false;
    const int nitems = up ? T->n_c2e_up : (far ? far->nitems : T->n_c2e_dn);
    if (nitems == 0) return true;
    const int4* items = up ? T->c2e_items_up.p : (far ? far->items.p : T->c2e_items_dn.p);
    const int* ids = up ? T->sleaf_ids.p : (far ? far->ids.p : T->xbox_ids.p);
    auto w1 = [&](const Operators& o) { return up ? o.uc2ue_w1_tc.p : o.dc2de_w1_tc.p; };
    auto w2 = [&](const Operators& o) { return up ? o.uc2ue_w2_tc.p : o.dc2de_w2_tc.p; };
    int parts = 0, ks = 0;
    tc_split(O.npad, parts, ks);
    if (ks > 1) {                     // the inner parts add up
        const size_t bytes = (size_t)T->nbox * O.npad * sizeof(float);
        PB_CUDA(cudaMemsetAsync(tmp, 0, bytes, st));
        if (O2) PB_CUDA(cudaMemsetAsync(tmp2, 0, bytes, st));
    }
    const int ns = O2 ? 2 : 1;
    TcSets p1{{w1(O), O2 ? w1(*O2) : nullptr}, {X, X2}, {tmp, tmp2}, 0, 1};
    TcSets p2{{w2(O), O2 ? w2(*O2) : nullptr}, {tmp, tmp2}, {Y, Y2}, 0, 1};
    if (!tc_dispatch(O.npad, items, nitems, ids, ids, p1, ns, err, st)) return false;
    return tc_dispatch(O.npad, items, nitems, ids, ids, p2, ns, err, st);
}

bool c2e_tc_launch(const fmm_tree* T, const Operators& O, bool up, const float* X, float* Y, float* tmp, int* err,
                   cudaStream_t st, const XFar* far) {
    return c2e_tc_launch2(T, O, nullptr, up, X, Y, tmp, nullptr, nullptr, nullptr, err, st, far);
}

}  // namespace pbfmm

// ---------------------------------------------------------------------------
// Self-test hooks (not part of the documented ABI)
// ---------------------------------------------------------------------------
namespace pbfmm {
static std::atomic<int> g_selftest_h{1};
bool m2l_h_supported(int npad);
void m2l_h_selftest(int nrows, int npad, const float* Q, const float* Op, const int* xs, float* D, int* err,
                    cudaStream_t st);
void m2l_h_info(int* out);
}  // namespace pbfmm
using namespace pbfmm;
extern "C" int pbfmm_test_tc_pair(int mode) { return g_selftest_h.exchange(mode ? 1 : 0); }

extern "C" int pbfmm_test_tc_pair_info(int* out) {
    try {
        m2l_h_info(out);
        return PB_OK;
    } catch (const Error& e) {
        std::fprintf(stderr, "pbfmm_test_tc_pair_info: %s\n", e.what());
        return e.code;
    }
}

extern "C" int pbfmm_selftest_m2l_tc(int nrows, int npad, const float* Q, const float* Op, float* D) {
    try {
        int ns_, ks_;
        if (nrows < 1 || !tc_split(npad, ns_, ks_)) return PB_EINVAL;
        cudaStream_t st = nullptr;
        DBuf<float> op, q, d;
        DBuf<int> e;
        op.alloc((size_t)npad * npad, st);
        PB_CUDA(cudaMemcpyAsync(op.p, Op, (size_t)npad * npad * 4, cudaMemcpyHostToDevice, st));
        q.alloc((size_t)nrows * npad, st);
        d.alloc((size_t)nrows * npad, st);
        d.zero(st);
        e.alloc(1, st);
        e.zero(st);
        PB_CUDA(cudaMemcpyAsync(q.p, Q, (size_t)nrows * npad * 4, cudaMemcpyHostToDevice, st));
        if (g_selftest_h.load() && m2l_h_supported(npad)) {
            m2l_h_selftest(nrows, npad, q.p, op.p, nullptr, d.p, e.p, st);
        } else {
            DBuf<float> packed;
            DBuf<int> ids;
            DBuf<int4> ditems;
            pack_tc(npad, 1, op.p, packed, st);
            std::vector<int> id(nrows);
            for (int i = 0; i < nrows; ++i) id[i] = i;
            std::vector<int4> items;
            for (int a = 0; a < nrows; a += kTcItemPairs)
                items.push_back(make_int4(a, std::min(kTcItemPairs, nrows - a), 0, 0));
            ids.alloc(nrows, st);
            ditems.alloc(items.size(), st);
            PB_CUDA(cudaMemcpyAsync(ids.p, id.data(), nrows * 4, cudaMemcpyHostToDevice, st));
            PB_CUDA(cudaMemcpyAsync(ditems.p, items.data(), items.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
            TcSets sets{{packed.p, nullptr}, {q.p, nullptr}, {d.p, nullptr}, 0, 0, 1, kTcItemPairs};
            if (!tc_dispatch(npad, ditems.p, (int)items.size(), ids.p, ids.p, sets, 1, e.p, st)) return PB_EINVAL;
            PB_CUDA(cudaStreamSynchronize(st));
        }
        int herr = 0;
        PB_CUDA(cudaMemcpyAsync(&herr, e.p, 4, cudaMemcpyDeviceToHost, st));
        PB_CUDA(cudaMemcpyAsync(D, d.p, (size_t)nrows * npad * 4, cudaMemcpyDeviceToHost, st));
        PB_CUDA(cudaStreamSynchronize(st));
        return herr ? PB_ETIMEOUT : PB_OK;
    } catch (const Error& e) {
        return e.code;
    }
}
