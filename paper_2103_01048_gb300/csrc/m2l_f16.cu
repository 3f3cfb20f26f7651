// M2L on the 5th-generation tensor cores in split half precision.
//
// Work (Sec. "Fast multipole method": interaction list I(B)): for every
// V-list pair (target t, source s) Qd[t] += M(offset, level) Qu[s], M the
// n_e x n_e operator with the DC2DE solve folded in.  The kernels 1/r and
// e^{-kr}/r are radial and the surfaces are grids on a cube, so for even p
// (no surface point on a coordinate plane) the operators of the up to eight
// offsets (+-a, +-b, +-c) are one matrix with its rows and columns permuted:
// with the points numbered 8 * orbit + (sign bits), M(o)[i][j] =
// M(|o|)[i ^ x][j ^ x], x the sign bits of o.  64 operator slots per level
// (56 used) instead of 343 (316); the pairs of a slot are 5.6 times as many,
// so an operator stays in shared memory for many row tiles and the whole
// set stays in L2 at ordinary sizes.  Odd p: one slot per offset, x = 0.
//
// Arithmetic: FP32 operands as hi + lo in half precision, three products
// hi*hi + hi*lo + lo*hi with FP32 accumulation.  Half has TF32's 11
// significant bits at twice its rate and half its bytes; its range is no
// limit because every source row and every operator is scaled by a power of
// two to a largest entry in [2^14, 2^15) first (undone exactly in the
// epilogue).  hi + lo then hold an entry to 2^-23 relative, or 2^-39 of the
// row's largest where lo leaves the normal range (spacing 2^-24, largest
// entry at least 2^14); the TF32 split that this replaces kept 2^-21 (lo
// truncated to 11 bits) of every entry.
//
// Layout: a K block is 32 columns; its row is 128 B = [32 hi halves | 32 lo
// halves], 128B-swizzled in shared memory.
//
// Floor: the reductions into Qd, n_e * 4 B per pair at the L2's rate for them
// (measured on random rows: 5.9 TB/s for 64-byte pieces of red.v4; 16-byte
// pieces 3.3, 32-byte 4.2); at p = 8 and 10 the MMAs (three products) take as
// long.  What bounds it: the producers' gathers of source rows from L2, two K
// blocks in flight (at 1M points, p = 6, long-scoreboard stalls lead, the
// tensor pipe is active 33% of the time and the L2 is 45% busy).  Before (TF32, one operator per offset, CTA pairs)
// -> now, both kernels: p = 4, 3M points 1.35 -> 0.62 ms; p = 6, 15,000 0.18
// -> 0.03, 240,000 0.40 -> 0.14, 4M 2.74 -> 1.62; p = 8, 500,000 1.98 -> 0.85;
// p = 10, 197,000 3.19 -> 1.01.
#include "fmm.cuh"
#include "tc_ptx.cuh"
#include <cuda_fp16.h>
#include <algorithm>

namespace pbfmm {

constexpr int kHRows = 128;                     // pairs per row tile (MMA M)
constexpr int kHProdWarps = 8, kHEpiWarps = 8;
constexpr int kHRowsPerThr = kHRows / (kHProdWarps * 4);  // rows a producer thread carries a 16-byte column of
constexpr int kHThreads = 32 * (kHProdWarps + kHEpiWarps + 1);
constexpr uint32_t kHStageBytes = kHRows * 128; // one K block of a row tile, hi and lo

// Per padded size: the operator is cut into NS row parts times KS column
// parts, each N = npad / NS rows by npad / KS columns (<= 128 KB as hi + lo
// halves), one of them held by a CTA at a time; STAGES A stages in the rest of
// the 227 KB.  Row parts gather every source row again, column parts add
// every target row again, and a narrow tile leaves the tensor core idle: six
// MMAs take 72 cycles each at N = 64 or 80 (32 and 40 of work), 84 at N = 160.
// Measured, NS x KS: p = 8 with 500,000 points 4 x 1 1.066 ms, 2 x 2 0.847;
// p = 10 with 197,000 points 8 x 1 1.52 ms, 4 x 2 1.051, 2 x 4 1.008.
template <int NPAD> struct HCfg;
template <> struct HCfg<32> { static constexpr int NS = 1, KS = 1, STAGES = 4; };
template <> struct HCfg<64> { static constexpr int NS = 1, KS = 1, STAGES = 8; };
template <> struct HCfg<128> { static constexpr int NS = 1, KS = 1, STAGES = 8; };
template <> struct HCfg<160> { static constexpr int NS = 1, KS = 1, STAGES = 6; };
template <> struct HCfg<320> { static constexpr int NS = 2, KS = 2, STAGES = 6; };
template <> struct HCfg<512> { static constexpr int NS = 2, KS = 4, STAGES = 5; };

bool m2l_h_supported(int npad) {
    return npad == 32 || npad == 64 || npad == 128 || npad == 160 || npad == 320 || npad == 512;
}
static void h_split(int npad, int& ns, int& ks) {
    ns = npad == 320 ? HCfg<320>::NS : (npad == 512 ? HCfg<512>::NS : 1);
    ks = npad == 320 ? HCfg<320>::KS : (npad == 512 ? HCfg<512>::KS : 1);
}

// 2^s with the largest scaled entry in [2^14, 2^15); 0 for zero, infinite or NaN rows
__device__ __forceinline__ int h_scale_exp(float m) {
    if (!(m > 0.f) || !(m < __int_as_float(0x7f800000))) return 0;
    const int e = (int)(__float_as_uint(m) >> 23) - 127;         // denormals: -127
    return min(126, 14 - e);
}
__device__ __forceinline__ float h_pow2(int s) { return __uint_as_float((uint32_t)(s + 127) << 23); }

// eight consecutive FP32 values as eight hi and eight lo halves
__device__ __forceinline__ void h_split8(const float* v, float sc, uint4& hi, uint4& lo) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float a = v[2 * i] * sc, b = v[2 * i + 1] * sc;
        const __half2 hh = __floats2half2_rn(a, b);
        const float2 back = __half22float2(hh);
        const __half2 ll = __floats2half2_rn(a - back.x, b - back.y);
        h[i] = *reinterpret_cast<const uint32_t*>(&hh);
        l[i] = *reinterpret_cast<const uint32_t*>(&ll);
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// Column order of a K block: 4 orbits x 8 sign patterns m as (m >> 1) * 8 +
// orbit * 2 + (m & 1), so that a reflection x exchanges whole 16-byte
// vectors (vector index ^ (x >> 1)) and, for x & 1, the halves of each 32-bit
// word: the gather pays an address and four byte permutations per vector.
// (Vectors that hold one orbit each cost twelve selects: the producers were
// issue-bound, M2L 1.13 against 0.83 ms without them at 500k points, p = 8.)
__device__ __forceinline__ int h_col(int vec, int e) { return (e >> 1) * 8 + vec * 2 + (e & 1); }   // vector, half -> natural column of the block

// Source rows: per box [K block][32 hi | 32 lo] halves and the inverse of
// the row's scale.  One warp per box, one 16-byte vector of hi and of lo per
// lane and step; grid y: operator set.  HBM-bound (reads and writes 4 B per
// entry).
struct HPack {
    const float* X[2];
    uint4* out[2];
    float* inv[2];
};
__global__ void __launch_bounds__(256) k_h_pack_rows(int nbox, int npad, HPack P) {
    const int b = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (b >= nbox) return;
    const float2* row = reinterpret_cast<const float2*>(P.X[blockIdx.y] + (size_t)b * npad);
    uint4* out = P.out[blockIdx.y] + (size_t)b * (npad / 4);
    const int ng = npad / 8;                    // <= 64
    float v[2][8];
    float m = 0.f;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int g = lane + 32 * k;
        if (g >= ng) continue;
        const float2* blk = row + (g >> 2) * 16 + (g & 3);
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            const float2 a = blk[4 * o];
            v[k][2 * o] = a.x;
            v[k][2 * o + 1] = a.y;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) m = fabsf(v[k][i]) > m || v[k][i] != v[k][i] ? fabsf(v[k][i]) : m;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const float y = __shfl_xor_sync(0xffffffffu, m, o);
        m = y > m || y != y ? y : m;
    }
    const int s = h_scale_exp(m);
    const float sc = h_pow2(s);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int g = lane + 32 * k;
        if (g >= ng) continue;
        uint4 hi, lo;
        h_split8(v[k], sc, hi, lo);
        out[(g >> 2) * 8 + (g & 3)] = hi;
        out[(g >> 2) * 8 + 4 + (g & 3)] = lo;
    }
    if (lane == 0) P.inv[blockIdx.y][b] = h_pow2(-s);
}

// Operators: [operator][part][K block][N rows][32 hi | 32 lo] halves,
// swizzled, and the inverse scales.  One CTA per operator; slot -> offset by
// the rule of the file's head.
__global__ void __launch_bounds__(256) k_h_pack_ops(int npad, int NS, int KS, int nslot, int level0, const float* __restrict__ m2l,
                                                    uint8_t* __restrict__ out, float* __restrict__ inv) {
    __shared__ float red[256];
    const int slot = blockIdx.x, lev = blockIdx.y;
    int off = slot;
    if (nslot == 64) off = ((slot >> 4) + 3) * 49 + (((slot >> 2) & 3) + 3) * 7 + ((slot & 3) + 3);
    const size_t m2 = (size_t)npad * npad;
    const float* M = m2l + ((size_t)(level0 + lev) * kNumOffsets + off) * m2;
    float m = 0.f;
    for (size_t i = threadIdx.x; i < m2; i += 256) m = fmaxf(m, fabsf(M[i]));
    red[threadIdx.x] = m;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] = fmaxf(red[threadIdx.x], red[threadIdx.x + o]);
        __syncthreads();
    }
    const int s = h_scale_exp(red[0]);
    const float sc = h_pow2(s);
    const size_t op = (size_t)lev * nslot + slot;
    if (threadIdx.x == 0) inv[op] = h_pow2(-s);
    uint8_t* base = out + op * m2 * 4;
    const int N = npad / NS, KB = npad / KS / 32, ng = npad / 8;
    for (int e = threadIdx.x; e < npad * ng; e += 256) {
        const int n = e / ng, g = e % ng;
        float v[8];
        for (int i = 0; i < 8; ++i) v[i] = M[(size_t)n * npad + 32 * (g >> 2) + h_col(g & 3, i)];
        uint4 hi, lo;
        h_split8(v, sc, hi, lo);
        const int r = n % N, kb = g >> 2, c = g & 3, part = (n / N) * KS + kb / KB;
        uint8_t* blk = base + ((size_t)part * KB + kb % KB) * N * 128 + (r >> 3) * 1024 + (r & 7) * 128;
        *reinterpret_cast<uint4*>(blk + ((c ^ (r & 7)) << 4)) = hi;
        *reinterpret_cast<uint4*>(blk + (((4 + c) ^ (r & 7)) << 4)) = lo;
    }
}

void pack_m2l_h(Operators& O, cudaStream_t st) {
    if (!m2l_h_supported(O.npad) || O.nlev <= 2) return;
    O.h_nslot = O.p % 2 == 0 ? 64 : kNumOffsets;
    O.h_single = O.kernel == FMM_LAPLACE;      // 1/r scales with the box: one level (2) serves all
    const int lev = O.h_single ? 1 : O.nlev, l0 = O.h_single ? 2 : 0;
    const size_t nop = (size_t)lev * O.h_nslot;
    O.m2l_h.alloc(nop * O.npad * O.npad * 4, st);
    O.m2l_h_inv.alloc(nop, st);
    int ns, ks;
    h_split(O.npad, ns, ks);
    k_h_pack_ops<<<dim3(O.h_nslot, lev), 256, 0, st>>>(O.npad, ns, ks, O.h_nslot, l0, O.m2l.p, O.m2l_h.p,
                                                       O.m2l_h_inv.p);
    PB_CHECK_LAUNCH();
}

struct HArgs {
    const uint8_t* ops[2];       // packed operators
    const float* iop[2];         // inverse operator scales
    const uint4* X[2];           // packed source rows
    const float* ix[2];          // inverse row scales
    float* Y[2];
    int single[2];               // 1: the set's operators do not depend on the level
    const int4* tiles;           // (first pair, count <= 128, slot * 32 + level, 0)
    const int* seg;              // [nseg + 1] first tile of each segment
    int nseg, nset, nslot, ncols;
    const int* tgt;
    const int* srcx;             // source box | x << 28
    long long wait_limit;
    int* err;
};

template <int STAGES>
struct HSmem {
    uint64_t barB, full[STAGES], empty[STAGES], accf[2], acce[2];
    uint32_t tmem_slot;
    int failed;
};

__device__ __forceinline__ bool h_wait(uint64_t* bar, uint32_t parity, volatile int* failed, long long limit) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (*failed) return false;
        if (clock64() - t0 > limit) {
            *failed = 1;
            return false;
        }
    }
    return true;
}
__device__ __forceinline__ void mma_f16(uint32_t dt, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(dt),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
        : "memory");
}
// one lane of a converged warp
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
    return p != 0;
}
// A CTA's share of the work: segment after segment (set-major), the units
// (part, tile) of each segment cut into gridDim.x equal contiguous ranges.
struct HCursor {
    int set, seg, part, tile, v, vend, t0, t1;
    __device__ void enter(const HArgs& A, int ns) {
        for (;;) {
            if (set == A.nset) return;
            t0 = A.seg[seg];
            t1 = A.seg[seg + 1];
            const long long n = (long long)(t1 - t0) * ns;
            v = (int)(n * blockIdx.x / gridDim.x);
            vend = (int)(n * (blockIdx.x + 1) / gridDim.x);
            if (v < vend) {
                part = v / (t1 - t0);
                tile = v - part * (t1 - t0) + t0;
                return;
            }
            if (++seg == A.nseg) { seg = 0; ++set; }
        }
    }
    __device__ void start(const HArgs& A, int ns) {
        set = seg = 0;
        enter(A, ns);
    }
    __device__ void next(const HArgs& A, int ns) {
        if (set == A.nset) return;
        if (++v == vend) {
            if (++seg == A.nseg) { seg = 0; ++set; }
            enter(A, ns);
        } else if (++tile == t1) {
            tile = t0;
            ++part;
        }
    }
};

// Persistent, one CTA per SM.  The row tiles come in segments of 8,192 target
// boxes (consecutive boxes of a level, hence neighbours), slot-major inside
// a segment: all CTAs work on one segment at a time, so its rows of Qu and
// Qd stay in L2 while its ~300 offsets pass over them, and a CTA reloads its
// operator part only where its contiguous range crosses a slot.  (Reductions
// by bulk copies from a staging buffer, which takes the place of A stages:
// 1.84 ms at 4M points, p = 6.)
//   warps 0-7   producers: gather source rows (16 B per lane, eight lanes per
//               128-byte K-block row), reflect them, write them swizzled
//               into a ring of A stages;
//   warps 8-15  epilogue: accumulator -> registers (lane = row), scale and
//               reflect, transpose 16 columns through shared memory, reduce
//               8 rows x 64 B per instruction;
//   warp 16     loads operator parts and issues the MMAs.
template <int NPAD>
__global__ void __launch_bounds__(kHThreads, 1) k_m2l_f16(const HArgs A) {
    using C = HCfg<NPAD>;
    constexpr int NP = C::NS * C::KS;            // operator parts
    constexpr int N = NPAD / C::NS, KB = NPAD / C::KS / 32, STAGES = C::STAGES;
    static_assert(N % 16 == 0 && N <= 256, "split");
    constexpr uint32_t BBYTES = KB * N * 128;
    constexpr uint32_t ACOLS = N <= 32 ? 32 : (N <= 64 ? 64 : (N <= 128 ? 128 : 256));
    constexpr uint32_t IDESC = (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kHRows >> 4) << 24);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* sB = smem;
    uint8_t* sA = sB + BBYTES;
    float* sE = (float*)(sA + STAGES * kHStageBytes);
    HSmem<STAGES>* S = (HSmem<STAGES>*)(sE + kHEpiWarps * 32 * 16);
    volatile int* failed = &S->failed;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long wl = A.wait_limit;
    int nu = 0;                                  // this CTA's units
    for (int k = 0; k < A.nseg; ++k) {
        const long long n = (long long)(A.seg[k + 1] - A.seg[k]) * NP;
        nu += (int)(n * (blockIdx.x + 1) / gridDim.x) - (int)(n * blockIdx.x / gridDim.x);
    }
    nu *= A.nset;

    if (tid == 0) {
        mbar_init(&S->barB, 1);
        for (int q = 0; q < STAGES; ++q) {
            mbar_init(&S->full[q], kHProdWarps);
            mbar_init(&S->empty[q], 1);
        }
        for (int q = 0; q < 2; ++q) {
            mbar_init(&S->accf[q], 1);
            mbar_init(&S->acce[q], 4);
        }
        S->failed = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(&S->tmem_slot, 2 * ACOLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = S->tmem_slot;

    HCursor cur;
    cur.start(A, NP);
    if (warp < kHProdWarps) {
        // PF K blocks of loads in flight in registers (more spill: 2.09
        // against 1.61 ms at 4M points, p = 6, with PF = 4)
        constexpr int PF = 2;
        const int l8 = lane & 7, rbase = warp * 4 + (lane >> 3);
        const int gend = nu * KB;
        // Units are resolved ahead, so that no load waits for another: the
        // cursor stands two units after fu (the unit being fetched), td is
        // the tile after fu's, sn the sources of that tile.
        auto tile_of = [&]() -> int2 {
            return cur.set < A.nset ? *reinterpret_cast<const int2*>(A.tiles + cur.tile) : make_int2(0, 0);
        };
        auto load_src = [&](int2 t, int* s) {
#pragma unroll
            for (int i = 0; i < kHRowsPerThr; ++i) {
                const int r = i * (kHProdWarps * 4) + rbase;
                s[i] = r < t.y ? A.srcx[t.x + r] : -1;
            }
        };
        uint4 v[PF][kHRowsPerThr];
        uint32_t xm[PF];
        int sc[kHRowsPerThr], sn[kHRowsPerThr];
        int fu = 0, fkb = 0;                     // the next block to fetch
        // a unit's set and column part of the source rows, and where these begin
        auto sp_of = [&]() { return cur.set * C::KS + cur.part % C::KS; };
        auto x_of = [&](int sp) {
            return sp < A.nset * C::KS ? A.X[sp / C::KS] + (sp % C::KS) * KB * 8 + l8 : nullptr;
        };
        int sp1 = sp_of(), sp2;                  // of the units fu + 1 and fu + 2
        const uint4* X = x_of(sp1);
        load_src(tile_of(), sc);
        cur.next(A, NP);
        sp1 = sp_of();
        load_src(tile_of(), sn);
        cur.next(A, NP);
        sp2 = sp_of();
        int2 td = tile_of();
        auto fetch = [&](uint4* d, uint32_t& x) {
            if (fkb == KB) {
                fkb = 0;
                ++fu;
                X = x_of(sp1);
#pragma unroll
                for (int i = 0; i < kHRowsPerThr; ++i) sc[i] = sn[i];
                load_src(td, sn);
                cur.next(A, NP);
                td = tile_of();
                sp1 = sp2;
                sp2 = sp_of();
            }
            x = 0;
            if (fu < nu) {
#pragma unroll
                for (int i = 0; i < kHRowsPerThr; ++i) {
                    d[i] = sc[i] >= 0 ? X[(size_t)(sc[i] & 0x0fffffff) * (NPAD / 4) + fkb * 8] : make_uint4(0, 0, 0, 0);
                    x |= (uint32_t)((sc[i] >> 28) & 7) << (4 * i);
                }
            }
            ++fkb;
        };
#pragma unroll
        for (int j = 0; j < PF; ++j) fetch(v[j], xm[j]);
        int g = 0, s = 0, ph = 1;            // stage and the parity of its last release (1: a fresh barrier passes)
        while (g < gend) {
#pragma unroll
            for (int j = 0; j < PF; ++j) {
                if (g < gend) {
                    if (!h_wait(&S->empty[s], ph, failed, wl)) goto prod_done;
                    uint8_t* a = sA + (size_t)s * kHStageBytes;
#pragma unroll
                    for (int i = 0; i < kHRowsPerThr; ++i) {
                        const int r = i * (kHProdWarps * 4) + rbase;
                        const uint32_t x = xm[j] >> (4 * i);
                        const uint32_t sel = (x & 1) ? 0x1032u : 0x3210u;
                        const int c = l8 ^ ((x >> 1) & 3);       // hi and lo vectors alike
                        *(uint4*)(a + (r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4)) =
                            make_uint4(__byte_perm(v[j][i].x, 0, sel), __byte_perm(v[j][i].y, 0, sel),
                                       __byte_perm(v[j][i].z, 0, sel), __byte_perm(v[j][i].w, 0, sel));
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&S->full[s]);
                    fetch(v[j], xm[j]);
                    ++g;
                    if (++s == STAGES) { s = 0; ph ^= 1; }
                }
            }
        }
    prod_done:
        __syncwarp();
    } else if (warp < kHProdWarps + kHEpiWarps) {
        // Groups of four warps take the units in turn.
        constexpr int EG = kHEpiWarps / 4;
        const int q = warp & 3, r = q * 32 + lane, eg = (warp - kHProdWarps) >> 2;
        float* buf = sE + (warp - kHProdWarps) * 32 * 16;
        // resolved ahead, as in the producers: tile of the group's unit after
        // next, target and source of its next, scale at this one's end
        auto tile_of = [&]() -> int4 { return cur.set < A.nset ? A.tiles[cur.tile] : make_int4(0, 0, 0, 0); };
        struct Row { int tgt, sx; };
        auto load_row = [&](int4 t) -> Row {
            return r < t.y ? Row{A.tgt[t.x + r], A.srcx[t.x + r]} : Row{-1, -1};
        };
        auto load_scale = [&](int set, int z, int sx) -> float {
            if (sx < 0) return 0.f;
            return A.ix[set][sx & 0x0fffffff] * A.iop[set][(A.single[set] ? 0 : (z & 31) * A.nslot) + (z >> 5)];
        };
        for (int i = 0; i < eg; ++i) cur.next(A, NP);
        int set = cur.set, part = cur.part;
        int4 t = tile_of();
        Row row = load_row(t);
        float f = load_scale(set, t.z, row.sx);
        for (int i = 0; i < EG; ++i) cur.next(A, NP);
        int set1 = cur.set, part1 = cur.part;
        t = tile_of();
        for (int k = eg; k < nu; k += EG) {
            const int a = k & 1;
            const int x = (row.sx >> 28) & 7;
            const Row row1 = load_row(t);
            const int z1 = t.z;
            for (int i = 0; i < EG; ++i) cur.next(A, NP);
            const int set2 = cur.set, part2 = cur.part;
            t = tile_of();
            // after the transpose a lane adds 16 B of the rows j * 8 + lane / 4
            float* y[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int tr = __shfl_sync(0xffffffffu, row.tgt, j * 8 + (lane >> 2));
                y[j] = tr >= 0 ? A.Y[set] + (size_t)tr * NPAD + (part / C::KS) * N + (lane & 3) * 4 : nullptr;
            }
            const int cmax = A.ncols - (part / C::KS) * N - (lane & 3) * 4;      // this lane's columns end
            const bool ok = h_wait(&S->accf[a], (k >> 1) & 1, failed, wl);
            if (!__all_sync(0xffffffffu, ok)) break;
            tc_fence_after();
            const uint32_t tb = taddr + ((uint32_t)(q * 32) << 16) + a * ACOLS;
            const bool x4 = x & 4, x2 = x & 2, x1 = x & 1;
            auto drain = [&](const uint32_t* e, int c0) {
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const float d0 = __uint_as_float(e[4 * h]) * f, d1 = __uint_as_float(e[4 * h + 1]) * f;
                    const float d2 = __uint_as_float(e[4 * h + 2]) * f, d3 = __uint_as_float(e[4 * h + 3]) * f;
                    const float g0 = x2 ? d2 : d0, g1 = x2 ? d3 : d1, g2 = x2 ? d0 : d2, g3 = x2 ? d1 : d3;
                    // 16-byte pieces exchanged by row so that neither side has bank conflicts
                    const int pos = (h ^ (int)x4) ^ ((lane >> 1) & 3);
                    *(float4*)(buf + lane * 16 + pos * 4) =
                        make_float4(x1 ? g1 : g0, x1 ? g0 : g1, x1 ? g3 : g2, x1 ? g2 : g3);
                }
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int rr = j * 8 + (lane >> 2);
                    const float4 w = *(const float4*)(buf + rr * 16 + (((lane & 3) ^ (rr >> 1)) & 3) * 4);
                    if (y[j] && c0 < cmax) red_add_v4(y[j] + c0, w.x, w.y, w.z, w.w);
                }
                __syncwarp();
            };
            // the next 16 columns load while these are added
            uint32_t da[16], db[16];
            tmem_ld16_issue(tb, da);
            tmem_wait16(da);
#pragma unroll 1
            for (int c0 = 0; c0 < N; c0 += 32) {
                if (c0 + 16 < N) tmem_ld16_issue(tb + c0 + 16, db);
                drain(da, c0);
                if (c0 + 16 >= N) break;
                tmem_wait16(db);
                if (c0 + 32 < N) tmem_ld16_issue(tb + c0 + 32, da);
                drain(db, c0 + 16);
                if (c0 + 32 < N) tmem_wait16(da);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S->acce[a]);
            row = row1;
            f = load_scale(set1, z1, row.sx);
            set = set1; part = part1;
            set1 = set2; part1 = part2;
        }
        __syncwarp();
    } else {
        // the whole warp runs the loop, one elected lane issues: the operands
        // of tcgen05.mma stay in uniform registers (84 against 91 cycles per
        // MMA at N = 160, 72 against 91 at N = 64, measured alone)
        uint64_t* last = nullptr;      // barrier of the last commit, and its phase parity
        uint32_t last_par = 0;
        int s = 0, nload = 0;
        uint32_t par = 0;
        bool ok = true;
        const uint8_t* held = nullptr;
        const uint64_t ad0 = sw128_desc(smem_u32(sA)), bd0 = sw128_desc(smem_u32(sB));
        int4 t = nu > 0 ? A.tiles[cur.tile] : make_int4(0, 0, 0, 0);
        for (int k = 0; ok && k < nu; ++k) {
            const int a = k & 1;
            const int op = (A.single[cur.set] ? 0 : (t.z & 31) * A.nslot) + (t.z >> 5);
            const uint8_t* want = A.ops[cur.set] + ((size_t)op * NP + cur.part) * BBYTES;
            cur.next(A, NP);
            if (k + 1 < nu) t = A.tiles[cur.tile];
            if (want != held) {
                // every MMA that reads the held part is done before it is overwritten
                if (last && !(ok = h_wait(last, last_par, failed, wl))) break;
                if (elect_one()) {
                    mbar_arrive_expect_tx(&S->barB, BBYTES);
                    for (int kb = 0; kb < KB; ++kb)
                        bulk_g2s(sB + (size_t)kb * N * 128, want + (size_t)kb * N * 128, N * 128, &S->barB);
                }
                __syncwarp();
                ++nload;
                if (!(ok = h_wait(&S->barB, (nload - 1) & 1, failed, wl))) break;
                held = want;
            }
            if (k > 1 && !(ok = h_wait(&S->acce[a], ((k >> 1) - 1) & 1, failed, wl))) break;
            const uint32_t dacc = taddr + a * ACOLS;
            uint64_t bd = bd0;
            for (int kb = 0; kb < KB; ++kb, bd += N * 8) {
                if (!(ok = h_wait(&S->full[s], par, failed, wl))) break;
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t ad = ad0 + s * (kHStageBytes >> 4);
#pragma unroll
                    for (int ks = 0; ks < 2; ++ks) {
                        const uint32_t h = ks * 2, l = 4 + ks * 2;       // 16-byte units in the 128-byte row
                        mma_f16(dacc, ad + h, bd + h, IDESC, (kb > 0 || ks > 0) ? 1u : 0u);
                        mma_f16(dacc, ad + h, bd + l, IDESC, 1u);
                        mma_f16(dacc, ad + l, bd + h, IDESC, 1u);
                    }
                    mma_commit(&S->empty[s]);
                    if (kb == KB - 1) mma_commit(&S->accf[a]);
                }
                __syncwarp();
                last = &S->empty[s];
                last_par = par;
                if (++s == STAGES) { s = 0; par ^= 1; }
            }
            if (ok) {
                last = &S->accf[a];
                last_par = (k >> 1) & 1;
            }
        }
        // every MMA and operator copy issued here ends before TMEM is freed
        // and the CTA's shared memory given up, whichever role gave up
        // waiting: an epilogue that timed out leaves the last ones in flight
        if (last) mbar_wait(last, last_par);
        if (nload) mbar_wait(&S->barB, (nload - 1) & 1);
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0 && S->failed) atomicExch(A.err, 1);
    if (warp == 0) tmem_dealloc(taddr, 2 * ACOLS);
}

template <int NPAD>
static constexpr size_t h_smem_bytes() {
    using C = HCfg<NPAD>;
    return 1024 + (size_t)(NPAD / C::KS) * (NPAD / C::NS) * 4 + C::STAGES * (size_t)kHStageBytes +
           kHEpiWarps * 32 * 16 * sizeof(float) + sizeof(HSmem<C::STAGES>);
}
static_assert(h_smem_bytes<128>() <= 232448 && h_smem_bytes<160>() <= 232448 && h_smem_bytes<320>() <= 232448 &&
                  h_smem_bytes<512>() <= 232448,
              "shared memory per CTA");

template <int NPAD>
static void h_launch(const HArgs& a, int ntile, int sm_count, cudaStream_t st) {
    static bool done[64] = {false};
    int dev = 0;
    PB_CUDA(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64 && !done[dev]) {
        PB_CUDA(cudaFuncSetAttribute(k_m2l_f16<NPAD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)h_smem_bytes<NPAD>()));
        done[dev] = true;
    }
    const int grid = (int)std::min<long long>(sm_count, (long long)ntile * HCfg<NPAD>::NS * HCfg<NPAD>::KS * a.nset);
    k_m2l_f16<NPAD><<<grid, kHThreads, h_smem_bytes<NPAD>(), st>>>(a);
    PB_CHECK_LAUNCH();
}

static bool h_dispatch(int npad, const HArgs& a, int ntile, int sms, cudaStream_t st) {
    switch (npad) {
        case 32: h_launch<32>(a, ntile, sms, st); return true;
        case 64: h_launch<64>(a, ntile, sms, st); return true;
        case 128: h_launch<128>(a, ntile, sms, st); return true;
        case 160: h_launch<160>(a, ntile, sms, st); return true;
        case 320: h_launch<320>(a, ntile, sms, st); return true;
        case 512: h_launch<512>(a, ntile, sms, st); return true;
        default: return false;
    }
}

// M2L for one operator set or two (O2) in one launch.  tmp / tmp2: packed
// source rows, n_box * (n_pad + 1) floats each.  False when this path does
// not apply to the operators.
bool m2l_h_launch(const fmm_tree* T, const Operators& O, const Operators* O2, const float* Qu, float* Qd, float* tmp,
                  const float* Qu2, float* Qd2, float* tmp2, int* err, cudaStream_t st) {
    if (!O.m2l_h.p || (O2 && (!O2->m2l_h.p || O2->npad != O.npad))) return false;
    const auto& P = T->m2l_pairs;
    const bool even = O.h_nslot == 64;
    HArgs a{};
    const int ntile = even ? P.ntile_even : P.ntile_odd;
    if (ntile == 0) return true;
    a.tiles = even ? P.tiles_even.p : P.tiles_odd.p;
    a.seg = even ? P.seg_even.p : P.seg_odd.p;
    a.nseg = P.nseg;
    a.nset = O2 ? 2 : 1;
    a.nslot = O.h_nslot;
    a.ncols = O.ne;
    a.tgt = P.tgt.p;
    a.srcx = even ? P.srcx.p : P.src.p;
    a.wait_limit = g_wait_limit.load();
    a.err = err;
    HPack pk{};
    const Operators* os[2] = {&O, O2};
    const float* qs[2] = {Qu, Qu2};
    float* ys[2] = {Qd, Qd2};
    float* ts[2] = {tmp, tmp2};
    for (int k = 0; k < a.nset; ++k) {
        a.ops[k] = os[k]->m2l_h.p;
        a.iop[k] = os[k]->m2l_h_inv.p;
        a.single[k] = os[k]->h_single ? 1 : 0;
        a.X[k] = reinterpret_cast<const uint4*>(ts[k]);
        a.ix[k] = ts[k] + (size_t)T->nbox * O.npad;
        a.Y[k] = ys[k];
        pk.X[k] = qs[k];
        pk.out[k] = reinterpret_cast<uint4*>(ts[k]);
        pk.inv[k] = ts[k] + (size_t)T->nbox * O.npad;
    }
    k_h_pack_rows<<<dim3(div_up(T->nbox, 8), a.nset), 256, 0, st>>>(T->nbox, O.npad, pk);
    PB_CHECK_LAUNCH();
    return h_dispatch(O.npad, a, ntile, T->ctx->sm_count, st);
}

// D[i][n ^ x_i] += sum_k Op[n][k] Q[i][k ^ x_i] through the kernel: device
// buffers, sign bits xs [nrows] on the host (null: 0), x only for n_pad
// orders of even p.  Used by the test hooks.
void m2l_h_selftest(int nrows, int npad, const float* Q, const float* Op, const int* xs, float* D, int* err,
                    cudaStream_t st) {
    constexpr int kSlot = 3 * 16 + 2 * 4 + 1, kOffset = 6 * 49 + 5 * 7 + 4;      // offset (3, 2, 1)
    const size_t m2 = (size_t)npad * npad;
    DBuf<float> m2l, inv, rows;
    DBuf<uint8_t> ops;
    DBuf<int> tgt, srcx, seg;
    DBuf<int4> tiles;
    m2l.alloc(kNumOffsets * m2, st);
    m2l.zero(st);
    PB_CUDA(cudaMemcpyAsync(m2l.p + kOffset * m2, Op, m2 * sizeof(float), cudaMemcpyDeviceToDevice, st));
    ops.alloc(64 * m2 * 4, st);
    inv.alloc(64, st);
    int ns, ks;
    h_split(npad, ns, ks);
    k_h_pack_ops<<<dim3(64, 1), 256, 0, st>>>(npad, ns, ks, 64, 0, m2l.p, ops.p, inv.p);
    PB_CHECK_LAUNCH();
    std::vector<int> ht(nrows), hs(nrows);
    for (int i = 0; i < nrows; ++i) { ht[i] = i; hs[i] = i | (xs ? xs[i] & 7 : 0) << 28; }
    std::vector<int4> htile;
    for (int i = 0; i < nrows; i += kHRows) htile.push_back(make_int4(i, std::min(kHRows, nrows - i), kSlot * 32, 0));
    const int hseg[3] = {0, (int)htile.size() / 2, (int)htile.size()};           // two segments
    tgt.alloc(nrows, st); srcx.alloc(nrows, st); tiles.alloc(htile.size(), st); seg.alloc(3, st);
    rows.alloc((size_t)nrows * (npad + 1), st);
    PB_CUDA(cudaMemcpyAsync(tgt.p, ht.data(), nrows * sizeof(int), cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaMemcpyAsync(srcx.p, hs.data(), nrows * sizeof(int), cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaMemcpyAsync(tiles.p, htile.data(), htile.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
    PB_CUDA(cudaMemcpyAsync(seg.p, hseg, sizeof(hseg), cudaMemcpyHostToDevice, st));
    HPack pk{{Q, nullptr}, {reinterpret_cast<uint4*>(rows.p), nullptr}, {rows.p + (size_t)nrows * npad, nullptr}};
    k_h_pack_rows<<<div_up(nrows, 8), 256, 0, st>>>(nrows, npad, pk);
    PB_CHECK_LAUNCH();
    HArgs a{};
    a.ops[0] = ops.p; a.iop[0] = inv.p; a.X[0] = pk.out[0]; a.ix[0] = pk.inv[0]; a.Y[0] = D;
    a.single[0] = 1;
    a.tiles = tiles.p; a.seg = seg.p; a.nseg = 2; a.nset = 1; a.nslot = 64; a.ncols = npad;
    a.tgt = tgt.p; a.srcx = srcx.p;
    a.wait_limit = g_wait_limit.load();
    a.err = err;
    int dev = 0, sms = 0;
    PB_CUDA(cudaGetDevice(&dev));
    PB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    h_dispatch(npad, a, (int)htile.size(), sms, st);
    PB_CUDA(cudaStreamSynchronize(st));                   // the host vectors go out of scope
}

// registers, max threads, static and dynamic shared bytes, resident CTAs
void m2l_h_info(int* out) {
    cudaFuncAttributes fa;
    PB_CUDA(cudaFuncSetAttribute(k_m2l_f16<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)h_smem_bytes<128>()));
    PB_CUDA(cudaFuncGetAttributes(&fa, k_m2l_f16<128>));
    int dev = 0, sms = 0, per = 0;
    PB_CUDA(cudaGetDevice(&dev));
    PB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    PB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_m2l_f16<128>, kHThreads, h_smem_bytes<128>()));
    out[0] = fa.numRegs;
    out[1] = fa.maxThreadsPerBlock;
    out[2] = (int)fa.sharedSizeBytes;
    out[3] = (int)h_smem_bytes<128>();
    out[4] = per * sms;
}

}  // namespace pbfmm

extern "C" int pbfmm_selftest_m2l_f16(int nrows, int npad, const float* Q, const float* Op, const int32_t* xs, float* D) {
    using namespace pbfmm;
    try {
        if (nrows < 1 || !m2l_h_supported(npad)) return PB_EINVAL;
        cudaStream_t st = nullptr;
        DBuf<float> q, op, d;
        DBuf<int> e;
        const size_t n = (size_t)nrows * npad;
        q.alloc(n, st); op.alloc((size_t)npad * npad, st); d.alloc(n, st); e.alloc(1, st);
        d.zero(st);
        e.zero(st);
        PB_CUDA(cudaMemcpyAsync(q.p, Q, n * 4, cudaMemcpyHostToDevice, st));
        PB_CUDA(cudaMemcpyAsync(op.p, Op, (size_t)npad * npad * 4, cudaMemcpyHostToDevice, st));
        m2l_h_selftest(nrows, npad, q.p, op.p, xs, d.p, e.p, st);
        int herr = 0;
        PB_CUDA(cudaMemcpyAsync(&herr, e.p, 4, cudaMemcpyDeviceToHost, st));
        PB_CUDA(cudaMemcpyAsync(D, d.p, n * 4, cudaMemcpyDeviceToHost, st));
        PB_CUDA(cudaStreamSynchronize(st));
        return herr ? PB_ETIMEOUT : PB_OK;
    } catch (const Error& ex) {
        return ex.code;
    }
}
