// ft_gemm.cu -- the folded tensor-core contraction (ft_gemm.cuh), its operand producers and the
// return from parity classes to planes.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cudaTypedefs.h>

#include <algorithm>
#include <type_traits>

#include "fft_pair.cuh"
#include "ft_gemm.cuh"
#include "tc_ptx.cuh"
#include "tcx_slices.cuh"

namespace coro {

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder();   // tc_gemm.cu

namespace {

constexpr int BM = 128;                     // rows per tile (UMMA M)
constexpr int XPAIR_BYTES = BM * 128;       // one plane pair of an X stage: 128 rows x 128 bytes
constexpr int MAX_STAGES = 6;

template <int FMT> struct FtCfg {
    static constexpr bool EXT = FMT == FT_EXT;
    static constexpr bool B16 = FMT != FT_TF32;
    static constexpr int S = FMT + 2;                         // planes per operand
    static constexpr int PAIRS = (S + 1) / 2;
    // 64-byte K slices per drain: 12 (FT_EXT: 40) MMAs, so that the accumulator truncates no more
    // often than one sum of three products over 16 K steps would
    static constexpr int CHUNK = FMT == FT_BF16 ? 1 : 2;
    static constexpr int KE = B16 ? 32 : 16;                  // elements of a 64-byte slice
    // two plane pairs fill the shared memory of one block per SM (and two-float sums its registers):
    // sixteen epilogue warps there, against eight on each of two blocks of FT_TF32, whose
    // prologues, drains and stores then hide one another
    static constexpr int PER_SM = FMT == FT_TF32 ? 2 : 1;
    static constexpr int EPI_WARPS = 16 / PER_SM;
    static constexpr int THREADS = 64 + 32 * EPI_WARPS;
    static constexpr int COLG = EPI_WARPS / 4;                // column groups
    static constexpr int PARTS = 128 / COLG / 8;              // 8-column parts per warp at the widest tile
    static constexpr uint32_t TMEM_COLS = EXT ? 512 : 256;    // 2 buffers x (1 or 2 levels) x 128
    static constexpr int SMEM_BUDGET = PER_SM == 1 ? 200 * 1024 : 98 * 1024;
};

// ------------------------------------------------------------------ stored values

template <int FMT> struct FtElem { using type = __nv_bfloat16; };
template <> struct FtElem<FT_TF32> { using type = float; };

__device__ __forceinline__ float tf32_rna(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

// Place of inner index k in a row (of the first plane of a pair; the second is KE elements on).
template <int FMT> __device__ __forceinline__ int slot(int k) { return k + (k & ~(FtCfg<FMT>::KE - 1)); }

// The planes of a value (FT_TF32: 22 bits, FT_BF16: 24); `pair` elements between plane pairs.
template <int FMT>
__device__ __forceinline__ void put(typename FtElem<FMT>::type* p, size_t pair, float v) {
    constexpr int KE = FtCfg<FMT>::KE;
    if constexpr (FMT == FT_TF32) {
        const float h = tf32_rna(v);
        p[0] = h;
        p[KE] = tf32_rna(v - h);
    } else {
        const __nv_bfloat16 h = __float2bfloat16_rn(v);
        const float r = v - __bfloat162float(h);
        const __nv_bfloat16 m = __float2bfloat16_rn(r);
        p[0] = h;
        p[KE] = m;
        p[pair] = __float2bfloat16_rn(r - __bfloat162float(m));
    }
}

__device__ __forceinline__ void put4(__nv_bfloat16* p, size_t pair, float h, float l, int ge) {
    constexpr int KE = FtCfg<FT_EXT>::KE;
    float s[4];
    make_slices(h, l, ge, s);
#pragma unroll
    for (int i = 0; i < 4; ++i) p[(i >> 1) * pair + (i & 1) * KE] = __float2bfloat16_rn(s[i]);
}

// The value back: (h, l), l = 0 outside FT_EXT.
template <int FMT>
__device__ __forceinline__ void get(const typename FtElem<FMT>::type* p, size_t pair, float& h, float& l) {
    constexpr int KE = FtCfg<FMT>::KE;
    if constexpr (FMT == FT_TF32) {
        h = p[0] + p[KE];
        l = 0.f;
    } else if constexpr (FMT == FT_BF16) {
        h = __bfloat162float(p[0]) + (__bfloat162float(p[KE]) + __bfloat162float(p[pair]));
        l = 0.f;
    } else {
        const float s0 = __bfloat162float(p[0]), s1 = __bfloat162float(p[KE]);
        const float s2 = __bfloat162float(p[pair]), s3 = __bfloat162float(p[pair + KE]);
        two_sum(s0 + s1, s2, h, l);                  // s0 + s1 is exact
        l += s3;
    }
}

// (h, l) += (bh, bl): sums that end in FP64 are kept like this, FP64 running at 1/64 of the FP32 rate
__device__ __forceinline__ void add22(float& h, float& l, float bh, float bl) {
    float s, e;
    two_sum(h, bh, s, e);
    h = s;
    l += e + bl;
}

// An infinite sum's low part is NaN and adds nothing.
__device__ __forceinline__ double sum22(float h, float l) { return (double)h + (l == l ? (double)l : 0.0); }

// ------------------------------------------------------------------ tiles

// K slices a tile runs: rows m0 ... of the flattened (q, c, i), columns n0 ...; none where the mask
// drops every output. Shared with the host-side count. (32-bit arithmetic: indices stay below 4100.)
__host__ __device__ inline int ft_slices(const FtItem& it, int R, int m0, int n0, int ke, bool masked) {
    const int last = m0 + BM - 1 < 4 * R - 1 ? m0 + BM - 1 : 4 * R - 1;
    const int near = m0 / R == last / R ? m0 % R : 0;
    if (near >= it.H || (masked && near * near + n0 * n0 > it.thr_out)) return 0;
    int K = it.K;
    if (it.thr_in >= 0) {
        const int rem = it.thr_in - near * near;
        if (rem < 0) return 0;
        int w = (int)sqrtf((float)rem);
        while (w * w > rem) --w;
        while ((w + 1) * (w + 1) <= rem) ++w;
        if (w + 1 < K) K = w + 1;
    }
    return (K + ke - 1) / ke;
}

// One half of a packed pair (`which` a constant).
__device__ __forceinline__ float pk_half(pk::u64 v, int which) {
    float a, b;
    pk::unpack(v, a, b);
    return which ? b : a;
}

struct FtTile {
    int b, p, m0, n0, slices;
    bool live;
};

// Tile t of the walk: items, parities, row tiles, column tiles fastest (neighbours share X rows).
template <int FMT, int EPI>
__device__ __forceinline__ FtTile ft_tile(const FtArgs& a, int t, int nt, int tiles_n, int tiles_m) {
    FtTile tl;
    const int mn = tiles_n * tiles_m;
    tl.b = t / (2 * mn);
    int r = t - tl.b * 2 * mn;
    tl.p = r / mn;
    r -= tl.p * mn;
    tl.m0 = (r / tiles_n) * BM;
    tl.n0 = (r % tiles_n) * nt;
    const FtItem& it = a.items[tl.b];
    tl.live = tl.n0 < it.N;
    tl.slices = tl.live ? ft_slices(it, a.R, tl.m0, tl.n0, FtCfg<FMT>::KE, EPI == FT_SPLIT || EPI == FT_BABINET || EPI == FT_SEED) : 0;
    return tl;
}

// Blocks walk the tiles blockIdx.x, + gridDim.x, ... Warp 0 streams 128-byte K slices of all plane pairs
// of X (128 rows) and W (nt rows) through a ring of `stages` shared buffers, one 4-D TMA each; warp 1
// issues the MMAs, those sharing an X plane back to back (A collector), into one of two TMEM buffers
// per CHUNK slices; the other warps add each drained buffer into registers and run the epilogue,
// while the MMAs of the following chunks (or tile) go on. All walk the tiles alike with running
// stage and drain counters.
//
// What bounds it: the epilogue warps' instructions. An output costs a packed half add per drain and
// some ten instructions at the end, against 26 x 18 tensor clocks for 128 x 96 of them at K = 410;
// the first form of the epilogue (masks and addresses in full per output, 65 instructions) ran the
// 168-item detector contraction in 1.06 ms, this one in 0.85. Measured and left out:
// clusters of two or four row tiles sharing W by multicast (1.05 / 1.32 ms: loads are not the limit).
template <int FMT, int EPI>
__global__ void __launch_bounds__(FtCfg<FMT>::THREADS, FtCfg<FMT>::PER_SM)
ft_gemm_kernel(const __grid_constant__ CUtensorMap mx, const __grid_constant__ CUtensorMap mw, const FtArgs a, int nt,
               int tiles_n, int tiles_m, int items, int stages) {
    using Cfg = FtCfg<FMT>;
    using E = typename FtElem<FMT>::type;
    constexpr int S = Cfg::S, PAIRS = Cfg::PAIRS, KE = Cfg::KE, PARTS = Cfg::PARTS;
    constexpr bool EXT = Cfg::EXT;
    const int total = 2 * tiles_n * tiles_m * items;
    const int wpair = nt * 128, x_bytes = PAIRS * XPAIR_BYTES, stage_bytes = x_bytes + PAIRS * wpair;

    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t full[MAX_STAGES], empty[MAX_STAGES], tfull[2], tempty[2];
    __shared__ uint32_t tslot;
    __shared__ uint32_t xmax[EXT ? Cfg::EPI_WARPS * PARTS * 8 : 1];

    // the warp index through a shuffle, which tells the compiler that it is uniform
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) { tc::mbar_init(&full[s], 1); tc::mbar_init(&empty[s], 1); }
        for (int s = 0; s < 2; ++s) { tc::mbar_init(&tfull[s], 1); tc::mbar_init(&tempty[s], Cfg::EPI_WARPS); }
        tc::fence_mbar_init();
        tc::prefetch_tmap(&mx);
        tc::prefetch_tmap(&mw);
    }
    if (warp == 1) {
        tc::tmem_alloc(&tslot, Cfg::TMEM_COLS);
        tc::tmem_relinquish();
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tbase = tslot;
    constexpr uint32_t BUF = EXT ? 256 : 128;        // TMEM columns of one buffer

    if (warp == 0) {
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
                const FtTile tl = ft_tile<FMT, EPI>(a, t, nt, tiles_n, tiles_m);
                const int w_idx = a.items[tl.b].w_idx;
                for (int k = 0; k < tl.slices; ++k) {
                    if (!(ok = tc::mbar_wait(&empty[s], ph ^ 1, a.err, 21))) break;
                    unsigned char* st = smem + s * stage_bytes;
                    tc::mbar_arrive_expect_tx(&full[s], stage_bytes);
                    tc::tma_load_4d(st, &mx, &full[s], k * 2 * KE, tl.m0, tl.p * PAIRS, tl.b);
                    tc::tma_load_4d(st + x_bytes, &mw, &full[s], k * 2 * KE, tl.n0, tl.p * PAIRS, w_idx);
                    if (++s == stages) { s = 0; ph ^= 1; }
                }
            }
            // no copy is in flight when the block ends, whatever wait expired: the last load of each stage
            // (a stage never loaded passes, its barrier being in its first phase)
#pragma unroll 1
            for (int x = 0; x < stages; ++x) tc::mbar_wait(&full[x], x < s ? ph : ph ^ 1, a.err, 25);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t ID = tc::idesc<Cfg::B16>(BM, nt, false);
            bool ok = true;
            int s = 0;
            uint32_t ph = 0;
            unsigned g = 0;                          // running drain counter
            for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
                const FtTile tl = ft_tile<FMT, EPI>(a, t, nt, tiles_n, tiles_m);
                for (int k = 0; k < tl.slices; ++k) {
                    const uint32_t buf = g & 1;
                    const bool first = k % Cfg::CHUNK == 0;
                    if (first) {
                        if (!(ok = tc::mbar_wait(&tempty[buf], ((g >> 1) & 1) ^ 1, a.err, 24))) break;
                        tc::tc_fence_after();
                    }
                    if (!(ok = tc::mbar_wait(&full[s], ph, a.err, 22))) break;
                    tc::tc_fence_after();
                    const uint32_t d0 = tbase + buf * BUF;
                    const uint32_t xa = tc::smem_u32(smem + s * stage_bytes), wa = xa + x_bytes;
                    const uint32_t keep = first ? 0u : 1u;
                    if constexpr (EXT) {
#pragma unroll
                        for (int kk = 0; kk < 2; ++kk) {             // two MMA K steps of 32 bytes
                            // plane and K-step offsets move the descriptor's start address only
                            const uint64_t dx = tc::sdesc_sw128(xa + kk * 32), dw = tc::sdesc_sw128(wa + kk * 32);
#pragma unroll
                            for (int i = 0; i < S; ++i) {
                                const uint64_t ad = dx + (uint64_t)(((i >> 1) * XPAIR_BYTES + (i & 1) * 64) >> 4);
                                const int last = S - 1 - i;          // products of planes i + j < S
#pragma unroll
                                for (int j = 0; j <= last; ++j) {
                                    const uint64_t bd = dw + (uint64_t)(((j >> 1) * wpair + (j & 1) * 64) >> 4);
                                    // level 0 alone, levels 1-3 in a second accumulator
                                    const uint32_t d = d0 + (i + j ? 128u : 0u);
                                    const uint32_t acc = kk == 0 && i == 0 && j <= 1 ? keep : 1u;
                                    if (last == 0) tc::umma_coll<Cfg::B16, tc::COLL_NONE>(d, ad, bd, ID, acc);
                                    else if (j == 0) tc::umma_coll<Cfg::B16, tc::COLL_FILL>(d, ad, bd, ID, acc);
                                    else if (j == last) tc::umma_coll<Cfg::B16, tc::COLL_LASTUSE>(d, ad, bd, ID, acc);
                                    else tc::umma_coll<Cfg::B16, tc::COLL_USE>(d, ad, bd, ID, acc);
                                }
                            }
                        }
                    } else {
                        // products with the lower planes of X first, those of its upper plane from the lowest
                        // plane of W up: every MMA cuts its sum off at the accumulator's last bit, so the
                        // small products go in while it is small (dark-hole sums of 3xTF32 Lyot images off
                        // by 1.6e-5 with the products from large to small, 1.2e-5 like this; 3xBF16 1.4e-5
                        // and 0.5e-5; same time)
                        const uint64_t dx = tc::sdesc_sw128(xa), dw = tc::sdesc_sw128(wa);
#pragma unroll
                        for (int i = S - 1; i >= 0; --i) {
                            const uint64_t di = dx + (uint64_t)(((i >> 1) * XPAIR_BYTES + (i & 1) * 64) >> 4);
#pragma unroll
                            for (int kk = 0; kk < 2; ++kk) {
                                const uint64_t ad = di + kk * 2;
#pragma unroll
                                for (int j = S - 1 - i; j >= 0; --j) {
                                    const uint64_t bd = dw + (uint64_t)(((j >> 1) * wpair + (j & 1) * 64) >> 4) + kk * 2;
                                    const uint32_t acc = kk == 0 && i == S - 1 ? keep : 1u;
                                    if (i == S - 1) tc::umma_coll<Cfg::B16, tc::COLL_NONE>(d0, ad, bd, ID, acc);
                                    else if (j == S - 1 - i) tc::umma_coll<Cfg::B16, tc::COLL_FILL>(d0, ad, bd, ID, acc);
                                    else if (j == 0) tc::umma_coll<Cfg::B16, tc::COLL_LASTUSE>(d0, ad, bd, ID, acc);
                                    else tc::umma_coll<Cfg::B16, tc::COLL_USE>(d0, ad, bd, ID, acc);
                                }
                            }
                        }
                    }
                    tc::umma_commit(&empty[s]);                  // frees the stage once these MMAs retire
                    if (++s == stages) { s = 0; ph ^= 1; }
                    if (k % Cfg::CHUNK == Cfg::CHUNK - 1 || k == tl.slices - 1) {
                        tc::umma_commit(&tfull[buf]);
                        ++g;
                    }
                }
            }
            // nor is an MMA, when the tensor memory is given back
            tc::mbar_wait(&empty[(s ? s : stages) - 1], s ? ph : ph ^ 1, a.err, 26);
        }
    } else {
        const int q = warp & 3;                      // TMEM lane quarter this warp may read
        const int cg = (warp - 2) >> 2;              // column group
        const int cols = nt / Cfg::COLG, np = cols / 8;
        const uint32_t lane_base = tbase + ((uint32_t)(q * 32) << 16) + cg * cols;
        bool ok = true;
        unsigned g = 0;
        // every epilogue warp walks every tile even after a wait has failed (no further waits or
        // stores then), so that partner warps always meet at their barriers
        for (int t = blockIdx.x; t < total; t += gridDim.x) {
            const FtTile tl = ft_tile<FMT, EPI>(a, t, nt, tiles_n, tiles_m);
            if (!tl.live) continue;
            const FtItem it = a.items[tl.b];
            pk::u64 acc[EXT ? 1 : PARTS * 4];        // pairs of columns (FT_TF32, FT_BF16)
            float h[EXT ? PARTS * 8 : 1], l[EXT ? PARTS * 8 : 1];
            if constexpr (EXT) {
#pragma unroll
                for (int j = 0; j < PARTS * 8; ++j) { h[j] = 0.f; l[j] = 0.f; }
            } else {
#pragma unroll
                for (int j = 0; j < PARTS * 4; ++j) acc[j] = 0ull;
            }
            const int row = tl.m0 + q * 32 + lane, qc = row / a.R, i = row - qc * a.R;
            const int qq = qc >> 1, cc = qc & 1, n_first = tl.n0 + cg * cols;
            constexpr bool BASE = EPI == FT_BABINET || EPI == FT_DIFF;
            const size_t bpair = (size_t)4 * a.base_R * 2 * a.base_ld;
            const E* bp = nullptr;                   // base at row i (clamped), column 0
            if (BASE && qc < 4)
                bp = reinterpret_cast<const E*>(a.base) + tl.b * a.base_bstride + (size_t)qq * PAIRS * bpair +
                     (size_t)(tl.p * 2 + cc) * a.base_R * 2 * a.base_ld + slot<FMT>(min(i, a.base_H - 1));
            if constexpr (BASE) {
                // its lines into L2 while the products run: the epilogue's loads are a serial part of the
                // tile (168-item Babinet: 3.3 ms without, 1.7 with). A warp's 32 rows of one column are one or two lines of each
                // plane: lane j asks for those of column j by the first and last rows' addresses
                const unsigned long long own = (unsigned long long)bp;
                const E* ends[2] = {(const E*)__shfl_sync(0xffffffffu, own, 0), (const E*)__shfl_sync(0xffffffffu, own, 31)};
                for (int j = lane; j < cols; j += 32) {
                    const size_t at = (size_t)min(n_first + j, a.base_H - 1) * 2 * a.base_ld;
#pragma unroll
                    for (int e = 0; e < 2; ++e)
                        if (ends[e])
#pragma unroll
                            for (int pr = 0; pr < PAIRS; ++pr) asm volatile("prefetch.global.L2 [%0];" ::"l"(ends[e] + pr * bpair + at));
                }
            }
            const int drains = (tl.slices + Cfg::CHUNK - 1) / Cfg::CHUNK;
            for (int c = 0; c < drains; ++c, ++g) {
                const uint32_t buf = g & 1;
                if (!ok || !(ok = tc::mbar_wait(&tfull[buf], (g >> 1) & 1, a.err, 23))) break;
                __syncwarp();
                tc::tc_fence_after();
                const uint32_t from = lane_base + buf * BUF;
                // two loads in flight before each wait (16 registers)
#pragma unroll
                for (int part = 0; part < PARTS; part += EXT ? 1 : 2) {
                    if (part < np) {
                        uint32_t r0[8], r1[8];
                        tc::tmem_ld8(from + part * 8, r0);
                        if constexpr (EXT) tc::tmem_ld8(from + 128 + part * 8, r1);
                        else if (part + 1 < np) tc::tmem_ld8(from + part * 8 + 8, r1);
                        tc::tmem_ld_wait();
                        if (part + (EXT ? 1 : 2) >= np) {                // the buffer is drained
                            tc::tc_fence_before();
                            __syncwarp();
                            if (lane == 0) tc::mbar_arrive(&tempty[buf]);
                        }
                        if constexpr (EXT) {
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                float s, e;
                                two_sum(h[part * 8 + j], __uint_as_float(r0[j]), s, e);
                                h[part * 8 + j] = s;
                                l[part * 8 + j] += e + __uint_as_float(r1[j]);
                            }
                        } else {
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                acc[part * 4 + j] = pk::add2(acc[part * 4 + j], pk::pack(__uint_as_float(r0[2 * j]), __uint_as_float(r0[2 * j + 1])));
                            if (part + 1 < np) {
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    acc[part * 4 + 4 + j] = pk::add2(acc[part * 4 + 4 + j], pk::pack(__uint_as_float(r1[2 * j]), __uint_as_float(r1[2 * j + 1])));
                            }
                        }
                    }
                }
            }
            // ---------------------------------------------------------------- epilogue
            const int ncols = min(cols, it.N - n_first);         // valid columns of this warp (uniform)
            const bool rows_in = ok && qc < 4 && i < it.H;
            const bool rows_out = ok && qc < 4 && i < a.dst_ld;      // the padding gets zeros: whole sectors
            const float sh = (float)it.scale, sl = EXT ? (float)(it.scale - (double)sh) : 0.f;
            // n^2 <= lim: valid row, and inside the disk where there is a mask (FT_DIFF: none)
            const int lim = !rows_in ? -1 : EPI == FT_DIFF ? 0x7fffffff : it.thr_out - i * i;
            if constexpr (EPI == FT_FLOAT) {
                if (rows_out) {
                    using F = typename std::conditional<EXT, float2, float>::type;
                    F* d = reinterpret_cast<F*>(a.dst) + tl.b * a.dst_bstride + ((size_t)(qq * 4 + tl.p * 2 + cc) * a.dst_R + n_first) * a.dst_ld + i;
#pragma unroll
                    for (int j = 0; j < PARTS * 8; ++j, d += a.dst_ld) {
                        if (j >= ncols) break;
                        if constexpr (EXT) *d = make_float2(h[j], l[j]);
                        else *d = pk_half(acc[j / 2], j & 1);
                    }
                }
            } else {
                constexpr bool DIFF = EPI == FT_DIFF;
                const size_t pair = (size_t)4 * a.dst_R * 2 * a.dst_ld;
                const size_t d_row = DIFF ? (size_t)a.dst_ld : (size_t)2 * a.dst_ld;
                E* d = nullptr;
                float* df = nullptr;
                if constexpr (DIFF)
                    df = reinterpret_cast<float*>(a.dst) + tl.b * a.dst_bstride + ((size_t)(qq * 4 + tl.p * 2 + cc) * a.dst_R + n_first) * a.dst_ld + i;
                else
                    d = reinterpret_cast<E*>(a.dst) + tl.b * a.dst_bstride + (size_t)qq * PAIRS * pair +
                        ((size_t)(tl.p * 2 + cc) * a.dst_R + n_first) * 2 * a.dst_ld + slot<FMT>(i);
                // w scale at n > 0, and half of it at n = 0 (w = 1: both the same)
                const float wi = a.weights && !DIFF ? (i ? 4.f : 2.f) : 1.f, w0 = a.weights && !DIFF ? 0.5f * wi : wi;
                const bool scaled = it.scale != 1.0 || (a.weights && !DIFF);
                const float ip = EPI == FT_SEED ? (float)it.inv_peak : 1.f;
                const float ipl = EPI == FT_SEED && EXT ? (float)(it.inv_peak - (double)ip) : 0.f;
                const int low = EPI == FT_SEED ? it.lo_out - i * i : 0;
                const bool based = BASE && bp && i < a.base_H;
                constexpr int AHEAD = 4;       // columns of the base loaded together
                float bh8[AHEAD], bl8[EXT ? AHEAD : 1];
                float dsh = 0.f, dsl = 0.f;              // FT_SEED: dark-hole sum
#pragma unroll
                for (int j = 0; j < PARTS * 8; ++j) {
                    if (j >= ncols) {
                        if constexpr (EXT) h[j] = 0.f;
                        continue;
                    }
                    const int n = n_first + j;
                    // the base of several columns at a time, all loads in flight together (clamped to its
                    // extent; values beyond are dropped)
                    if (BASE && j % AHEAD == 0 && bp) {
#pragma unroll
                        for (int e = 0; e < AHEAD; ++e) {
                            float low = 0.f;
                            get<FMT>(bp + (size_t)min(n + e, a.base_H - 1) * 2 * a.base_ld, bpair, bh8[e], low);
                            if constexpr (EXT) bl8[e] = low;
                        }
                    }
                    const bool keep = n * n <= lim && (EPI != FT_SEED || n * n >= low);
                    const float w = n ? wi : w0;
                    float vh, vl = 0.f;
                    if constexpr (EXT) {
                        // both normalise the pair, which the slices need
                        if (scaled) mul22(h[j], l[j], sh * w, sl * w, vh, vl);
                        else two_sum(h[j], l[j], vh, vl);
                    } else {
                        vh = pk_half(acc[j / 2], j & 1) * (sh * w);
                    }
                    if constexpr (EPI == FT_SEED) {
                        // w T'^2 / peak with T' = scale Y; vh, vl = w T'
                        const float yh = vh, yl = vl;
                        if constexpr (EXT) mul22(vh, vl, ip, ipl, vh, vl);
                        else vh *= ip;
                        if (keep) {
                            const float iw = (i ? 0.5f : 1.f) * (n ? 0.5f : 1.f);
                            float th, tl = 0.f;
                            if constexpr (EXT) mul22(vh, vl, yh, yl, th, tl);
                            else th = vh * yh;
                            add22(dsh, dsl, th * iw, tl * iw);
                        }
                    }
                    if constexpr (BASE) {
                        float bh = 0.f, bl = 0.f;
                        if (based && n < a.base_H) {
                            const float iw = DIFF ? (i ? 0.5f : 1.f) * (n ? 0.5f : 1.f) : 1.f;
                            bh = bh8[j % AHEAD] * iw;
                            if constexpr (EXT) bl = bl8[j % AHEAD] * iw;
                        }
                        if constexpr (EXT) {
                            float s, e;
                            two_sum(bh, -vh, s, e);
                            vl = e + (bl - vl);
                            vh = s;
                        } else {
                            vh = bh - vh;
                        }
                    }
                    if (!keep) { vh = 0.f; vl = 0.f; }
                    if constexpr (DIFF) {
                        if (rows_out) df[j * d_row] = vh + vl;
                    } else if constexpr (EXT) {
                        h[j] = vh;
                        l[j] = vl;
                    } else if (rows_out) {
                        put<FMT>(d + j * d_row, pair, vh);
                    }
                }
                if constexpr (EPI == FT_SEED) {
                    double dh = sum22(dsh, dsl);
                    for (int o = 16; o > 0; o >>= 1) dh += __shfl_down_sync(0xffffffffu, dh, o);
                    if (lane == 0 && dh != 0.0 && a.dh_acc) atomicAdd(a.dh_acc + tl.b, dh);
                }
                if constexpr (EXT && !DIFF) {
                    // the scaling group of a value is 64 consecutive i of its (q, c): the rows of
                    // this warp and of its partner (quarters 2h and 2h + 1, same column group)
                    const int ew = warp - 2, partner = 4 * cg + (((q ^ 1) + 2) & 3), bar = 1 + cg * 2 + (q >> 1);
#pragma unroll
                    for (int j = 0; j < PARTS * 8; ++j) {
                        if (j >= cols) break;
                        const uint32_t m = warp_max_bits(fabsf(h[j]));
                        if (lane == 0) xmax[ew * PARTS * 8 + j] = m;
                    }
                    asm volatile("bar.sync %0, 64;" ::"r"(bar) : "memory");
                    if (rows_out) {
#pragma unroll
                        for (int j = 0; j < PARTS * 8; ++j) {
                            if (j >= ncols) break;
                            put4(d + j * d_row, pair, h[j], l[j], group_exp_of(max(xmax[ew * PARTS * 8 + j], xmax[partner * PARTS * 8 + j])));
                        }
                    }
                    // both have read the maxima before either writes the next tile's
                    asm volatile("bar.sync %0, 64;" ::"r"(bar) : "memory");
                }
            }
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tbase, Cfg::TMEM_COLS);
    }
}

// ------------------------------------------------------------------ producers

// Exponents of V values over the 64-element groups of two consecutive warps (blocks of 128).
template <int V>
__device__ __forceinline__ void group_exps(const float (&v)[V], int (&e)[V], uint32_t (*sh)[4]) {
    const int w = threadIdx.x >> 5;
#pragma unroll
    for (int j = 0; j < V; ++j) {
        const uint32_t m = warp_max_bits(fabsf(v[j]));
        if ((threadIdx.x & 31) == 0) sh[j][w] = m;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < V; ++j) e[j] = group_exp_of(max(sh[j][w & ~1], sh[j][w | 1]));
}

template <int FMT>
__global__ void __launch_bounds__(128)
ft_fold_kernel(const float2* __restrict__ src, long long sb, int sld, int n, int h, int keep_r2,
               typename FtElem<FMT>::type* dst, int R, int ld, long long stride) {
    constexpr bool EXT = FMT == FT_EXT;
    __shared__ uint32_t sh[EXT ? 8 : 1][4];
    const int kx = blockIdx.x * 128 + threadIdx.x, ky = blockIdx.y, b = blockIdx.z, hn = n / 2;
    float2 f[4] = {};                                // samples at (+-ky, +-kx): pp, pm, mp, mm
    if (kx < h && (keep_r2 < 0 || kx * kx + ky * ky <= keep_r2)) {
        const float2* s = src + b * sb;
        const bool py = hn + ky < n, px = hn + kx < n;
        if (py && px) f[0] = s[(size_t)(hn + ky) * sld + hn + kx];
        if (py && kx) f[1] = s[(size_t)(hn + ky) * sld + hn - kx];
        if (ky && px) f[2] = s[(size_t)(hn - ky) * sld + hn + kx];
        if (ky && kx) f[3] = s[(size_t)(hn - ky) * sld + hn - kx];
    }
    // class (px, py), component c at v[px * 4 + py * 2 + c]
    float v[8], lo[8] = {};
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const float pp = c ? f[0].y : f[0].x, pm = c ? f[1].y : f[1].x, mp = c ? f[2].y : f[2].x, mm = c ? f[3].y : f[3].x;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int px = k >> 1, py = k & 1, at = px * 4 + py * 2 + c;
            const float sx = px ? -1.f : 1.f, sy = py ? -1.f : 1.f;
            if constexpr (EXT) {
                float s0, e0, s1, e1, s, e;
                two_sum(pp, sx * pm, s0, e0);
                two_sum(mp, sx * mm, s1, e1);
                two_sum(s0, sy * s1, s, e);
                v[at] = s;
                lo[at] = e + (e0 + sy * e1);
            } else {
                v[at] = (pp + sx * pm) + sy * (mp + sx * mm);
            }
            if ((px && kx == 0) || (py && ky == 0)) { v[at] = 0.f; lo[at] = 0.f; }
        }
    }
    int ge[8];
    if constexpr (EXT) group_exps(v, ge, sh);
    if (kx >= ld) return;                            // h ... ld - 1: zeros
    const size_t pair = (size_t)4 * R * 2 * ld;
#pragma unroll
    for (int at = 0; at < 8; ++at) {
        typename FtElem<FMT>::type* d = dst + b * stride + (size_t)(at >> 2) * FtCfg<FMT>::PAIRS * pair +
                                        (size_t)((at & 3) * R + ky) * 2 * ld + slot<FMT>(kx);
        if constexpr (EXT) put4(d, pair, v[at], lo[at], ge[at]);
        else put<FMT>(d, pair, v[at]);
    }
}

template <int FMT>
__global__ void __launch_bounds__(128)
ft_basis_kernel(double c, const FtItem* __restrict__ items, int K, typename FtElem<FMT>::type* w, long long stride, int R, int ld) {
    constexpr bool EXT = FMT == FT_EXT;
    __shared__ uint32_t sh[EXT ? 2 : 1][4];
    const int k = blockIdx.x * 128 + threadIdx.x, n = blockIdx.y;
    if (items) c = items[blockIdx.z].scale;
    w += blockIdx.z * stride;
    double s = 0.0, co = 0.0;
    if (k < K) {
        double cyc = (double)((long long)k * n) * c;
        cyc -= rint(cyc);
        sincospi(2.0 * cyc, &s, &co);
    }
    const float v[2] = {(float)co, (float)s};
    int ge[2];
    if constexpr (EXT) group_exps(v, ge, sh);
    if (k >= ld) return;
    const size_t pair = (size_t)R * 2 * ld;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        typename FtElem<FMT>::type* d = w + (size_t)p * FtCfg<FMT>::PAIRS * pair + (size_t)n * 2 * ld + slot<FMT>(k);
        if constexpr (EXT) put4(d, pair, v[p], (float)((p ? s : co) - (double)v[p]), ge[p]);
        else put<FMT>(d, pair, v[p]);
    }
}

// ------------------------------------------------------------------ back to planes

// One thread per |u| and PLANE_ROWS |v|: eight class values in, four pixels out. (One row per block spent
// its time in the blocks' ends: 168 images of 512^2 0.31 ms, with eight 0.23.)
constexpr int PLANE_ROWS = 8, PLANE_MAX = 320;

inline int plane_threads(int h) {                    // blocks along u all alike, whole warps
    const int blocks = (h + PLANE_MAX - 1) / PLANE_MAX;
    return ((h + blocks - 1) / blocks + 31) / 32 * 32;
}

template <bool EXT>
__global__ void __launch_bounds__(PLANE_MAX) ft_plane_kernel(const FtPlane p) {
    const int hm = p.m / 2, b = blockIdx.z, u = blockIdx.x * blockDim.x + threadIdx.x;
    const FtItem it = p.items[b];
    const float sh = (float)it.scale, sl = EXT ? (float)(it.scale - (double)sh) : 0.f;
    const float ph = (float)it.inv_peak, pl = EXT ? (float)(it.inv_peak - (double)ph) : 0.f;
    float dsh = 0.f, dsl = 0.f;
    // the largest value as two floats, FP64 after the loop (in it, even predicated off, it held the FP64
    // pipe: 61^2 -> 1099^2 of six fields at 3xBF16, where this kernel takes two fifths: 90 us, like this 77)
    float toph = 0.f, topl = 0.f;
    const int v_end = min((int)(blockIdx.y + 1) * PLANE_ROWS, hm + 1);
    for (int v = blockIdx.y * PLANE_ROWS; u <= hm && v < v_end; ++v) {
        float th[8], tl[8] = {};                     // class (px, py), component c at px * 4 + py * 2 + c
        const size_t cls = (size_t)p.R * p.ld, at = b * p.bstride + (size_t)v * p.ld + u;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if constexpr (EXT) {
                const float2 t = reinterpret_cast<const float2*>(p.T)[at + k * cls];
                th[k] = t.x;
                tl[k] = t.y;
            } else {
                th[k] = reinterpret_cast<const float*>(p.T)[at + k * cls];
            }
        }
        const float sg = p.sign < 0 ? -1.f : 1.f;
        const int r2 = u * u + v * v;
        // The dark-hole sum over the four signs is that of the classes alone, w_u w_v |T|^2 (their cross
        // terms cancel), summed as the seed's contraction does.
        if (p.dh && r2 >= it.lo_out && r2 <= it.thr_out) {
            const float w = (u ? 2.f : 1.f) * (v ? 2.f : 1.f), iw = w == 1.f ? 1.f : w == 2.f ? 0.5f : 0.25f;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                float yh = th[k], yl = tl[k], vh, vl = 0.f;
                if constexpr (EXT) {
                    mul22(yh, yl, sh * w, sl * w, yh, yl);
                    mul22(yh, yl, ph, pl, vh, vl);
                } else {
                    yh *= sh * w;
                    vh = yh * ph;
                }
                float sum, low = 0.f;
                if constexpr (EXT) mul22(vh, vl, yh, yl, sum, low);
                else sum = vh * yh;
                add22(dsh, dsl, sum * iw, low * iw);
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {                // signs: bit 0 of u, bit 1 of v
            const bool nu = k & 1, nv = k & 2;
            if ((nu && u == 0) || (nv && v == 0)) continue;
            if ((!nu && hm + u >= p.m) || (!nv && hm + v >= p.m)) continue;
            const float su = nu ? -sg : sg, sv = nv ? -sg : sg;
            // F = T00 + i (su T10 + sv T01) - su sv T11 (first index: parity in x), sg^2 = 1
            float rh = th[0], rl = tl[0], ih = th[1], il = tl[1];
            const float suv = su * sv;
            if constexpr (EXT) {
                add22(rh, rl, -su * th[5], -su * tl[5]);
                add22(rh, rl, -sv * th[3], -sv * tl[3]);
                add22(rh, rl, -suv * th[6], -suv * tl[6]);
                add22(ih, il, su * th[4], su * tl[4]);
                add22(ih, il, sv * th[2], sv * tl[2]);
                add22(ih, il, -suv * th[7], -suv * tl[7]);
                mul22(rh, rl, sh, sl, rh, rl);
                mul22(ih, il, sh, sl, ih, il);
            } else {
                rh = ((rh - suv * th[6]) - (su * th[5] + sv * th[3])) * sh;
                ih = ((ih - suv * th[7]) + (su * th[4] + sv * th[2])) * sh;
            }
            const size_t o = (size_t)b * p.m * p.m + (size_t)(nv ? hm - v : hm + v) * p.m + (nu ? hm - u : hm + u);
            if (p.field) p.field[o] = make_float2(rh + rl, ih + il);
            if constexpr (EXT) {
                // |v|^2 = re^2 + im^2 in two-float, times 1 / peak
                const float q0 = rh * rh, q1 = ih * ih, e0 = fmaf(rh, rh, -q0), e1 = fmaf(ih, ih, -q1);
                float nh, nl;
                two_sum(q0, q1, nh, nl);
                nl += e0 + e1 + 2.f * (rh * rl + ih * il);
                mul22(nh, nl, ph, pl, nh, nl);
                if (p.image) p.image[o] = nh + nl;
                if (p.peak64 && nl == nl && (nh > toph || (nh == toph && nl > topl))) { toph = nh; topl = nl; }
            } else {
                const float inten = (rh * rh + ih * ih) * ph;
                if (p.image) p.image[o] = inten;
                if (p.peak) toph = fmaxf(toph, inten);
            }
        }
    }
    if (!p.dh && !p.peak && !p.peak64) return;       // uniform
    double dh = 0.0;                                 // warps without a dark-hole pixel skip the FP64 sum
    if (__any_sync(0xffffffffu, dsh != 0.f || dsl != 0.f)) {
        dh = sum22(dsh, dsl);
        for (int o = 16; o > 0; o >>= 1) dh += __shfl_down_sync(0xffffffffu, dh, o);
    }
    double top = 0.0;
    if (p.peak || p.peak64) {
        top = (double)toph + (double)topl;
        for (int o = 16; o > 0; o >>= 1) top = fmax(top, __shfl_down_sync(0xffffffffu, top, o));
    }
    __shared__ double sd[PLANE_MAX / 32], st[PLANE_MAX / 32];
    __shared__ bool last;
    const int warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    auto total = [&]() {
        double s = 0.0;
        for (int w = 0; w < warps; ++w) s += sd[w];
        return s;
    };
    if ((threadIdx.x & 31) == 0) { sd[warp] = dh; st[warp] = top; }
    __syncthreads();
    const int blocks = gridDim.x * gridDim.y;
    double* part = p.dh_part + (size_t)b * blocks;
    if (threadIdx.x == 0) {
        for (int w = 0; w < warps; ++w) top = fmax(top, st[w]);
        // non-negative values order like their bit patterns
        if (p.peak) atomicMax(reinterpret_cast<int*>(p.peak) + b, __float_as_int((float)top));
        if (p.peak64) atomicMax(reinterpret_cast<unsigned long long*>(p.peak64) + b, (unsigned long long)__double_as_longlong(top));
        if (p.dh) {
            part[blockIdx.y * gridDim.x + blockIdx.x] = total();
            __threadfence();
            last = atomicAdd(p.dh_count + b, 1u) == (unsigned)blocks - 1;
        }
    }
    if (!p.dh) return;
    __syncthreads();
    if (!last) return;
    // the item's last block adds the partial sums in their order: every run gives the same bits
    __threadfence();
    dh = 0.0;
    for (int i = threadIdx.x; i < blocks; i += blockDim.x) dh += part[i];
    for (int o = 16; o > 0; o >>= 1) dh += __shfl_down_sync(0xffffffffu, dh, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sd[warp] = dh;
    __syncthreads();
    if (threadIdx.x == 0) {
        p.dh[b] = total();
        p.dh_count[b] = 0;                           // ready for the next launch
    }
}

__global__ void __launch_bounds__(128)
ft_unfold_kernel(const float* __restrict__ T, int R, int ld, long long bstride, int n, float2* __restrict__ dst, int dld,
                 long long db) {
    const int hn = n / 2, b = blockIdx.z, ky = blockIdx.y, kx = blockIdx.x * 128 + threadIdx.x;
    if (kx > hn) return;
    const size_t cls = (size_t)R * ld;
    const float* t = T + b * bstride + (size_t)ky * ld + kx;
    const float2 t00 = make_float2(t[0], t[cls]), t01 = make_float2(t[2 * cls], t[3 * cls]);
    const float2 t10 = make_float2(t[4 * cls], t[5 * cls]), t11 = make_float2(t[6 * cls], t[7 * cls]);   // (px, py)
    float2* o = dst + b * db;
    auto put = [&](int y, int x, float sx, float sy) {
        o[(size_t)y * dld + x] = make_float2((t00.x + sx * t10.x) + sy * (t01.x + sx * t11.x),
                                             (t00.y + sx * t10.y) + sy * (t01.y + sx * t11.y));
    };
    const bool px = hn + kx < n, py = hn + ky < n;
    if (px && py) put(hn + ky, hn + kx, 1.f, 1.f);
    if (kx && py) put(hn + ky, hn - kx, -1.f, 1.f);
    if (px && ky) put(hn - ky, hn + kx, 1.f, -1.f);
    if (kx && ky) put(hn - ky, hn - kx, -1.f, -1.f);
}

// ------------------------------------------------------------------ host side

cudaError_t make_map(int fmt, const void* base, int ld, int rows, int pairs, int items, int box_rows, int box_pairs,
                     CUtensorMap* map) {
    auto fn = tensor_map_encoder();
    if (!fn) return cudaErrorNotSupported;
    const cuuint64_t es = ft_elem(fmt), row = 2 * ld * es;
    if (((uintptr_t)base & 15) || row % 128) return cudaErrorInvalidValue;
    cuuint64_t dims[4] = {(cuuint64_t)2 * ld, (cuuint64_t)rows, (cuuint64_t)pairs, (cuuint64_t)items};
    cuuint64_t strides[3] = {row, rows * row, pairs * rows * row};
    cuuint32_t box[4] = {(cuuint32_t)(128 / es), (cuuint32_t)box_rows, (cuuint32_t)box_pairs, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = fn(map, fmt == FT_TF32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4,
                    const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

int device_sms() {
    static int sms[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
    if (sms[dev] == 0) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1) return 148;
        sms[dev] = v;
    }
    return sms[dev];
}

template <int FMT, int EPI>
cudaError_t launch_t(const FtGemm& g, const FtArgs& a, cudaStream_t stream) {
    using Cfg = FtCfg<FMT>;
    static unsigned long long attr_done = 0;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(attr_done & bit)) {
        e = cudaFuncSetAttribute(ft_gemm_kernel<FMT, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM_BUDGET + 1024);
        if (e != cudaSuccess) return e;
        attr_done |= bit;
    }
    const int smem = g.stages * Cfg::PAIRS * (XPAIR_BYTES + g.nt * 128) + 1024;
    // PER_SM blocks share an SM (and its 512 tensor-memory columns); the occupancy query counts one
    // for any kernel that allocates tensor memory, but they do run side by side
    const int total = 2 * g.tiles_n * g.tiles_m * g.items, slots = device_sms() * Cfg::PER_SM;
    ft_gemm_kernel<FMT, EPI><<<std::min(total, slots), Cfg::THREADS, smem, stream>>>(g.mx, g.mw, a, g.nt, g.tiles_n, g.tiles_m,
                                                                                   g.items, g.stages);
    return cudaGetLastError();
}

template <int FMT>
cudaError_t launch_f(const FtGemm& g, int epi, const FtArgs& a, cudaStream_t s) {
    switch (epi) {
        case FT_SPLIT: return launch_t<FMT, FT_SPLIT>(g, a, s);
        case FT_BABINET: return launch_t<FMT, FT_BABINET>(g, a, s);
        case FT_FLOAT: return launch_t<FMT, FT_FLOAT>(g, a, s);
        case FT_DIFF: return launch_t<FMT, FT_DIFF>(g, a, s);
        case FT_SEED: return launch_t<FMT, FT_SEED>(g, a, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

FtOperand ft_operand(int fmt, int items, int rows, int cols) {
    FtOperand o;
    o.items = items;
    o.R = ft_pitch(fmt, rows);
    o.cols = cols;
    o.ld = ft_pitch(fmt, cols);
    o.stride = (long long)2 * ft_pairs(fmt) * 4 * o.R * 2 * o.ld;
    return o;
}

FtOperand ft_basis_operand(int fmt, int bases, int rows, int cols) {
    FtOperand o;
    o.items = bases;
    o.R = rows;
    o.cols = cols;
    o.ld = ft_pitch(fmt, cols);
    o.stride = (long long)2 * ft_pairs(fmt) * o.R * 2 * o.ld;
    return o;
}

// Tile width: the columns in as few tiles as `max_nt` allows, all alike (101 -> 112, 257 -> 3 x 96,
// 410 -> 4 x 112), a multiple of the epilogue's column groups; narrower, down to 32, while there are
// fewer tiles than resident blocks.
cudaError_t ft_make(int fmt, const FtOperand& x, const FtOperand& w, int items, int max_n, int max_nt, FtGemm* g) {
    const int slots = device_sms() * (fmt == FT_TF32 ? 2 : 1), P = ft_pairs(fmt), unit = fmt == FT_TF32 ? 16 : 32;
    g->fmt = fmt;
    g->items = items;
    g->tiles_m = (4 * x.R + BM - 1) / BM;
    auto width = [&](int tiles) { return (((max_n + tiles - 1) / tiles) + unit - 1) / unit * unit; };
    int tiles = (max_n + max_nt - 1) / max_nt;
    while (width(tiles) > 32 && 2LL * g->tiles_m * tiles * items < slots) ++tiles;
    g->nt = width(tiles);
    g->tiles_n = (max_n + g->nt - 1) / g->nt;
    if (2LL * g->tiles_m * g->tiles_n * items > 0x7fffffffLL) return cudaErrorInvalidValue;
    const int stage = P * (XPAIR_BYTES + g->nt * 128);
    const int budget = fmt == FT_TF32 ? FtCfg<FT_TF32>::SMEM_BUDGET : FtCfg<FT_EXT>::SMEM_BUDGET;   // FT_BF16 alike
    g->stages = std::min(MAX_STAGES, budget / stage);
    cudaError_t e = make_map(fmt, x.base, x.ld, 4 * x.R, 2 * P, x.items, BM, P, &g->mx);
    if (e == cudaSuccess) e = make_map(fmt, w.base, w.ld, w.R, 2 * P, w.items, g->nt, P, &g->mw);
    return e;
}

cudaError_t ft_launch(const FtGemm& g, int epi, const FtArgs& a, cudaStream_t stream) {
    switch (g.fmt) {
        case FT_TF32: return launch_f<FT_TF32>(g, epi, a, stream);
        case FT_BF16: return launch_f<FT_BF16>(g, epi, a, stream);
        case FT_EXT: return launch_f<FT_EXT>(g, epi, a, stream);
    }
    return cudaErrorInvalidValue;
}

void ft_count_flops(const FtGemm& g, int epi, const FtItem* items, int R, double* useful, double* issued) {
    const int ke = g.fmt == FT_TF32 ? 16 : 32, products = ft_planes(g.fmt) * (ft_planes(g.fmt) + 1) / 2;
    const bool masked = epi == FT_SPLIT || epi == FT_BABINET || epi == FT_SEED;
    for (int b = 0; b < g.items; ++b) {
        const FtItem& it = items[b];
        for (int tm = 0; tm < g.tiles_m; ++tm)
            for (int n0 = 0; n0 < it.N; n0 += g.nt) {
                const int sl = ft_slices(it, R, tm * BM, n0, ke, masked);
                *issued += 2.0 * 2.0 * products * BM * g.nt * (double)sl * ke;
                if (!sl) continue;
                int rows = 0;
                for (int r = tm * BM; r < tm * BM + BM && r < 4 * R; ++r) rows += r % R < it.H;
                *useful += 2.0 * 2.0 * products * rows * std::min(g.nt, it.N - n0) * (double)std::min(it.K, sl * ke);
            }
    }
}

cudaError_t ft_fold(int fmt, const float2* src, long long sb, int sld, int n, int h, int keep_r2, const FtOperand& d,
                    cudaStream_t stream) {
    const dim3 grid((d.ld + 127) / 128, h, d.items);
    if (fmt == FT_TF32) ft_fold_kernel<FT_TF32><<<grid, 128, 0, stream>>>(src, sb, sld, n, h, keep_r2, (float*)d.base, d.R, d.ld, d.stride);
    else if (fmt == FT_BF16) ft_fold_kernel<FT_BF16><<<grid, 128, 0, stream>>>(src, sb, sld, n, h, keep_r2, (__nv_bfloat16*)d.base, d.R, d.ld, d.stride);
    else ft_fold_kernel<FT_EXT><<<grid, 128, 0, stream>>>(src, sb, sld, n, h, keep_r2, (__nv_bfloat16*)d.base, d.R, d.ld, d.stride);
    return cudaGetLastError();
}

static cudaError_t basis_launch(int fmt, double c, const FtItem* items, int K, int N, const FtOperand& w, int first, int count,
                                cudaStream_t stream) {
    if (K > w.ld || N > w.R || first < 0 || first + count > w.items) return cudaErrorInvalidValue;
    const dim3 grid((w.ld + 127) / 128, N, count);
    const size_t at = (size_t)first * w.stride;
    if (fmt == FT_TF32) ft_basis_kernel<FT_TF32><<<grid, 128, 0, stream>>>(c, items, K, (float*)w.base + at, w.stride, w.R, w.ld);
    else if (fmt == FT_BF16) ft_basis_kernel<FT_BF16><<<grid, 128, 0, stream>>>(c, items, K, (__nv_bfloat16*)w.base + at, w.stride, w.R, w.ld);
    else ft_basis_kernel<FT_EXT><<<grid, 128, 0, stream>>>(c, items, K, (__nv_bfloat16*)w.base + at, w.stride, w.R, w.ld);
    return cudaGetLastError();
}

cudaError_t ft_basis(int fmt, double c, int K, int N, const FtOperand& w, int index, cudaStream_t stream) {
    return basis_launch(fmt, c, nullptr, K, N, w, index, 1, stream);
}

cudaError_t ft_bases(int fmt, const FtItem* items, int K, int N, const FtOperand& w, cudaStream_t stream) {
    return basis_launch(fmt, 0.0, items, K, N, w, 0, w.items, stream);
}

size_t ft_plane_parts(int m) {
    const int h = m / 2 + 1;
    return (size_t)((h + PLANE_MAX - 1) / PLANE_MAX) * ((h + PLANE_ROWS - 1) / PLANE_ROWS);
}

cudaError_t ft_plane(const FtPlane& p, int items, cudaStream_t stream) {
    const int h = p.m / 2 + 1, threads = plane_threads(h);
    const dim3 grid((h + threads - 1) / threads, (h + PLANE_ROWS - 1) / PLANE_ROWS, items);
    if (p.ext) ft_plane_kernel<true><<<grid, threads, 0, stream>>>(p);
    else ft_plane_kernel<false><<<grid, threads, 0, stream>>>(p);
    return cudaGetLastError();
}

cudaError_t ft_unfold(const float* T, int R, int ld, long long bstride, int n, int items, float2* dst, int dst_ld,
                      long long dst_bstride, cudaStream_t stream) {
    const int h = n / 2 + 1;
    ft_unfold_kernel<<<dim3((h + 127) / 128, h, items), 128, 0, stream>>>(T, R, ld, bstride, n, dst, dst_ld, dst_bstride);
    return cudaGetLastError();
}

}  // namespace coro
