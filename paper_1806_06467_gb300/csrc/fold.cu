// fold.cu -- kernels of the folded matrix Fourier transform on the CUDA cores (fold.cuh): basis
// and fold, the real-basis contraction in FP32 and FP64, and the expansion to the full plane.
#include <cuda_runtime.h>

#include <algorithm>

#include "fft_engine.cuh"
#include "fft_pair.cuh"
#include "fold.cuh"

namespace coro {
namespace {

// Per-item constants travel in the launch (no upload); larger batches take several launches.
constexpr int kConsts = 64;
struct Consts {
    double v[kConsts];
};

constexpr int PREP_THREADS = 128;

// Blocks [0, basis_blocks) fill W (one thread a (k, n) pair: one FP64 sincospi serves both
// parities; a quarter of the pairs of the unfolded basis, which is what bounds small transforms at
// GB300's FP64 rate); the rest fold the field.
template <typename C>
__global__ void __launch_bounds__(PREP_THREADS)
fold_prepare_kernel(const C* __restrict__ in, int n, int h, long long keep_r2, C* __restrict__ F, Consts c, int K,
                    int N, int ldw, typename real_of<C>::type* __restrict__ W, int basis_blocks) {
    using R = typename real_of<C>::type;
    const int b = blockIdx.y;
    if ((int)blockIdx.x < basis_blocks) {
        const long long i = (long long)blockIdx.x * PREP_THREADS + threadIdx.x;
        const int k = (int)(i / ldw), u = (int)(i % ldw);
        if (k >= K) return;
        double s = 0.0, co = 0.0;
        if (u < N) {
            double cyc = (double)((long long)k * u) * c.v[b];
            cyc -= rint(cyc);
            sincospi(2.0 * cyc, &s, &co);
        }
        R* w = W + (size_t)b * 2 * K * ldw + (size_t)k * ldw + u;
        w[0] = (R)co;
        w[(size_t)K * ldw] = (R)s;
        return;
    }
    const long long i = (long long)(blockIdx.x - basis_blocks) * PREP_THREADS + threadIdx.x;
    const int ky = (int)(i / h), kx = (int)(i % h);
    if (ky >= h) return;
    const int hn = n / 2;
    const C z = mk<C>((R)0, (R)0);
    const C* f = in + (size_t)b * n * n;
    C pp = z, pm = z, mp = z, mm = z;                  // samples at (+-ky, +-kx)
    if (keep_r2 < 0 || (long long)ky * ky + (long long)kx * kx <= keep_r2) {
        const bool py = hn + ky < n, px = hn + kx < n;
        if (py && px) pp = f[(size_t)(hn + ky) * n + hn + kx];
        if (py && kx) pm = f[(size_t)(hn + ky) * n + hn - kx];
        if (ky && px) mp = f[(size_t)(hn - ky) * n + hn + kx];
        if (ky && kx) mm = f[(size_t)(hn - ky) * n + hn - kx];
    }
    const C se = cadd(pp, pm), de = csub(pp, pm);      // row +ky, even and odd in x
    const C so = cadd(mp, mm), dd = csub(mp, mm);      // row -ky
    C* o = F + (size_t)b * 4 * h * h + (size_t)ky * 2 * h + kx;
    const size_t odd_y = (size_t)h * 2 * h;
    o[0] = cadd(se, so);
    o[h] = kx ? cadd(de, dd) : z;
    o[odd_y] = ky ? csub(se, so) : z;
    o[odd_y + h] = ky && kx ? csub(de, dd) : z;
}

// What a contraction writes at row m = (pm, km), column (p, n).
template <typename C, typename R>
__device__ __forceinline__ C fold_out(const FoldGemm<C>& g, const C* base, C v, int m, int p, int n) {
    if (g.epi == FOLD_PLAIN) return v;
    const int H = g.M / 2, pm = m >= H, km = m - pm * H;
    if ((long long)km * km + (long long)n * n > g.thr) return mk<C>((R)0, (R)0);
    const R w = (km ? (R)2 : (R)1) * (n ? (R)2 : (R)1);
    if (g.epi == FOLD_MASK) return mk<C>(w * v.x, w * v.y);
    const C a = base[(((size_t)pm * g.base_h + km) * 2 + p) * g.base_h + n];
    const R s = w * g.scale;
    return mk<C>(a.x - s * v.x, a.y - s * v.y);
}

// ---------------------------------------------------------------------------- FP32
//
// 64 rows (of M) x 32 columns per block, K in slices of 16, each thread 4 x 4 complex outputs. One
// packed FMA is one complex x real multiply-add, so a k step is 16 packed FMAs against 3 shared
// 16-byte loads; the next slice's global loads are in flight while this one is multiplied. 32
// columns because half an occulter or camera field is some 100-250 wide: wider tiles pad more.
// Sums run over RUN terms and are then added to the total: with one running sum over all of
// K = 501 the 1000^2 to 301^2 transform is 4.4e-7 off its 64-bit value, like this 2.2e-7.
constexpr int BM = 64, BN = 32, BK = 16, GT = 128;
constexpr int RUN = 64;

__global__ void __launch_bounds__(GT) fold_cgemm_kernel(const FoldGemm<float2> g, int splits, int kc, float2* part) {
    __shared__ __align__(16) float2 Xs[2][BK][BM];
    __shared__ __align__(16) float Ws[2][BK][BN];
    const int zp = blockIdx.z / splits, sp = blockIdx.z % splits, b = zp >> 1, p = zp & 1;
    const int k_lo = sp * kc, k_hi = min(g.K, k_lo + kc);
    const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
    const float2* X = g.X + b * g.sX + (size_t)p * g.K * g.M;
    const float* W = g.W + b * g.sW + (size_t)p * g.K * g.ldw;
    const int t = threadIdx.x;
    // loads of a slice: rows of 32 float4 (64 samples) of X, 8 float4 of W; M is even, so a
    // float4 of two samples is inside or outside as a whole
    const int xc = t & 31, xr = t >> 5, wc = t & 7, wr = t >> 3;
    const bool xin = m0 + 2 * xc < g.M;
    float4 rx[4], rw;
    auto fetch = [&](int k0) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int k = k0 + xr + 4 * r;
            rx[r] = xin && k < k_hi ? *reinterpret_cast<const float4*>(X + (size_t)k * g.M + m0 + 2 * xc)
                                    : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const int k = k0 + wr;
        rw = k < k_hi ? *reinterpret_cast<const float4*>(W + (size_t)k * g.ldw + n0 + 4 * wc) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    auto stash = [&](int s) {
#pragma unroll
        for (int r = 0; r < 4; ++r) *reinterpret_cast<float4*>(&Xs[s][xr + 4 * r][2 * xc]) = rx[r];
        *reinterpret_cast<float4*>(&Ws[s][wr][4 * wc]) = rw;
    };
    const int tx = t & 15, ty = t >> 4;                // rows 2 tx + {0, 1, 32, 33}, columns 4 ty ...
    pk::u64 acc[4][4], sum[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { acc[i][j] = 0ull; sum[i][j] = 0ull; }
    fetch(k_lo);
    stash(0);
    __syncthreads();
    int s = 0;
    for (int k0 = k_lo; k0 < k_hi; k0 += BK, s ^= 1) {
        const bool more = k0 + BK < k_hi;
        if (more) fetch(k0 + BK);
#pragma unroll
        for (int k = 0; k < BK; ++k) {
            const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(&Xs[s][k][2 * tx]);
            const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(&Xs[s][k][32 + 2 * tx]);
            const float4 w = *reinterpret_cast<const float4*>(&Ws[s][k][4 * ty]);
            const pk::u64 a[4] = {a0.x, a0.y, a1.x, a1.y};
            const pk::u64 ww[4] = {pk::pack(w.x, w.x), pk::pack(w.y, w.y), pk::pack(w.z, w.z), pk::pack(w.w, w.w)};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = pk::fma2(a[i], ww[j], acc[i][j]);
        }
        if (more) stash(s ^ 1);
        if (!more || (k0 + BK - k_lo) % RUN == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    sum[i][j] = pk::add2(sum[i][j], acc[i][j]);
                    acc[i][j] = 0ull;
                }
        }
        __syncthreads();
    }
    const bool whole = splits == 1;
    float2* Y = whole ? g.Y + b * g.sY : part + ((size_t)sp * g.items + b) * (size_t)g.M * 2 * g.N;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + 2 * tx + (i & 1) + 32 * (i >> 1);
        if (m >= g.M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + 4 * ty + j;
            float2 v;
            pk::unpack(sum[i][j], v.x, v.y);
            if (n < g.N) Y[((size_t)m * 2 + p) * g.N + n] = v;
        }
    }
}

// ---------------------------------------------------------------------------- FP64
//
// The 1024^2 / 256^2 / 512^2 Lyot image takes 1.72 ms (11.48 ms with complex bases on the full
// planes); its widest contraction (820 x 257 x 410, both parities) runs at 0.9 of the FMA rate.
//
// GB300 issues two FP64 FMAs per SM and clock, so nothing but the number of multiply-adds and
// their even spread over the SMs counts: each warp takes 32 rows x NT columns straight from L1 / L2
// (a k step is 2 NT warp FMAs, 32 NT clocks, against one 512-byte row read), the four warps of a
// block take every fourth k and add up in shared memory in a fixed order. NT is 8, or 4 where 8
// would leave SMs without a block (launcher).
template <int NT>
__global__ void __launch_bounds__(128) fold_zgemm_kernel(const FoldGemm<double2> g) {
    __shared__ double2 red[3][NT][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.z >> 1, p = blockIdx.z & 1;
    const int m = blockIdx.x * 32 + lane, n0 = blockIdx.y * NT;
    // rows of this block nearest to the axis (0 where the two parities meet): known zeros of X end
    // its k range, and a block whose outputs the mask drops has nothing to sum
    const int H = g.M / 2, first = blockIdx.x * 32, last = min(first + 31, g.M - 1);
    const long long near = first < H && last >= H ? 0 : first >= H ? first - H : first;
    int K = g.K;
    if (g.thr_in >= 0) {
        const long long rem = g.thr_in - near * near;
        K = rem < 0 ? 0 : min(K, (int)sqrt((double)rem) + 2);
    }
    if (g.epi != FOLD_PLAIN && near * near + (long long)n0 * n0 > g.thr) K = 0;
    const double2* X = g.X + b * g.sX + (size_t)p * g.K * g.M + min(m, g.M - 1);
    const double* W = g.W + b * g.sW + (size_t)p * g.K * g.ldw + n0;
    double2 acc[NT];
#pragma unroll
    for (int j = 0; j < NT; ++j) acc[j] = make_double2(0.0, 0.0);
#pragma unroll 4
    for (int k = warp; k < K; k += 4) {
        const double2 x = __ldg(X + (size_t)k * g.M);
        const double2* w = reinterpret_cast<const double2*>(W + (size_t)k * g.ldw);
#pragma unroll
        for (int j = 0; j < NT / 2; ++j) {
            const double2 ww = __ldg(w + j);
            acc[2 * j].x = fma(x.x, ww.x, acc[2 * j].x);
            acc[2 * j].y = fma(x.y, ww.x, acc[2 * j].y);
            acc[2 * j + 1].x = fma(x.x, ww.y, acc[2 * j + 1].x);
            acc[2 * j + 1].y = fma(x.y, ww.y, acc[2 * j + 1].y);
        }
    }
    if (warp) {
#pragma unroll
        for (int j = 0; j < NT; ++j) red[warp - 1][j][lane] = acc[j];
    }
    __syncthreads();
    if (warp || m >= g.M) return;
    const double2* base = g.base;
    double2* Y = g.Y + b * g.sY + ((size_t)m * 2 + p) * g.N;
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        double2 v = acc[j];
        for (int q = 0; q < 3; ++q) { v.x += red[q][j][lane].x; v.y += red[q][j][lane].y; }
        if (n0 + j < g.N) Y[n0 + j] = fold_out<double2, double>(g, base, v, m, p, n0 + j);
    }
}

// Y = sum of the K splits in order.
__global__ void fold_reduce_kernel(const FoldGemm<float2> g, int splits, const float2* __restrict__ part) {
    const size_t per = (size_t)g.M * 2 * g.N, total = per * g.items;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        float2 v = part[i];
        for (int s = 1; s < splits; ++s) {
            const float2 q = part[(size_t)s * total + i];
            v.x += q.x;
            v.y += q.y;
        }
        const size_t b = i / per;
        g.Y[b * g.sY + (i - b * per)] = v;
    }
}

// out = scale * (T00 + su sigma i T01 + sv sigma i T10 - su sv T11) at the four signs.
template <typename C>
__global__ void fold_expand_kernel(const C* __restrict__ T, int m, int sign, Consts scale, C* __restrict__ out) {
    using R = typename real_of<C>::type;
    const int h = m / 2 + 1, hm = m / 2;
    const int u = blockIdx.x * blockDim.x + threadIdx.x, v = blockIdx.y, b = blockIdx.z;
    if (u >= h) return;
    const C* t = T + (size_t)b * 4 * h * h + (size_t)v * 2 * h + u;
    const size_t odd = (size_t)h * 2 * h;
    const R s = (R)scale.v[b], si = sign < 0 ? -s : s;
    C t00 = t[0], t01 = t[h], t10 = t[odd], t11 = t[odd + h];
    t00 = mk<C>(s * t00.x, s * t00.y);
    t11 = mk<C>(s * t11.x, s * t11.y);
    t01 = mk<C>(-si * t01.y, si * t01.x);              // sigma i T01
    t10 = mk<C>(-si * t10.y, si * t10.x);
    C* o = out + (size_t)b * m * m;
    const C e = csub(t00, t11), f = cadd(t00, t11), gsum = cadd(t01, t10), gdif = csub(t01, t10);
    const bool pv = hm + v < m, pu = hm + u < m;
    if (pv && pu) o[(size_t)(hm + v) * m + hm + u] = cadd(e, gsum);
    if (pv) o[(size_t)(hm + v) * m + hm - u] = csub(f, gdif);
    if (pu) o[(size_t)(hm - v) * m + hm + u] = cadd(f, gdif);
    o[(size_t)(hm - v) * m + hm - u] = csub(e, gsum);
}

int sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 148;
    return sms;
}

// K splits of the FP32 contraction: enough blocks for four on every SM (a block is one warp per
// scheduler), at least 64 of K each. 1000^2 to 301^2 with two per SM: 39 + 13 us for the two
// contractions and 4 us for the sums of splits; with four 25 + 14 and 10 us.
int fold_splits(int M, int N, int K, int items) {
    const long long tiles = (long long)((M + BM - 1) / BM) * ((N + BN - 1) / BN) * 2 * items;
    const long long want = 4LL * sm_count() / tiles;
    return (int)std::max(1LL, std::min<long long>(want, K / 64));
}

}  // namespace

size_t fold_part_elems(int M, int N, int K, int items) {
    const int s = fold_splits(M, N, K, items);
    return s > 1 ? (size_t)s * items * M * 2 * N : 0;
}

cudaError_t fold_gemm(const FoldGemm<float2>& g, float2* part, cudaStream_t stream) {
    if (g.epi != FOLD_PLAIN || g.items > 32767) return cudaErrorInvalidValue;
    int splits = fold_splits(g.M, g.N, g.K, g.items);
    if (!part || (long long)splits * 2 * g.items > 65535) splits = 1;
    const int kc = ((g.K + splits - 1) / splits + BK - 1) / BK * BK;
    splits = (g.K + kc - 1) / kc;
    dim3 grid((g.M + BM - 1) / BM, (g.N + BN - 1) / BN, 2 * g.items * splits);
    fold_cgemm_kernel<<<grid, GT, 0, stream>>>(g, splits, kc, part);
    if (splits > 1) {
        const size_t total = (size_t)g.items * g.M * 2 * g.N;
        fold_reduce_kernel<<<(int)std::min<size_t>((total + 255) / 256, 2048), 256, 0, stream>>>(g, splits, part);
    }
    return cudaGetLastError();
}

cudaError_t fold_gemm(const FoldGemm<double2>& g, double2*, cudaStream_t stream) {
    if (g.items > 32767) return cudaErrorInvalidValue;
    const int sms = sm_count();
    auto rounds = [&](int nt) {                        // FMA time of the fullest SM, in columns
        const long long blocks = (long long)((g.M + 31) / 32) * ((g.N + nt - 1) / nt) * 2 * g.items;
        return (blocks + sms - 1) / sms * nt;
    };
    const int nt = rounds(4) < rounds(8) ? 4 : 8;
    dim3 grid((g.M + 31) / 32, (g.N + nt - 1) / nt, 2 * g.items);
    if (nt == 8) fold_zgemm_kernel<8><<<grid, 128, 0, stream>>>(g);
    else fold_zgemm_kernel<4><<<grid, 128, 0, stream>>>(g);
    return cudaGetLastError();
}

template <typename C>
cudaError_t fold_prepare(const C* in, int n, int h, long long keep_r2, C* F, const double* c, int K, int N,
                         typename FoldReal<C>::type* W, int batch, cudaStream_t stream) {
    const int ldw = fold_ldw(N);
    for (int b0 = 0; b0 < batch; b0 += kConsts) {
        const int nb = std::min(kConsts, batch - b0);
        Consts cc{};
        if (c) std::copy(c + b0, c + b0 + nb, cc.v);
        const int bb = W ? (int)(((long long)K * ldw + PREP_THREADS - 1) / PREP_THREADS) : 0;
        const int fb = F ? (int)(((long long)h * h + PREP_THREADS - 1) / PREP_THREADS) : 0;
        fold_prepare_kernel<C><<<dim3(bb + fb, nb), PREP_THREADS, 0, stream>>>(
            F ? in + (size_t)b0 * n * n : nullptr, n, h, keep_r2, F ? F + (size_t)b0 * 4 * h * h : nullptr, cc, K, N, ldw,
            W ? W + (size_t)b0 * 2 * K * ldw : nullptr, bb);
    }
    return cudaGetLastError();
}

template <typename C>
cudaError_t fold_expand(const C* T, int m, int sign, const double* scale, C* out, int batch, cudaStream_t stream) {
    const int h = fold_len(m);
    for (int b0 = 0; b0 < batch; b0 += kConsts) {
        const int nb = std::min(kConsts, batch - b0);
        Consts s{};
        std::copy(scale + b0, scale + b0 + nb, s.v);
        fold_expand_kernel<C><<<dim3((h + 127) / 128, h, nb), 128, 0, stream>>>(T + (size_t)b0 * 4 * h * h, m, sign, s,
                                                                               out + (size_t)b0 * m * m);
    }
    return cudaGetLastError();
}

template cudaError_t fold_prepare<float2>(const float2*, int, int, long long, float2*, const double*, int, int, float*, int, cudaStream_t);
template cudaError_t fold_prepare<double2>(const double2*, int, int, long long, double2*, const double*, int, int, double*, int, cudaStream_t);
template cudaError_t fold_expand<float2>(const float2*, int, int, const double*, float2*, int, cudaStream_t);
template cudaError_t fold_expand<double2>(const double2*, int, int, const double*, double2*, int, cudaStream_t);

}  // namespace coro
