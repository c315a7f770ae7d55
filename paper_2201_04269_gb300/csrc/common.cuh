// common.cuh - block reductions, site loading and small pivoted LU determinants shared by
// the kernels of libmbc (internal).
#pragma once
#include "device.cuh"
#include "numeric.cuh"

namespace mbc {

// --------------------------------------------------------------------- reductions
__device__ __forceinline__ kacc kacc_shfl_down(kacc v, int off) {
    kacc o;
    o.hi = __shfl_down_sync(0xffffffffu, v.hi, off);
    o.lo = __shfl_down_sync(0xffffffffu, v.lo, off);
    return o;
}

// Deterministic compensated block sum of one complex double per thread; the result is valid
// in thread 0.  The values go through buf (blockDim values, free after the barrier the caller
// has passed); warp 0 adds the real parts, the last warp the imaginary parts, every 32nd value
// per lane and then a shuffle tree: an FP64 warp instruction takes 64 cycles of the pipe
// whatever its active lanes, so a shuffle tree in every warp costs far more.  red: 4 doubles.
__device__ __forceinline__ void block_sum(cd v, kacc& out_re, kacc& out_im, double* red, cd* buf) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, last = (blockDim.x >> 5) - 1;
    buf[threadIdx.x] = v;
    __syncthreads();
    for (int part = 0; part < 2; ++part) {
        if (warp != (part ? last : 0)) continue;
        kacc k = {0.0, 0.0};
        for (int i = lane; i < (int)blockDim.x; i += 32) kacc_add(k, part ? buf[i].im : buf[i].re);
        for (int off = 16; off > 0; off >>= 1) kacc_merge(k, kacc_shfl_down(k, off));
        if (lane == 0) {
            red[2 * part] = k.hi;
            red[2 * part + 1] = k.lo;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        out_re = kacc{red[0], red[1]};
        out_im = kacc{red[2], red[3]};
    }
    __syncthreads();
}

__device__ __forceinline__ double block_max(double v, double* red) {
    for (int off = 16; off > 0; off >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, off));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double m = 0.0;
    for (int w = 0; w < nw; ++w) m = fmax(m, red[w]);
    __syncthreads();
    return m;
}

// Exponents e with max |re|, |im| of each of two 12x12 blocks in [0.5, 1) after scaling by 2^-e,
// from the high words of the values (no FP64 arithmetic): true when both maxima are well inside
// the normal range (or zero), the same for every thread.  ru: 64 words of shared memory.
__device__ __forceinline__ bool block_exponents(const double* __restrict__ a, const double* __restrict__ b,
                                                unsigned* ru, int& ea, int& eb) {
    unsigned ma = 0u, mb = 0u;
    for (int i = threadIdx.x; i < 288; i += blockDim.x) {
        const double2 v = __ldg(reinterpret_cast<const double2*>(i < 144 ? a : b) + (i < 144 ? i : i - 144));
        // (the lowest bit keeps a subnormal number below 2^-1042, whose high word is zero, from counting as zero)
        const unsigned m = max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu) |
                           ((__double2loint(v.x) | __double2loint(v.y)) != 0);
        if (i < 144) ma = max(ma, m);
        else mb = max(mb, m);
    }
    ma = __reduce_max_sync(0xffffffffu, ma);
    mb = __reduce_max_sync(0xffffffffu, mb);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane == 0) {
        ru[warp] = ma;
        ru[32 + warp] = mb;
    }
    __syncthreads();
    ma = __reduce_max_sync(0xffffffffu, lane < nw ? ru[lane] : 0u);
    mb = __reduce_max_sync(0xffffffffu, lane < nw ? ru[32 + lane] : 0u);
    ea = ma ? (int)(ma >> 20) - 1022 : 0;
    eb = mb ? (int)(mb >> 20) - 1022 : 0;
    auto plain = [](unsigned m) { return m == 0u || ((m >> 20) >= 200u && (m >> 20) < 2047u); };
    return plain(ma) && plain(mb);
}
// x 2^-e for an entry of a block whose exponent block_exponents gave, by the exponent field (0
// where that is far below the float range)
__device__ __forceinline__ double scaled_entry(double x, int e) {
    const int hi = __double2hiint(x);
    return ((hi >> 20) & 0x7ff) - e < 800 ? 0.0 : __hiloint2double(hi - (e << 20), __double2loint(x));
}

// Load two 12x12 complex double blocks (flavour matrices of one site) into shared memory
// as precision-P values; for the mixed precision each block is first scaled by an exact
// power of two so that its largest |re|, |im| lies in [0.5, 1); the exponents are
// returned (0, 0 for FP64).
template <class P>
__device__ __forceinline__ void load_pair(const double* __restrict__ a, const double* __restrict__ b,
                                          typename P::V* sa, typename P::V* sb, double* red, int& ea, int& eb) {
    // entry (r, c) goes to [r * kLd + c]
    if (P::scaled() && block_exponents(a, b, reinterpret_cast<unsigned*>(red), ea, eb)) {
        for (int i = threadIdx.x; i < 288; i += blockDim.x) {
            const int e = i < 144 ? i : i - 144;
            const double2 v = __ldg(reinterpret_cast<const double2*>(i < 144 ? a : b) + e);
            const int sc = i < 144 ? ea : eb;
            (i < 144 ? sa : sb)[(e / 12) * kLd + e % 12] = P::from_scaled(cd_make(scaled_entry(v.x, sc), scaled_entry(v.y, sc)));
        }
        __syncthreads();
        return;
    }
    if (P::scaled()) __syncthreads();           // (red is written again)
    cd* ra = reinterpret_cast<cd*>(sa);
    cd* rb = reinterpret_cast<cd*>(sb);
    double ma = 0.0, mb = 0.0;
    for (int i = threadIdx.x; i < 288; i += blockDim.x) {
        const int e = i < 144 ? i : i - 144;
        const int o = (e / 12) * kLd + e % 12;
        const double2 v = __ldg(reinterpret_cast<const double2*>(i < 144 ? a : b) + e);
        if (i < 144) { ra[o] = cd_make(v.x, v.y); ma = fmax(ma, fmax(fabs(v.x), fabs(v.y))); }
        else { rb[o] = cd_make(v.x, v.y); mb = fmax(mb, fmax(fabs(v.x), fabs(v.y))); }
    }
    if (!P::scaled()) { ea = eb = 0; __syncthreads(); return; }
    ma = block_max(ma, red);
    mb = block_max(mb, red);
    ea = block_exponent(ma);
    eb = block_exponent(mb);
    for (int i = threadIdx.x; i < 288; i += blockDim.x) {
        const int e = i < 144 ? i : i - 144;
        const int o = (e / 12) * kLd + e % 12;
        if (i < 144) sa[o] = P::from_cd(ra[o], -ea);
        else sb[o] = P::from_cd(rb[o], -eb);
    }
    __syncthreads();
}

// --------------------------------------------------------------------- LU determinants
// det of the N x N matrix m[rows[i]][cols[k]] gathered from a 12x12 block, by Gaussian
// elimination with partial pivoting (pivot = largest |re| + |im|, first on ties; a row
// swap flips the sign; an exactly zero pivot gives 0, and so does, in the mixed
// arithmetic, a pivot below P::tiny()).
template <class P, int N, int LD>
__device__ __forceinline__ typename P::V det_gather(const typename P::V* m, const int8_t* rows, const int8_t* cols) {
    typedef typename P::V V;
    V a[N][N];
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int k = 0; k < N; ++k) a[i][k] = m[rows[i] * LD + cols[k]];
    V det = P::zero();
    bool first = true;
    int sign = 1;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        int p = k;
        auto best = P::mag(a[k][k]);
#pragma unroll
        for (int i = k + 1; i < N; ++i) {
            auto mg = P::mag(a[i][k]);
            if (mg > best) { best = mg; p = i; }
        }
        if (best <= P::tiny()) return P::zero();
#pragma unroll
        for (int i = k + 1; i < N; ++i) {
            if (i == p) {
#pragma unroll
                for (int c = k; c < N; ++c) { V t = a[k][c]; a[k][c] = a[i][c]; a[i][c] = t; }
                sign = -sign;
            }
        }
        det = first ? a[k][k] : P::mul(det, a[k][k]);
        first = false;
        if (k + 1 < N) {
            V inv = P::div(P::one(), a[k][k]);
#pragma unroll
            for (int i = k + 1; i < N; ++i) {
                V f = P::mul(a[i][k], inv);
#pragma unroll
                for (int c = k + 1; c < N; ++c) {
                    typename P::A acc;
                    P::acc_zero(acc);
                    P::add(acc, a[i][c]);
                    P::fms(acc, f, a[k][c]);
                    a[i][c] = P::get(acc);
                }
            }
        }
    }
    return sign < 0 ? P::neg(det) : det;
}

// (N: the largest n the caller needs)
template <class P, int LD, int N = 6>
__device__ __forceinline__ typename P::V det_n(int n, const typename P::V* m, const int8_t* rows, const int8_t* cols) {
    switch (n) {
        case 1: return m[rows[0] * LD + cols[0]];
        // 2 x 2 without elimination: the pivoted LU's division was most of the work
        // (proton direct sweep in FP64, 512 sites: 205 -> 127 us)
        case 2: return P::det2(m[rows[0] * LD + cols[0]], m[rows[0] * LD + cols[1]], m[rows[1] * LD + cols[0]],
                               m[rows[1] * LD + cols[1]]);
        case 3: return det_gather<P, N < 3 ? 1 : 3, LD>(m, rows, cols);
        case 4: return det_gather<P, N < 4 ? 1 : 4, LD>(m, rows, cols);
        case 5: return det_gather<P, N < 5 ? 1 : 5, LD>(m, rows, cols);
        case 6: return det_gather<P, N < 6 ? 1 : 6, LD>(m, rows, cols);
        default: return P::one();   // n = 0: empty product
    }
}

__device__ __forceinline__ void store_partial(d4* dst, const kacc& re, const kacc& im, int scale_exp) {
    d4 v;
    v.x = ldexp(re.hi, scale_exp); v.y = ldexp(re.lo, scale_exp);
    v.z = ldexp(im.hi, scale_exp); v.w = ldexp(im.lo, scale_exp);
    *dst = v;
}

}  // namespace mbc
