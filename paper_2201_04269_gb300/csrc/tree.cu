// tree.cu - factor-tree evaluation (arXiv 2201.04269 Sec. 4).
//
// The planner's linearised factor tree (factors in depth-first order, children counts,
// leaf coefficients; Fig. 5) has the up minors det U[R_u, C_u] at level 1 and the down
// minors det D[R_d, C_d] at the leaves.  Evaluation has two kernels per wave of sites:
//
//  1. every factor (distinct minor) once per site into a scratch table laid out
//     [minor][site], so that the tree walk's gathers for 32 consecutive sites are one
//     contiguous 512-byte access: by shared Laplace steps level by level (entry_kernel, then
//     minor_level_kernel per level and flavour; minor_levels.hpp), or, for a flavour whose few
//     scattered minors share too little, by one pivoted LU per minor (minor_table_kernel).
//  2. tree_walk_kernel: one block per (32 sites, chunk of level-1 subtrees), its warps
//     taking runs of the chunk's subtrees; lane = site.
//     The tree arrays are read warp-uniformly (broadcast), the factor values gathered
//     from the table; a level-1 vertex multiplies the sum of its leaves
//     (coefficient x leaf factor) -- the sum over root-to-leaf paths of Sec. 4.
#include "common.cuh"

namespace mbc {

static constexpr int kTreeSites = 32;              // sites per block / warp
static constexpr int kPad = 145;                   // padded 12x12 block stride (values)

template <class P>
__global__ void __launch_bounds__(256) minor_table_kernel(TreeDev d, int flavour, const double* __restrict__ M,
                                                          int64_t site0, int64_t n_sites, int64_t wave,
                                                          typename P::V* __restrict__ table, int64_t table_off,
                                                          int* __restrict__ exps) {
    typedef typename P::V V;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* sm = reinterpret_cast<V*>(smem_raw);        // [32][kPad]
    __shared__ int s_exp[kTreeSites];
    const int n = flavour == 0 ? d.n_u : d.n_d;
    const int64_t n_minors = d.n_minors[flavour];
    const int64_t g0 = (int64_t)blockIdx.y * kTreeSites;   // first site of this block within the wave
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    // stage 32 sites (one warp per site at a time), with the per-site exponent
    for (int s = warp; s < kTreeSites; s += nw) {
        const int64_t site = site0 + g0 + s;
        double m = 0.0;
        cd raw[5];
        for (int i = 0; i < 5; ++i) {
            const int e = lane + 32 * i;
            raw[i] = cd_make(0.0, 0.0);
            if (e < 144 && g0 + s < n_sites) {
                const double2 v = __ldg(reinterpret_cast<const double2*>(M + site * 288) + e);
                raw[i] = cd_make(v.x, v.y);
                m = fmax(m, fmax(fabs(v.x), fabs(v.y)));
            }
        }
        for (int off = 16; off > 0; off >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, off));
        const int e = P::scaled() ? block_exponent(m) : 0;
        for (int i = 0; i < 5; ++i) {
            const int k = lane + 32 * i;
            if (k < 144) sm[s * kPad + k] = P::from_cd(raw[i], -e);
        }
        if (lane == 0) s_exp[s] = e;
    }
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x < kTreeSites && g0 + threadIdx.x < n_sites)
        exps[(g0 + threadIdx.x) * 2 + flavour] = s_exp[threadIdx.x];
    // minors: warp w takes minors blockIdx.x * nw + w, + gridDim.x * nw, ...
    const bool live = g0 + lane < n_sites;
    for (int64_t mi = (int64_t)blockIdx.x * nw + warp; mi < n_minors; mi += (int64_t)gridDim.x * nw) {
        int8_t rows[6], cols[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            if (i < n) { rows[i] = d.minor_rows[flavour][mi * n + i]; cols[i] = d.minor_cols[flavour][mi * n + i]; }
        }
        const V v = det_n<P, 12>(n, sm + lane * kPad, rows, cols);
        if (live) table[(table_off + mi) * wave + g0 + lane] = v;
    }
}

// The site's blocks as level 1 of the tables: entry e of flavour f of site s at row f * 144 + e
// of `table` (scaled by the per-site exponent in the mixed arithmetic).  One warp per (site,
// flavour) reads its block whole; the transposed 16-byte stores meet in L2.
template <class P>
__global__ void __launch_bounds__(256) entry_kernel(const double* __restrict__ U, const double* __restrict__ D,
                                                    int64_t n_sites, int64_t wave, typename P::V* __restrict__ table,
                                                    int* __restrict__ exps) {
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t s = w >> 1;
    const int f = (int)(w & 1);
    if (s >= n_sites) return;
    const double2* m = reinterpret_cast<const double2*>((f == 0 ? U : D) + s * 288);
    cd raw[5];
    double top = 0.0;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const int e = lane + 32 * i;
        raw[i] = cd_make(0.0, 0.0);
        if (e < 144) {
            const double2 v = __ldg(m + e);
            raw[i] = cd_make(v.x, v.y);
            top = fmax(top, fmax(fabs(v.x), fabs(v.y)));
        }
    }
    for (int off = 16; off > 0; off >>= 1) top = fmax(top, __shfl_xor_sync(0xffffffffu, top, off));
    const int ex = P::scaled() ? block_exponent(top) : 0;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const int e = lane + 32 * i;
        if (e < 144) table[(int64_t)(f * 144 + e) * wave + s] = P::from_cd(raw[i], -ex);
    }
    if (lane == 0) exps[s * 2 + f] = ex;
}

// One level of one flavour: entry e's result from K parents (rows of `below`) and K matrix
// entries (rows of `entries`), lane = site, so every table access is one coalesced 512-byte
// row segment and the record (K + 1 words) is the same for the warp.  A warp takes kLevelRun
// consecutive entries, which share a column set and so most parents (L1).  Bound by the
// multiply-adds: 3He_I needs 1.1e6 of them a site where one LU per minor took 6.8e6 and
// divisions (512 sites in double-float: 22.4 -> 1.24 ms for
// both flavours).
constexpr int kLevelRun = 4;
template <class P, int K>
__global__ void __launch_bounds__(256) minor_level_kernel(const uint32_t* __restrict__ words, int64_t n_entries,
                                                          const typename P::V* __restrict__ entries,
                                                          const typename P::V* __restrict__ below,
                                                          typename P::V* __restrict__ out, int64_t wave) {
    const int64_t s = (int64_t)blockIdx.y * 32 + (threadIdx.x & 31);
    int64_t e = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kLevelRun;
    const int64_t end = min(e + kLevelRun, n_entries);
    for (; e < end; ++e) {
        const uint32_t* w = words + e * (K + 1);
        typename P::V a[K], p[K];
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const uint32_t x = __ldg(w + i);
            a[i] = entries[(int64_t)(x & 0xFFu) * wave + s];
            p[i] = below[(int64_t)(x >> 8) * wave + s];
        }
        const uint32_t to = __ldg(w + K);
        typename P::A acc;
        P::acc_zero(acc);
#pragma unroll
        for (int i = 0; i < K; ++i) {
            if (i & 1) P::fms(acc, a[i], p[i]);
            else P::fma(acc, a[i], p[i]);
        }
        out[(int64_t)(to >> 1) * wave + s] = P::flip(P::get(acc), (to & 1u) ? -1 : 1);
    }
}

template <class P>
void launch_level(int k, const uint32_t* words, int64_t n, const typename P::V* entries, const typename P::V* below,
                  typename P::V* out, int64_t wave, cudaStream_t s) {
    const int64_t per_block = 8 * kLevelRun;
    const dim3 grid((unsigned)((n + per_block - 1) / per_block), (unsigned)(wave / 32));
    switch (k) {
        case 2: minor_level_kernel<P, 2><<<grid, 256, 0, s>>>(words, n, entries, below, out, wave); break;
        case 3: minor_level_kernel<P, 3><<<grid, 256, 0, s>>>(words, n, entries, below, out, wave); break;
        case 4: minor_level_kernel<P, 4><<<grid, 256, 0, s>>>(words, n, entries, below, out, wave); break;
        case 5: minor_level_kernel<P, 5><<<grid, 256, 0, s>>>(words, n, entries, below, out, wave); break;
        default: minor_level_kernel<P, 6><<<grid, 256, 0, s>>>(words, n, entries, below, out, wave); break;
    }
}

// The levels of the flavours that have them, in the rows after the tree's minors.
template <class P>
cudaError_t launch_levels(const TreeDev& d, const double* U, const double* D, int64_t n, int64_t wave,
                          typename P::V* table, int* exps, cudaStream_t s, int64_t* launches) {
    typename P::V* entries = table + (d.n_minors[0] + d.n_minors[1]) * wave;
    entry_kernel<P><<<(unsigned)((2 * n + 7) / 8), 256, 0, s>>>(U, D, n, wave, entries, exps);
    ++*launches;
    typename P::V* free_rows = entries + 288 * wave;
    for (int f = 0; f < 2; ++f) {
        const TreeLevelsDev& l = d.levels[f];
        if (!l.n) continue;
        const typename P::V* ent = entries + f * 144 * wave;
        const typename P::V* below = ent;
        for (int k = 2; k <= l.n; ++k) {
            typename P::V* out = k == l.n ? table + (f == 0 ? 0 : d.n_minors[0]) * wave : free_rows;
            launch_level<P>(k, l.words[k], l.entries[k], ent, below, out, wave, s);
            ++*launches;
            below = out;
            if (k < l.n) free_rows += l.entries[k] * wave;
        }
    }
    return cudaGetLastError();
}

// REAL: the coefficients are real scalars of the arithmetic (d.coef_s), half the multiply-adds.
// Leaves are taken four at a time so that their table reads are in flight together.
template <class P, bool REAL>
__global__ void __launch_bounds__(32 * kTreeSplit) tree_walk_kernel(TreeDev d, const typename P::V* __restrict__ table,
                                                        int64_t site0, int64_t n_sites, int64_t wave,
                                                        const int* __restrict__ exps, Partials out) {
    typedef typename P::V V;
    __shared__ cd sum[kTreeSplit][32];
    const int lane = threadIdx.x & 31, run = threadIdx.x >> 5;
    // chunks of one site group side by side: the blocks in flight (about 450) then read the
    // minors of one or two groups, which stay in L2 (3He_I: 99 MB a group), each about 12
    // times; with the groups side by side every read came from DRAM (512 sites: 2.0 -> 1.5 ms)
    const int c = (int)(blockIdx.x % d.n_chunks);
    const int64_t s = (int64_t)(blockIdx.x / d.n_chunks) * 32 + lane;
    const bool live = s < n_sites;
    const int64_t col = live ? s : 0;
    int64_t k = d.run_node[c * kTreeSplit + run];
    int64_t leaf = d.run_leaf[c * kTreeSplit + run];
    const int count = d.run_count[c * kTreeSplit + run];
    typename P::A acc;
    P::acc_zero(acc);
    for (int v1 = 0; v1 < count; ++v1) {
        const int32_t f1 = __ldg(d.factors + k);
        const int32_t nch = __ldg(d.children + k);
        ++k;
        const V u = table[(int64_t)f1 * wave + col];
        typename P::A inner;
        P::acc_zero(inner);
        auto leaf_add = [&](int64_t l, V v) {
            if (REAL) P::fma_s(inner, __ldg(reinterpret_cast<const typename P::S*>(d.coef_s) + l), v);
            else P::fma(inner, ldv<V>(d.coefficients, l), v);
        };
        int i = 0;
        for (; i + 4 <= nch; i += 4) {
            V v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = table[(int64_t)__ldg(d.factors + k + i + u) * wave + col];
#pragma unroll
            for (int u = 0; u < 4; ++u) leaf_add(leaf + i + u, v[u]);
        }
        for (; i < nch; ++i) leaf_add(leaf + i, table[(int64_t)__ldg(d.factors + k + i) * wave + col]);
        k += nch;
        leaf += nch;
        P::fma(acc, u, P::get(inner));
    }
    sum[run][lane] = P::to_cd(P::get(acc));
    __syncthreads();
    if (run == 0 && live) {
        kacc re = {0.0, 0.0}, im = {0.0, 0.0};
        for (int r = 0; r < kTreeSplit; ++r) {
            kacc_add(re, sum[r][lane].re);
            kacc_add(im, sum[r][lane].im);
        }
        store_partial(out.part + (site0 + s) * out.n_chunks + c, re, im,
                      exps[s * 2 + 0] * d.n_u + exps[s * 2 + 1] * d.n_d);
    }
}

size_t tree_value_bytes(int) { return 16; }

cudaError_t launch_tree(const TreeDev& d, int prec, const double* U, const double* D, Geometry g, void* scratch,
                        int64_t scratch_sites, int* exps, Partials out, int threads, cudaStream_t s,
                        int64_t* launches) {
    const int64_t total = g.n_sites();
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const size_t smem = (size_t)kTreeSites * kPad * 16;
    cudaError_t attr = prec == 0 ? cudaFuncSetAttribute(minor_table_kernel<FP64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                                 : cudaFuncSetAttribute(minor_table_kernel<MIXED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (attr != cudaSuccess) return attr;
    cudaMemsetAsync(exps, 0, sizeof(int) * 2 * (size_t)std::min(total, scratch_sites), s);
    for (int64_t site0 = 0; site0 < total; site0 += scratch_sites) {
        const int64_t n = std::min(scratch_sites, total - site0);
        const int64_t wave = (n + 31) / 32 * 32;
        const int64_t gy = wave / 32;
        if (d.levels[0].n || d.levels[1].n) {
            const cudaError_t e =
                prec == 0 ? launch_levels<FP64>(d, U + site0 * 288, D + site0 * 288, n, wave, (cd*)scratch, exps, s, launches)
                          : launch_levels<MIXED>(d, U + site0 * 288, D + site0 * 288, n, wave, (cdf*)scratch, exps, s, launches);
            if (e != cudaSuccess) return e;
        }
        for (int f = 0; f < 2; ++f) {
            if (d.n_minors[f] == 0 || d.levels[f].n) continue;
            const int64_t per_block = (int64_t)(threads / 32) * 16;            // minors per block (16 rounds)
            int64_t gx = (d.n_minors[f] + per_block - 1) / per_block;
            gx = std::max<int64_t>(1, std::min<int64_t>(gx, std::max<int64_t>(1, (int64_t)sms * 16 / gy)));
            dim3 grid((unsigned)gx, (unsigned)gy);
            const double* M = (f == 0 ? U : D) + site0 * 288;
            const int64_t off = f == 0 ? 0 : d.n_minors[0];
            if (prec == 0)
                minor_table_kernel<FP64><<<grid, threads, smem, s>>>(d, f, M, 0, n, wave, (cd*)scratch, off, exps);
            else
                minor_table_kernel<MIXED><<<grid, threads, smem, s>>>(d, f, M, 0, n, wave, (cdf*)scratch, off, exps);
            ++*launches;
        }
        const int64_t blocks = (n + 31) / 32 * d.n_chunks;
#define MBC_WALK_ARGS site0, n, wave, exps, out
        if (prec == 0 && d.coef_s)
            tree_walk_kernel<FP64, true><<<(unsigned)blocks, 32 * kTreeSplit, 0, s>>>(d, (const cd*)scratch, MBC_WALK_ARGS);
        else if (prec == 0)
            tree_walk_kernel<FP64, false><<<(unsigned)blocks, 32 * kTreeSplit, 0, s>>>(d, (const cd*)scratch, MBC_WALK_ARGS);
        else if (d.coef_s)
            tree_walk_kernel<MIXED, true><<<(unsigned)blocks, 32 * kTreeSplit, 0, s>>>(d, (const cdf*)scratch, MBC_WALK_ARGS);
        else
            tree_walk_kernel<MIXED, false><<<(unsigned)blocks, 32 * kTreeSplit, 0, s>>>(d, (const cdf*)scratch, MBC_WALK_ARGS);
#undef MBC_WALK_ARGS
        ++*launches;
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

}  // namespace mbc
