// mc_importance.cu -- the token importance of Sec. 2.3.2 (Eq. 6), the mask of the
// most important tokens that ODP never prunes, and the Eq. 5 threshold taken from
// calibration routing weights (Sec. 2.3.1).
//
//   I_j = ||t_j||_1 * (1 / (L - j)) * sum_{i=j}^{L-1} Abar[i][j]      (0-based j)
//   Abar = the mean over the nh heads of the attention probabilities attn[h][i][j]
//          (query i, key j; a causal map, so key j is seen by queries i >= j)
//
// colsum_kernel: one CTA per (32 V key columns, head, 128-row chunk), V = 4, 2 or 1
//   floats per lane by the alignment of the map's rows; each CTA adds its partial
//   column sums to a fixed-point (2^-40) int64 accumulator with integer atomics,
//   which commute, so the result does not depend on the order the CTAs run in
//   (the partial of a CTA is a fixed sequence of fp32 adds).
// importance_kernel: one warp per token: the l1 norm of t_j, times the column mean.
// rank_select_kernel (L <= 8192): the mask from each token's rank, the number of
//   tokens with a larger bit pattern or an equal one at a lower index (floats >= 0
//   order like their bit patterns), one warp per token.
// select_kernel (larger L, where the L^2 comparisons outgrow it): one CTA: radix
//   select of the n-th largest importance, 8 bits per pass, then the mask: every
//   token above that value and, among the tokens equal to it, the lowest indices
//   until n are chosen.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "mc_host.h"
#include "mc_kernels.h"
#include "mc_profile.h"

namespace mc {

constexpr int kRowChunk = 128, kColWarps = 8;
constexpr double kFix = 1099511627776.0;  // 2^40: fixed-point scale of the column sums

// The first launch of the step: it lets the next one start only after its own
// wait, so that a kernel behind it may read the caller's inputs (t) before its wait.
__global__ void zero_kernel(unsigned long long *acc, int L)
{
    pdl_wait();
    pdl_trigger();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < L) acc[j] = 0ull;
}

template <int V>
struct ColVec;
template <>
struct ColVec<4> {
    using T = float4;
    static __device__ __forceinline__ void get(const T &v, float (&f)[4]) { f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w; }
};
template <>
struct ColVec<2> {
    using T = float2;
    static __device__ __forceinline__ void get(const T &v, float (&f)[2]) { f[0] = v.x; f[1] = v.y; }
};
template <>
struct ColVec<1> {
    using T = float;
    static __device__ __forceinline__ void get(const T &v, float (&f)[1]) { f[0] = v; }
};

// V floats per lane (a row starts V-aligned when V divides L), every warp 16 rows
// of the chunk with 8 loads in flight.  Bound by HBM on the causal half of the map:
// at L = 2048, 32 heads (268 MB, 40 us at the measured copy rate) the whole call,
// this kernel most of it, takes 53.6 us; with 4-byte loads in 32-column tiles, the
// scalar l1 norm and the one-CTA select it took 84.7 us.
template <int V>
__global__ void __launch_bounds__(32 * kColWarps) colsum_kernel(const float *attn, int L, unsigned long long *acc)
{
    constexpr int kTile = 32 * V;
    __shared__ float part[kColWarps][kTile];
    pdl_trigger();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int j0 = blockIdx.x * kTile, j = j0 + V * lane;
    const int i0 = max(j0, (int)blockIdx.z * kRowChunk), i1 = min(L, ((int)blockIdx.z + 1) * kRowChunk);
    if (i0 >= i1) return;  // the chunk lies above the tile's diagonal (whole CTA)
    pdl_wait();
    const float *a = attn + (size_t)blockIdx.y * L * L;
    float s[V];
#pragma unroll
    for (int k = 0; k < V; ++k) s[k] = 0.f;
    if (j < L) {
        using Vec = typename ColVec<V>::T;
#pragma unroll 8
        for (int i = i0 + warp; i < i1; i += kColWarps) {
            float f[V];
            ColVec<V>::get(__ldcs(reinterpret_cast<const Vec *>(a + (size_t)i * L + j)), f);
#pragma unroll
            for (int k = 0; k < V; ++k) s[k] += i >= j + k ? f[k] : 0.f;
        }
    }
#pragma unroll
    for (int k = 0; k < V; ++k) part[warp][V * lane + k] = s[k];
    __syncthreads();
    for (int c = threadIdx.x; c < kTile && j0 + c < L; c += 32 * kColWarps) {
        float t = 0.f;
#pragma unroll
        for (int q = 0; q < kColWarps; ++q) t += part[q][c];
        atomicAdd(acc + j0 + c, (unsigned long long)llrint((double)t * kFix));
    }
}

// VEC: 16-byte loads of the token's row (H % 8 == 0 and t 16-byte aligned).  The l1
// norm is formed before the wait for the column sums: t is an input of the call, and
// zero_kernel let the launches behind it start only after its own wait.
template <bool VEC>
__global__ void __launch_bounds__(256) importance_kernel(const __nv_bfloat16 *t, int L, int H, int nh,
                                                         const unsigned long long *acc, float *imp)
{
    pdl_trigger();
    const int lane = threadIdx.x & 31, j = blockIdx.x * 8 + (threadIdx.x >> 5);
    float l1 = 0.f;
    if (j < L) {
        const __nv_bfloat16 *row = t + (size_t)j * H;
        if (VEC) {
            const uint4 *r4 = reinterpret_cast<const uint4 *>(row);
#pragma unroll 8
            for (int c = lane; c < H / 8; c += 32) {
                const uint4 v = r4[c];
                const __nv_bfloat162 *b2 = reinterpret_cast<const __nv_bfloat162 *>(&v);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float2 f = __bfloat1622float2(b2[k]);
                    l1 += fabsf(f.x);
                    l1 += fabsf(f.y);
                }
            }
        } else {
            for (int h = lane; h < H; h += 32) l1 += fabsf(__bfloat162float(row[h]));
        }
    }
    for (int m = 16; m >= 1; m >>= 1) l1 += __shfl_xor_sync(0xffffffffu, l1, m);
    pdl_wait();
    if (j < L && lane == 0) imp[j] = (float)((double)l1 * ((double)acc[j] / kFix) / ((double)nh * (double)(L - j)));
}

__global__ void __launch_bounds__(1024) select_kernel(const float *imp, int L, int n, uint8_t *mask)
{
    __shared__ int hist[256];
    __shared__ unsigned s_prefix, s_bits;
    __shared__ int s_k, s_base;
    __shared__ int wsum[32];
    pdl_trigger();
    pdl_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        s_prefix = 0;
        s_bits = 0;
        s_k = n;
    }
    __syncthreads();
    // the n-th largest key (n >= 1): 4 passes of 8 bits, most significant first
    for (int shift = 24; shift >= 0; shift -= 8) {
        for (int b = tid; b < 256; b += blockDim.x) hist[b] = 0;
        __syncthreads();
        const unsigned prefix = s_prefix, bits = s_bits;
        for (int j = tid; j < L; j += blockDim.x) {
            const unsigned u = __float_as_uint(imp[j]);
            if ((u & bits) == prefix) atomicAdd(&hist[(u >> shift) & 255], 1);
        }
        __syncthreads();
        if (tid == 0) {
            int k = s_k, cum = 0, b = 255;
            for (; b > 0; --b) {
                if (cum + hist[b] >= k) break;
                cum += hist[b];
            }
            s_k = k - cum;  // still to take among the keys of bin b
            s_prefix = prefix | ((unsigned)b << shift);
            s_bits = bits | (255u << shift);
        }
        __syncthreads();
    }
    const unsigned key = s_prefix;
    const int k = s_k;  // tokens equal to key to select, lowest indices first
    if (tid == 0) s_base = 0;
    __syncthreads();
    for (int j0 = 0; j0 < L; j0 += blockDim.x) {
        const int j = j0 + tid;
        const unsigned u = j < L ? __float_as_uint(imp[j]) : 0u;
        const int eq = j < L && u == key;
        // exclusive prefix count of eq over the chunk, in index order
        const unsigned bal = __ballot_sync(0xffffffffu, eq);
        if (lane == 0) wsum[warp] = __popc(bal);
        __syncthreads();
        int before = s_base + __popc(bal & ((1u << lane) - 1));
        for (int w = 0; w < warp; ++w) before += wsum[w];
        if (j < L) mask[j] = (u > key || (eq && before < k)) ? 1 : 0;
        __syncthreads();
        if (tid == 0) {
            int s = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += wsum[w];
            s_base += s;
        }
        __syncthreads();
    }
}

// One warp per token, so that the L^2 comparisons spread over every SM, where the
// radix select runs in one CTA with four serial bin scans.  The limit is where the
// comparisons (L^2 / 32 warp steps over 608 schedulers) would come to some ten
// microseconds; the map of such a call is 256 MB per head, which outweighs both.
constexpr int kRankMaxL = 8192;

__global__ void __launch_bounds__(256) rank_select_kernel(const float *imp, int L, int n, uint8_t *mask)
{
    pdl_trigger();
    pdl_wait();
    const int lane = threadIdx.x & 31, j = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (j >= L) return;
    const unsigned kj = __float_as_uint(imp[j]);
    int r = 0;
#pragma unroll 8
    for (int i = lane; i < L; i += 32) {
        const unsigned ki = __float_as_uint(imp[i]);
        r += ki > kj || (ki == kj && i < j);
    }
    r = __reduce_add_sync(0xffffffffu, r);
    if (lane == 0) mask[j] = r < n ? 1 : 0;
}

__global__ void fill_kernel(uint8_t *mask, int L, uint8_t v)
{
    pdl_trigger();
    pdl_wait();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < L) mask[j] = v;
}

}  // namespace mc

using namespace mc;

extern "C" {

size_t mc_token_importance_workspace_size(int L) { return L <= 0 ? 0 : (((size_t)L * 8 + 255) & ~(size_t)255); }

int mc_token_importance(const void *t, const float *attn, int L, int H, int nh, float protect_frac,
                        float *importance, uint8_t *mask, void *workspace, size_t ws_bytes, void *stream)
{
    clear_error();
    if (L < 0 || H <= 0 || nh <= 0 || nh > 65535 || !(protect_frac >= 0.f && protect_frac <= 1.f))
        return set_error(MC_ERR_INVALID_ARG, "L=%d H=%d nh=%d protect_frac=%g", L, H, nh, (double)protect_frac);
    if (L == 0) return MC_OK;
    if (!t || !attn || !importance || !workspace) return set_error(MC_ERR_INVALID_ARG, "NULL pointer argument");
    if (ws_bytes < mc_token_importance_workspace_size(L))
        return set_error(MC_ERR_INVALID_ARG, "workspace has %zu bytes, needs %zu", ws_bytes,
                         mc_token_importance_workspace_size(L));
    if ((double)nh * L * L > 9.0e18 / 4 || (double)nh * L > 2.0e9 * 256)
        return set_error(MC_ERR_INVALID_ARG, "attention map too large");
    cudaStream_t st = (cudaStream_t)stream;
    unsigned long long *acc = (unsigned long long *)workspace;
    // loads as wide as the rows' alignment allows
    const int V = L % 4 == 0 && aligned(attn, 16) ? 4 : L % 2 == 0 && aligned(attn, 8) ? 2 : 1;
    auto colsum = V == 4 ? colsum_kernel<4> : V == 2 ? colsum_kernel<2> : colsum_kernel<1>;
    auto rows = H % 8 == 0 && aligned(t, 16) ? importance_kernel<true> : importance_kernel<false>;
    const dim3 grid((L + 32 * V - 1) / (32 * V), nh, (L + kRowChunk - 1) / kRowChunk);
    profile_begin(kKImportance, st);
    cudaError_t err = launch_k(zero_kernel, dim3((L + 255) / 256), dim3(256), 0, st, acc, L);
    profile_end(kKImportance, st);
    if (err == cudaSuccess) {
        profile_begin(kKImportance, st);
        err = launch_k(colsum, grid, dim3(32 * kColWarps), 0, st, attn, L, acc);
        profile_end(kKImportance, st);
    }
    if (err == cudaSuccess) {
        profile_begin(kKImportance, st);
        err = launch_k(rows, dim3((L + 7) / 8), dim3(256), 0, st, (const __nv_bfloat16 *)t, L, H, nh,
                       (const unsigned long long *)acc, importance);
        profile_end(kKImportance, st);
    }
    if (err == cudaSuccess && mask) {
        // ceil(frac * L); a product within 1e-6 of an integer counts as that integer
        const int n = (int)ceil((double)protect_frac * L - 1e-6);
        profile_begin(kKImportance, st);
        if (n <= 0 || n >= L)
            err = launch_k(fill_kernel, dim3((L + 255) / 256), dim3(256), 0, st, mask, L, (uint8_t)(n > 0));
        else if (L <= kRankMaxL)
            err = launch_k(rank_select_kernel, dim3((L + 7) / 8), dim3(256), 0, st, (const float *)importance, L, n, mask);
        else
            err = launch_k(select_kernel, dim3(1), dim3(1024), 0, st, (const float *)importance, L, n, mask);
        profile_end(kKImportance, st);
    }
    if (err != cudaSuccess) return set_error(MC_ERR_CUDA, "importance launch: %s", cudaGetErrorString(err));
    return MC_OK;
}

int mc_odp_threshold_host(const float *w_host, const uint8_t *mask_host, int T, double q, float *mu_out)
{
    clear_error();
    if (T < 0 || !(q >= 0.0 && q <= 1.0)) return set_error(MC_ERR_INVALID_ARG, "T=%d q=%g", T, q);
    if (!w_host || !mu_out) return set_error(MC_ERR_INVALID_ARG, "NULL pointer argument");
    std::vector<double> r;
    r.reserve((size_t)T);
    for (int t = 0; t < T; ++t) {
        if (mask_host && mask_host[t] != 0) continue;  // protected or dropped: never pruned
        const double w0 = w_host[2 * t], w1 = w_host[2 * t + 1];
        if (w0 > 0.0) r.push_back(w1 / w0);
    }
    if (r.empty()) return set_error(MC_ERR_INVALID_ARG, "no prunable token with a positive primary weight");
    std::sort(r.begin(), r.end());
    // linear interpolation between the order statistics around q * (n - 1)
    const double pos = q * (double)(r.size() - 1);
    const size_t lo = (size_t)floor(pos), hi = std::min(lo + 1, r.size() - 1);
    *mu_out = (float)(r[lo] + (pos - (double)lo) * (r[hi] - r[lo]));
    return MC_OK;
}

}  // extern "C"
