// sm_103a kernels of the Fermi operator expansion of the density kernel (App. "Fermi
// operator expansion"; Sec. "Density kernel optimization"), FP64 on the sparsity
// pattern of H and S (CSR: rows a, ascending columns b; the pattern is symmetric and
// holds the diagonal).  Every matrix is a vector of values on that pattern.
//
//   k_foe_prep    H~ = sigma (H - tau S) and the Taylor S^-1/2 = (3 I - S) / 2
//   k_triple      Y = X A X restricted to the pattern: per row i, w = X_i. A is summed
//                 exactly (over every column it reaches) in a per-CTA dense row of the
//                 scratch, then Y_il = sum_m w_m X_ml for the pattern's l
//   k_cheb        one Chebyshev step for every column l of the pattern:
//                 t_l^{j+1} = alpha H~' t_l^j - t_l^{j-1}, kept on pattern column l;
//                 the columns are stored transposed (column l of T on row l of the CSR)
//   k_traces      sums of the diagonal entries of the T_j (a CTA per matrix, fixed order)
//   k_kernel_sum  K'(transposed) = c_0/2 I + sum_j c_j T_j(transposed) from the stored T_j
//   k_axpy_t      K'(transposed) += c T_j(transposed), where they are not stored
//   k_transpose   values on (i, l) <- values on (l, i)
//   k_ebs         E_BS = sum_{il} K_il (H~_li / sigma + tau S_li) (partial sums, then one CTA)
//
// The functions of an atom have the same pattern row (a "group" of rows), so matrices are
// blocks of groups and index work is done once per pair of groups: k_cheb and k_triple_g give
// a warp the outputs (i, l) of a pair (I, L) as lanes and list the common columns once.
// FP64 products (1/64 of the FP32 rate) are the bound that remains.
#include <algorithm>
#include <cstdint>

#include "lsw_device.h"
#include "lsw_internal.h"

namespace lsw {

__global__ void k_foe_prep(const double* __restrict__ H, const double* __restrict__ S, const int64_t* __restrict__ row_ptr,
                           const int32_t* __restrict__ col, int n, double sigma, double tau, double* __restrict__ Ht,
                           double* __restrict__ X) {
    const int a = blockIdx.x * blockDim.y + threadIdx.y;
    if (a >= n) return;
    for (int64_t k = row_ptr[a] + threadIdx.x; k < row_ptr[a + 1]; k += blockDim.x) {
        Ht[k] = sigma * (H[k] - tau * S[k]);
        X[k] = 0.5 * (3.0 * (col[k] == a ? 1.0 : 0.0) - S[k]);
    }
}

__device__ __forceinline__ double warp_sum_d(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

constexpr int FOE_WARPS = 8;

// Lane layout of the outputs (i, l) of a pair of groups, `no` of them from o0: lane = o + no g, the
// sum of an output split over G = 2^k <= 32 / no parts g.
struct FoeLanes {
    int no, G, o, g;
    bool on;
    __device__ __forceinline__ FoeLanes(int total, int o0, int lane) {
        no = min(total - o0, 32);
        G = 1;
        while (2 * G * no <= 32) G *= 2;
        g = lane / no;
        o = o0 + lane - g * no;
        on = g < G;
    }
    __device__ __forceinline__ double sum(double v) const {       // over the parts; valid on g = 0
        for (int s = G >> 1; s > 0; s >>= 1) v += __shfl_down_sync(0xffffffffu, v, s * no);
        return v;
    }
};

// Y = X A X on the pattern, a CTA per group I with its rows of w = X A (dense, every column) in
// shared memory: a warp per neighbour K adds sum_{k in K} X_ik A_km for all m of K's rows, then a
// warp per pair (I, L) sums Y_il = sum_m w_im X_ml (X_ml = X[tpos]).  400 atoms (1,348 functions,
// 161 k entries): 223 us, 318 with a CTA per row and global atomics (k_triple, which
// stays for patterns whose rows of w do not fit).
constexpr int FOE_TWARPS = 16;
__global__ void __launch_bounds__(32 * FOE_TWARPS) k_triple_g(FoeLaunch a, const double* __restrict__ X,
                                                             const double* __restrict__ A, double* __restrict__ Y) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 14;
    extern __shared__ __align__(16) double foe_w[];               // [n_i][n]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int I = blockIdx.x;
    const int i0 = LD(a.gfirst, I, a.ng + 1), nI = LD(a.gfirst, I + 1, a.ng + 1) - i0;
    const int64_t r0 = LD(a.row_ptr, i0, a.n + 1);
    const int len = static_cast<int>(LD(a.row_ptr, i0 + 1, a.n + 1) - r0);
    const int t0 = LD(a.nptr, I, a.ng + 1), nt = LD(a.nptr, I + 1, a.ng + 1) - t0;
    [[maybe_unused]] const int64_t wn = static_cast<int64_t>(nI) * a.n;
    for (int e = threadIdx.x; e < nI * a.n; e += blockDim.x) ST(foe_w, e, wn, 0.0);
    __syncthreads();
    for (int t = warp; t < nt; t += FOE_TWARPS) {
        const int K = LD(a.ngrp, t0 + t, a.nn), qK = LD(a.npos, t0 + t, a.nn);
        const int k0 = LD(a.gfirst, K, a.ng + 1), nK = LD(a.gfirst, K + 1, a.ng + 1) - k0;
        const int64_t s0 = LD(a.row_ptr, k0, a.n + 1);
        const int lenK = static_cast<int>(LD(a.row_ptr, k0 + 1, a.n + 1) - s0);
        for (int p = lane; p < lenK; p += 32) {
            const int m = LD(a.col, s0 + p, a.nnz);
            for (int i = 0; i < nI; ++i) {
                double v = 0.0;
                for (int k = 0; k < nK; ++k)
                    v = fma(LD(X, r0 + static_cast<int64_t>(i) * len + qK + k, a.nnz),
                            LD(A, s0 + static_cast<int64_t>(k) * lenK + p, a.nnz), v);
                atomicAdd(&foe_w[i * a.n + m], v);
            }
        }
    }
    __syncthreads();
    for (int t = warp; t < nt; t += FOE_TWARPS) {
        const int L = LD(a.ngrp, t0 + t, a.nn), qL = LD(a.npos, t0 + t, a.nn);
        const int l0 = LD(a.gfirst, L, a.ng + 1), nL = LD(a.gfirst, L + 1, a.ng + 1) - l0;
        const int64_t s0 = LD(a.row_ptr, l0, a.n + 1);
        const int lenL = static_cast<int>(LD(a.row_ptr, l0 + 1, a.n + 1) - s0);
        for (int o0 = 0; o0 < nI * nL; o0 += 32) {
            const FoeLanes f(nI * nL, o0, lane);
            const int i = f.o / nL, l = f.o - i * nL;
            double acc = 0.0;
            if (f.on)
#pragma unroll 8
                for (int p = f.g; p < lenL; p += f.G) {
                    const int64_t e = s0 + static_cast<int64_t>(l) * lenL + p;
                    acc = fma(LD(foe_w, i * a.n + LD(a.col, e, a.nnz), wn), LD(X, LD(a.tpos, e, a.nnz), a.nnz), acc);
                }
            acc = f.sum(acc);
            if (f.on && f.g == 0) ST(Y, r0 + static_cast<int64_t>(i) * len + qL + l, a.nnz, acc);
        }
    }
}

// Y = X A X on the pattern; tpos[q] = position of the transposed entry of q.  Each CTA
// owns the dense row scratch w + blockIdx.x * n (zero on entry, zero again on exit).
__global__ void __launch_bounds__(256) k_triple(FoeLaunch a, const double* __restrict__ X, const double* __restrict__ A,
                                                double* __restrict__ Y) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 14;
    double* w = a.scratch + static_cast<int64_t>(blockIdx.x) * a.n;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int i = blockIdx.x; i < a.n; i += gridDim.x) {
        const int64_t r0 = LD(a.row_ptr, i, a.n + 1), r1 = LD(a.row_ptr, i + 1, a.n + 1);
        // w_m = sum_k X_ik A_km
        for (int64_t q = r0 + warp; q < r1; q += nw) {
            const int k = LD(a.col, q, a.nnz);
            const double x = LD(X, q, a.nnz);
            const int64_t s0 = LD(a.row_ptr, k, a.n + 1), s1 = LD(a.row_ptr, k + 1, a.n + 1);
            for (int64_t p = s0 + lane; p < s1; p += 32) {
                const int m = LD(a.col, p, a.nnz);
                atomicAdd(&w[m], x * LD(A, p, a.nnz));
            }
        }
        __syncthreads();
        // Y_il = sum_m w_m X_ml, m over row l of the transposed X (X_ml = X[tpos[q]])
        for (int64_t q = r0 + warp; q < r1; q += nw) {
            const int l = LD(a.col, q, a.nnz);
            const int64_t s0 = LD(a.row_ptr, l, a.n + 1), s1 = LD(a.row_ptr, l + 1, a.n + 1);
            double acc = 0.0;
            for (int64_t p = s0 + lane; p < s1; p += 32) {
                const int m = LD(a.col, p, a.nnz);
                acc += LD(w, m, a.n) * LD(X, LD(a.tpos, p, a.nnz), a.nnz);
            }
            acc = warp_sum_d(acc);
            if (lane == 0) ST(Y, q, a.nnz, acc);
        }
        __syncthreads();
        for (int64_t q = r0 + warp; q < r1; q += nw) {
            const int k = LD(a.col, q, a.nnz);
            const int64_t s0 = LD(a.row_ptr, k, a.n + 1), s1 = LD(a.row_ptr, k + 1, a.n + 1);
            for (int64_t p = s0 + lane; p < s1; p += 32) ST(w, LD(a.col, p, a.nnz), a.n, 0.0);
        }
        __syncthreads();
    }
}

// One Chebyshev step on every column (transposed storage: Tc[pos(l, k)] = T_kl):
//   Tn[pos(l, i)] = alpha sum_k Htp_ik Tc[pos(l, k)] - (Tp ? Tp[pos(l, i)] : 0)
// A CTA per group L of columns; map (shared, a.n ints, -1 outside) gives the position of k in
// the group's rows.  A warp takes a neighbour I of L: it lists, a.chunk entries of I's rows at a
// time, the columns that both have (position in I's row, position in L's row), and sums the
// outputs (i, l) over the list, a lane each (several lanes where there are fewer than 32).
// A group is split over several CTAs where there are few (one each: too few warps to cover its
// loads).  400 atoms (1,348 functions, 161 k entries): 62 us a step, 86 unsplit, 181 with a warp per
// entry (i, l) that looks every column up for itself.
__global__ void __launch_bounds__(32 * FOE_WARPS) k_cheb(FoeLaunch a, const double* __restrict__ Htp,
                                                         const double* __restrict__ Tc, const double* __restrict__ Tp,
                                                         double alpha, double* __restrict__ Tn) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 15;
    extern __shared__ int map[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // [FOE_WARPS][chunk]: position in I's row << 16 | position in L's (rows are shorter than 2^16)
    uint32_t* list = reinterpret_cast<uint32_t*>(map + a.n) + warp * a.chunk;
    for (int i = threadIdx.x; i < a.n; i += blockDim.x) map[i] = -1;
    __syncthreads();
    for (int it = blockIdx.x; it < a.ng * a.split; it += gridDim.x) {
        const int L = it / a.split, part = it - L * a.split;       // a share of L's neighbours per CTA
        const int l0 = LD(a.gfirst, L, a.ng + 1), nL = LD(a.gfirst, L + 1, a.ng + 1) - l0;
        const int64_t r0 = LD(a.row_ptr, l0, a.n + 1);
        const int len = static_cast<int>(LD(a.row_ptr, l0 + 1, a.n + 1) - r0);
        for (int q = threadIdx.x; q < len; q += blockDim.x) ST(map, LD(a.col, r0 + q, a.nnz), a.n, q);
        __syncthreads();
        const int t0 = LD(a.nptr, L, a.ng + 1), nt = LD(a.nptr, L + 1, a.ng + 1) - t0;
        for (int t = warp + FOE_WARPS * part; t < nt; t += FOE_WARPS * a.split) {
            const int I = LD(a.ngrp, t0 + t, a.nn), qI = LD(a.npos, t0 + t, a.nn);
            const int i0 = LD(a.gfirst, I, a.ng + 1), nI = LD(a.gfirst, I + 1, a.ng + 1) - i0;
            const int64_t s0 = LD(a.row_ptr, i0, a.n + 1);
            const int lenI = static_cast<int>(LD(a.row_ptr, i0 + 1, a.n + 1) - s0);
            for (int o0 = 0; o0 < nI * nL; o0 += 32) {
                const FoeLanes f(nI * nL, o0, lane);
                const int i = f.o / nL, l = f.o - i * nL;
                const int64_t hrow = s0 + static_cast<int64_t>(i) * lenI, trow = r0 + static_cast<int64_t>(l) * len;
                double acc = 0.0;
                for (int p0 = 0; p0 < lenI; p0 += a.chunk) {
                    int cnt = 0;
                    __syncwarp();                                 // the previous chunk's readers are done
                    for (int p = p0; p < min(p0 + a.chunk, lenI); p += 32) {
                        const int q = p + lane;
                        const int j = q < lenI ? LD(map, LD(a.col, s0 + q, a.nnz), a.n) : -1;
                        const unsigned m = __ballot_sync(0xffffffffu, j >= 0);
                        if (j >= 0) list[cnt + __popc(m & ((1u << lane) - 1))] = static_cast<uint32_t>(q) << 16 | j;
                        cnt += __popc(m);
                    }
                    __syncwarp();
                    if (f.on)
#pragma unroll 8
                        for (int k = f.g; k < cnt; k += f.G) {
                            const uint32_t e = list[k];
                            acc = fma(LD(Htp, hrow + (e >> 16), a.nnz), LD(Tc, trow + (e & 0xffff), a.nnz), acc);
                        }
                }
                acc = f.sum(acc);
                if (f.on && f.g == 0) {
                    const int64_t q = trow + qI + i;
                    ST(Tn, q, a.nnz, alpha * acc - (Tp ? LD(Tp, q, a.nnz) : 0.0));
                }
            }
        }
        __syncthreads();
        for (int q = threadIdx.x; q < len; q += blockDim.x) ST(map, LD(a.col, r0 + q, a.nnz), a.n, -1);
        __syncthreads();
    }
}

__device__ double block_sum_d(double v) {
    __shared__ double part[32];
    v = warp_sum_d(v);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < static_cast<int>(blockDim.x >> 5); ++i) s += part[i];
    return s;
}

// out[b] = sum of the diagonal entries of matrix b (T + b nnz; positions diag[0 .. n))
__global__ void __launch_bounds__(1024) k_traces(const double* __restrict__ T, int64_t nnz, const int64_t* __restrict__ diag,
                                                 int n, double* __restrict__ out) {
    T += blockIdx.x * nnz;
    double v = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) v += T[diag[i]];
    const double s = block_sum_d(v);
    if (threadIdx.x == 0) out[blockIdx.x] = s;
}

// K = c_0/2 I + sum_{j = 1 .. m} c_j T_j (T_j at T + (j - 1) nnz; c on the device), one read of each
__global__ void __launch_bounds__(256) k_kernel_sum(const double* __restrict__ I, const double* __restrict__ T,
                                                    const double* __restrict__ c, int m, int64_t nnz,
                                                    double* __restrict__ K) {
    for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; k < nnz;
         k += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        double v = 0.5 * c[0] * I[k];
#pragma unroll 8
        for (int j = 1; j <= m; ++j) v = fma(c[j], T[(j - 1) * nnz + k], v);
        K[k] = v;
    }
}

__global__ void k_axpy_t(double* __restrict__ K, const double* __restrict__ T, double c, int64_t nnz) {
    for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; k < nnz;
         k += static_cast<int64_t>(gridDim.x) * blockDim.x)
        K[k] += c * T[k];
}

__global__ void k_transpose(const double* __restrict__ src, const int64_t* __restrict__ tpos, double* __restrict__ dst,
                            int64_t nnz) {
    for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; k < nnz;
         k += static_cast<int64_t>(gridDim.x) * blockDim.x)
        dst[k] = src[tpos[k]];
}

// E_BS = sum over pattern entries (i, l) of K_il (Ht_li / sigma + tau S_li): partial sums of the
// CTAs, then k_sum adds them in order
__global__ void __launch_bounds__(256) k_ebs(const double* __restrict__ K, const double* __restrict__ Ht,
                                             const double* __restrict__ S, const int64_t* __restrict__ tpos, int64_t nnz,
                                             double sigma, double tau, double* __restrict__ part) {
    double v = 0.0;
    for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; k < nnz;
         k += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t t = tpos[k];
        v += K[k] * (Ht[t] / sigma + tau * S[t]);
    }
    const double s = block_sum_d(v);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}
__global__ void __launch_bounds__(256) k_sum(const double* __restrict__ part, int n, double* __restrict__ out) {
    double v = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) v += part[i];
    const double s = block_sum_d(v);
    if (threadIdx.x == 0) *out = s;
}

// ---------------------------------------------------------------- host wrappers

cudaError_t configure_foe_kernels(size_t max_smem) {
    cudaError_t e;
    const void* ks[] = {reinterpret_cast<const void*>(k_cheb), reinterpret_cast<const void*>(k_triple_g)};
    for (const void* k : ks) {
        cudaFuncAttributes fa;
        if ((e = cudaFuncGetAttributes(&fa, k)) != cudaSuccess) return e;
        if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      static_cast<int>(max_smem - fa.sharedSizeBytes))) != cudaSuccess)
            return e;
    }
    return cudaSuccess;
}

cudaError_t foe_prep(const FoeLaunch& a, const double* H, const double* S, double sigma, double tau, double* Ht,
                     double* X, cudaStream_t s) {
    k_foe_prep<<<(a.n + 7) / 8, dim3(32, 8), 0, s>>>(H, S, a.row_ptr, a.col, a.n, sigma, tau, Ht, X);
    return cudaGetLastError();
}

cudaError_t foe_triple(const FoeLaunch& a, const double* X, const double* A, double* Y, cudaStream_t s) {
    if (a.triple_smem) k_triple_g<<<a.ng, 32 * FOE_TWARPS, a.triple_smem, s>>>(a, X, A, Y);
    else k_triple<<<a.triple_ctas, 256, 0, s>>>(a, X, A, Y);
    return cudaGetLastError();
}

cudaError_t foe_cheb(const FoeLaunch& a, const double* Htp, const double* Tc, const double* Tp, double alpha, double* Tn,
                     cudaStream_t s) {
    k_cheb<<<a.cheb_ctas, 32 * FOE_WARPS, foe_cheb_smem(a.n, a.chunk), s>>>(a, Htp, Tc, Tp, alpha, Tn);
    return cudaGetLastError();
}

// traces of `count` matrices, nnz values apart
cudaError_t foe_traces(const FoeLaunch& a, const double* T, int count, double* out, cudaStream_t s) {
    k_traces<<<count, 1024, 0, s>>>(T, a.nnz, a.diag, a.n, out);
    return cudaGetLastError();
}

cudaError_t foe_kernel_sum(const FoeLaunch& a, const double* I, const double* T, const double* c, int m, double* K,
                           cudaStream_t s) {
    k_kernel_sum<<<static_cast<unsigned>(std::min<int64_t>((a.nnz + 255) / 256, 8192)), 256, 0, s>>>(I, T, c, m, a.nnz, K);
    return cudaGetLastError();
}

cudaError_t foe_axpy_t(const FoeLaunch& a, double* K, const double* T, double c, cudaStream_t s) {
    k_axpy_t<<<static_cast<unsigned>(std::min<int64_t>((a.nnz + 255) / 256, 8192)), 256, 0, s>>>(K, T, c, a.nnz);
    return cudaGetLastError();
}

cudaError_t foe_transpose(const FoeLaunch& a, const double* src, double* dst, cudaStream_t s) {
    k_transpose<<<static_cast<unsigned>(std::min<int64_t>((a.nnz + 255) / 256, 8192)), 256, 0, s>>>(src, a.tpos, dst, a.nnz);
    return cudaGetLastError();
}

cudaError_t foe_ebs(const FoeLaunch& a, const double* K, const double* Ht, const double* S, double sigma, double tau,
                    double* part, double* out, cudaStream_t s) {
    const int ctas = static_cast<int>(std::min<int64_t>((a.nnz + 255) / 256, FOE_PARTS));
    k_ebs<<<ctas, 256, 0, s>>>(K, Ht, S, a.tpos, a.nnz, sigma, tau, part);
    k_sum<<<1, 256, 0, s>>>(part, ctas, out);
    return cudaGetLastError();
}

}  // namespace lsw
