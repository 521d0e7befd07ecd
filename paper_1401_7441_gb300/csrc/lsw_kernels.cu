// sm_103a kernels of the localized Hamiltonian application and the sparse H/S build.
//
// H phi = L' (T + W^T M^T diag(V) M W) L phi   (Sec. II.A, II.B Eq. phi, III.B)
//
//   k_uncompress  compressed phi on L (segment keys) -> dense 8-type box D (L box)
//   k_fwd_xy      per coarse z plane: synthesis+magic along x then y, i.e. the
//                 combined filters (w*h), (w*g) (u_j = sum_i (w*h)_{j-2i} s_i + ...)
//   k_z           per (x', y') column: the same along z -> real-space u; v = V u
//                 (E_pot += V u^2); then the transposed filters back to coarse z on
//                 the L' box
//   k_kin_z       per (x, y) column of L: kinetic arm along z (T = -1/(2h^2) sum_d
//                 T_{b_d b'_d} along d, Galerkin blocks of the two-level basis) -> G
//   k_bwd_xy      per coarse z plane of L': transposed filters along y then x, plus
//                 the kinetic arms along x and y, plus G; written straight into the
//                 compressed H phi on the members of L'; E_kin partials
// (the sparse S_ab, H_ab build is in lsw_panels.cu)
//
// Density rho = sum_ab K_ab phi_a phi_b on the fine grid (Sec. II.A Eq. density):
//   k_z_dens      the forward half of k_z: real-space values u of every function into
//                 a store (after k_uncompress and k_fwd_xy)
//   k_density     per tile of grid points: sum over chunk pairs of the functions whose
//                 blocks meet the tile of K_ab u_a u_b, FP64 total per point
//
// All kernels are templated on the storage/compute type T (double or float); energy
// and matrix accumulations are FP64.  Device-side checks set bits of a status word
// (never trap).
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "lsw_internal.h"
#include "lsw_device.h"
#include "lsw_tc.h"

namespace lsw {

__constant__ double c_fwd_d[2][FWD_TAPS];
__constant__ float c_fwd_f[2][FWD_TAPS];
__constant__ double c_kin_d[4][KIN_TAPS];
__constant__ float c_kin_f[4][KIN_TAPS];
// Tap pairs for the packed (two-lane) FP32 FMA of the blocks below: the two outputs of a
// block that read the same input element, side by side.
__constant__ float2 c_fwd2_bwd[FWD_TAPS];          // (F_0[m], F_1[m])
__constant__ float2 c_fwd2_up[2][16];              // (F_b[2k], F_b[2k+1]), F_b[31] = 0
__constant__ float2 c_kin2[2][KIN_TAPS];           // (K_0(l), K_2(l)), (K_1(l), K_3(l))

template <class T>
struct Tab;
template <>
struct Tab<double> {
    __device__ static __forceinline__ double fwd(int b, int m) { return c_fwd_d[b][m]; }
    __device__ static __forceinline__ double kin(int k, int l) { return c_kin_d[k][l]; }
};
template <>
struct Tab<float> {
    __device__ static __forceinline__ float fwd(int b, int m) { return c_fwd_f[b][m]; }
    __device__ static __forceinline__ float kin(int k, int l) { return c_kin_f[k][l]; }
};

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

#define FWD(b, m) Tab<T>::fwd(b, m)
#ifdef LSW_CHECKED
#undef FWD
#define FWD(b, m) (((m) >= 0 && (m) < FWD_TAPS) ? Tab<T>::fwd(b, m) : (lsw_report(ST_, KID, __LINE__, (m), FWD_TAPS), T(0)))
#endif

// Element copy global -> shared without a register round trip (cp.async, 4 or 8 bytes):
// a staging loop issues all its copies back to back, so every load of a plane is in
// flight at once; cp_wait() completes this thread's copies (a barrier then publishes
// them to the block).  The checked build copies through the bounds-checked accessors.
#ifdef LSW_CHECKED
#define CPA(dst, di, dn, src, si, sn) ST(dst, di, dn, LD(src, si, sn))
#else
#define CPA(dst, di, dn, src, si, sn) cp_async(&(dst)[di], &(src)[si])
#endif
template <class T>
__device__ __forceinline__ void cp_async(T* dst, const T* src) {
    static_assert(sizeof(T) == 4 || sizeof(T) == 8, "cp.async element of 4 or 8 bytes");
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
    if constexpr (sizeof(T) == 4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// wait until at most N committed groups of this thread's copies are still in flight
template <int N>
__device__ __forceinline__ void cp_wait_group() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }


// Bulk copy global -> shared (both 16-byte aligned, a multiple of 16 bytes) signalled on an
// mbarrier with one arrival: bulk_fence orders earlier shared accesses of the block (behind a
// barrier) before the copy, bulk_expect arrives and announces the bytes.
__device__ __forceinline__ void bulk_fence() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
__device__ __forceinline__ void bulk_expect(uint32_t mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(mbar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mbar)
                 : "memory");
}

// ---------------------------------------------------------------- uncompress / compress

// Bound: the chain of loads ahead of a row's stores (record, rows, segments, values), then DRAM.  An
// atom's functions have the same rows: with `group` functions per grid slot the tables are read
// once for those of one atom (FP32, 6 CTAs an SM): 1.75 -> 1.35 ms for 1,200 atoms of radii 5-8
// bohr, 4.11 -> 2.92 ms for 3,000 dense ones.
template <class T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 6 : 4) k_uncompress(HphiLaunch a, int group) {
    // Warp per (y, z) row of the L box: writes all 8 types of the row, the members' values
    // from the compressed phi (one coarse segment per row of the sphere, a few fine
    // segments) and zero elsewhere, so the box needs no separate clearing.
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = blockIdx.x * (blockDim.x >> 5) + warp;
    const int fe = min(static_cast<int>(blockIdx.y + 1) * group, a.nfn);
    for (int f = blockIdx.y * group; f < fe;) {
        const int atom = a.fn[f].atom, first = f;
        do {
            ++f;
        } while (f < fe && a.fn[f].atom == atom);
        const FnRec& r = a.fn[first];
        const AtomRec& at = a.atoms[atom];
        const int nx = r.n[0], nrows = r.n[1] * r.n[2];
        if (row >= nrows) continue;
        const int64_t plane = static_cast<int64_t>(nx) * nrows;
        const int c0 = LD(a.rowptr, at.rowLc + row, a.rowptr_n), c1 = LD(a.rowptr, at.rowLc + row + 1, a.rowptr_n);
        const int f0 = LD(a.rowptr, at.rowLf + row, a.rowptr_n), f1 = LD(a.rowptr, at.rowLf + row + 1, a.rowptr_n);
        Seg cs{};
        cs.x0 = 1;
        cs.x1 = 0;                                     // empty unless the row has members
        if (c1 > c0) {
            cs = LD(a.seg, at.segLc + c0, a.seg_n);
            if (c1 - c0 > 1 || cs.x0 < 0 || cs.x1 >= nx || cs.row != row) {
                if (lane == 0) atomicOr(a.status, ST_BAD_SEG);
                continue;
            }
        }
        for (int x = lane; x < nx; x += 32) {
            // wavelet types: the fine segment of this row holding x, if any
            int64_t fo = -1;
            for (int q = f0; q < f1; ++q) {
                const Seg fs = LD(a.seg, at.segLf + q, a.seg_n);
                if (x >= fs.x0 && x <= fs.x1) fo = fs.off + (x - fs.x0);
            }
            for (int k = first; k < f; ++k) {
                T* D = static_cast<T*>(a.ws) + a.fn[k].ws_D + static_cast<int64_t>(row) * nx;
                const T* phi = static_cast<const T*>(a.phi) + a.fn[k].off_phi;
                const int64_t phi_room = a.phi_n - a.fn[k].off_phi;
                T v[8];
                v[0] = x >= cs.x0 && x <= cs.x1 ? LD(phi, cs.off + (x - cs.x0), phi_room) : T(0);
#pragma unroll
                for (int t = 1; t < 8; ++t)
                    v[t] = fo >= 0 ? LD(phi, at.ncL + static_cast<int64_t>(t - 1) * at.nfL + fo, phi_room) : T(0);
#pragma unroll
                for (int t = 0; t < 8; ++t) ST(D, t * plane + x, 8 * plane - static_cast<int64_t>(row) * nx, v[t]);
            }
        }
    }
}

// Division by a loop-invariant divisor d (1 <= d < 2^16) for dividends n < 2^16:
// q = umulhi(n, ceil(2^32 / d)) is exact there (the error term n / 2^32 < 2^-16 cannot
// reach the next integer).  Replaces the ~20-instruction integer division in index math.
struct FastDiv {
    uint32_t m;
    int d;
    __device__ __forceinline__ explicit FastDiv(int dd) : m(dd > 1 ? 0xFFFFFFFFu / static_cast<uint32_t>(dd) + 1u : 0u), d(dd) {}
    __device__ __forceinline__ int div(int n) const {
        return d > 1 ? static_cast<int>(__umulhi(static_cast<uint32_t>(n), m)) : n;
    }
};

// ---------------------------------------------------------------- register-blocked 1D blocks
//
// Forward (synthesis + magic filter, upsampling by 2): u[2p+e] = sum_{k} F_b[2k+e] in_b[p-k],
// k = 0..15 (e = 0) or 0..14 (e = 1), summed over the two input types b (s and d).  A
// block produces the 8 outputs 2p0 .. 2p0+7 from the window in_b[p0-15 .. p0+3] (19
// values per type) held in registers; taps are compile-time immediates.
constexpr int FB = 4;                 // coarse steps per forward block (8 outputs)
constexpr int FW = FB + 15;           // forward window
constexpr int BB = 4;                 // outputs per kinetic block
constexpr int KW = BB + 2 * KIN_HALF; // kinetic window
#ifndef LSW_Z_NB
#define LSW_Z_NB 4                    // outputs per backward block in the z stage (FP32)
#endif
template <class T, int Stage>         // Stage 0: z stage, 1: backward plane kernel
struct Blk {                          // outputs per backward (decimating) block
    static constexpr int NB = sizeof(T) == 4 ? (Stage == 0 ? LSW_Z_NB : BWD_NB_F32) : BWD_NB_F64;
    static constexpr int W = 2 * NB + 29;
};
template <class T>
struct ZCols { static constexpr int C = sizeof(T) == 8 ? ZCOLS_F64 : ZCOLS_F32; };

// Window w[i] = p[off + (first + i) * stride] for positions first + i in [0, n), 0 outside.
// When the whole window is inside (the common, warp-uniform case) the loads carry no
// bounds test.
#ifdef LSW_CHECKED
#define WLD(p, i, room) ld_chk(p, static_cast<int64_t>(i), static_cast<int64_t>(room), st, 11, __LINE__)
#else
#define WLD(p, i, room) ((p)[i])
#endif
template <int N, class T>
__device__ __forceinline__ void win(T (&w)[N], const T* p, int64_t off, int stride, int first, int n,
                                    [[maybe_unused]] int64_t room, [[maybe_unused]] int* st) {
    if (first >= 0 && first + N <= n) {
        const T* q = p + off + static_cast<int64_t>(first) * stride;
#pragma unroll
        for (int i = 0; i < N; ++i) w[i] = WLD(q, static_cast<int64_t>(i) * stride, room - off - static_cast<int64_t>(first) * stride);
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int pos = first + i;
            w[i] = (pos >= 0 && pos < n) ? WLD(p, off + static_cast<int64_t>(pos) * stride, room) : T(0);
        }
    }
}

// The same for a window in shared memory, with 32-bit offsets (shared addresses are
// 32-bit; keeping the index math in int lets loads fold their offsets).
template <int N, class T>
__device__ __forceinline__ void swin(T (&w)[N], const T* p, int off, int stride, int first, int n,
                                     [[maybe_unused]] int64_t room, [[maybe_unused]] int* st) {
    if (first >= 0 && first + N <= n) {
        const int b = off + first * stride;
#pragma unroll
        for (int i = 0; i < N; ++i) w[i] = WLD(p, b + i * stride, room);
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int pos = first + i;
            w[i] = (pos >= 0 && pos < n) ? WLD(p, off + pos * stride, room) : T(0);
        }
    }
}

template <class T>
__device__ __forceinline__ void fwd_block(const T (&w0)[FW], const T (&w1)[FW], T (&u)[2 * FB]) {
#pragma unroll
    for (int j = 0; j < FB; ++j) {
        T ue = 0, uo = 0;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            ue += Tab<T>::fwd(0, 2 * k) * w0[j + 15 - k];
            ue += Tab<T>::fwd(1, 2 * k) * w1[j + 15 - k];
            if (k < 15) {
                uo += Tab<T>::fwd(0, 2 * k + 1) * w0[j + 15 - k];
                uo += Tab<T>::fwd(1, 2 * k + 1) * w1[j + 15 - k];
            }
        }
        u[2 * j] = ue;
        u[2 * j + 1] = uo;
    }
}

// Backward (transposed filters, decimation by 2): s_j = sum_m F_0[m] v[2j+m],
// d_j = sum_m F_1[m] v[2j+m], m = 0..30, from the window v[0 .. 2*NB+28].
template <class T, int NB>
__device__ __forceinline__ void bwd_block(const T (&w)[2 * NB + 29], T (&s)[NB], T (&d)[NB]) {
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        T a0 = 0, a1 = 0;
#pragma unroll
        for (int m = 0; m < FWD_TAPS; ++m) {
            a0 += Tab<T>::fwd(0, m) * w[2 * j + m];
            a1 += Tab<T>::fwd(1, m) * w[2 * j + m];
        }
        s[j] = a0;
        d[j] = a1;
    }
}

// Kinetic arm along one axis for the two types of a pair differing in that axis' bit:
// out_o[j] += sum_l K_{o,0}(l) in_0[j+14+l] + K_{o,1}(l) in_1[j+14+l], o = 0, 1.
template <class T>
__device__ __forceinline__ void kin_block(const T (&k0)[KW], const T (&k1)[KW], T (&o0)[BB], T (&o1)[BB]) {
#pragma unroll
    for (int j = 0; j < BB; ++j) {
        T a0 = 0, a1 = 0;
#pragma unroll
        for (int l = 0; l < KIN_TAPS; ++l) {
            a0 += Tab<T>::kin(0, l) * k0[j + l];
            a0 += Tab<T>::kin(1, l) * k1[j + l];
            a1 += Tab<T>::kin(2, l) * k0[j + l];
            a1 += Tab<T>::kin(3, l) * k1[j + l];
        }
        o0[j] = a0;
        o1[j] = a1;
    }
}

// FP32 versions on the packed two-lane FMA (__ffma2_rn: each lane one FMA rounded to
// nearest, so every accumulator sees the same operations in the same order as above and
// the results are the same bits).  The two lanes are the two outputs of a block that read
// the same input element.
#ifndef LSW_FFMA2
#define LSW_FFMA2 1
#endif
#if LSW_FFMA2
template <>
__device__ __forceinline__ void fwd_block<float>(const float (&w0)[FW], const float (&w1)[FW], float (&u)[2 * FB]) {
#pragma unroll
    for (int j = 0; j < FB; ++j) {
        float2 acc = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const float a = w0[j + 15 - k], b = w1[j + 15 - k];
            acc = __ffma2_rn(c_fwd2_up[0][k], make_float2(a, a), acc);
            acc = __ffma2_rn(c_fwd2_up[1][k], make_float2(b, b), acc);
        }
        u[2 * j] = acc.x;
        u[2 * j + 1] = acc.y;
    }
}
// The tap loop outside, the NB independent accumulators inside: each accumulator sees the
// same operations in the same order (same bits), and consecutive instructions belong to
// different dependency chains.
template <int NB>
__device__ __forceinline__ void bwd_block_f2(const float (&w)[2 * NB + 29], float (&s)[NB], float (&d)[NB]) {
    float2 acc[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) acc[j] = make_float2(0.f, 0.f);
#pragma unroll
    for (int m = 0; m < FWD_TAPS; ++m) {
        const float2 t = c_fwd2_bwd[m];
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            const float a = w[2 * j + m];
            acc[j] = __ffma2_rn(t, make_float2(a, a), acc[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        s[j] = acc[j].x;
        d[j] = acc[j].y;
    }
}
template <>
__device__ __forceinline__ void bwd_block<float, 4>(const float (&w)[37], float (&s)[4], float (&d)[4]) {
    bwd_block_f2<4>(w, s, d);
}
template <>
__device__ __forceinline__ void bwd_block<float, 8>(const float (&w)[45], float (&s)[8], float (&d)[8]) {
    bwd_block_f2<8>(w, s, d);
}
template <>
__device__ __forceinline__ void kin_block<float>(const float (&k0)[KW], const float (&k1)[KW], float (&o0)[BB],
                                                 float (&o1)[BB]) {
    float2 acc[BB];
#pragma unroll
    for (int j = 0; j < BB; ++j) acc[j] = make_float2(0.f, 0.f);
#pragma unroll
    for (int l = 0; l < KIN_TAPS; ++l) {
        const float2 t0 = c_kin2[0][l], t1 = c_kin2[1][l];
#pragma unroll
        for (int j = 0; j < BB; ++j) {
            const float a = k0[j + l], b = k1[j + l];
            acc[j] = __ffma2_rn(t0, make_float2(a, a), acc[j]);
            acc[j] = __ffma2_rn(t1, make_float2(b, b), acc[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < BB; ++j) {
        o0[j] = acc[j].x;
        o1[j] = acc[j].y;
    }
}
#endif

// FP64 forms (bound by the FP64 pipe, 1/64 of the FP32 rate): products only where the input can
// be nonzero, decided position by position.  8 outputs of the upsampling block at coarse step
// q0 + 15 from the inputs ld(b, q), q within [l0, h0] for the first type, [l1, h1] for the second.
template <class T, class Ld>
__device__ __forceinline__ void fwd_range(T (&u)[2 * FB], Ld ld, int q0, int l0, int h0, int l1, int h1) {
#pragma unroll
    for (int k = 0; k < 2 * FB; ++k) u[k] = T(0);
#pragma unroll
    for (int i = 0; i < FW; ++i) {
        const int q = q0 + i;
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            if (q < (b ? l1 : l0) || q > (b ? h1 : h0)) continue;
            const T v = ld(b, q);
#pragma unroll
            for (int j = 0; j < FB; ++j) {
                const int k = j + 15 - i;
                if (k < 0 || k > 15) continue;
                u[2 * j] += Tab<T>::fwd(b, 2 * k) * v;
                if (k < 15) u[2 * j + 1] += Tab<T>::fwd(b, 2 * k + 1) * v;
            }
        }
    }
}

// The transposed filters of N coarse outputs from the window starting at position `first` of a
// line of n values.  FP32: as bwd_block.  FP64 (bound by the FP64 pipe): positions outside the
// line are skipped, not multiplied as zeros.
template <class T, int NB>
__device__ __forceinline__ void bwd_window(const T* p, int off, int stride, int first, int n, T (&s)[NB], T (&d)[NB],
                                           int64_t room, int* st) {
    if constexpr (sizeof(T) == 4) {
        T w[2 * NB + 29];
        swin(w, p, off, stride, first, n, room, st);
        bwd_block<T, NB>(w, s, d);
    } else {
#pragma unroll
        for (int j = 0; j < NB; ++j) s[j] = d[j] = T(0);
#pragma unroll
        for (int m = 0; m < 2 * NB + 29; ++m) {
            const int pos = first + m;
            if (pos < 0 || pos >= n) continue;
            const T v = WLD(p, off + pos * stride, room);
#pragma unroll
            for (int j = 0; j < NB; ++j)
                if (m - 2 * j >= 0 && m - 2 * j < FWD_TAPS) {
                    s[j] += Tab<T>::fwd(0, m - 2 * j) * v;
                    d[j] += Tab<T>::fwd(1, m - 2 * j) * v;
                }
        }
    }
}

// ---------------------------------------------------------------- forward x, y

template <class T>
__device__ __forceinline__ void fwd_plane(const HphiLaunch& a, int fl, int z, int bz) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 2;
    int* st = a.status;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    const FnRec r = a.fn[fl];
    if (z >= r.n[2]) return;
    const int nx = r.n[0], ny = r.n[1], nz = r.n[2];
    const int X = 2 * nx + 29, Y = 2 * ny + 29;
    const int RS = nx | 1;                   // odd row stride: rows land in different banks
    T* in = sm;                              // [4][ny][RS], type tb = bx + 2 by
    T* mid = sm + 4 * ny * RS;               // [2][ny][X]
    const int64_t smem_n = static_cast<int64_t>(a.smem_fwd / sizeof(T));
    const int64_t mid_n = smem_n - 4 * ny * RS;
    const T* D = static_cast<const T*>(a.ws) + r.ws_D;
    const int64_t plane = static_cast<int64_t>(nx) * ny * nz;
    const int pn = nx * ny;
    {
        const FastDiv fd_pn(pn), fd_nx(nx);
        for (int i = threadIdx.x; i < 4 * pn; i += blockDim.x) {
            const int tb = fd_pn.div(i), rem = i - tb * pn;
            const int y = fd_nx.div(rem), x = rem - y * nx;
            CPA(in, (tb * ny + y) * RS + x, smem_n, D, (tb + 4 * bz) * plane + static_cast<int64_t>(z) * pn + rem,
                8 * plane);
        }
    }
    // x pass work list.  Row (by, y) holds the types (bz, by, 0), (bz, by, 1) of D, which are
    // zero off L's members in the row: the coarse segment where the pair holds type 0
    // (bz = 0, by = 0), else the fine segments.  Block blk (inputs x = 4 blk - 15 ..
    // 4 blk + 3) is computed for the rows whose nonzero range meets its window; per (by,
    // blk) the hull of those rows is listed (block-major, consecutive rows on consecutive
    // threads), and the rest of mid is zero.
    const int nbx = (nx + 15 + FB - 1) / FB;
    __shared__ int16_t ix0[2][256], ix1[2][256];
    __shared__ int hlo[128], hhi[128], hp[129];
    const bool listed = a.fwd_list && 2 * nbx <= 128 && ny <= 256;   // else every (row, block)
    if (listed) {
        const AtomRec& at = a.atoms[r.atom];
        for (int y = threadIdx.x; y < ny; y += blockDim.x) {
            const int64_t crow = at.rowLc + y + static_cast<int64_t>(ny) * z;
            const int64_t frow = at.rowLf + y + static_cast<int64_t>(ny) * z;
            const int c0 = LD(a.rowptr, crow, a.rowptr_n), c1 = LD(a.rowptr, crow + 1, a.rowptr_n);
            const int q0 = LD(a.rowptr, frow, a.rowptr_n), q1 = LD(a.rowptr, frow + 1, a.rowptr_n);
            const int cx0 = c1 > c0 ? LD(a.seg, at.segLc + c0, a.seg_n).x0 : -1;
            const int cx1 = c1 > c0 ? LD(a.seg, at.segLc + c1 - 1, a.seg_n).x1 : -1;
            const int fx0 = q1 > q0 ? LD(a.seg, at.segLf + q0, a.seg_n).x0 : -1;
            const int fx1 = q1 > q0 ? LD(a.seg, at.segLf + q1 - 1, a.seg_n).x1 : -1;
            ix0[0][y] = static_cast<int16_t>(bz == 0 ? cx0 : fx0);
            ix1[0][y] = static_cast<int16_t>(bz == 0 ? cx1 : fx1);
            ix0[1][y] = static_cast<int16_t>(fx0);
            ix1[1][y] = static_cast<int16_t>(fx1);
        }
        for (int e = threadIdx.x; e < 2 * nbx; e += blockDim.x) {
            hlo[e] = ny;
            hhi[e] = -1;
        }
        for (int i = threadIdx.x; i < 2 * ny * X; i += blockDim.x) ST(mid, i, mid_n, T(0));
    }
    __syncthreads();
    if (listed) {
        for (int row = threadIdx.x; row < 2 * ny; row += blockDim.x) {
            const int by = row >= ny, y = row - by * ny;
            const int x0 = ix0[by][y];
            if (x0 < 0) continue;
            const int k1 = min(nbx - 1, (ix1[by][y] + 15) / FB);
            for (int k = x0 / FB; k <= k1; ++k) {
                atomicMin(&hlo[by * nbx + k], y);
                atomicMax(&hhi[by * nbx + k], y);
            }
        }
    }
    cp_wait();
    __syncthreads();
    if (listed && threadIdx.x == 0) {
        hp[0] = 0;
        for (int e = 0; e < 2 * nbx; ++e) hp[e + 1] = hp[e] + max(0, hhi[e] - hlo[e] + 1);
    }
    __syncthreads();
    // x pass: rows (by, y), blocks of 8 outputs along x'
    {
        const FastDiv fd_2ny(2 * ny), fd_ny(ny);
        const int ntk = listed ? hp[2 * nbx] : 2 * ny * nbx;
        for (int task = threadIdx.x; task < ntk; task += blockDim.x) {
            int by, y, blk;
            if (listed) {
                int lo = 0, hi = 2 * nbx - 1;              // the entry e with hp[e] <= task < hp[e + 1]
                while (lo < hi) {
                    const int m = (lo + hi + 1) >> 1;
                    if (hp[m] <= task) lo = m;
                    else hi = m - 1;
                }
                by = lo >= nbx;
                blk = lo - by * nbx;
                y = hlo[lo] + (task - hp[lo]);
            } else {
                blk = fd_2ny.div(task);
                const int rw = task - blk * 2 * ny;
                by = fd_ny.div(rw);
                y = rw - by * ny;
            }
            const int row = by * ny + y;
            const int p0 = blk * FB;
            const int s0 = ((2 * by) * ny + y) * RS, d0 = s0 + ny * RS;
            T u[2 * FB];
            if constexpr (sizeof(T) == 4) {
                T w0[FW], w1[FW];
                swin(w0, in, s0, 1, p0 - 15, nx, smem_n, st);
                swin(w1, in, d0, 1, p0 - 15, nx, smem_n, st);
                fwd_block(w0, w1, u);
            } else {
                // the row's members where they are listed (of both types: the second's are fine)
                const int l0 = listed ? ix0[by][y] : 0, h0 = listed ? ix1[by][y] : nx - 1;
                const int l1 = listed ? ix0[1][y] : 0, h1 = listed ? ix1[1][y] : nx - 1;
                fwd_range<T>(u, [&](int b, int q) { return LD(in, (b ? d0 : s0) + q, smem_n); }, p0 - 15, max(l0, 0),
                             l0 < 0 ? -1 : h0, max(l1, 0), l1 < 0 ? -1 : h1);
            }
#pragma unroll
            for (int k = 0; k < 2 * FB; ++k) {
                const int xo = 2 * p0 + k;
                if (xo < X) ST(mid, row * X + xo, mid_n, u[k]);
            }
        }
    }
    // rows with members, per y type (FP64: the y pass sums over them)
    [[maybe_unused]] __shared__ int yh[4];
    if constexpr (sizeof(T) == 8) {
        if (threadIdx.x < 2) {
            int lo = 0, hi = ny - 1;
            if (listed) {
                lo = ny;
                hi = -1;
                for (int y = 0; y < ny; ++y)
                    if (ix0[threadIdx.x][y] >= 0) {
                        lo = min(lo, y);
                        hi = y;
                    }
            }
            yh[2 * threadIdx.x] = lo;
            yh[2 * threadIdx.x + 1] = hi;
        }
    }
    __syncthreads();
    // y pass: columns x', blocks of 8 outputs along y'
    T* Bf = static_cast<T*>(a.ws) + r.ws_Bf + (static_cast<int64_t>(bz) * nz + z) * Y * X;
    const int64_t bf_room = 2LL * nz * Y * X - (static_cast<int64_t>(bz) * nz + z) * Y * X;
    const int nby = (ny + 15 + FB - 1) / FB;
    const FastDiv fd_X(X);
    for (int task = threadIdx.x; task < X * nby; task += blockDim.x) {
        const int blk = fd_X.div(task), xo = task - blk * X;
        const int p0 = blk * FB;
        T u[2 * FB];
        if constexpr (sizeof(T) == 4) {
            T w0[FW], w1[FW];
            swin(w0, mid, xo, X, p0 - 15, ny, mid_n, st);
            swin(w1, mid, ny * X + xo, X, p0 - 15, ny, mid_n, st);
            fwd_block(w0, w1, u);
        } else {
            fwd_range<T>(u, [&](int b, int q) { return LD(mid, (b * ny + q) * X + xo, mid_n); }, p0 - 15, yh[0], yh[1], yh[2],
                         yh[3]);
        }
#pragma unroll
        for (int k = 0; k < 2 * FB; ++k) {
            const int yo = 2 * p0 + k;
            if (yo < Y) ST(Bf, static_cast<int64_t>(yo) * X + xo, bf_room, u[k]);
        }
    }
}

// Item k of a persistent plane kernel: the next index of the queue counter (one atomic per
// CTA, broadcast through shared memory), so CTAs take the batch's planes largest first
// as they free up.  The caller's next barrier orders the read before the next write.
__device__ __forceinline__ int next_item(int* counter, int* s_item) {
    if (threadIdx.x == 0) *s_item = atomicAdd(counter, 1);
    __syncthreads();
    return *s_item;
}

// Persistent form (a.items_fwd set): a grid of as many CTAs as fit on the GPU loops over
// the batch's (function, z plane, z type) items; otherwise one CTA per grid slot
// (blockIdx.x = 2 z + b_z, blockIdx.y = function).
template <class T>
__global__ void __launch_bounds__(256) k_fwd_xy(HphiLaunch a) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 2;
    if (a.items_fwd) {
        __shared__ int s_item;
        for (;;) {
            const int k = next_item(a.queue, &s_item);
            if (k >= a.n_items_fwd) break;
            const int2 it = LD(a.items_fwd, k, a.n_items_fwd);
            fwd_plane<T>(a, it.x, (it.y >> 1) & 1023, it.y & 1);
            __syncthreads();   // shared memory and s_item are reused by the next item
        }
    } else {
        fwd_plane<T>(a, blockIdx.y, blockIdx.x >> 1, blockIdx.x & 1);
    }
}

// ---------------------------------------------------------------- z stage with V

// One thread per real-space column (x', y'): 8 outputs u of the synthesis + magic filter at a
// time from the column's coefficients, times V, then the transposed filters back.  The column
// lives in one shared buffer of 2 n_z + 30 slots per thread: input (b, q) starts in slot
// 30 + 2 q + b, and the block of outputs 2 p0 .. 2 p0 + 7 overwrites slots that no later block
// reads (the next one starts at input p0 - 11, slot 2 p0 + 8).  With the inputs and the
// products in buffers of their own, shared memory held 8 warps per SM and the kernel waited on
// its own latencies (issue 54 %): 3.0 -> 2.4 us per function at radii 5-8 bohr.  V is fetched a
// block ahead into registers.
// FP64 (bound by the FP64 pipe): products run over the hull of the warp's nonzero inputs, per
// type, and within the column, not over zeros: 82 -> 53 us per function at 6 bohr.
constexpr int Z_HEAD = 30;            // slots ahead of the inputs
template <class T>
__global__ void __launch_bounds__(ZCols<T>::C) k_z(HphiLaunch a) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 3;
    constexpr int NB = Blk<T, 0>::NB;
    constexpr int W = Blk<T, 0>::W;
    constexpr int C = ZCols<T>::C;       // columns per block = threads; a compile-time
                                         // stride turns window offsets into immediates
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);   // [2 nz + 30][C] (each thread owns its column)
    const FnRec r = a.fn[blockIdx.y];
    const int nx = r.n[0], ny = r.n[1], nz = r.n[2];
    const int X = 2 * nx + 29, Y = 2 * ny + 29, Z = 2 * nz + 29;
    const int cols = X * Y;
    const int c = blockIdx.x * C + threadIdx.x;
    if (blockIdx.x * C >= cols) return;
    const bool valid = c < cols;
    const int t = threadIdx.x;
    [[maybe_unused]] const int64_t smem_n = static_cast<int64_t>(a.smem_z / sizeof(T));
    const T* Bf = static_cast<const T*>(a.ws) + r.ws_Bf;
    T epot_t = 0;   // per-thread partial in the kernel's precision (no FP64 in FP32 loops)
    int hl[2] = {0, 0}, hh[2] = {nz - 1, nz - 1};
    if (valid)
        for (int q = 0; q < nz; ++q)
#pragma unroll
            for (int b = 0; b < 2; ++b)
                CPA(sm, (Z_HEAD + 2 * q + b) * C + t, smem_n, Bf, static_cast<int64_t>(b * nz + q) * cols + c, 2LL * nz * cols);
    cp_wait();   // each thread reads only its own column: no barrier needed
    if constexpr (sizeof(T) == 8) {
        const unsigned all = __ballot_sync(0xffffffffu, valid);
        if (valid)
            for (int b = 0; b < 2; ++b) {
                hl[b] = nz;
                hh[b] = -1;
                for (int q = 0; q < nz; ++q)
                    if (__any_sync(all, (__double_as_longlong(LD(sm, (Z_HEAD + 2 * q + b) * C + t, smem_n)) << 1) != 0)) {
                        hl[b] = min(hl[b], q);
                        hh[b] = q;
                    }
            }
    }
    if (valid) {
        const int xo = c % X, yo = c / X;
        const int64_t jx = 2LL * r.lo[0] - V_REACH + xo - a.vlo[0];
        const int64_t jy = 2LL * r.lo[1] - V_REACH + yo - a.vlo[1];
        const int64_t jz0 = 2LL * r.lo[2] - V_REACH - a.vlo[2];
        const T* V = static_cast<const T*>(a.V);
        const int64_t vstride = a.vn[0] * a.vn[1];
        const int64_t v0 = jz0 * vstride + jy * a.vn[0] + jx;
        T vn[2 * FB];
#pragma unroll
        for (int k = 0; k < 2 * FB; ++k) vn[k] = k < Z ? LD(V, v0 + k * vstride, a.v_n) : T(0);
        for (int p0 = 0; 2 * p0 < Z; p0 += FB) {
            T u[2 * FB], vv[2 * FB];
            const int q0 = p0 - 15;
#pragma unroll
            for (int k = 0; k < 2 * FB; ++k) {
                vv[k] = vn[k];
                const int zo = 2 * (p0 + FB) + k;
                if (zo < Z) vn[k] = LD(V, v0 + zo * vstride, a.v_n);
            }
            if constexpr (sizeof(T) == 4) {
                T w0[FW], w1[FW];
                if (q0 >= 0 && q0 + FW <= nz) {
#pragma unroll
                    for (int i = 0; i < FW; ++i) {
                        w0[i] = LD(sm, (Z_HEAD + 2 * (q0 + i)) * C + t, smem_n);
                        w1[i] = LD(sm, (Z_HEAD + 2 * (q0 + i) + 1) * C + t, smem_n);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < FW; ++i) {
                        const int q = q0 + i;
                        const bool ok = q >= 0 && q < nz;
                        w0[i] = ok ? LD(sm, (Z_HEAD + 2 * q) * C + t, smem_n) : T(0);
                        w1[i] = ok ? LD(sm, (Z_HEAD + 2 * q + 1) * C + t, smem_n) : T(0);
                    }
                }
                fwd_block(w0, w1, u);
            } else {
                fwd_range<T>(u, [&](int b, int q) { return LD(sm, (Z_HEAD + 2 * q + b) * C + t, smem_n); }, q0, hl[0], hh[0],
                             hl[1], hh[1]);
            }
#pragma unroll
            for (int k = 0; k < 2 * FB; ++k) {
                const int zo = 2 * p0 + k;
                if (zo < Z) {
                    const T v = vv[k] * u[k];
                    epot_t += v * u[k];
                    ST(sm, zo * C + t, smem_n, v);
                }
            }
        }
        const int nzp = r.np[2];
        const int dz = r.lop[2] - r.lo[2];
        T* Bb = static_cast<T*>(a.ws) + r.ws_Bb;
        for (int b0 = 0; b0 < nzp; b0 += NB) {
            T s[NB], d[NB];
            const int z0 = 2 * (b0 + dz);
            if constexpr (sizeof(T) == 4) {
                T w[W];
                if (z0 >= 0 && z0 + W <= Z) {
#pragma unroll
                    for (int i = 0; i < W; ++i) w[i] = LD(sm, (z0 + i) * C + t, smem_n);
                } else {
#pragma unroll
                    for (int i = 0; i < W; ++i) {
                        const int zo = z0 + i;
                        w[i] = (zo >= 0 && zo < Z) ? LD(sm, zo * C + t, smem_n) : T(0);
                    }
                }
                bwd_block<T, NB>(w, s, d);
            } else {
                bwd_window<T, NB>(sm, t, C, z0, Z, s, d, smem_n, a.status);
            }
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                const int b = b0 + j;
                if (b < nzp) {
                    ST(Bb, static_cast<int64_t>(b) * cols + c, 2LL * nzp * cols, s[j]);
                    ST(Bb, static_cast<int64_t>(nzp + b) * cols + c, 2LL * nzp * cols, d[j]);
                }
            }
        }
    }
    const double epot = warp_sum(static_cast<double>(epot_t));
    if ((threadIdx.x & 31) == 0 && epot != 0.0) atomicAdd(a.e_pot + r.f, epot);
}

// ---------------------------------------------------------------- density: real-space values

// The forward half of k_z for the density (Eq. density): per (x', y') column, synthesis +
// magic filter along z, and the real-space values u written to the function's block of
// the density store (no potential, no backward pass).
template <class T>
__global__ void __launch_bounds__(ZCols<T>::C) k_z_dens(HphiLaunch a) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 12;
    constexpr int C = ZCols<T>::C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* cin = reinterpret_cast<T*>(smem_raw);   // [2][nz][C] (each thread owns its column)
    const FnRec r = a.fn[blockIdx.y];
    const int nx = r.n[0], ny = r.n[1], nz = r.n[2];
    const int X = 2 * nx + 29, Y = 2 * ny + 29, Z = 2 * nz + 29;
    const int cols = X * Y;
    const int c = blockIdx.x * C + threadIdx.x;
    if (c >= cols) return;   // no barrier below: threads leave independently
    const int t = threadIdx.x;
    [[maybe_unused]] const int64_t smem_n = static_cast<int64_t>(a.smem_z / sizeof(T));
    const T* Bf = static_cast<const T*>(a.ws) + r.ws_Bf;
    const DensFn df = a.dfn[r.f];
    T* U = static_cast<T*>(a.U) + df.off;
    [[maybe_unused]] const int64_t room = a.U_n - df.off;
    for (int q = 0; q < 2 * nz; ++q)
        CPA(cin, q * C + t, smem_n, Bf, static_cast<int64_t>(q) * cols + c, 2LL * nz * cols);
    cp_wait();
    for (int p0 = 0; 2 * p0 < Z; p0 += FB) {
        T w0[FW], w1[FW], u[2 * FB];
        const int q0 = p0 - 15;
#pragma unroll
        for (int i = 0; i < FW; ++i) {
            const int q = q0 + i;
            const bool ok = q >= 0 && q < nz;
            w0[i] = ok ? LD(cin, q * C + t, smem_n) : T(0);
            w1[i] = ok ? LD(cin, (nz + q) * C + t, smem_n) : T(0);
        }
        fwd_block(w0, w1, u);
#pragma unroll
        for (int k = 0; k < 2 * FB; ++k) {
            const int zo = 2 * p0 + k;
            if (zo < Z) ST(U, static_cast<int64_t>(zo) * cols + c, room, u[k]);
        }
    }
}

// ---------------------------------------------------------------- z stage on tensor cores
//
// The z stage of k_z cast as two band-Toeplitz products per tile of 128 real-space
// columns c (the MMA rows, M = 128), with the filter matrices as the N x K operand:
//   U[c][o]  = sum_k A1[c][k] F1[o][k],   k = b nz + q,      F1[o][k] = F_b[o - 2q]
//   v[c][o]  = V(o, c) U[c][o]            (E_pot += v U)
//   Bb[c][j] = sum_o v[c][o] F2[j][o],    j = b' nz' + b,     F2[j][o] = F_b'[o - 2(b + dz)]
// F_b are the combined synthesis + magic filters (w*h), (w*g) of k_z.  Every FP32
// operand x is split into NS bfloat16 parts x = x_0 + x_1 (+ x_2) (each part the
// rounding of what the previous ones leave); the products of parts whose orders add up
// to at most NS - 1 are accumulated in FP32 in tensor memory: NS = 2 takes 3 products
// (relative error of a product about 2^-17), NS = 3 takes 6 (about 2^-24).
//
// One CTA of 8 warps loops over tiles of one function.  Warp w reads tensor-memory
// lanes 32 (w mod 4) .. + 31 (the hardware's lane quarters), so thread (w, lane) owns
// column 32 (w mod 4) + lane of the tile and half w / 4 of each K or N range.  Per tile:
// inputs (prefetched into registers during the previous tile) -> bfloat16 parts in
// shared memory; V of the tile -> shared memory by cp.async; forward MMAs; U from
// tensor memory -> v -> parts; backward MMAs; result from tensor memory -> Bb.  Waits on
// MMA completion are bounded (about 1 s) and end in a status bit, never a hang.

// (the tcgen05 helpers, namespace tc, are in lsw_tc.h)

// Dynamic shared memory of k_z_tc for a function with L extent nz, L' extent nzp
// (host mirror in lsw_host.cpp: ztc_smem).
template <int NS>
__global__ void __launch_bounds__(256, 1) k_z_tc(HphiLaunch a) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 8;
    using tc::TILE;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const FnRec r = a.fn[blockIdx.y];
    const int nx = r.n[0], ny = r.n[1], nz = r.n[2];
    const int X = 2 * nx + 29, Y = 2 * ny + 29, Z = 2 * nz + 29;
    const int cols = X * Y;
    const int ntiles = (cols + TILE - 1) / TILE;
    if (static_cast<int>(blockIdx.x) >= ntiles) return;   // uniform over the CTA
    const int nzp = r.np[2], dz = r.lop[2] - r.lo[2];
    const int K1 = (2 * nz + 15) & ~15, N1 = (Z + 15) & ~15, K2 = N1, N2 = (2 * nzp + 15) & ~15;
    const int KA = max(K1, K2);
    const int A_PART = TILE * KA * 2, B1_PART = N1 * K1 * 2, B2_PART = N2 * K2 * 2;
    unsigned char* sA = smem_raw + tc::HEAD;
    unsigned char* sB1 = sA + NS * A_PART;
    unsigned char* sB2 = sB1 + NS * B1_PART;
    float* sV = reinterpret_cast<float*>(sB2 + NS * B2_PART);   // [Z][TILE]
    const int64_t room = static_cast<int64_t>(a.smem_ztc);
    [[maybe_unused]] const int64_t sv_n = (room - (reinterpret_cast<unsigned char*>(sV) - smem_raw)) / 4;
    int* st = a.status;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = (warp & 3) * 32 + lane;    // tile column = tensor-memory lane
    const int half = warp >> 2;
    const uint32_t mbar = tc::saddr(smem_raw);
    const uint32_t tslot = tc::saddr(smem_raw + 8);
    const int ncols = max(N1, N2) <= 128 ? 128 : 256;
    float* taps = reinterpret_cast<float*>(smem_raw + 16);     // [2][FWD_TAPS]
    if (warp == 0) tc::tmem_alloc(tslot, ncols);
    if (threadIdx.x == 32) tc::mbar_init(mbar);
    if (threadIdx.x >= 64 && threadIdx.x < 64 + 2 * FWD_TAPS) {
        const int i = threadIdx.x - 64;
        taps[i] = Tab<float>::fwd(i / FWD_TAPS, i % FWD_TAPS);
    }
    __syncthreads();

    // filter operands F1 (N1 x K1) and F2 (N2 x K2), zero outside the filter support
    for (int ci = threadIdx.x; ci < N1 * (K1 >> 3); ci += blockDim.x) {
        const int o = ci / (K1 >> 3), k0 = (ci - o * (K1 >> 3)) * 8;
        float x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int k = k0 + e, b = k >= nz ? 1 : 0, q = k - b * nz, m = o - 2 * q;
            x[e] = (k < 2 * nz && m >= 0 && m < FWD_TAPS) ? taps[b * FWD_TAPS + m] : 0.f;
        }
        tc::put8<NS>(sB1, B1_PART, tc::core_off(o, k0, K1), x, st, room - (sB1 - smem_raw));
    }
    for (int ci = threadIdx.x; ci < N2 * (K2 >> 3); ci += blockDim.x) {
        const int j = ci / (K2 >> 3), o0 = (ci - j * (K2 >> 3)) * 8;
        const int bp = j >= nzp ? 1 : 0, b = j - bp * nzp;
        float x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int o = o0 + e, m = o - 2 * (b + dz);
            x[e] = (j < 2 * nzp && o < Z && m >= 0 && m < FWD_TAPS) ? taps[bp * FWD_TAPS + m] : 0.f;
        }
        tc::put8<NS>(sB2, B2_PART, tc::core_off(j, o0, K2), x, st, room - (sB2 - smem_raw));
    }

    const float* Bf = static_cast<const float*>(a.ws) + r.ws_Bf;
    float* Bb = static_cast<float*>(a.ws) + r.ws_Bb;
    const float* V = static_cast<const float*>(a.V);
    const int64_t vstride = a.vn[0] * a.vn[1];
    const int64_t jz0 = 2LL * r.lo[2] - V_REACH - a.vlo[2];
    const int kh = K1 >> 1, k_lo = half * kh;          // this thread's half of K1
    const int nh1 = N1 >> 1, o_lo = half * nh1;        // its half of N1 (= K2)
    const int nh2 = N2 >> 1, j_lo = half * nh2;        // its half of N2
    float xin[tc::MAX_KH];
    auto load_in = [&](int tile) {
        const int c = tile * TILE + row;
        const bool ok = c < cols;
#pragma unroll
        for (int i0 = 0; i0 < tc::MAX_KH; i0 += 8) {
            if (i0 >= kh) break;            // uniform: whole chunks of 8 past the half are skipped
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int k = k_lo + i0 + e;
                xin[i0 + e] = (ok && k < 2 * nz) ? LD(Bf, static_cast<int64_t>(k) * cols + c, 2LL * nz * cols) : 0.f;
            }
        }
    };
    load_in(blockIdx.x);
    tc::fence_smem();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem_raw + 8);
    const uint32_t tlane = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    uint32_t phase = 0;
    float epot_t = 0.f;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int c = tile * TILE + row;
        const bool valid = c < cols;
        // V(o, c) for o in this thread's half -> sV (cp.async; read back by this thread only)
        if (valid) {
            const int xo = c % X, yo = c / X;
            const int64_t vrow = (2LL * r.lo[1] - V_REACH + yo - a.vlo[1]) * a.vn[0] + (2LL * r.lo[0] - V_REACH + xo - a.vlo[0]);
            const int o1 = min(o_lo + nh1, Z);
#ifdef LSW_CHECKED
            for (int o = o_lo; o < o1; ++o) CPA(sV, o * TILE + row, sv_n, V, (jz0 + o) * vstride + vrow, a.v_n);
#else
            const float* vp = V + (jz0 + o_lo) * vstride + vrow;
            float* sp = sV + o_lo * TILE + row;
#pragma unroll 4
            for (int o = o_lo; o < o1; ++o, vp += vstride, sp += TILE) cp_async(sp, vp);
#endif
        }
        // inputs -> A1 parts (row `row`, k in this thread's half)
#pragma unroll
        for (int i = 0; i < tc::MAX_KH; i += 8) {
            if (i >= kh) break;
            float x[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) x[e] = xin[i + e];
            tc::put8<NS>(sA, A_PART, tc::core_off(row, k_lo + i, K1), x, st, room - (sA - smem_raw));
        }
        tc::fence_smem();
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
        if (threadIdx.x == 0) {
            const uint32_t id = tc::idesc(TILE, N1);
            for (int s = 0; s < (K1 >> 4); ++s)
#pragma unroll
                for (int t = 0; t < tc::Terms<NS>::n; ++t)
                    tc::mma(tmem, tc::sdesc(tc::saddr(sA + tc::Terms<NS>::a(t) * A_PART + s * 256), K1),
                            tc::sdesc(tc::saddr(sB1 + tc::Terms<NS>::b(t) * B1_PART + s * 256), K1), id,
                            s > 0 || t > 0);
            tc::commit(mbar);
        }
        if (tile + static_cast<int>(gridDim.x) < ntiles) load_in(tile + gridDim.x);   // prefetch
        bool ok = tc::mbar_wait(mbar, phase);
        phase ^= 1;
        cp_wait();
        if (!__syncthreads_and(ok)) {
            if (threadIdx.x == 0) atomicOr(st, ST_WAIT_TIMEOUT);
            break;
        }
        tc::fence_after();
        // U -> v = V U -> A2 parts (row `row`, o in this thread's half of K2 = N1)
        for (int ch = 0; ch < nh1; ch += 8) {
            float u[8], x[8];
            tc::tmem_ld8(tlane + o_lo + ch, u);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int o = o_lo + ch + e;
                const float v = (valid && o < Z) ? LD(sV, o * TILE + row, sv_n) * u[e] : 0.f;
                epot_t += v * u[e];
                x[e] = v;
            }
            tc::put8<NS>(sA, A_PART, tc::core_off(row, o_lo + ch, K2), x, st, room - (sA - smem_raw));
        }
        tc::fence_smem();
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
        if (threadIdx.x == 0) {
            const uint32_t id = tc::idesc(TILE, N2);
            for (int s = 0; s < (K2 >> 4); ++s)
#pragma unroll
                for (int t = 0; t < tc::Terms<NS>::n; ++t)
                    tc::mma(tmem, tc::sdesc(tc::saddr(sA + tc::Terms<NS>::a(t) * A_PART + s * 256), K2),
                            tc::sdesc(tc::saddr(sB2 + tc::Terms<NS>::b(t) * B2_PART + s * 256), K2), id,
                            s > 0 || t > 0);
            tc::commit(mbar);
        }
        ok = tc::mbar_wait(mbar, phase);
        phase ^= 1;
        if (!__syncthreads_and(ok)) {
            if (threadIdx.x == 0) atomicOr(st, ST_WAIT_TIMEOUT);
            break;
        }
        tc::fence_after();
        // result -> Bb (row j = b' nz' + b of the coarse z output, column c)
        const int j1 = valid ? min(j_lo + nh2, 2 * nzp) : j_lo;    // rows this thread stores
        for (int ch = 0; ch < nh2; ch += 8) {
            float d[8];
            tc::tmem_ld8(tlane + j_lo + ch, d);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int j = j_lo + ch + e;
                if (j < j1) ST(Bb, static_cast<int64_t>(j) * cols + c, 2LL * nzp * cols, d[e]);
            }
        }
        tc::fence_before();
        __syncthreads();   // every read of this tile's tensor memory and V is done
        tc::fence_after();
    }
    const double epot = warp_sum(static_cast<double>(epot_t));
    if (lane == 0 && epot != 0.0) atomicAdd(a.e_pot + r.f, epot);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (warp == 0) tc::tmem_free(tmem, ncols);
}

// ---------------------------------------------------------------- forward x, y on tensor cores
//
// k_fwd_xy as two band-Toeplitz tensor-core products per (z, b_z) plane with split-
// bfloat16 operands (NS parts) and FP32 accumulation in tensor memory:
//   M1[y'][i] = sum_k Fy[y'][k] Din[k][i],   k = by n_y + y,  i = bx n_x + q,  Fy[y'][k] = F_by[y' - 2y]
//   U[y'][x'] = sum_i M1[y'][i] Fx[x'][i],   Fx[x'][i] = F_bx[x' - 2q]
// with Din[k][i] = D[bx + 2 by][z][y][q] of this plane; U is the plane of Bf.  Thread
// (warp w, lane l) owns row y' = 32 (w mod 4) + l of both products and half w / 4 of each
// K or N range.  256 threads; the operands take about 90 KB, so two blocks share an SM.
template <int NS>
__global__ void __launch_bounds__(256) k_fwd_xy_tc(HphiLaunch a) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 2;
    int* st = a.status;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const FnRec r = a.fn[blockIdx.y];
    const int z = blockIdx.x >> 1, bz = blockIdx.x & 1;
    if (z >= r.n[2]) return;   // uniform over the CTA, before any allocation
    const int nx = r.n[0], ny = r.n[1], nz = r.n[2];
    const int X = 2 * nx + 29, Y = 2 * ny + 29;
    const int K1 = (2 * ny + 15) & ~15, N1 = (2 * nx + 15) & ~15, K2 = N1, N2 = (X + 15) & ~15;
    const int FY_PART = 128 * K1 * 2, FX_PART = N2 * K2 * 2, P_PART = N1 * K1 * 2, M_PART = 128 * K2 * 2;
    unsigned char* sFy = smem_raw + tc::HEAD;
    unsigned char* sFx = sFy + NS * FY_PART;
    unsigned char* sXr = sFx + NS * FX_PART;
    const int64_t room = static_cast<int64_t>(a.smem_fwd_tc);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = (warp & 3) * 32 + lane, half = warp >> 2;
    const uint32_t mbar = tc::saddr(smem_raw);
    float* taps = reinterpret_cast<float*>(smem_raw + 16);
    if (warp == 0) tc::tmem_alloc(tc::saddr(smem_raw + 8), 128);
    if (threadIdx.x == 32) tc::mbar_init(mbar);
    if (threadIdx.x >= 64 && threadIdx.x < 64 + 2 * FWD_TAPS) {
        const int i = threadIdx.x - 64;
        taps[i] = Tab<float>::fwd(i / FWD_TAPS, i % FWD_TAPS);
    }
    __syncthreads();
    // Fy[y'][k] = F_by[y' - 2y], k = by n_y + y
    for (int ci = threadIdx.x; ci < 128 * (K1 >> 3); ci += blockDim.x) {
        const int yo = ci / (K1 >> 3), k0 = (ci - yo * (K1 >> 3)) * 8;
        float x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int k = k0 + e, by = k >= ny ? 1 : 0, y = k - by * ny, m = yo - 2 * y;
            x[e] = (yo < Y && k < 2 * ny && m >= 0 && m < FWD_TAPS) ? taps[by * FWD_TAPS + m] : 0.f;
        }
        tc::put8<NS>(sFy, FY_PART, tc::core_off(yo, k0, K1), x, st, room - (sFy - smem_raw));
    }
    // Fx[x'][i] = F_bx[x' - 2q], i = bx n_x + q
    for (int ci = threadIdx.x; ci < N2 * (K2 >> 3); ci += blockDim.x) {
        const int xo = ci / (K2 >> 3), i0 = (ci - xo * (K2 >> 3)) * 8;
        float x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int i = i0 + e, bx = i >= nx ? 1 : 0, q = i - bx * nx, m = xo - 2 * q;
            x[e] = (xo < X && i < 2 * nx && m >= 0 && m < FWD_TAPS) ? taps[bx * FWD_TAPS + m] : 0.f;
        }
        tc::put8<NS>(sFx, FX_PART, tc::core_off(xo, i0, K2), x, st, room - (sFx - smem_raw));
    }
    // Din[k][i] as the N1 x K1 operand (row i, column k); consecutive threads take
    // consecutive q (contiguous in D)
    const float* D = static_cast<const float*>(a.ws) + r.ws_D;
    const int64_t plane = static_cast<int64_t>(nx) * ny * nz;
    for (int ci = threadIdx.x; ci < N1 * (K1 >> 3); ci += blockDim.x) {
        const int c = ci / N1, i = ci - c * N1, k0 = c * 8;
        const int bx = i >= nx ? 1 : 0, q = i - bx * nx;
        float x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int k = k0 + e, by = k >= ny ? 1 : 0, y = k - by * ny;
            x[e] = (i < 2 * nx && k < 2 * ny)
                       ? LD(D, (bx + 2 * by + 4 * bz) * plane + (static_cast<int64_t>(z) * ny + y) * nx + q, 8 * plane)
                       : 0.f;
        }
        tc::put8<NS>(sXr, P_PART, tc::core_off(i, k0, K1), x, st, room - (sXr - smem_raw));
    }
    tc::fence_smem();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem_raw + 8);
    const uint32_t tlane = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    if (threadIdx.x == 0) {
        const uint32_t id = tc::idesc(128, N1);
        for (int k = 0; k < (K1 >> 4); ++k)
#pragma unroll
            for (int t = 0; t < tc::Terms<NS>::n; ++t)
                tc::mma(tmem, tc::sdesc(tc::saddr(sFy + tc::Terms<NS>::a(t) * FY_PART + k * 256), K1),
                        tc::sdesc(tc::saddr(sXr + tc::Terms<NS>::b(t) * P_PART + k * 256), K1), id, k > 0 || t > 0);
        tc::commit(mbar);
    }
    bool ok = tc::mbar_wait(mbar, 0);
    if (__syncthreads_and(ok)) {
        tc::fence_after();
        for (int c = half; c < (N1 >> 3); c += 2) {
            float u[8];
            tc::tmem_ld8(tlane + c * 8, u);
            tc::put8<NS>(sXr, M_PART, tc::core_off(row, c * 8, K2), u, st, room - (sXr - smem_raw));
        }
        tc::fence_smem();
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
        if (threadIdx.x == 0) {
            const uint32_t id = tc::idesc(128, N2);
            for (int k = 0; k < (K2 >> 4); ++k)
#pragma unroll
                for (int t = 0; t < tc::Terms<NS>::n; ++t)
                    tc::mma(tmem, tc::sdesc(tc::saddr(sXr + tc::Terms<NS>::a(t) * M_PART + k * 256), K2),
                            tc::sdesc(tc::saddr(sFx + tc::Terms<NS>::b(t) * FX_PART + k * 256), K2), id,
                            k > 0 || t > 0);
            tc::commit(mbar);
        }
        ok = tc::mbar_wait(mbar, 1);
        if (__syncthreads_and(ok)) {
            tc::fence_after();
            float* Bf = static_cast<float*>(a.ws) + r.ws_Bf + (static_cast<int64_t>(bz) * nz + z) * Y * X;
            [[maybe_unused]] const int64_t bf_room = 2LL * nz * Y * X - (static_cast<int64_t>(bz) * nz + z) * Y * X;
            for (int c = half; c < (N2 >> 3); c += 2) {
                float u[8];
                tc::tmem_ld8(tlane + c * 8, u);
                if (row < Y) {
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (c * 8 + e < X) ST(Bf, static_cast<int64_t>(row) * X + c * 8 + e, bf_room, u[e]);
                }
            }
        } else if (threadIdx.x == 0) {
            atomicOr(st, ST_WAIT_TIMEOUT);
        }
    } else if (threadIdx.x == 0) {
        atomicOr(st, ST_WAIT_TIMEOUT);
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (warp == 0) tc::tmem_free(tmem, 128);
}

// Kinetic arm of N outputs (both types of a pair) from the window positions p = 0 .. NP - 1 of two
// lines: position p of the first line is D[off(p)], of the second D[off(p) + dist].  [s0, e0), [s1,
// e1): the positions of either line that can be nonzero, uniform over the warp, the second
// within the first.  c0, c1: the lines' values at the outputs.
template <class T>
struct KinArm {
    static constexpr int N = Blk<T, 1>::NB;            // outputs per block, both arms
    static constexpr int NP = N + 2 * KIN_HALF;        // window positions
    // positions per group: FP32 12 (4, with a test of the second line's range too, measured 2 % slower)
    static constexpr int G = sizeof(T) == 4 ? 12 : 1;
    template <class Off>
    static __device__ __forceinline__ void run(T (&o0)[N], T (&o1)[N], T (&c0)[N], T (&c1)[N], const T* D, int64_t dn,
                                               int dist, Off off, int s0, int e0, int s1, int e1,
                                               [[maybe_unused]] int* st) {
        [[maybe_unused]] int* ST_ = st;
        [[maybe_unused]] constexpr int KID = 4;
        float2 acc[sizeof(T) == 4 ? N : 1];
#pragma unroll
        for (int j = 0; j < N; ++j) {
            o0[j] = o1[j] = c0[j] = c1[j] = T(0);
            if constexpr (sizeof(T) == 4) acc[j] = make_float2(0.f, 0.f);
        }
        auto add = [&](int p, int src, T v) {
#pragma unroll
            for (int j = 0; j < N; ++j) {
                if (p - j < 0 || p - j >= KIN_TAPS) continue;
                if constexpr (sizeof(T) == 4) {
                    acc[j] = __ffma2_rn(c_kin2[src][p - j], make_float2(v, v), acc[j]);
                } else {
                    o0[j] += Tab<T>::kin(src, p - j) * v;
                    o1[j] += Tab<T>::kin(2 + src, p - j) * v;
                }
            }
        };
#pragma unroll
        for (int g = 0; g < NP; g += G) {
            if (g + G - 1 < s0 || g >= e0) continue;
            int at[G];
#pragma unroll
            for (int k = 0; k < G; ++k) {
                at[k] = off(g + k);
                const T v = LD(D, at[k], dn);
                if (g + k >= KIN_HALF && g + k < KIN_HALF + N) c0[(g + k - KIN_HALF) & (N - 1)] = v;
                add(g + k, 0, v);
            }
            if (G == 1 && (g < s1 || g >= e1)) continue;
#pragma unroll
            for (int k = 0; k < G; ++k) {
                const T v = LD(D, at[k] + dist, dn);
                if (g + k >= KIN_HALF && g + k < KIN_HALF + N) c1[(g + k - KIN_HALF) & (N - 1)] = v;
                add(g + k, 1, v);
            }
        }
        if constexpr (sizeof(T) == 4) {
#pragma unroll
            for (int j = 0; j < N; ++j) {
                o0[j] = acc[j].x;
                o1[j] = acc[j].y;
            }
        }
    }
};

// ---------------------------------------------------------------- kinetic z arm

// Per (x, y) column of the L box and type pair (t, t + 4): the kinetic arm along z,
// written to G on the L' box column (G holds only this arm; the backward plane kernel
// adds the rest).  Runs before the backward plane kernel.  The column pair is staged in
// shared memory; a column pair that is zero (outside the L sphere, or wavelet types off
// the fine region) only clears its flag, and the plane kernel then skips its G.  Products run
// over the hull of a warp's nonzero inputs, 8 planes (FP64: 4) per block: with the whole window,
// its bounds tests and 4 planes per block it issued about twice the instructions.
// 0.79 -> 0.61 us per function at radii 5-8 bohr, FP64 27 -> 11 us at 6 bohr.
template <class T>
__global__ void __launch_bounds__(128) k_kin_z(HphiLaunch a) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 5;
    int* st = a.status;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const FnRec r = a.fn[blockIdx.y];
    const int nx = r.n[0], ny = r.n[1], nz = r.n[2];
    const int nxp = r.np[0], nyp = r.np[1], nzp = r.np[2];
    const int dx = r.lop[0] - r.lo[0], dy = r.lop[1] - r.lo[1], dz = r.lop[2] - r.lo[2];
    const int pn = nx * ny;
    if (static_cast<int>(blockIdx.x) * 128 >= pn) return;
    const int t = threadIdx.x;
    const int c = blockIdx.x * 128 + t;                    // column (x, y) of the L box
    const int tb = blockIdx.z;                             // type pair (tb, tb + 4)
    T* col = reinterpret_cast<T*>(smem_raw);               // [2][nz + 1][128]: this thread's column pair, each with a zero row
    using Arm = KinArm<T>;
    [[maybe_unused]] const int64_t col_n = static_cast<int64_t>(a.smem_kin / sizeof(T));
    unsigned char* flag = reinterpret_cast<unsigned char*>(static_cast<T*>(a.ws) + r.ws_Gf) + tb * pn;
    T ekin_t = 0;
    int hl[2] = {nz, nz}, hh[2] = {-1, -1};                // hulls of the pair's nonzero inputs
    int zlo = nzp, zhi = -1;                               // planes of L' this column writes
    int64_t gcol = 0;
    ST(col, nz * 128 + t, col_n, T(0));
    ST(col, (2 * nz + 1) * 128 + t, col_n, T(0));
    if (c < pn) {
        const T* D = static_cast<const T*>(a.ws) + r.ws_D;
        const int64_t plane = static_cast<int64_t>(nx) * ny * nz;
        for (int q = 0; q < nz; ++q) {
            CPA(col, q * 128 + t, col_n, D, tb * plane + static_cast<int64_t>(q) * pn + c, 8 * plane);
            CPA(col, (nz + 1 + q) * 128 + t, col_n, D, (tb + 4) * plane + static_cast<int64_t>(q) * pn + c, 8 * plane);
        }
        cp_wait();
        for (int q = 0; q < nz; ++q)
#pragma unroll
            for (int b = 0; b < 2; ++b)
                if (LD(col, (b * (nz + 1) + q) * 128 + t, col_n) != T(0)) {
                    hl[b] = min(hl[b], q);
                    hh[b] = q;
                }
        const bool nonzero = max(hh[0], hh[1]) >= 0;
        ST(flag, c, 4LL * pn, nonzero ? 1 : 0);
        const int y = c / nx, x = c - y * nx;
        const int xb = x - dx, yb = y - dy;             // the same column in the L' box
        if (nonzero && xb >= 0 && xb < nxp && yb >= 0 && yb < nyp) {
            gcol = static_cast<int64_t>(yb) * nxp + xb;
            // the planes of this column the compressed H phi reads: the coarse members' z
            // range where the pair holds type 0 (tb = 0), else the fine members' z hull (the
            // D values of the pair are zero off those, so E_kin loses no term)
            zlo = 0;
            zhi = nzp - 1;
            if (a.colz) {
                const ColZ cz = LD(a.colz, a.atoms[r.atom].colz + gcol, a.colz_n);
                zlo = tb == 0 ? cz.c0 : cz.f0;
                zhi = tb == 0 ? cz.c1 : cz.f1;
                if (zlo < 0) zlo = nzp;
            }
        }
    }
    // a warp's columns together: the blocks of planes any of them needs, products over the hull
    // of their nonzero inputs (positions outside the column read the zero row)
    const int z0 = __reduce_min_sync(0xffffffffu, zlo), z1 = __reduce_max_sync(0xffffffffu, zhi);
    const int l0 = __reduce_min_sync(0xffffffffu, hl[0]), h0 = __reduce_max_sync(0xffffffffu, hh[0]);
    const int l1 = __reduce_min_sync(0xffffffffu, hl[1]), h1 = __reduce_max_sync(0xffffffffu, hh[1]);
    T* G = static_cast<T*>(a.ws) + r.ws_G;
    const int64_t gplane = static_cast<int64_t>(nxp) * nyp * nzp;
    const int64_t pnp = static_cast<int64_t>(nxp) * nyp;
    const T ks = static_cast<T>(a.kin_scale);
    for (int b0 = (z0 / Arm::N) * Arm::N; b0 <= z1; b0 += Arm::N) {
        const int f0 = b0 + dz - KIN_HALF;              // window position p is input f0 + p
        T o0[Arm::N], o1[Arm::N], c0[Arm::N], c1[Arm::N];
        // both types' ranges within one for the first type (the run's condition)
        Arm::run(o0, o1, c0, c1, col, col_n, (nz + 1) * 128,
                 [&](int p) { const int q = f0 + p; return (q >= 0 && q < nz ? q : nz) * 128 + t; },
                 min(l0, l1) - f0, max(h0, h1) - f0 + 1, l1 - f0, h1 - f0 + 1, st);
#pragma unroll
        for (int j = 0; j < Arm::N; ++j) {
            const int b = b0 + j;
            if (b >= zlo && b <= zhi) {
                o0[j] *= ks;
                o1[j] *= ks;
                ST(G, tb * gplane + b * pnp + gcol, 8 * gplane, o0[j]);
                ST(G, (tb + 4) * gplane + b * pnp + gcol, 8 * gplane, o1[j]);
                ekin_t += c0[j] * o0[j] + c1[j] * o1[j];
            }
        }
    }
    const double ekin = warp_sum(static_cast<double>(ekin_t));
    if ((threadIdx.x & 31) == 0 && ekin != 0.0) atomicAdd(a.e_kin + r.f, ekin);
}

// ---------------------------------------------------------------- backward y, x + kinetic x, y + compress

// Per plane (z'', bz) of the L' box: transposed filters along y then x (potential part)
// plus the kinetic arms along x and y of the four output types with z bit bz, plus the
// z arm that k_kin_z left in G; the sum is written straight into the compressed H phi
// on the members of L' in this plane.  Only member rows (and, per row, the x range of
// its member segment: L' is a sphere clipped by the box) are computed; kinetic type
// pairs whose input rows or columns of D are all zero (wavelet types off the fine
// region) are skipped.  Each phase first lists its tasks in shared memory, so skipped
// work frees whole rounds.
constexpr int BWD_MAX_TASKS = 2048;   // of the tensor-core version

// Potential part of the backward plane kernel on the tensor cores (the two products
// described at k_bwd_xy): builds the filter operands Fy (128 x K1) and Fx (N2 x K2) and
// the plane operand P (N1 x K1: row x', column y') from Bb, runs both products and writes
// Gs[bx + 2 by][b][b2] for every b < n_y', b2 < n_x'.  512 threads.  Returns false (for
// every thread) if a completion wait ran out.
template <int NS>
__device__ bool bwd_tc_potential(const float* Bb, [[maybe_unused]] int64_t bb_room, int X, int Y, int nyp, int nxp,
                                 int dx, int dy, int K1, int N1, int K2, int N2, int FY_PART, int FX_PART,
                                 [[maybe_unused]] int XR, unsigned char* sFy, unsigned char* sFx, unsigned char* sXr,
                                 float* Gs, unsigned char* smem_raw, int64_t room, int* st) {
    [[maybe_unused]] int* ST_ = st;
    [[maybe_unused]] constexpr int KID = 4;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = (warp & 3) * 32 + lane, part = warp >> 2;
    const int P_PART = N1 * K1 * 2, M_PART = 128 * K2 * 2;
    const float* taps = reinterpret_cast<const float*>(smem_raw + 16);
    const uint32_t mbar = tc::saddr(smem_raw);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem_raw + 8);
    const uint32_t tlane = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    // Fy[j][y'] = F_by[y' - 2 (b + dy)], j = by n_y' + b
    for (int ci = threadIdx.x; ci < 128 * (K1 >> 3); ci += blockDim.x) {
        const int j = ci / (K1 >> 3), y0 = (ci - j * (K1 >> 3)) * 8;
        const int by = j >= nyp ? 1 : 0, b = j - by * nyp;
        float x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int m = y0 + e - 2 * (b + dy);
            x[e] = (j < 2 * nyp && y0 + e < Y && m >= 0 && m < FWD_TAPS) ? taps[by * FWD_TAPS + m] : 0.f;
        }
        tc::put8<NS>(sFy, FY_PART, tc::core_off(j, y0, K1), x, st, room - (sFy - smem_raw));
    }
    // Fx[i][x'] = F_bx[x' - 2 (b2 + dx)], i = bx n_x' + b2
    for (int ci = threadIdx.x; ci < N2 * (K2 >> 3); ci += blockDim.x) {
        const int i = ci / (K2 >> 3), x0 = (ci - i * (K2 >> 3)) * 8;
        const int bx = i >= nxp ? 1 : 0, b2 = i - bx * nxp;
        float x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int m = x0 + e - 2 * (b2 + dx);
            x[e] = (i < 2 * nxp && x0 + e < X && m >= 0 && m < FWD_TAPS) ? taps[bx * FWD_TAPS + m] : 0.f;
        }
        tc::put8<NS>(sFx, FX_PART, tc::core_off(i, x0, K2), x, st, room - (sFx - smem_raw));
    }
    // P[x'][y'] = Bb plane (y', x'); consecutive threads take consecutive x' (coalesced)
    for (int ci = threadIdx.x; ci < N1 * (K1 >> 3); ci += blockDim.x) {
        const int c = ci / N1, xo = ci - c * N1, y0 = c * 8;
        float x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e)
            x[e] = (xo < X && y0 + e < Y) ? LD(Bb, static_cast<int64_t>(y0 + e) * X + xo, bb_room) : 0.f;
        tc::put8<NS>(sXr, P_PART, tc::core_off(xo, y0, K1), x, st, room - (sXr - smem_raw));
    }
    tc::fence_smem();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (threadIdx.x == 0) {
        const uint32_t id = tc::idesc(128, N1);
        for (int k = 0; k < (K1 >> 4); ++k)
#pragma unroll
            for (int t = 0; t < tc::Terms<NS>::n; ++t)
                tc::mma(tmem, tc::sdesc(tc::saddr(sFy + tc::Terms<NS>::a(t) * FY_PART + k * 256), K1),
                        tc::sdesc(tc::saddr(sXr + tc::Terms<NS>::b(t) * P_PART + k * 256), K1), id, k > 0 || t > 0);
        tc::commit(mbar);
    }
    bool ok = tc::mbar_wait(mbar, 0);
    if (!__syncthreads_and(ok)) return false;
    tc::fence_after();
    // M1 row `row` -> operand of the second product (the P operand is dead)
    for (int c = part; c < (N1 >> 3); c += 4) {
        float u[8];
        tc::tmem_ld8(tlane + c * 8, u);
        tc::put8<NS>(sXr, M_PART, tc::core_off(row, c * 8, K2), u, st, room - (sXr - smem_raw));
    }
    tc::fence_smem();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (threadIdx.x == 0) {
        const uint32_t id = tc::idesc(128, N2);
        for (int k = 0; k < (K2 >> 4); ++k)
#pragma unroll
            for (int t = 0; t < tc::Terms<NS>::n; ++t)
                tc::mma(tmem, tc::sdesc(tc::saddr(sXr + tc::Terms<NS>::a(t) * M_PART + k * 256), K2),
                        tc::sdesc(tc::saddr(sFx + tc::Terms<NS>::b(t) * FX_PART + k * 256), K2), id, k > 0 || t > 0);
        tc::commit(mbar);
    }
    ok = tc::mbar_wait(mbar, 1);
    if (!__syncthreads_and(ok)) return false;
    tc::fence_after();
    // Q row `row` -> Gs (the M1 operand is dead)
    const int by = row >= nyp ? 1 : 0, b = row - by * nyp;
    [[maybe_unused]] const int64_t gs_n = 4LL * nyp * nxp;
    for (int c = part; c < (N2 >> 3); c += 4) {
        float q[8];
        tc::tmem_ld8(tlane + c * 8, q);
        if (row < 2 * nyp) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int i = c * 8 + e;
                if (i < 2 * nxp) {
                    const int bx = i >= nxp ? 1 : 0, b2 = i - bx * nxp;
                    ST(Gs, ((bx + 2 * by) * nyp + b) * nxp + b2, gs_n, q[e]);
                }
            }
        }
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    return true;
}

// Split-bfloat16 systems, option "xy_tc": the transposed y and x filters as two band-Toeplitz
// tensor-core products per plane with split-bfloat16 operands (NS = 2 or 3 parts) and FP32
// accumulation in tensor memory, as in k_z_tc (512 threads, one block per SM):
//   M1[j][x'] = sum_y' Fy[j][y'] P[y'][x'],   j = by n_y' + b,  Fy[j][y'] = F_by[y' - 2(b + dy)]
//   Q[j][i]   = sum_x' M1[j][x'] Fx[i][x'],   i = bx n_x' + b2, Fx[i][x'] = F_bx[x' - 2(b2 + dx)]
// with P the plane of Bb; thread (warp w, lane l) owns row j = 32 (w mod 4) + l of both
// products and quarter w / 4 of each K or N range.
template <int NS>
__device__ __forceinline__ void bwd_plane_tc(const HphiLaunch& a, int fl, int zb, int bz) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 4;
    using T = float;
    int* st = a.status;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int16_t rx0[256], rx1[256];         // member x range per row (L' plane), -1: none
    __shared__ int roff[256];                      // coefficient offset of the row's coarse segment
    __shared__ int fr0[256], fr1[256];             // fine segment range of the row (L' keys)
    __shared__ int16_t fx0[256], fx1[256];         // hull of the row's fine members, -1: none
    __shared__ int rq0[128], rq1[128], rqp[129];   // kinetic y arm, per (x type, block of BB rows): the same
    __shared__ int ntask2, ylo, yhi;
    __shared__ unsigned char rowf[4][128], colf[4][128];   // D plane: nonzero per (type, row / column)
    const FnRec r = a.fn[fl];
    if (zb >= r.np[2]) return;
    const AtomRec& at = a.atoms[r.atom];
    const int nx = r.n[0], ny = r.n[1], nz = r.n[2];
    const int X = 2 * nx + 29, Y = 2 * ny + 29;
    const int nxp = r.np[0], nyp = r.np[1], nzp = r.np[2];
    const int dx = r.lop[0] - r.lo[0], dy = r.lop[1] - r.lo[1], dz = r.lop[2] - r.lo[2];
    const int RS = nx | 1;
    // layout: header, Fy parts, Fx parts, a region holding the P operand, then
    // the M1 operand, then Gs; Dp
    const int K1 = (Y + 15) & ~15, N1 = (X + 15) & ~15, K2 = N1, N2 = (2 * nxp + 15) & ~15;
    const int FY_PART = 128 * K1 * 2, FX_PART = N2 * K2 * 2, P_PART = N1 * K1 * 2, M_PART = 128 * K2 * 2;
    const int XR = (max(max(NS * P_PART, NS * M_PART), 16 * nyp * nxp) + 15) & ~15;
    unsigned char* sFy = smem_raw + tc::HEAD;
    unsigned char* sFx = sFy + NS * FY_PART;
    unsigned char* sXr = sFx + NS * FX_PART;
    // task list of the kinetic x arm, later the plane's fine segments for the compressed
    // write: the filter operands' region, dead once the potential part is done
    // (NS * FY_PART >= 2 * 128 * 16 * 2 bytes = BWD_MAX_TASKS ints; 16-byte aligned)
    int* task = reinterpret_cast<int*>(sFy);
    T* Gs = reinterpret_cast<T*>(sXr);
    T* Dp = reinterpret_cast<T*>(sXr + XR);
    const int64_t smem_n = static_cast<int64_t>(a.smem_bwd_tc / sizeof(T));
    {
        if ((threadIdx.x >> 5) == 0) tc::tmem_alloc(tc::saddr(smem_raw + 8), 128);
        if (threadIdx.x == 32) tc::mbar_init(tc::saddr(smem_raw));
        float* taps = reinterpret_cast<float*>(smem_raw + 16);
        if (threadIdx.x >= 64 && threadIdx.x < 64 + 2 * FWD_TAPS) {
            const int i = threadIdx.x - 64;
            taps[i] = Tab<float>::fwd(i / FWD_TAPS, i % FWD_TAPS);
        }
    }
    const int zL = zb + dz;
    const bool dplane = zL >= 0 && zL < nz;
    if (threadIdx.x == 0) {
        ylo = nyp;
        yhi = -1;
    }
    for (int i = threadIdx.x; i < 4 * 128; i += blockDim.x) {
        rowf[i >> 7][i & 127] = 0;
        colf[i >> 7][i & 127] = 0;
    }
    __syncthreads();
    // staging copies first (they fly while the row records below are read): the D plane and
    // the z-arm column flags
    const T* Bb = static_cast<const T*>(a.ws) + r.ws_Bb + (static_cast<int64_t>(bz) * nzp + zb) * Y * X;
    const int64_t bb_room = 2LL * nzp * Y * X - (static_cast<int64_t>(bz) * nzp + zb) * Y * X;
    const T* D = static_cast<const T*>(a.ws) + r.ws_D;
    const int64_t plane = static_cast<int64_t>(nx) * ny * nz;
    const int pn = nx * ny;
    const int64_t dp_n = smem_n - (reinterpret_cast<unsigned char*>(Dp) - smem_raw) / static_cast<int64_t>(sizeof(T));
    if (dplane) {
        const FastDiv fd_pn(pn), fd_nx(nx);
        for (int i = threadIdx.x; i < 4 * pn; i += blockDim.x) {
            const int tb = fd_pn.div(i), rem = i - tb * pn;
            const int y = fd_nx.div(rem), x = rem - y * nx;
            CPA(Dp, (tb * ny + y) * RS + x, dp_n, D, (tb + 4 * bz) * plane + static_cast<int64_t>(zL) * pn + rem,
                8 * plane);
        }
    }
    // z-arm column flags of the L box (written by k_kin_z)
    const uint32_t* gsrc = reinterpret_cast<const uint32_t*>(static_cast<const T*>(a.ws) + r.ws_Gf);
    uint32_t* gfl = reinterpret_cast<uint32_t*>(Dp + 4 * ny * RS);
    [[maybe_unused]] const int64_t gfl_n = (smem_n * static_cast<int64_t>(sizeof(T)) -
                                            (reinterpret_cast<unsigned char*>(gfl) - smem_raw)) / 4;
    for (int i = threadIdx.x; i < pn; i += blockDim.x) CPA(gfl, i, gfl_n, gsrc, i, pn);
    // member x range of each row of this plane (coarse part of L')
    for (int y = threadIdx.x; y < nyp; y += blockDim.x) {
        const int64_t row = at.rowPc + y + static_cast<int64_t>(nyp) * zb;
        const int s0 = LD(a.rowptr, row, a.rowptr_n), s1 = LD(a.rowptr, row + 1, a.rowptr_n);
        int lo = -1, hi = -1, off = 0;
        if (s1 > s0) {
            const Seg sg = LD(a.seg, at.segPc + s0, a.seg_n);
            lo = sg.x0;
            off = sg.off;
            hi = LD(a.seg, at.segPc + s1 - 1, a.seg_n).x1;
            atomicMin(&ylo, y);
            atomicMax(&yhi, y);
        }
        rx0[y] = static_cast<int16_t>(lo);
        rx1[y] = static_cast<int16_t>(hi);
        roff[y] = off;
        const int64_t frow = at.rowPf + y + static_cast<int64_t>(nyp) * zb;
        const int q0 = LD(a.rowptr, frow, a.rowptr_n), q1 = LD(a.rowptr, frow + 1, a.rowptr_n);
        fr0[y] = q0;
        fr1[y] = q1;
        fx0[y] = static_cast<int16_t>(q1 > q0 ? LD(a.seg, at.segPf + q0, a.seg_n).x0 : -1);
        fx1[y] = static_cast<int16_t>(q1 > q0 ? LD(a.seg, at.segPf + q1 - 1, a.seg_n).x1 : -1);
    }
    if (threadIdx.x == 0) ntask2 = 0;
    __syncthreads();
    const int64_t gs_n = 4LL * nyp * nxp;
    const T ks = static_cast<T>(a.kin_scale);
    T ekin_t = 0;
    const int ylo_ = ylo, yhi_ = yhi;
    // The x range of row b whose outputs of the y-type pair `by` (types 2 by, 2 by + 1 of
    // this plane) the compressed write reads: the coarse members where the pair holds the
    // scaling type 0 (bz = 0, by = 0), else the hull of the row's fine members (the wavelet
    // types are stored on fine members only).  lo < 0: none.
    auto need = [&](int by, int b, int& lo, int& hi) {
        if (bz == 0 && by == 0) {
            lo = rx0[b];
            hi = rx1[b];
        } else {
            lo = fx0[b];
            hi = fx1[b];
        }
    };
    // ---- column ranges of the kinetic y arm per x type bx (the pair of types bx, bx + 2) and
    //      block of BB rows, with their prefix sums: the hull of the rows' needed ranges, the
    //      coarse members where the pair holds type 0, else the fine members
    const int nbyk = (yhi_ - ylo_ + BB) / BB;
    if (yhi_ >= 0) {
        const int t2 = static_cast<int>(threadIdx.x) - 128;
        if (t2 >= 0 && t2 < 2 * nbyk) {
            const int bx = t2 >= nbyk, q = t2 - bx * nbyk;
            const bool coarse = bz == 0 && bx == 0;
            int c0 = nxp, c1 = -1;
            for (int b = ylo_ + q * BB; b < min(ylo_ + (q + 1) * BB, yhi_ + 1); ++b) {
                const int lo = coarse ? rx0[b] : fx0[b], hi = coarse ? rx1[b] : fx1[b];
                if (lo < 0) continue;
                c0 = min(c0, lo);
                c1 = max(c1, hi);
            }
            rq0[t2] = c0;
            rq1[t2] = c1;
        }
        __syncthreads();
        if (threadIdx.x == 32) {
            rqp[0] = 0;
            for (int i = 0; i < 2 * nbyk; ++i) rqp[i + 1] = rqp[i] + max(0, rq1[i] - rq0[i] + 1);
        }
        __syncthreads();
    }
    {
        // ---- potential part on the tensor cores -> Gs (every row and column of the plane)
        if (yhi_ >= 0 && !bwd_tc_potential<NS>(reinterpret_cast<const float*>(Bb), bb_room, X, Y, nyp, nxp, dx, dy,
                                                K1, N1, K2, N2, FY_PART, FX_PART, XR, sFy, sFx, sXr,
                                                reinterpret_cast<float*>(Gs), smem_raw, smem_n * 4, st)) {
            if (threadIdx.x == 0) atomicOr(st, ST_WAIT_TIMEOUT);
        }
    }
    if (yhi_ >= 0) {
        // the D plane and the flags have landed (their copies flew during the passes above)
        cp_wait();
        __syncthreads();
        if (dplane) {   // zero flags of the staged D plane
            const FastDiv fd_pn(pn), fd_nx(nx);
            for (int i = threadIdx.x; i < 4 * pn; i += blockDim.x) {
                const int tb = fd_pn.div(i), rem = i - tb * pn;
                const int y = fd_nx.div(rem), x = rem - y * nx;
                if (LD(Dp, (tb * ny + y) * RS + x, dp_n) != T(0)) {
                    rowf[tb][y & 127] = 1;
                    colf[tb][x & 127] = 1;
                }
            }
        }
        if (dplane) {
            int nt;
            __syncthreads();   // the D plane's zero flags
            // ---- kinetic x arm: (by, row b, x block of BB) over the needed range of rows whose
            //      D rows are nonzero
            for (int b = ylo_ + threadIdx.x; b <= yhi_; b += blockDim.x) {
                const int y = b + dy;
                if (y < 0 || y >= ny) continue;
                for (int by = 0; by < 2; ++by) {
                    if (!rowf[2 * by][y & 127] && !rowf[2 * by + 1][y & 127]) continue;
                    int lo, hi;
                    need(by, b, lo, hi);
                    if (lo < 0) continue;
                    const int k0 = lo / BB, k1 = hi / BB;
                    const int base = atomicAdd(&ntask2, k1 - k0 + 1);
                    for (int k = k0; k <= k1; ++k)
                        if (base + k - k0 < BWD_MAX_TASKS) task[base + k - k0] = (by << 24) | (b << 12) | k;
                }
            }
            __syncthreads();
            nt = min(ntask2, BWD_MAX_TASKS);
            if (ntask2 > BWD_MAX_TASKS && threadIdx.x == 0) atomicOr(a.status, ST_BAD_BOX);
            for (int it = threadIdx.x; it < nt; it += blockDim.x) {
                const int code = task[it];
                const int by = code >> 24, b = (code >> 12) & 4095, x0 = (code & 4095) * BB;
                const int y = b + dy;
                T k0[KW], k1[KW], o0[BB], o1[BB];
                const int r0 = ((2 * by) * ny + y) * RS, r1 = r0 + ny * RS;
                swin(k0, Dp, r0, 1, x0 + dx - KIN_HALF, nx, dp_n, st);
                swin(k1, Dp, r1, 1, x0 + dx - KIN_HALF, nx, dp_n, st);
                kin_block(k0, k1, o0, o1);
#pragma unroll
                for (int j = 0; j < BB; ++j) {
                    const int xb = x0 + j;
                    if (xb < nxp) {
                        o0[j] *= ks;
                        o1[j] *= ks;
                        const int64_t g0 = ((0 + 2 * by) * nyp + b) * nxp + xb;
                        const int64_t g1 = ((1 + 2 * by) * nyp + b) * nxp + xb;
                        ST(Gs, g0, gs_n, LD(Gs, g0, gs_n) + o0[j]);
                        ST(Gs, g1, gs_n, LD(Gs, g1, gs_n) + o1[j]);
                        const int x = x0 + dx + j;
                        if (x >= 0 && x < nx) ekin_t += k0[KIN_HALF + j] * o0[j] + k1[KIN_HALF + j] * o1[j];
                    }
                }
            }
            __syncthreads();   // the x arm's Gs updates are done
            // ---- kinetic y arm: tasks (x type bx, block q of BB rows, column) over the column
            //      ranges listed above, consecutive columns on consecutive threads
            nt = rqp[2 * nbyk];
            for (int it = threadIdx.x; it < nt; it += blockDim.x) {
                int lo = 0, hi = 2 * nbyk - 1;              // the entry i with rqp[i] <= it < rqp[i + 1]
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (rqp[mid] <= it) lo = mid;
                    else hi = mid - 1;
                }
                const int bx = lo >= nbyk, q = lo - bx * nbyk;
                const int xb = rq0[lo] + (it - rqp[lo]), b0 = ylo_ + q * BB;
                const int x = xb + dx;
                if (x < 0 || x >= nx) continue;
                if (!colf[bx][x & 127] && !colf[bx + 2][x & 127]) continue;
                T k0[KW], k1[KW], o0[BB], o1[BB];
                swin(k0, Dp, bx * ny * RS + x, RS, b0 + dy - KIN_HALF, ny, dp_n, st);
                swin(k1, Dp, (bx + 2) * ny * RS + x, RS, b0 + dy - KIN_HALF, ny, dp_n, st);
                kin_block(k0, k1, o0, o1);
#pragma unroll
                for (int j = 0; j < BB; ++j) {
                    const int b = b0 + j;
                    if (b <= yhi_) {
                        o0[j] *= ks;
                        o1[j] *= ks;
                        const int64_t g0 = (static_cast<int64_t>(bx + 0) * nyp + b) * nxp + xb;
                        const int64_t g1 = (static_cast<int64_t>(bx + 2) * nyp + b) * nxp + xb;
                        ST(Gs, g0, gs_n, LD(Gs, g0, gs_n) + o0[j]);
                        ST(Gs, g1, gs_n, LD(Gs, g1, gs_n) + o1[j]);
                        const int y = b + dy;
                        if (y >= 0 && y < ny) ekin_t += k0[KIN_HALF + j] * o0[j] + k1[KIN_HALF + j] * o1[j];
                    }
                }
            }
        }
    }
    cp_wait();
    __syncthreads();
    // ---- compress: members of this plane -> H phi (plus the z arm left in G by k_kin_z).  Coarse members (type 0)
    //      row by row, a warp per row (one segment of up to n_x' members each); fine members
    //      flattened over the CTA, one member per thread and type: the plane's fine
    //      segments (many short chords of the fine spheres) are staged in shared memory and
    //      each member finds its segment by a binary search, so every lane writes and
    //      consecutive lanes write consecutive H phi elements.
    if (yhi_ >= 0) {
        const T* G = static_cast<const T*>(a.ws) + r.ws_G;
        const unsigned char* gflag = reinterpret_cast<const unsigned char*>(gfl);
        const int64_t gplane = static_cast<int64_t>(nxp) * nyp * nzp;
        T* out = static_cast<T*>(a.hphi) + r.off_hphi;
        const int64_t out_room = a.hphi_n - r.off_hphi;
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (bz == 0) {   // scaling part s (type 0) on the coarse members
            for (int b = ylo_ + warp; b <= yhi_; b += (blockDim.x >> 5)) {
                if (rx0[b] < 0) continue;
                const int y = b + dy;
                const bool yin = y >= 0 && y < ny;
                const int64_t grow = (static_cast<int64_t>(zb) * nyp + b) * nxp;
                for (int xb = rx0[b] + lane; xb <= rx1[b]; xb += 32) {
                    const int x = xb + dx;
                    T v = LD(Gs, static_cast<int64_t>(b) * nxp + xb, gs_n);
                    if (yin && x >= 0 && x < nx && LD(gflag, y * nx + x, 4LL * pn))
                        v += LD(G, grow + xb, 8 * gplane);
                    ST(out, roff[b] + (xb - rx0[b]), out_room, v);
                }
            }
        }
        // wavelet parts on the fine members of this plane: segments [q0, q1) hold members
        // [m0, m1) of each type's block
        const int q0 = fr0[ylo_], q1 = fr1[yhi_];
        if (q1 > q0) {
            constexpr int SEG_CAP = BWD_MAX_TASKS / 4;    // Seg records in the task array
            int4* sseg = reinterpret_cast<int4*>(task);
            const int nq = q1 - q0;
            const bool staged = nq <= SEG_CAP;
            if (staged)
                for (int i = threadIdx.x; i < nq; i += blockDim.x) {
                    const Seg g = LD(a.seg, at.segPf + q0 + i, a.seg_n);
                    sseg[i] = make_int4(g.x0, g.x1, g.row, g.off);
                }
            __syncthreads();
            auto seg_at = [&](int i) -> int4 {
                if (staged) return sseg[i];
                const Seg g = LD(a.seg, at.segPf + q0 + i, a.seg_n);
                return make_int4(g.x0, g.x1, g.row, g.off);
            };
            const int4 sl = seg_at(nq - 1);
            const int m0 = seg_at(0).w, m1 = sl.w + (sl.y - sl.x + 1);
            const int64_t zrow = static_cast<int64_t>(nyp) * zb;
            for (int m = m0 + static_cast<int>(threadIdx.x); m < m1; m += blockDim.x) {
                int lo = 0, hi = nq - 1;                     // the segment with off <= m
                while (lo < hi) {
                    const int mid_ = (lo + hi + 1) >> 1;
                    if (seg_at(mid_).w <= m) lo = mid_;
                    else hi = mid_ - 1;
                }
                const int4 g = seg_at(lo);
                const int xb = g.x + (m - g.w);
                const int b = static_cast<int>(g.z - zrow);
                const int y = b + dy, x = xb + dx;
                const bool zin = y >= 0 && y < ny && x >= 0 && x < nx;
                const int64_t grow = (static_cast<int64_t>(zb) * nyp + b) * nxp;
#pragma unroll
                for (int tb = 0; tb < 4; ++tb) {
                    const int t = tb + 4 * bz;
                    if (t == 0) continue;
                    T v = LD(Gs, (static_cast<int64_t>(tb) * nyp + b) * nxp + xb, gs_n);
                    if (zin && LD(gflag, (t & 3) * pn + y * nx + x, 4LL * pn))
                        v += LD(G, t * gplane + grow + xb, 8 * gplane);
                    ST(out, at.ncP + static_cast<int64_t>(t - 1) * at.nfP + m, out_room, v);
                }
            }
        }
    }
    const double ekin = warp_sum(static_cast<double>(ekin_t));
    if ((threadIdx.x & 31) == 0 && ekin != 0.0) atomicAdd(a.e_kin + r.f, ekin);
    {
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
        if ((threadIdx.x >> 5) == 0) tc::tmem_free(*reinterpret_cast<volatile uint32_t*>(smem_raw + 8), 128);
    }
}

template <int NS>
__global__ void __launch_bounds__(512, 1) k_bwd_xy_tc(HphiLaunch a) {
    bwd_plane_tc<NS>(a, blockIdx.y, blockIdx.x >> 1, blockIdx.x & 1);
}

// The FMA version.  An item is a plane (z'', b_z) of an atom's L' box for `cnt` consecutive
// functions of the atom: the functions share every table below, so the tables are built once
// per item and the item loops over the functions.
//
// Bound: instruction issue and its latencies (two CTAs per SM by registers and shared memory).
// What is not arithmetic is kept small:
//   - the planes of Bb and of the z arm arrive by bulk copies (one instruction each; the copy
//     starts at the 16-byte boundary below the plane, the remainder becomes the first index);
//   - the kinetic x arm is computed by the thread that computes the transposed x filter of the
//     same outputs: one store, and one barrier for both;
//   - kinetic sums skip window positions outside the hull of L's members (per row along x, per
//     column along y), in groups of 12 positions, uniformly over a warp; neighbouring lanes take
//     neighbouring rows (columns) of the same block, so their hulls nearly agree.  Positions
//     outside the box read a zero beside the D plane;
//   - the y pass, the x pass and the kinetic y arm are one loop body run in three phases: as three
//     bodies their unrolled code (40 KB) missed the instruction caches (17 % of the stalls);
//   - the compressed write's fine members come from a list built once per item;
//   - the tables are one chain of loads (a row and part per thread), ranges by atomics, prefix
//     sums and tasks by warps, while the first function's planes arrive (built ahead of them by one
//     thread per table they took 15 % of an item, 32 % of one with a single function).  The next
//     item is fetched during the last write, no earlier: a CTA that holds an item unbegun delays
//     the end (64 atoms in FP64: 11.1 ms a step, so 10.0).
// Measured (GB300, 2,070 MHz, 1,024 functions a batch): 4.4 us per function at radii 5-8 bohr (n_x' to
// 52), 5.4 us at 7 bohr in a dense system (n_x' 47, more fine members); with an element per copy, an
// item per function and the arms apart: 9.5 and 7.3.

#ifndef LSW_BWD_THREADS
#define LSW_BWD_THREADS 256
#endif
constexpr int BWD_THREADS = LSW_BWD_THREADS;

// (out of line: the kernel's time depends on what its loops share the instruction caches with)
static __device__ __noinline__ void bwd_last_wait(uint32_t mbar, uint32_t parity) { (void)tc::mbar_wait(mbar, parity); }

template <class T>
__device__ __forceinline__ void bwd_plane(const HphiLaunch& a, int fl, int cnt, int zb, int bz, uint32_t& phase, int& dead,
                                          int2* s_next) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 4;
    int* st = a.status;
    constexpr int NB = Blk<T, 1>::NB;
    using Arm = KinArm<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int ylo, yhi;
    const FnRec r0 = a.fn[fl];
    if (zb >= r0.np[2]) return;
    const AtomRec& at = a.atoms[r0.atom];
    const int nx = r0.n[0], ny = r0.n[1], nz = r0.n[2];
    const int X = 2 * nx + 29, Y = 2 * ny + 29;
    const int nxp = r0.np[0], nyp = r0.np[1], nzp = r0.np[2];
    const int dx = r0.lop[0] - r0.lo[0], dy = r0.lop[1] - r0.lo[1], dz = r0.lop[2] - r0.lo[2];
    const BwdLayout L = bwd_layout(nx, ny, nxp, nyp, sizeof(T), NB, a.gstage, a.lists);
    const int RS = L.RS, PS = L.PS;
    T* const plb = reinterpret_cast<T*>(smem_raw + L.o_pl);     // Bb plane [Y][X], later Gs [4][nyp][nxp]
    T* const Gs = plb;
    T* const mid = reinterpret_cast<T*>(smem_raw + L.o_mid);    // [2][nyp][X], later the z-arm plane
    T* const Dp = reinterpret_cast<T*>(smem_raw + L.o_D);       // [4][PS]: rows [ny][RS], then a zero
    uint16_t* const task = reinterpret_cast<uint16_t*>(smem_raw + L.o_task);   // x pass: block entry << kx | row
    uint16_t* const taskk = task + L.taskN;                     // kinetic y arm: block entry << ky | column
    int* const roff = reinterpret_cast<int*>(smem_raw + L.o_roff);
    int* const cq0 = reinterpret_cast<int*>(smem_raw + L.o_blk);   // y pass, per block of NB rows: column range, prefix
    int* const cq1 = cq0 + L.nb_y;
    int* const pq = cq1 + L.nb_y;                               // [nb_y + 1]
    int* const rq0 = pq + L.nb_y + 1;                           // kinetic y arm, per (x type, block of N rows): the same
    int* const rq1 = rq0 + 2 * L.nb_y;
    int* const rqp = rq1 + 2 * L.nb_y;                          // [2 nb_y + 1]
    int* const hlo = rqp + 2 * L.nb_y + 1;                      // x pass, per (y type, block of NB columns): row hull, prefix
    int* const hhi = hlo + 2 * L.nb_x;
    int* const hp = hhi + 2 * L.nb_x;                           // [2 nb_x + 1]
    int16_t* const rx0 = reinterpret_cast<int16_t*>(smem_raw + L.o_row);   // member x range per row (L' plane), -1: none
    int16_t* const rx1 = rx0 + nyp;
    int16_t* const fx0 = rx1 + nyp;                             // hull of the row's fine members, -1: none
    int16_t* const fx1 = fx0 + nyp;
    int* const lxr = reinterpret_cast<int*>(fx1 + nyp);         // [2][ny]: hull of L's coarse, fine members per row of the D plane
    int* const cyr = lxr + 2 * ny;                              // [2][nx]: the same per column; first << 16 | last, -1: none
    uint16_t* const memb = reinterpret_cast<uint16_t*>(smem_raw + L.o_mem);   // b n_x' + x of the plane's fine members
    const int kx = 32 - __clz(max(nyp - 1, 1)), ky = 32 - __clz(max(nxp - 1, 1));   // (n_x' n_y' < 2^14: codes < 2^16)
    const uint32_t mbar = tc::saddr(smem_raw);
    const int zL = zb + dz;
    const bool dplane = zL >= 0 && zL < nz;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t smem_n = static_cast<int64_t>(a.smem_bwd / sizeof(T));
    [[maybe_unused]] const int64_t pl_n = smem_n - L.o_pl / sizeof(T), mid_n = smem_n - L.o_mid / sizeof(T),
                                   dp_n = smem_n - L.o_D / sizeof(T);
    const int pn = nx * ny;
    const int64_t dplane_n = static_cast<int64_t>(pn) * nz;
    // the D plane of function f (types tb + 4 bz), an element per copy into the padded rows
    auto stage_D = [&](const FnRec& r) {
        const T* D = static_cast<const T*>(a.ws) + r.ws_D + 4LL * bz * dplane_n + static_cast<int64_t>(zL) * pn;
        for (int row = warp; row < 4 * ny; row += blockDim.x >> 5) {
            const int tb = (row >= 2 * ny ? 2 : 0) + (row >= 3 * ny || (row >= ny && row < 2 * ny) ? 1 : 0);
            const int y = row - tb * ny;
            for (int x = lane; x < nx; x += 32)
                CPA(Dp, tb * PS + y * RS + x, dp_n, D, tb * dplane_n + y * nx + x, 8 * dplane_n);
        }
    };
    // the copies of the first function's planes are in flight while the tables are built
    auto load_Bb = [&](const FnRec& r) {                       // one thread
        const T* Bb = static_cast<const T*>(a.ws) + r.ws_Bb + (static_cast<int64_t>(bz) * nzp + zb) * Y * X;
        const int rem = static_cast<int>((reinterpret_cast<uintptr_t>(Bb) & 15) / sizeof(T));
        const uint32_t bytes = static_cast<uint32_t>((static_cast<size_t>(rem + Y * X) * sizeof(T) + 15) & ~size_t(15));
        if (dead) return;
        bulk_fence();                                          // Gs was read and written there
        bulk_expect(mbar, bytes);
        bulk_load(tc::saddr(plb), Bb - rem, bytes, mbar);
    };
    // For the bulk copies in flight.  Once a wait has run out (dead: 1 + the phase that is still open) no
    // thread waits any more and the first one, behind the CTA's next barrier, announces no more
    // copies: a phase may be opened again only once it is complete.
    auto wait = [&]() {
#ifndef LSW_CHECKED
        if (!dead && (a.wait_out || !tc::mbar_wait(mbar, phase))) {
            atomicOr(st, ST_WAIT_TIMEOUT);
            dead = 1 + static_cast<int>(phase);
        }
        phase ^= 1;
#endif
    };
#ifndef LSW_CHECKED
    if (tid == 0) load_Bb(r0);
#endif
    // the CTA's next item, by the last thread: taken no earlier than at the end of this one (a CTA
    // that holds a second item unbegun delays the last ones)
    const bool fetch = s_next && tid == blockDim.x - 1;
    auto item = [&](int k) { return k < a.n_items_bwd ? a.items_bwd[k] : make_int2(0, -1); };
    if (tid == 0) {
        ylo = nyp;
        yhi = -1;
    }
    for (int i = tid; i < 2 * L.nb_x; i += blockDim.x) {
        hlo[i] = nyp;
        hhi[i] = -1;
    }
    for (int i = tid; i < 2 * L.nb_y; i += blockDim.x) {
        if (i < L.nb_y) {
            cq0[i] = X;
            cq1[i] = -1;
        }
        rq0[i] = nxp;
        rq1[i] = -1;
    }
    if (dplane) stage_D(r0);
    const int64_t crow0 = at.rowPc + static_cast<int64_t>(nyp) * zb, frow0 = at.rowPf + static_cast<int64_t>(nyp) * zb;
    const int q0 = LD(a.rowptr, frow0, a.rowptr_n), q1 = LD(a.rowptr, frow0 + nyp, a.rowptr_n);
    __syncthreads();
    // member x range of each row of this plane (coarse part of L', fine hull) and of the D plane
    // (coarse and fine members of L), a row and part per thread: one chain of loads for all
    for (int i = tid; i < 2 * nyp + (dplane ? 2 * ny : 0); i += blockDim.x) {
        const bool inP = i < 2 * nyp;
        const int part = inP ? i >= nyp : i - 2 * nyp >= ny, y = inP ? i - part * nyp : i - 2 * nyp - part * ny;
        const int64_t row = inP ? (part ? frow0 : crow0) + y : (part ? at.rowLf : at.rowLc) + y + static_cast<int64_t>(ny) * zL;
        const int64_t sg = inP ? (part ? at.segPf : at.segPc) : (part ? at.segLf : at.segLc);
        const int s0 = LD(a.rowptr, row, a.rowptr_n), s1 = LD(a.rowptr, row + 1, a.rowptr_n);
        int lo = -1, hi = -1, off = 0;
        if (s1 > s0) {
            const Seg first = LD(a.seg, sg + s0, a.seg_n);
            lo = first.x0;
            off = first.off;
            hi = LD(a.seg, sg + s1 - 1, a.seg_n).x1;
        }
        if (!inP) {
            lxr[part * ny + y] = lo < 0 ? -1 : lo << 16 | hi;
            continue;
        }
        (part ? fx0 : rx0)[y] = static_cast<int16_t>(lo);
        (part ? fx1 : rx1)[y] = static_cast<int16_t>(hi);
        if (!part) roff[y] = off;
        if (lo >= 0 && part == (bz != 0)) {                    // rows that the compressed write reads
            atomicMin(&ylo, y);
            atomicMax(&yhi, y);
        }
    }
    if (dplane && tid < 4) ST(Dp, tid * PS + PS - 1, dp_n, T(0));
    // the plane's fine members: m0 .. m0 + nm - 1 of each type's block
    int m0 = 0, nm = 0;
    if (q1 > q0) {
        const Seg sl = LD(a.seg, at.segPf + q1 - 1, a.seg_n);
        m0 = LD(a.seg, at.segPf + q0, a.seg_n).off;
        nm = sl.off + (sl.x1 - sl.x0 + 1) - m0;
    }
    const bool listed = nm <= L.memN;
    if (listed)
        for (int q = q0 + static_cast<int>(blockDim.x) - 1 - tid; q < q1; q += blockDim.x) {
            const Seg g = LD(a.seg, at.segPf + q, a.seg_n);
            const int at0 = static_cast<int>(g.row - static_cast<int64_t>(nyp) * zb) * nxp;
            for (int x = g.x0; x <= g.x1; ++x) ST(memb, g.off - m0 + (x - g.x0), L.memN, static_cast<uint16_t>(at0 + x));
        }
    __syncthreads();
    const int ylo_ = ylo, yhi_ = yhi;
    if (yhi_ < 0) {                                            // uniform; nothing to write in this plane
        wait();
        cp_wait();
        if (fetch) *s_next = item(atomicAdd(a.queue + 1, 1));
        __syncthreads();
        return;
    }
    // The x range of row b whose outputs of the y-type pair `by` (types 2 by, 2 by + 1 of
    // this plane) the compressed write reads: the coarse members where the pair holds the
    // scaling type 0 (bz = 0, by = 0), else the hull of the row's fine members (the wavelet
    // types are stored on fine members only).  lo < 0: none.
    auto need = [&](int by, int b, int& lo, int& hi) {
        const bool c = bz == 0 && by == 0;
        lo = c ? rx0[b] : fx0[b];
        hi = c ? rx1[b] : fx1[b];
    };
    // ---- ranges: the y pass's columns per block of NB rows (for row b and pair by its blocks
    //      k = lo/NB .. hi/NB of the needed range read x' in [2 (k NB + dx),
    //      2 (k NB + NB - 1 + dx) + 30]); the kinetic y arm's columns (per x type bx, the pair of
    //      types bx, bx + 2, and block of rows: the hull of the rows' needed ranges); the x pass's
    //      rows per (pair, block of NB columns); beside them, on other warps first, the hulls of
    //      D's columns
    const int nbb = (yhi_ - ylo_ + NB) / NB;
    for (int i = static_cast<int>(blockDim.x) - 1 - tid; i < 2 * (yhi_ - ylo_ + 1); i += blockDim.x) {
        const int by = i & 1, b = ylo_ + (i >> 1), q = (b - ylo_) / NB;
        int lo, hi;
        need(by, b, lo, hi);                                   // (the same rule for x types)
        if (lo < 0) continue;
        atomicMin(&cq0[q], 2 * ((lo / NB) * NB + dx));
        atomicMax(&cq1[q], 2 * ((hi / NB) * NB + NB - 1 + dx) + 30);
        atomicMin(&rq0[by * nbb + q], lo);
        atomicMax(&rq1[by * nbb + q], hi);
        for (int k = lo / NB; k <= hi / NB; ++k) {
            atomicMin(&hlo[by * L.nb_x + k], b);
            atomicMax(&hhi[by * L.nb_x + k], b);
        }
    }
    if (dplane)
        for (int i = tid; i < 2 * nx; i += blockDim.x) {
            const int part = i >= nx, x = i - part * nx;
            const int* rows = lxr + part * ny;
            int lo = -1, hi = 0;
#pragma unroll 8
            for (int y = 0; y < ny; ++y) {
                const int v = rows[y];
                if (v >= 0 && x >= v >> 16 && x <= (v & 0xffff)) {
                    if (lo < 0) lo = y;
                    hi = y;
                }
            }
            cyr[i] = lo < 0 ? -1 : lo << 16 | hi;
        }
    __syncthreads();
    // pre[e] = the counts of entries before e (a warp)
    auto scan = [&](int* pre, int n, auto count) {
        if (lane == 0) pre[0] = 0;
        int base = 0;
        for (int k = 0; k < n; k += 32) {
            int v = k + lane < n ? count(k + lane) : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += u;
            }
            if (k + lane < n) pre[k + lane + 1] = base + v;
            base += __shfl_sync(0xffffffffu, v, 31);
        }
    };
    if (warp == 0)
        scan(pq, nbb, [&](int q) {
            cq0[q] = max(cq0[q], 0);
            cq1[q] = min(cq1[q], X - 1);
            return max(0, cq1[q] - cq0[q] + 1);
        });
    if (warp == 1)
        scan(rqp, 2 * nbb, [&](int i) {
            rq0[i] = max(rq0[i], -dx);                         // columns of the D plane
            rq1[i] = min(rq1[i], nx - 1 - dx);
            return max(0, rq1[i] - rq0[i] + 1);
        });
    if (warp == 2) scan(hp, 2 * L.nb_x, [&](int e) { return max(0, hhi[e] - hlo[e] + 1); });
    __syncthreads();
    // tasks, block-major: consecutive rows (columns) of a block on consecutive lanes (odd row
    // strides: no bank conflicts, and nearly equal kinetic hulls); a warp per block
    const int ntx = hp[2 * L.nb_x], nty = rqp[2 * nbb], nwarp = blockDim.x >> 5;
    for (int e = warp; e < 2 * L.nb_x; e += nwarp)
        for (int b = hlo[e] + lane; b <= hhi[e]; b += 32)
            ST(task, hp[e] + b - hlo[e], L.taskN, static_cast<uint16_t>((e << kx) | b));
    for (int e = nwarp - 1 - warp; e < 2 * nbb; e += nwarp)
        for (int x = rq0[e] + lane; x <= rq1[e]; x += 32)
            ST(taskk, rqp[e] + x - rq0[e], L.taskkN, static_cast<uint16_t>((e << ky) | x));
    const T ks = static_cast<T>(a.kin_scale);
    const int pnp = nyp * nxp;
    const int64_t gplane = static_cast<int64_t>(pnp) * nzp;
    const FastDiv fd_nxp(nxp);
    for (int c = 0; c < cnt; ++c) {
        const FnRec r = a.fn[fl + c];
        const T* Bb = static_cast<const T*>(a.ws) + r.ws_Bb + (static_cast<int64_t>(bz) * nzp + zb) * Y * X;
        [[maybe_unused]] const int64_t bb_room = 2LL * nzp * Y * X - (static_cast<int64_t>(bz) * nzp + zb) * Y * X;
        // ---- the Bb plane
#ifdef LSW_CHECKED
        T* const pl = plb;
        for (int i = tid; i < Y * X; i += blockDim.x) CPA(pl, i, pl_n, Bb, i, bb_room);
#else
        const int rem = static_cast<int>((reinterpret_cast<uintptr_t>(Bb) & 15) / sizeof(T));
        T* const pl = plb + rem;
        if (tid == 0 && c > 0) load_Bb(r);
        wait();
#endif
#ifdef LSW_CHECKED
        cp_wait();
        __syncthreads();
#endif
        T ekin_t = 0;
        const T* G = static_cast<const T*>(a.ws) + r.ws_G;
        const int g_r0 = ylo_ * nxp, g_n = (yhi_ - ylo_ + 1) * nxp;
        const int slot = (pnp + 15) & ~7;                      // a type's place in mid (16-byte multiple)
        auto g_rem = [&](int tb) -> int {
#ifdef LSW_CHECKED
            return 0;
#else
            const T* src = G + (tb + 4 * bz) * gplane + static_cast<int64_t>(zb) * pnp + g_r0;
            return static_cast<int>((reinterpret_cast<uintptr_t>(src) & 15) / sizeof(T));
#endif
        };
        // ---- phase 0, y pass: blocks of NB rows b within [ylo, yhi], the listed columns -> mid;
        //      phase 1, x pass and kinetic x arm: the listed (y type, block of columns, row) -> Gs;
        //      phase 2, kinetic y arm: the listed (x type, block of rows, column), added to Gs
#pragma unroll 1
        for (int ph = 0; ph < 3; ++ph) {
            const int nt = ph == 0 ? pq[nbb] : ph == 1 ? ntx : dplane ? nty : 0;
            for (int i0 = warp * 32; i0 < nt; i0 += blockDim.x) {   // whole warps: kinetic ranges are a warp's
                const bool on = i0 + lane < nt;
                const int it = on ? i0 + lane : i0;
                // the window: position m of the filter is at first + m on a line of n values at wp + woff
                const T* wp = pl;
                int woff, wstride, first, n;
                // the arm: D row or column a0 (stride sd), window position p is D position f0 + p of kn
                int a0 = 0, sd = 1, f0 = 0, kn = 0, dist = 0, h0 = 0, h1 = 0;
                const int* hull = lxr;
                int out, ostep, onum, odist;                    // outputs j < onum at out + j ostep (+ odist)
                if (ph == 0) {
                    int q = 0;
                    while (it >= pq[q + 1]) ++q;
                    const int xo = cq0[q] + (it - pq[q]), b0 = ylo_ + q * NB;
                    woff = xo;
                    wstride = X;
                    first = 2 * (b0 + dy);
                    n = Y;
                    out = b0 * X + xo;
                    ostep = X;
                    odist = nyp * X;
                    onum = yhi_ + 1 - b0;
                } else if (ph == 1) {
                    const int code = task[it], e = code >> kx, b = code & ((1 << kx) - 1);
                    const int by = e >= L.nb_x, x0 = (e - by * L.nb_x) * NB, y = b + dy;
                    wp = mid;
                    woff = (by * nyp + b) * X;
                    wstride = 1;
                    first = 2 * (x0 + dx);
                    n = X;
                    out = ((2 * by) * nyp + b) * nxp + x0;
                    ostep = 1;
                    odist = pnp;
                    onum = nxp - x0;
                    f0 = x0 + dx - KIN_HALF;
                    const bool in = dplane && y >= 0 && y < ny;
                    kn = in ? nx : 0;
                    a0 = 2 * by * PS + (in ? y * RS : 0);
                    dist = PS;
                    h0 = (bz == 0 && by == 0 ? 0 : ny) + y;
                    h1 = ny + y;
                } else {
                    const int code = taskk[it], e = code >> ky, xb = code & ((1 << ky) - 1);
                    const int bx = e >= nbb, b0 = ylo_ + (e - bx * nbb) * NB, x = xb + dx;
                    woff = wstride = first = n = 0;
                    out = (bx * nyp + b0) * nxp + xb;
                    ostep = nxp;
                    odist = 2 * pnp;
                    onum = yhi_ + 1 - b0;
                    f0 = b0 + dy - KIN_HALF;
                    kn = ny;
                    a0 = bx * PS + x;
                    sd = RS;
                    dist = 2 * PS;
                    hull = cyr;
                    h0 = (bz == 0 && bx == 0 ? 0 : nx) + x;
                    h1 = nx + x;
                }
                T s[NB], d[NB];
                if (ph < 2) {
                    bwd_window<T, NB>(wp, woff, wstride, first, n, s, d, ph ? mid_n : pl_n, st);
                } else {
#pragma unroll
                    for (int j = 0; j < NB; ++j) s[j] = d[j] = T(0);
                }
                if (ph > 0 && dplane) {
                    int s0 = Arm::NP, e0 = 0, s1 = Arm::NP, e1 = 0;
                    if (on && kn) {
                        const int v0 = hull[h0], v1 = hull[h1];
                        if (v0 >= 0) s0 = (v0 >> 16) - f0, e0 = (v0 & 0xffff) - f0 + 1;
                        if (v1 >= 0) s1 = (v1 >> 16) - f0, e1 = (v1 & 0xffff) - f0 + 1;
                    }
                    s0 = __reduce_min_sync(0xffffffffu, s0);
                    e0 = __reduce_max_sync(0xffffffffu, e0);
                    s1 = __reduce_min_sync(0xffffffffu, s1);
                    e1 = __reduce_max_sync(0xffffffffu, e1);
                    // window positions inside the box, a bit each; the others read the zero after
                    // the first type's rows and, `dist` further, after the rows of another
                    const int plo = min(max(-f0, 0), 63), phi = min(max(kn - f0, 0), Arm::NP);
                    const uint64_t in = phi > plo ? ((1ull << phi) - 1) & ~((1ull << plo) - 1) : 0;
                    const uint32_t in0 = static_cast<uint32_t>(in), in1 = static_cast<uint32_t>(in >> 32);
                    const int base = a0 + f0 * sd;
                    T o0[NB], o1[NB], c0[NB], c1[NB];
                    Arm::run(o0, o1, c0, c1, Dp, dp_n, dist,
                             [&](int p) { return (p < 32 ? in0 >> (p & 31) : in1 >> (p & 31)) & 1 ? base + p * sd : PS - 1; },
                             s0, e0, s1, e1, st);
#pragma unroll
                    for (int j = 0; j < NB; ++j) {
                        o0[j] *= ks;
                        o1[j] *= ks;
                        s[j] += o0[j];
                        d[j] += o1[j];
                        if (on && j < onum) ekin_t += c0[j] * o0[j] + c1[j] * o1[j];
                    }
                }
                if (on) {
                    T* const dst = ph == 0 ? mid : Gs;
                    [[maybe_unused]] const int64_t dst_n = ph == 0 ? mid_n : pl_n;
#pragma unroll
                    for (int j = 0; j < NB; ++j)
                        if (j < onum) {
                            const int o = out + j * ostep;
                            if (ph == 2) {
                                s[j] += LD(dst, o, dst_n);
                                d[j] += LD(dst, o + odist, dst_n);
                            }
                            ST(dst, o, dst_n, s[j]);
                            ST(dst, o + odist, dst_n, d[j]);
                        }
                }
            }
            if (ph == 0) cp_wait();                            // the D plane
            if (ph < 2) __syncthreads();                       // pl is dead after phase 0 (Gs reuses it), mid after 1
            if (ph == 1 && a.gstage) {
                // the z-arm plane G (types tb + 4 bz, member rows) into mid
#ifdef LSW_CHECKED
                for (int tb = 0; tb < 4; ++tb)
                    for (int i = tid; i < g_n; i += blockDim.x)
                        CPA(mid, tb * slot + i, mid_n, G, (tb + 4 * bz) * gplane + static_cast<int64_t>(zb) * pnp + g_r0 + i,
                            8 * gplane);
#else
                if (tid == 0 && !dead) {
                    bulk_fence();
                    uint32_t total = 0;
#pragma unroll
                    for (int tb = 0; tb < 4; ++tb)
                        total += static_cast<uint32_t>((static_cast<size_t>(g_rem(tb) + g_n) * sizeof(T) + 15) & ~size_t(15));
                    bulk_expect(mbar, total);
#pragma unroll
                    for (int tb = 0; tb < 4; ++tb) {
                        const int gr = g_rem(tb);
                        const uint32_t bytes = static_cast<uint32_t>((static_cast<size_t>(gr + g_n) * sizeof(T) + 15) & ~size_t(15));
                        bulk_load(tc::saddr(mid + tb * slot),
                                  G + (tb + 4 * bz) * gplane + static_cast<int64_t>(zb) * pnp + g_r0 - gr, bytes, mbar);
                    }
                }
#endif
            }
        }
        if (a.gstage) {
#ifdef LSW_CHECKED
            cp_wait();
#endif
            wait();
        }
        __syncthreads();
        if (c + 1 < cnt && dplane) stage_D(a.fn[fl + c + 1]);  // the D plane is dead; in flight during the write
        // ---- compress: members of this plane -> H phi, plus the z arm left in G by k_kin_z
        //      where its flag says so.  Coarse members (type 0) row by row, a warp per row; fine
        //      members flattened over the CTA, consecutive lanes on consecutive H phi elements.
        const unsigned char* gflag = reinterpret_cast<const unsigned char*>(static_cast<const T*>(a.ws) + r.ws_Gf);
        T* out = static_cast<T*>(a.hphi) + r.off_hphi;
        [[maybe_unused]] const int64_t out_room = a.hphi_n - r.off_hphi;
        auto zarm = [&](int t, int i) -> T {                   // type t (of 8), plane index i = b n_x' + x
            if (a.gstage) return LD(mid, (t & 3) * slot + g_rem(t & 3) + i - g_r0, mid_n);
            return LD(G, t * gplane + static_cast<int64_t>(zb) * pnp + i, 8 * gplane);
        };
        int nk = 0;
        int2 ni = make_int2(0, -1);
        if (fetch && c + 1 == cnt) nk = atomicAdd(a.queue + 1, 1);
        if (bz == 0) {                                         // scaling part s (type 0) on the coarse members
            for (int b = ylo_ + warp; b <= yhi_; b += (blockDim.x >> 5)) {
                if (rx0[b] < 0) continue;
                const int y = b + dy;
                const bool yin = y >= 0 && y < ny;
                for (int xb = rx0[b] + lane; xb <= rx1[b]; xb += 32) {
                    const int x = xb + dx;
                    T v = LD(Gs, b * nxp + xb, pl_n);
                    if (yin && x >= 0 && x < nx && LD(gflag, y * nx + x, 4LL * pn)) v += zarm(0, b * nxp + xb);
                    ST(out, roff[b] + (xb - rx0[b]), out_room, v);
                }
            }
        }
        if (fetch && c + 1 == cnt) ni = item(nk);
        for (int m = tid; m < nm; m += blockDim.x) {
            int i;
            if (listed) {
                i = LD(memb, m, L.memN);
            } else {                                           // more members than the list holds: find the segment
                int lo = q0, hi = q1 - 1;
                while (lo < hi) {
                    const int k = (lo + hi + 1) >> 1;
                    if (LD(a.seg, at.segPf + k, a.seg_n).off - m0 <= m) lo = k;
                    else hi = k - 1;
                }
                const Seg g = LD(a.seg, at.segPf + lo, a.seg_n);
                i = static_cast<int>(g.row - static_cast<int64_t>(nyp) * zb) * nxp + g.x0 + (m - (g.off - m0));
            }
            const int b = fd_nxp.div(i), xb = i - b * nxp;
            const int y = b + dy, x = xb + dx;
            const bool zin = y >= 0 && y < ny && x >= 0 && x < nx;
#pragma unroll
            for (int tb = 0; tb < 4; ++tb) {
                const int t = tb + 4 * bz;
                if (t == 0) continue;
                T v = LD(Gs, tb * pnp + i, pl_n);
                if (zin && LD(gflag, tb * pn + y * nx + x, 4LL * pn)) v += zarm(t, i);
                ST(out, at.ncP + static_cast<int64_t>(t - 1) * at.nfP + m0 + m, out_room, v);
            }
        }
        if (fetch && c + 1 == cnt) *s_next = ni;
        const double ekin = warp_sum(static_cast<double>(ekin_t));
        if (lane == 0 && ekin != 0.0) atomicAdd(a.e_kin + r.f, ekin);
        __syncthreads();                                       // Gs and mid are free for the next function
    }
}

// Persistent form (a.items_bwd set): the batch's (atom's functions, z'' plane, z type) items,
// largest first, from the second queue counter; otherwise one CTA per grid slot (blockIdx.x =
// 2 z'' + b_z, blockIdx.y = function).  Two CTAs of 8 warps per SM (128 registers).
template <class T>
__global__ void __launch_bounds__(BWD_THREADS, 2) k_bwd_xy(HphiLaunch a) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int dead;                       // 1 + the phase that a wait ran out on; 0: none did
    if (threadIdx.x == 0) {
        tc::mbar_init(tc::saddr(smem_raw));
        dead = 0;
    }
    __syncthreads();
    uint32_t phase = 0;
    if (a.items_bwd) {
        __shared__ int2 s_item;
        if (threadIdx.x == 0) {
            const int k = atomicAdd(a.queue + 1, 1);
            s_item = k < a.n_items_bwd ? a.items_bwd[k] : make_int2(0, -1);
        }
        __syncthreads();
        for (;;) {
            const int2 it = s_item;   // (the next one is written behind the plane's barriers)
            if (it.y < 0) break;
            bwd_plane<T>(a, it.x, it.y >> 11, (it.y >> 1) & 1023, it.y & 1, phase, dead, &s_item);
        }
    } else {
        bwd_plane<T>(a, blockIdx.y, 1, blockIdx.x >> 1, blockIdx.x & 1, phase, dead, nullptr);
    }
    // the copies still in flight write to this CTA's shared memory: end behind them (or the limit)
    if (threadIdx.x == 0 && dead) bwd_last_wait(tc::saddr(smem_raw), dead - 1);
}

// ---------------------------------------------------------------- density: pair products
//
// rho_j = sum_ab K_ab u_a(j) u_b(j) (Eq. density) per tile of DT_X x DT_Y x DT_Z grid
// points, over the functions whose real-space blocks meet the tile (App. D: the density
// is formed like the scalar products, from the functions present at each point).  The
// quadratic form depends only on the symmetric part of K, so the functions of a tile are
// taken in chunks of DT_MC and every pair of chunks A <= B once: the coefficient block is
// K_ab for A = B and K_ab + K_ba for A < B.  Each thread owns DT_PP points and keeps the
// B chunk's values there in registers; the coefficient block sits in shared memory and is
// read as a broadcast.  Products and the chunk-pair partial sums run in T, the total per
// point in FP64; every point of the grid is written (0 where no block reaches).
//
// The chunks (32 functions of the tile's list in order) fix the sums; what is left out adds exact
// zeros.  Bound: instruction issue and its latencies at two CTAs an SM (128 registers: a chunk's
// values at two points are 64 of them).  So:
//   - a warp takes a block of 8 x 4 x 2 points (a row of 32 meets nearly every function of the tile)
//     and forms only the products of A functions with a value there, with groups of four B
//     functions that have one and are in the pattern;
//   - the pattern is searched once per pair of atoms of a tile (an atom's functions have equal
//     pattern rows and consecutive columns), the next pair's coefficients are copied during the
//     products into a second block, one barrier per pair, four A functions at a time;
//   - a chunk's values are loaded where their boxes meet the warp's block, all loads before the
//     first test of a value (7.1 ms with each tested as it arrives).
// 300 atoms (1,038 functions) in FP32: 5.1 ms; every function of the tile at rows of 32 points, a
// search per coefficient: 13.0.

struct __align__(16) DensRec {       // one function of a chunk
    int64_t off;                     // block in the store
    int o[3], d[3];
    int64_t rp;                      // first pattern entry
    int f;
    int lead, grp;                   // first entry of its atom, number of its atom (in the chunk or tile)
};

// u_f at the thread's points (x, y, z + i); 0 outside f's block.
template <class T, class Rec>
__device__ __forceinline__ void dens_u(const DensLaunch& a, const Rec& df, int x, int y, int z, T (&u)[DT_PP]) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 13;
    const int lx = x - df.o[0], ly = y - df.o[1], lz = z - df.o[2];
    const bool in = static_cast<unsigned>(lx) < static_cast<unsigned>(df.d[0]) &&
                    static_cast<unsigned>(ly) < static_cast<unsigned>(df.d[1]);
    const T* U = static_cast<const T*>(a.U);
    // 32 bits hold a place in the block (its planes fit in shared memory), and are used only inside it
    const uint32_t n = static_cast<uint32_t>(df.d[0]) * df.d[1], at = lz * n + static_cast<uint32_t>(ly) * df.d[0] + lx;
#pragma unroll
    for (int i = 0; i < DT_PP; ++i)
        u[i] = in && static_cast<unsigned>(lz + i) < static_cast<unsigned>(df.d[2]) ? LD(U, df.off + static_cast<int64_t>(at + i * n), a.U_n) : T(0);
}

// Records of the chunk of n functions tfn[at ..] (one warp); returns the number of atoms.
__device__ __forceinline__ int dens_records(const DensLaunch& a, int64_t at, int n, DensRec* rec, int* leads) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 13;
    const int lane = threadIdx.x & 31;
    int atom = -1;
    if (lane < n) {
        DensRec& r = rec[lane];
        r.f = LD(a.tfn, at + lane, a.tfn_n);
        const DensFn df = LD(a.fn, r.f, a.fn_n);
        r.off = df.off;
        r.rp = LD(a.row_ptr, r.f, a.rowp_n);
        for (int k = 0; k < 3; ++k) r.o[k] = df.o[k], r.d[k] = df.d[k];
        atom = LD(a.sf_atom, r.f, a.fn_n);
    }
    const int before = __shfl_up_sync(0xffffffffu, atom, 1);
    const unsigned m = __ballot_sync(0xffffffffu, lane < n && (lane == 0 || atom != before));
    if (lane < n) {
        const unsigned up = m & (0xffffffffu >> (31 - lane));
        rec[lane].lead = 31 - __clz(up);
        rec[lane].grp = __popc(up) - 1;
        if (m >> lane & 1) leads[__popc(up) - 1] = lane;
    }
    return __popc(m);
}

// Position of column fb in row fa of the pattern, from the row's start; -1 outside the pattern.
__device__ __forceinline__ int dens_find(const DensLaunch& a, int64_t rp, int fa, int fb) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 13;
    int64_t lo = rp, hi = LD(a.row_ptr, fa + 1, a.rowp_n);
    const int64_t end = hi;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (LD(a.col, mid, a.nnz) < fb)
            lo = mid + 1;
        else
            hi = mid;
    }
    return (lo < end && LD(a.col, lo, a.nnz) == fb) ? static_cast<int>(lo - rp) : -1;
}

__device__ __forceinline__ void lds16(const float* p, float (&v)[4]) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
}
__device__ __forceinline__ void lds16(const double* p, double (&v)[2]) {
    const double2 t = *reinterpret_cast<const double2*>(p);
    v[0] = t.x, v[1] = t.y;
}

// The points of a thread and their sums, and the values of the B chunk there.  A warp's points
// are a block of 8 x 4 x DT_PP.
template <class T>
struct DensPoints {
    int x, y, z;
    double acc[DT_PP];
    T ub[DT_MC][DT_PP];
    unsigned fmask;            // B functions with a nonzero value at some point of the warp
    __device__ __forceinline__ void init(const DensLaunch& a) {
        static_assert(DT_X == 32 && DT_Y == 4 && DT_PP * DT_THREADS == DT_X * DT_Y * DT_Z, "a warp's block of points");
        const int tile = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const int tx = tile % a.ntile[0];
        const int ty = (tile / a.ntile[0]) % a.ntile[1];
        const int tz = tile / (a.ntile[0] * a.ntile[1]);
        x = tx * DT_X + (warp & 3) * 8 + (lane & 7);
        y = ty * DT_Y + (lane >> 3);
        z = tz * DT_Z + (warp >> 2) * DT_PP;
#pragma unroll
        for (int i = 0; i < DT_PP; ++i) acc[i] = 0.0;
    }
    __device__ __forceinline__ void load_b(const DensLaunch& a, const DensRec* rb, int nb) {
        const int lane = threadIdx.x & 31;
        bool meets = false;                        // lane j: the box of function j and the warp's block of points
        if (lane < nb) {
            const DensRec& r = rb[lane];
            const int bx = x - (lane & 7) - r.o[0], by = y - (lane >> 3) - r.o[1], bz = z - r.o[2];
            meets = bx + 8 > 0 && bx < r.d[0] && by + 4 > 0 && by < r.d[1] && bz + DT_PP > 0 && bz < r.d[2];
        }
        const unsigned bmask = __ballot_sync(0xffffffffu, meets);
#pragma unroll
        for (int j = 0; j < DT_MC; ++j) {
            if (bmask >> j & 1) {
                dens_u<T>(a, rb[j], x, y, z, ub[j]);
            } else {
#pragma unroll
                for (int i = 0; i < DT_PP; ++i) ub[j][i] = T(0);
            }
        }
        fmask = 0;
#pragma unroll
        for (int j = 0; j < DT_MC; ++j) {
            bool any = false;
#pragma unroll
            for (int i = 0; i < DT_PP; ++i) any |= ub[j][i] != T(0);
            if (__any_sync(0xffffffffu, any)) fmask |= 1u << j;
        }
    }
    // acc += sum over the A chunk of u_a sum_b kb_ab u_b (partial sums of the pair of chunks in T).
    // amask: the A functions with a nonzero value at some point of the warp; kmask: the B
    // functions within the pattern, per A function.  RW rows (A functions) at a time, each a chain of
    // its own: one row's products depend on one another (up to 32 in a row).
    __device__ __forceinline__ void products(const DensLaunch& a, const DensRec* ra, unsigned amask, const T* kb,
                                             const unsigned* kmask) {
        constexpr int VW = 16 / sizeof(T), NG = DT_MC / 4, RW = sizeof(T) == 4 ? 4 : 1;
        const int lane = threadIdx.x & 31;
        unsigned rows = __ballot_sync(0xffffffffu, (amask >> lane & 1) && (kmask[lane] & fmask));
        if (rows == 0) return;                     // every product is an exact zero
        T part[DT_PP], next[RW][DT_PP];
        int id[RW];
        auto take = [&]() {
#pragma unroll
            for (int w = 0; w < RW; ++w) {
                id[w] = __ffs(rows) - 1;
                rows &= rows - 1;
                if (id[w] >= 0) {
                    dens_u<T>(a, ra[id[w]], x, y, z, next[w]);
                } else {
#pragma unroll
                    for (int i = 0; i < DT_PP; ++i) next[w][i] = T(0);
                }
            }
        };
#pragma unroll
        for (int i = 0; i < DT_PP; ++i) part[i] = T(0);
        take();
        while (id[0] >= 0) {
            T ua[RW][DT_PP], zz[RW][DT_PP];
            const T* row[RW];
            unsigned on = 0;
#pragma unroll
            for (int w = 0; w < RW; ++w) {
                const int r = id[w] >= 0 ? id[w] : id[0];
                on |= kmask[r];
                row[w] = kb + r * DT_MC;
#pragma unroll
                for (int i = 0; i < DT_PP; ++i) {
                    ua[w][i] = next[w][i];
                    zz[w][i] = T(0);
                }
            }
            take();
            on &= fmask;
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                if (!(on >> (4 * g) & 15)) continue;
#pragma unroll
                for (int q = 4 * g; q < 4 * g + 4; q += VW) {
                    T k[RW][VW];
#pragma unroll
                    for (int w = 0; w < RW; ++w) lds16(row[w] + q, k[w]);
#pragma unroll
                    for (int e = 0; e < VW; ++e)
#pragma unroll
                        for (int w = 0; w < RW; ++w) {
                            if constexpr (sizeof(T) == 4 && DT_PP == 2) {   // both points in one packed FMA: the same bits
                                const float2 t = __ffma2_rn(make_float2(k[w][e], k[w][e]), make_float2(ub[q + e][0], ub[q + e][1]),
                                                            make_float2(zz[w][0], zz[w][1]));
                                zz[w][0] = t.x, zz[w][1] = t.y;
                            } else {
#pragma unroll
                                for (int i = 0; i < DT_PP; ++i) zz[w][i] += k[w][e] * ub[q + e][i];
                            }
                        }
                }
            }
#pragma unroll
            for (int w = 0; w < RW; ++w)
#pragma unroll
                for (int i = 0; i < DT_PP; ++i) part[i] += ua[w][i] * zz[w][i];
        }
#pragma unroll
        for (int i = 0; i < DT_PP; ++i) acc[i] += static_cast<double>(part[i]);
    }
    __device__ __forceinline__ void store(const DensLaunch& a) const {
        [[maybe_unused]] int* ST_ = a.status;
        [[maybe_unused]] constexpr int KID = 13;
#pragma unroll
        for (int i = 0; i < DT_PP; ++i)
            if (x < a.gn[0] && y < a.gn[1] && z + i < a.gn[2])
                ST(a.rho, ((z + i) * a.gn[1] + y) * a.gn[0] + x, a.rho_n, acc[i]);
    }
};

// Row ia of the coefficient block (a warp): the value of lane b, and whether (a, b) is in the pattern.
template <class T>
__device__ __forceinline__ void dens_row(T* kb, unsigned* kmask, int ia, double v, bool in) {
    const int lane = threadIdx.x & 31;
    kb[ia * DT_MC + lane] = static_cast<T>(v);
    const unsigned m = __ballot_sync(0xffffffffu, in);
    if (lane == 0) kmask[ia] = m;
}

constexpr int DENS_MASKS = 64;       // chunks whose masks a warp keeps (the others' functions all count as present)

// The records of all functions of the tile and the pattern positions of all pairs of their
// atoms in shared memory (a.max_m functions, a.max_g atoms at most), built once per tile; the
// coefficients of the next pair of chunks are copied during the products of this one.
template <class T>
__global__ void __launch_bounds__(DT_THREADS) k_density(DensLaunch a) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 13;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* kraw = reinterpret_cast<double*>(smem_raw);                  // [2][MC][MC]: K_ab, K_ba
    T* kb = reinterpret_cast<T*>(kraw + 2 * DT_MC * DT_MC);              // [2][MC][MC], in turn
    DensRec* rec = reinterpret_cast<DensRec*>(kb + 2 * DT_MC * DT_MC);   // [max_m]
    int* rel = reinterpret_cast<int*>(rec + a.max_m);                    // [atoms][RS]
    const int RS = a.max_g | 1;                                          // odd: a column's entries in different banks
    int* lead = rel + a.max_g * RS;                                 // [max_g]
    __shared__ unsigned um[DT_THREADS / 32][DENS_MASKS];
    __shared__ unsigned kmask[2][DT_MC];        // per A function, a bit per B function: the pair is in the pattern
    __shared__ int s_ng;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t t0 = LD(a.tptr, blockIdx.x, a.tptr_n);
    const int m = static_cast<int>(LD(a.tptr, blockIdx.x + 1, a.tptr_n) - t0);
    DensPoints<T> P;
    P.init(a);
    auto all = [&](int ca) { return 0xffffffffu >> (DT_MC - min(DT_MC, m - ca)); };
    for (int k = threadIdx.x; k < m; k += DT_THREADS) {
        DensRec& r = rec[k];
        r.f = LD(a.tfn, t0 + k, a.tfn_n);
        const DensFn df = LD(a.fn, r.f, a.fn_n);
        r.off = df.off;
        r.rp = LD(a.row_ptr, r.f, a.rowp_n);
        for (int d = 0; d < 3; ++d) r.o[d] = df.o[d], r.d[d] = df.d[d];
        r.grp = LD(a.sf_atom, r.f, a.fn_n);    // its atom, renumbered below
    }
    __syncthreads();
    if (warp == 0) {                           // atoms of the list, numbered in order
        int runs = 0, first = 0, last = -1;
        for (int b = 0; b < m; b += 32) {
            const int k = b + lane;
            const int at = k < m ? rec[k].grp : -2;
            int before = __shfl_up_sync(0xffffffffu, at, 1);
            if (lane == 0) before = last;
            const unsigned mk = __ballot_sync(0xffffffffu, k < m && at != before);
            const unsigned up = mk & (0xffffffffu >> (31 - lane));
            if (k < m) {
                rec[k].lead = up ? b + 31 - __clz(up) : first;
                rec[k].grp = runs + __popc(up) - 1;
                if (mk >> lane & 1) lead[rec[k].grp] = k;
            }
            if (mk) first = b + 31 - __clz(mk);
            runs += __popc(mk);
            last = __shfl_sync(0xffffffffu, at, 31);
        }
        if (lane == 0) s_ng = runs;
    }
    __syncthreads();
    const int ng = s_ng;
    for (int e = threadIdx.x; e < ng * ng; e += DT_THREADS) {
        const DensRec &A = rec[lead[e / ng]], &B = rec[lead[e % ng]];
        rel[e / ng * RS + e % ng] = dens_find(a, A.rp, A.f, B.f);
    }
    __syncthreads();
    // coefficients of the pair of chunks (ca, cb): each thread copies its own entries
    unsigned in = 0;                           // per row of this warp: the lane's pair is in the pattern
    int ib = -1, gb = 0;                       // the lane's B function and what belongs to it
    int64_t rb = 0;
    int ob = 0;
    auto issue = [&](int ca, int cb) {
        in = 0;
        if (ib != cb + lane) {
            ib = cb + lane;
            if (ib < m) gb = rec[ib].grp, rb = rec[ib].rp, ob = ib - rec[ib].lead;
        }
#pragma unroll
        for (int k = 0; k < DT_MC * 32 / DT_THREADS; ++k) {
            const int ia = warp + k * (DT_THREADS / 32);
            int64_t ab = -1, ba = -1;
            if (ca + ia < m && ib < m) {
                const DensRec& A = rec[ca + ia];
                const int r = rel[A.grp * RS + gb], q = ca != cb ? rel[gb * RS + A.grp] : -1;
                if (r >= 0) ab = A.rp + (r + ob);
                if (q >= 0) ba = rb + (q + ca + ia - A.lead);
                if (r >= 0 || q >= 0) in |= 1u << k;
            }
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int64_t at = s ? ba : ab;
                const int to = (s * DT_MC + ia) * DT_MC + lane;
                if (at >= 0) CPA(kraw, to, 2 * DT_MC * DT_MC, a.K, at, a.nnz);
                else kraw[to] = 0.0;
            }
        }
    };
    auto finish = [&](int to) {
        cp_wait();
#pragma unroll
        for (int k = 0; k < DT_MC * 32 / DT_THREADS; ++k) {
            const int ia = warp + k * (DT_THREADS / 32);
            dens_row(kb + to * DT_MC * DT_MC, kmask[to], ia, kraw[ia * DT_MC + lane] + kraw[(DT_MC + ia) * DT_MC + lane], in >> k & 1);
        }
        __syncthreads();
    };
    int cur = 0;
    if (m > 0) {
        issue(0, 0);
        finish(0);
    }
    for (int cb = 0; cb < m; cb += DT_MC) {
        P.load_b(a, rec + cb, min(DT_MC, m - cb));
        if (cb / DT_MC < DENS_MASKS && lane == 0) um[warp][cb / DT_MC] = P.fmask;
        __syncwarp();
        for (int ca = 0; ca <= cb; ca += DT_MC) {
            const bool more = ca < cb || cb + DT_MC < m;
            if (more) issue(ca < cb ? ca + DT_MC : 0, ca < cb ? cb : cb + DT_MC);
            P.products(a, rec + ca, ca / DT_MC < DENS_MASKS ? um[warp][ca / DT_MC] : all(ca), kb + cur * DT_MC * DT_MC, kmask[cur]);
            cur ^= 1;                          // the other block's readers passed the last barrier
            if (more) finish(cur);
        }
    }
    P.store(a);
}

// The same for grids with a tile whose tables do not fit: a chunk's records at a time, the pattern
// searched per pair of chunks (300 atoms in FP32: 6.9 ms where the tables give 5.1; 60 atoms 1.18, 0.93).
template <class T>
__global__ void __launch_bounds__(DT_THREADS) k_density_big(DensLaunch a) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 13;
    __shared__ __align__(16) T kb[DT_MC * DT_MC];
    __shared__ DensRec ra[DT_MC], rb[DT_MC];
    __shared__ int la[DT_MC], lb[DT_MC], rel[2][DT_MC * DT_MC], ng[2];
    __shared__ unsigned um[DT_THREADS / 32][DENS_MASKS];
    __shared__ unsigned kmask[DT_MC];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t t0 = LD(a.tptr, blockIdx.x, a.tptr_n);
    const int m = static_cast<int>(LD(a.tptr, blockIdx.x + 1, a.tptr_n) - t0);
    DensPoints<T> P;
    P.init(a);
    auto all = [&](int ca) { return 0xffffffffu >> (DT_MC - min(DT_MC, m - ca)); };
    for (int cb = 0; cb < m; cb += DT_MC) {
        const int nb = min(DT_MC, m - cb);
        __syncthreads();       // the previous chunk's readers of rb are done
        if (warp == 0) {
            const int g = dens_records(a, t0 + cb, nb, rb, lb);
            if (lane == 0) ng[1] = g;
        }
        __syncthreads();
        P.load_b(a, rb, nb);
        if (cb / DT_MC < DENS_MASKS && lane == 0) um[warp][cb / DT_MC] = P.fmask;
        __syncwarp();
        for (int ca = 0; ca <= cb; ca += DT_MC) {
            const int na = min(DT_MC, m - ca);
            __syncthreads();   // the previous block's readers are done
            if (warp == 0) {
                const int g = dens_records(a, t0 + ca, na, ra, la);
                if (lane == 0) ng[0] = g;
            }
            __syncthreads();
            for (int e = threadIdx.x; e < ng[0] * ng[1]; e += DT_THREADS) {
                const int ga = e / ng[1], gb = e - ga * ng[1];
                const DensRec &A = ra[la[ga]], &B = rb[lb[gb]];
                rel[0][ga * DT_MC + gb] = dens_find(a, A.rp, A.f, B.f);
                if (ca != cb) rel[1][ga * DT_MC + gb] = dens_find(a, B.rp, B.f, A.f);
            }
            __syncthreads();
            for (int ia = warp; ia < DT_MC; ia += DT_THREADS / 32) {
                double v = 0.0;
                bool in = false;
                if (ia < na && lane < nb) {
                    const DensRec &A = ra[ia], &B = rb[lane];
                    const int r = rel[0][A.grp * DT_MC + B.grp];
                    if (r >= 0) v = LD(a.K, A.rp + r + (lane - B.lead), a.nnz), in = true;
                    if (ca != cb) {
                        const int q = rel[1][A.grp * DT_MC + B.grp];
                        if (q >= 0) v += LD(a.K, B.rp + q + (ia - A.lead), a.nnz), in = true;
                    }
                }
                dens_row(kb, kmask, ia, v, in);
            }
            __syncthreads();
            P.products(a, ra, ca / DT_MC < DENS_MASKS ? um[warp][ca / DT_MC] : all(ca), kb, kmask);
        }
    }
    P.store(a);
}

// Grids whose tiles hold at most M functions: every coefficient looked up by a thread of its own
// while the threads load the functions' values, one barrier.  There the tables and the masks above
// are only a longer chain of loads and barriers.  Kernel times with them, with M = 8 and with M = 16:
// one function on a 31^3 box FP32 33.8, 6.1, 8.1 us, FP64 103, 17, 30; two atoms (8 functions) FP32
// 47, 15, 23, FP64 194, 111, 209; four atoms (13 functions) FP32 68, -, 30, FP64 343, -, 360: up to
// 16 in FP32, up to 8 in FP64.  The same sums in the same order as for one chunk.
template <class T, int M>
__global__ void __launch_bounds__(DT_THREADS) k_density_few(DensLaunch a) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 13;
    __shared__ T kb[M * M];
    const int64_t t0 = LD(a.tptr, blockIdx.x, a.tptr_n);
    const int m = static_cast<int>(LD(a.tptr, blockIdx.x + 1, a.tptr_n) - t0);
    DensPoints<T> P;
    P.init(a);
    for (int e = threadIdx.x; e < m * m; e += DT_THREADS) {
        const int ia = e / m, ib = e - ia * m;
        const int fa = LD(a.tfn, t0 + ia, a.tfn_n), fb = LD(a.tfn, t0 + ib, a.tfn_n);
        const int64_t rp = LD(a.row_ptr, fa, a.rowp_n);
        const int r = dens_find(a, rp, fa, fb);
        kb[ia * M + ib] = r >= 0 ? static_cast<T>(LD(a.K, rp + r, a.nnz)) : T(0);
    }
    T u[M][DT_PP];
#pragma unroll
    for (int j = 0; j < M; ++j) {
#pragma unroll
        for (int i = 0; i < DT_PP; ++i) u[j][i] = T(0);
        if (j < m) {
            const DensFn df = LD(a.fn, LD(a.tfn, t0 + j, a.tfn_n), a.fn_n);
            dens_u<T>(a, df, P.x, P.y, P.z, u[j]);
        }
    }
    __syncthreads();
    T part[DT_PP];
#pragma unroll
    for (int i = 0; i < DT_PP; ++i) part[i] = T(0);
#pragma unroll
    for (int ia = 0; ia < M; ++ia) {
        if (ia >= m) break;
        T zz[DT_PP];
#pragma unroll
        for (int i = 0; i < DT_PP; ++i) zz[i] = T(0);
#pragma unroll
        for (int ib = 0; ib < M; ++ib)
            if (ib < m)
#pragma unroll
                for (int i = 0; i < DT_PP; ++i) zz[i] += kb[ia * M + ib] * u[ib][i];
#pragma unroll
        for (int i = 0; i < DT_PP; ++i) part[i] += u[ia][i] * zz[i];
    }
#pragma unroll
    for (int i = 0; i < DT_PP; ++i) P.acc[i] = static_cast<double>(part[i]);
    P.store(a);
}

// Dynamic shared memory of k_density.
size_t density_smem(int prec, int max_m, int max_g) {
    return static_cast<size_t>(DT_MC) * DT_MC * 2 * (sizeof(double) + (prec == 0 ? sizeof(double) : sizeof(float))) +
           static_cast<size_t>(max_m) * sizeof(DensRec) + (static_cast<size_t>(max_g) * (max_g | 1) + max_g) * sizeof(int);
}

// ---------------------------------------------------------------- peak probes
//
// Denominators of the rooflines, measured on the running GPU: a dependent-chain FMA
// loop (8 independent chains per thread, operands from memory so nothing folds) and a
// 16-byte streaming copy.

template <class T>
__global__ void __launch_bounds__(256) k_fma_peak(const T* in, T* out, int iters) {
    T x = in[0], y = in[1];
    T acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = in[2 + i] + static_cast<T>(threadIdx.x);
    for (int it = 0; it < iters; ++it)
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] = acc[i] * x + y;
    T sum = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) sum += acc[i];
    if (sum == static_cast<T>(-1.2345)) out[blockIdx.x * blockDim.x + threadIdx.x] = sum;   // keeps the loop live
}

__global__ void __launch_bounds__(256) k_copy_peak(const float4* __restrict__ src, float4* __restrict__ dst, int64_t n) {
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        dst[i] = src[i];
}

cudaError_t measure_peaks(int n_sm, double* fp32_tflops, double* fp64_tflops, double* copy_gbs) {
    cudaError_t e;
    const int64_t n4 = (1LL << 30) / 16;       // 1 GiB per buffer
    float4 *a = nullptr, *b = nullptr;
    double* io = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    auto done = [&](cudaError_t r) {
        if (a) cudaFree(a);
        if (b) cudaFree(b);
        if (io) cudaFree(io);
        if (e0) cudaEventDestroy(e0);
        if (e1) cudaEventDestroy(e1);
        return r;
    };
    if ((e = cudaMalloc(&a, n4 * 16)) != cudaSuccess) return done(e);
    if ((e = cudaMalloc(&b, n4 * 16)) != cudaSuccess) return done(e);
    if ((e = cudaMalloc(&io, 4096)) != cudaSuccess) return done(e);
    if ((e = cudaMemset(a, 0, n4 * 16)) != cudaSuccess) return done(e);
    {
        const double hv[10] = {0.999999, 1e-7, 1, 2, 3, 4, 5, 6, 7, 8};
        const float hf[10] = {0.999999f, 1e-7f, 1, 2, 3, 4, 5, 6, 7, 8};
        if ((e = cudaMemcpy(io, hv, sizeof(hv), cudaMemcpyHostToDevice)) != cudaSuccess) return done(e);
        if ((e = cudaMemcpy(reinterpret_cast<char*>(io) + 128, hf, sizeof(hf), cudaMemcpyHostToDevice)) != cudaSuccess)
            return done(e);
    }
    if ((e = cudaEventCreate(&e0)) != cudaSuccess || (e = cudaEventCreate(&e1)) != cudaSuccess) return done(e);
    const int blocks = n_sm * 8;
    auto best_ms = [&](auto launch, float* out_ms) -> cudaError_t {
        float best = 1e30f;
        for (int r = 0; r < 6; ++r) {
            cudaEventRecord(e0);
            launch();
            cudaEventRecord(e1);
            cudaError_t le = cudaEventSynchronize(e1);
            if (le != cudaSuccess) return le;
            if ((le = cudaGetLastError()) != cudaSuccess) return le;
            float ms = 0;
            cudaEventElapsedTime(&ms, e0, e1);
            if (r > 0) best = std::min(best, ms);
        }
        *out_ms = best;
        return cudaSuccess;
    };
    float ms;
    const int it32 = 1 << 16, it64 = 1 << 12;
    float* io32 = reinterpret_cast<float*>(reinterpret_cast<char*>(io) + 128);
    if ((e = best_ms([&] { k_fma_peak<float><<<blocks, 256>>>(io32, io32 + 64, it32); }, &ms)) != cudaSuccess)
        return done(e);
    *fp32_tflops = 2.0 * 8.0 * it32 * blocks * 256.0 / (ms * 1e-3) / 1e12;
    if ((e = best_ms([&] { k_fma_peak<double><<<blocks, 256>>>(io, io + 128, it64); }, &ms)) != cudaSuccess)
        return done(e);
    *fp64_tflops = 2.0 * 8.0 * it64 * blocks * 256.0 / (ms * 1e-3) / 1e12;
    if ((e = best_ms([&] { k_copy_peak<<<n_sm * 16, 256>>>(a, b, n4); }, &ms)) != cudaSuccess) return done(e);
    *copy_gbs = 2.0 * n4 * 16.0 / (ms * 1e-3) / 1e9;
    return done(cudaSuccess);
}

// ---------------------------------------------------------------- reformat

// Reuse of support functions on a shifted geometry: warp per destination segment of
// L_dst(f); each member point p takes the source value at p - shift(atom) if that point
// is a member of L_src(f) (coarse part for s, fine part for d^1..d^7), else 0.
template <class T>
__global__ void k_reformat(ReformatLaunch a) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 10;
    const FnRec r = a.fn[blockIdx.y];
    const AtomRec& ad = a.atoms_dst[r.atom];
    const AtomRec& as = a.atoms_src[r.atom];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sidx = blockIdx.x * (blockDim.x >> 5) + warp;
    const int nseg = ad.nsegLc + ad.nsegLf;
    if (sidx >= nseg) return;
    const bool fine = sidx >= ad.nsegLc;
    const Seg sg = LD(a.seg_dst, fine ? ad.segLf + (sidx - ad.nsegLc) : ad.segLc + sidx, a.seg_dst_n);
    const int sx = a.shift[3 * r.atom], sy = a.shift[3 * r.atom + 1], sz = a.shift[3 * r.atom + 2];
    // destination row -> global (y, z)
    const int yl = sg.row % ad.n[1], zl = sg.row / ad.n[1];
    const int gy = ad.lo[1] + yl - sy, gz = ad.lo[2] + zl - sz;     // source row
    const int ys = gy - as.lo[1], zs = gz - as.lo[2];
    const bool row_in = ys >= 0 && zs >= 0 && ys < as.n[1] && zs < as.n[2];
    int s0 = 0, s1 = 0;
    if (row_in) {
        const int64_t rrow = (fine ? as.rowLf : as.rowLc) + ys + static_cast<int64_t>(as.n[1]) * zs;
        s0 = LD(a.rowptr_src, rrow, a.rowptr_src_n);
        s1 = LD(a.rowptr_src, rrow + 1, a.rowptr_src_n);
    }
    const T* src = static_cast<const T*>(a.phi_src) + LD(a.off_src, r.f, a.nfn + 1);
    T* dst = static_cast<T*>(a.phi_dst) + r.off_phi;
    const int64_t src_room = a.src_n - LD(a.off_src, r.f, a.nfn + 1);
    const int64_t dst_room = a.dst_n - r.off_phi;
    const int64_t seg0 = fine ? as.segLf : as.segLc;
    const int len = sg.x1 - sg.x0 + 1;
    for (int k = lane; k < len; k += 32) {
        const int xs = ad.lo[0] + sg.x0 + k - sx - as.lo[0];          // source box-local x
        int64_t off = -1;
        for (int q = s0; q < s1; ++q) {
            const Seg ss = LD(a.seg_src, seg0 + q, a.seg_src_n);
            if (xs >= ss.x0 && xs <= ss.x1) off = ss.off + (xs - ss.x0);
        }
        if (!fine) {
            ST(dst, sg.off + k, dst_room, off >= 0 ? LD(src, off, src_room) : T(0));
        } else {
#pragma unroll
            for (int t = 0; t < 7; ++t)
                ST(dst, ad.ncL + static_cast<int64_t>(t) * ad.nfL + sg.off + k, dst_room,
                   off >= 0 ? LD(src, as.ncL + static_cast<int64_t>(t) * as.nfL + off, src_room) : T(0));
        }
    }
}

cudaError_t enqueue_reformat(const ReformatLaunch& a, cudaStream_t s) {
    if (a.nfn == 0) return cudaSuccess;
    const dim3 grid((a.max_seg + 7) / 8, a.nfn);
    if (a.prec == 0)
        k_reformat<double><<<grid, 256, 0, s>>>(a);
    else
        k_reformat<float><<<grid, 256, 0, s>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- fixed device scratch

// Workspace of lsw_apply_hamiltonian_noalloc: a file-scope device array, so that this
// entry point never allocates.  Every GPU that loads the library holds it until exit.
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_SCRATCH_BYTES];

// Device address of the array on `device` (which must be current).  The first call for
// a device looks the address up with cudaGetSymbolAddress (this may load the module, so
// it belongs before any stream capture); later calls return the cached address.
cudaError_t noalloc_scratch(int device, void** ptr) {
    static std::mutex mu;
    static void* addr[NOALLOC_MAX_DEVICES] = {};
    if (device < 0 || device >= NOALLOC_MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (addr[device] == nullptr) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        addr[device] = p;
    }
    *ptr = addr[device];
    return cudaSuccess;
}

// Records of one batch of the allocation-free path, built on the device: boxes and
// offsets are copied from the system's resident per-function records (all[f0 ..
// f0 + nb)), and the workspace offsets are laid out again, function after function, in
// the order and sizes the host validated (D boxes first, then Bf, Bb, G and the z-arm
// flags of each function; every region a multiple of 64 elements).  One thread: nb is
// at most NOALLOC_MAX_BATCH.
__global__ void k_noalloc_records(const FnRec* __restrict__ all, int64_t f0, int nb, int64_t esize,
                                  FnRec* __restrict__ out) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    auto al = [](int64_t x) { return (x + ALIGN_ELEMS - 1) / ALIGN_ELEMS * ALIGN_ELEMS; };
    int64_t o = 0;
    for (int k = 0; k < nb; ++k) {
        FnRec r = all[f0 + k];
        r.ws_D = o;
        o += al(8LL * r.n[0] * r.n[1] * r.n[2]);
        out[k] = r;
    }
    for (int k = 0; k < nb; ++k) {
        FnRec& r = out[k];
        const int64_t X = 2 * r.n[0] + 29, Y = 2 * r.n[1] + 29;
        r.ws_Bf = o;
        o += al(2LL * r.n[2] * Y * X);
        r.ws_Bb = o;
        o += al(2LL * r.np[2] * Y * X);
        r.ws_G = o;
        o += al(8LL * r.np[0] * r.np[1] * r.np[2]);
        r.ws_Gf = o;
        o += al((4LL * r.n[0] * r.n[1] + esize - 1) / esize);
    }
}

cudaError_t enqueue_noalloc_records(const FnRec* all, int64_t f0, int nb, int64_t esize, FnRec* out, cudaStream_t s) {
    k_noalloc_records<<<1, 32, 0, s>>>(all, f0, nb, esize, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- host entry points

cudaError_t upload_filters(const FilterSet& fs, int device) {
    cudaError_t e = cudaSetDevice(device);
    if (e != cudaSuccess) return e;
    float f32[2][FWD_TAPS];
    float k32[4][KIN_TAPS];
    for (int b = 0; b < 2; ++b)
        for (int i = 0; i < FWD_TAPS; ++i) f32[b][i] = static_cast<float>(fs.fwd[b][i]);
    for (int b = 0; b < 4; ++b)
        for (int i = 0; i < KIN_TAPS; ++i) k32[b][i] = static_cast<float>(fs.kin[b][i]);
    if ((e = cudaMemcpyToSymbol(c_fwd_d, fs.fwd, sizeof(fs.fwd))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_kin_d, fs.kin, sizeof(fs.kin))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_fwd_f, f32, sizeof(f32))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_kin_f, k32, sizeof(k32))) != cudaSuccess) return e;
    float2 bwd2[FWD_TAPS], up2[2][16], kin2[2][KIN_TAPS];
    for (int m = 0; m < FWD_TAPS; ++m) bwd2[m] = make_float2(f32[0][m], f32[1][m]);
    for (int b = 0; b < 2; ++b)
        for (int k = 0; k < 16; ++k) up2[b][k] = make_float2(f32[b][2 * k], 2 * k + 1 < FWD_TAPS ? f32[b][2 * k + 1] : 0.f);
    for (int l = 0; l < KIN_TAPS; ++l) {
        kin2[0][l] = make_float2(k32[0][l], k32[2][l]);
        kin2[1][l] = make_float2(k32[1][l], k32[3][l]);
    }
    if ((e = cudaMemcpyToSymbol(c_fwd2_bwd, bwd2, sizeof(bwd2))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_fwd2_up, up2, sizeof(up2))) != cudaSuccess) return e;
    return cudaMemcpyToSymbol(c_kin2, kin2, sizeof(kin2));
}

cudaError_t configure_kernels(size_t max_smem) {
    // dynamic shared memory may use what the kernel's static shared memory leaves
    cudaError_t e;
#define SETMAX(K)                                                                               \
    {                                                                                           \
        cudaFuncAttributes fa;                                                                  \
        if ((e = cudaFuncGetAttributes(&fa, K)) != cudaSuccess) return e;                       \
        const int m = static_cast<int>(max_smem - fa.sharedSizeBytes);                          \
        if ((e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, m)) != cudaSuccess) \
            return e;                                                                           \
    }
    SETMAX(k_density<double>) SETMAX(k_density<float>)
    SETMAX(k_fwd_xy<double>) SETMAX(k_fwd_xy<float>)
    SETMAX(k_z<double>) SETMAX(k_z<float>)
    SETMAX(k_kin_z<double>) SETMAX(k_kin_z<float>)
    SETMAX(k_z_tc<2>) SETMAX(k_z_tc<3>)
    SETMAX(k_fwd_xy_tc<2>) SETMAX(k_fwd_xy_tc<3>)
    SETMAX(k_bwd_xy<double>) SETMAX(k_bwd_xy<float>)
    SETMAX(k_bwd_xy_tc<2>) SETMAX(k_bwd_xy_tc<3>)
    SETMAX(k_z_dens<double>) SETMAX(k_z_dens<float>)
#undef SETMAX
    // the plans size the plane kernels' dynamic shared memory against these bounds
#define STATIC_BOUND(K, B)                                                                     \
    {                                                                                          \
        cudaFuncAttributes fa;                                                                 \
        if ((e = cudaFuncGetAttributes(&fa, K)) != cudaSuccess) return e;                      \
        if (fa.sharedSizeBytes > (B)) return cudaErrorInvalidConfiguration;                     \
    }
    STATIC_BOUND(k_fwd_xy<double>, FWD_STATIC_SMEM) STATIC_BOUND(k_fwd_xy<float>, FWD_STATIC_SMEM)
    STATIC_BOUND(k_bwd_xy<double>, BWD_STATIC_SMEM) STATIC_BOUND(k_bwd_xy<float>, BWD_STATIC_SMEM)
    STATIC_BOUND(k_bwd_xy_tc<2>, BWD_TC_STATIC_SMEM) STATIC_BOUND(k_bwd_xy_tc<3>, BWD_TC_STATIC_SMEM)
#undef STATIC_BOUND
    return cudaSuccess;
}

cudaError_t plane_kernel_blocks(int prec, size_t smem_fwd, size_t smem_bwd, int* fwd, int* bwd) {
    cudaError_t e;
    if (prec == 0) {
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(fwd, k_fwd_xy<double>, 256, smem_fwd)) != cudaSuccess)
            return e;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(bwd, k_bwd_xy<double>, BWD_THREADS, smem_bwd);
    }
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(fwd, k_fwd_xy<float>, 256, smem_fwd)) != cudaSuccess)
        return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(bwd, k_bwd_xy<float>, BWD_THREADS, smem_bwd);
}

#define TRACED(TR, KIND, S, LAUNCH) \
    do {                                \
        trace_begin(TR, KIND, S);       \
        LAUNCH;                         \
        trace_end(TR, S);               \
    } while (0)

// Functions per grid slot of k_uncompress: eight where that leaves eight waves of CTAs (six an SM), else
// four (batches of 32 functions, 64 atoms: 89 us with four, 119 with one or eight).
static int uncompress_group(const HphiLaunch& a) {
    return static_cast<int64_t>(a.nfn) * ((a.max_rowsL + 7) / 8) >= 8LL * 8 * 6 * a.n_sm ? 8 : 4;
}

template <class T>
static cudaError_t hphi_batch(const HphiLaunch& a, cudaStream_t s) {
    const int nf = a.nfn;
    const int ug = uncompress_group(a);
    TRACED(a.tr, TK_UNCOMPRESS, s, (k_uncompress<T><<<dim3((a.max_rowsL + 7) / 8, (nf + ug - 1) / ug), 256, 0, s>>>(a, ug)));
    const dim3 gfwd = a.items_fwd ? dim3(a.grid_fwd) : dim3(2 * a.max_nz, nf);
    const dim3 gbwd = a.items_bwd ? dim3(a.grid_bwd) : dim3(2 * a.max_nzp, nf);
    if constexpr (sizeof(T) == 4) {
        if (a.xy_tc && a.zsplit == 3)
            TRACED(a.tr, TK_FWD_XY, s, (k_fwd_xy_tc<3><<<dim3(2 * a.max_nz, nf), 256, a.smem_fwd_tc, s>>>(a)));
        else if (a.xy_tc && a.zsplit == 2)
            TRACED(a.tr, TK_FWD_XY, s, (k_fwd_xy_tc<2><<<dim3(2 * a.max_nz, nf), 256, a.smem_fwd_tc, s>>>(a)));
        else
            TRACED(a.tr, TK_FWD_XY, s, (k_fwd_xy<T><<<gfwd, 256, a.smem_fwd, s>>>(a)));
    } else {
        TRACED(a.tr, TK_FWD_XY, s, (k_fwd_xy<T><<<gfwd, 256, a.smem_fwd, s>>>(a)));
    }
    if constexpr (sizeof(T) == 4) {
        if (a.zsplit) {
            // several tiles per CTA: the filter operands are built once per CTA
            const int gx = ((a.max_cols + tc::TILE - 1) / tc::TILE + tc::TILES_PER_CTA - 1) / tc::TILES_PER_CTA;
            if (a.zsplit == 3)
                TRACED(a.tr, TK_Z, s, (k_z_tc<3><<<dim3(gx, nf), 256, a.smem_ztc, s>>>(a)));
            else
                TRACED(a.tr, TK_Z, s, (k_z_tc<2><<<dim3(gx, nf), 256, a.smem_ztc, s>>>(a)));
        } else {
            TRACED(a.tr, TK_Z, s, (k_z<T><<<dim3((a.max_cols + a.zcols - 1) / a.zcols, nf), a.zcols, a.smem_z, s>>>(a)));
        }
    } else {
        TRACED(a.tr, TK_Z, s, (k_z<T><<<dim3((a.max_cols + a.zcols - 1) / a.zcols, nf), a.zcols, a.smem_z, s>>>(a)));
    }
    TRACED(a.tr, TK_KINETIC, s,
           (k_kin_z<T><<<dim3(static_cast<unsigned>((a.max_colsL + 127) / 128), nf, 4), 128, a.smem_kin, s>>>(a)));
    if constexpr (sizeof(T) == 4) {
        if (a.xy_tc && a.zsplit == 3)
            TRACED(a.tr, TK_BWD_XY, s, (k_bwd_xy_tc<3><<<dim3(2 * a.max_nzp, nf), 512, a.smem_bwd_tc, s>>>(a)));
        else if (a.xy_tc && a.zsplit == 2)
            TRACED(a.tr, TK_BWD_XY, s, (k_bwd_xy_tc<2><<<dim3(2 * a.max_nzp, nf), 512, a.smem_bwd_tc, s>>>(a)));
        else
            TRACED(a.tr, TK_BWD_XY, s, (k_bwd_xy<T><<<gbwd, BWD_THREADS, a.smem_bwd, s>>>(a)));
    } else {
        TRACED(a.tr, TK_BWD_XY, s, (k_bwd_xy<T><<<gbwd, BWD_THREADS, a.smem_bwd, s>>>(a)));
    }
    return cudaGetLastError();
}

cudaError_t enqueue_hphi_batch(const HphiLaunch& a, cudaStream_t s) {
    return a.prec == 0 ? hphi_batch<double>(a, s) : hphi_batch<float>(a, s);
}

// Density, per batch: uncompress, forward x, y (FMA plane kernel in every precision) and
// the density z stage writing u into the store.
template <class T>
static cudaError_t dens_batch(HphiLaunch a, cudaStream_t s) {
    const int nf = a.nfn;
    const int ug = uncompress_group(a);
    constexpr int C = ZCols<T>::C;
    a.items_fwd = a.items_bwd = nullptr;       // one CTA per grid slot here
    a.queue = nullptr;
    a.smem_z = sizeof(T) * 2 * static_cast<size_t>(a.max_nz) * C;
    TRACED(a.tr, TK_UNCOMPRESS, s, (k_uncompress<T><<<dim3((a.max_rowsL + 7) / 8, (nf + ug - 1) / ug), 256, 0, s>>>(a, ug)));
    TRACED(a.tr, TK_FWD_XY, s, (k_fwd_xy<T><<<dim3(2 * a.max_nz, nf), 256, a.smem_fwd, s>>>(a)));
    TRACED(a.tr, TK_DENS_U, s, (k_z_dens<T><<<dim3((a.max_cols + C - 1) / C, nf), C, a.smem_z, s>>>(a)));
    return cudaGetLastError();
}

cudaError_t enqueue_dens_batch(const HphiLaunch& a, cudaStream_t s) {
    return a.prec == 0 ? dens_batch<double>(a, s) : dens_batch<float>(a, s);
}

cudaError_t enqueue_density(const DensLaunch& a, cudaStream_t s) {
    const int64_t nt = static_cast<int64_t>(a.ntile[0]) * a.ntile[1] * a.ntile[2];
    if (nt == 0) return cudaSuccess;
    const unsigned g = static_cast<unsigned>(nt);
    // tables in shared memory where two CTAs an SM fit with the tile of most functions
    if (a.max_m > 0 && a.max_m <= (a.prec == 0 ? 8 : 16)) {
        if (a.prec == 0)
            TRACED(a.tr, TK_DENSITY, s, (k_density_few<double, 8><<<g, DT_THREADS, 0, s>>>(a)));
        else if (a.max_m <= 8)
            TRACED(a.tr, TK_DENSITY, s, (k_density_few<float, 8><<<g, DT_THREADS, 0, s>>>(a)));
        else
            TRACED(a.tr, TK_DENSITY, s, (k_density_few<float, 16><<<g, DT_THREADS, 0, s>>>(a)));
    } else if (a.max_m > 0) {
        const size_t smem = density_smem(a.prec, a.max_m, a.max_g);
        if (a.prec == 0)
            TRACED(a.tr, TK_DENSITY, s, (k_density<double><<<g, DT_THREADS, smem, s>>>(a)));
        else
            TRACED(a.tr, TK_DENSITY, s, (k_density<float><<<g, DT_THREADS, smem, s>>>(a)));
    } else if (a.prec == 0) {
        TRACED(a.tr, TK_DENSITY, s, (k_density_big<double><<<g, DT_THREADS, 0, s>>>(a)));
    } else {
        TRACED(a.tr, TK_DENSITY, s, (k_density_big<float><<<g, DT_THREADS, 0, s>>>(a)));
    }
    return cudaGetLastError();
}


}  // namespace lsw
