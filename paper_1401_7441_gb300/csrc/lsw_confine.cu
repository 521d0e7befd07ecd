// sm_103a kernels of the quartic confinement and the preconditioning equation (Sec.
// "Support function optimization": H_alpha = H_KS + a_alpha (r - R_alpha)^4 in the first
// iterations, "evaluated via convolutions in the same manner as the kinetic energy";
// Eq. precond: (-1/2 nabla^2 + a_alpha (r - R_alpha)^4 - eps_alpha) g_prec = -g).
//
// The operator on a function's two-level coefficients, types t = bx + 2 by + 4 bz:
//   Q = a [ sum_d X_d^4 + 2 sum_{d<e} X_d^2 X_e^2 ],  X_d = x_d - R_d,
// each X_d^m a 1D operator along d between the scaling/wavelet functions of coarse
// points i, j (band |j - i| <= 14), its entries depending on i (tables from the moment
// overlaps F^p of the filter set); T = -1/(2h^2) sum_d K_d with the Galerkin kinetic blocks.
//
// What bounds it: the FP64 pipe (1/64 of the FP32 rate: one warp instruction per 16 clocks
// of an SM), in every precision, since sums and tables are FP64.  So the design removes
// FP64 operations and lets loads and index arithmetic take care of themselves:
//   - 1D operators along different dimensions commute, so the cross terms share factors:
//       A = 2a X_z^2 P,  B = A + 2a X_y^2 P,
//       Q P = sum_d a X_d^4 P + X_y^2 A + X_x^2 B,
//     7 passes instead of 9 (and the kinetic arms are added into the X^4 tables of a
//     function, 7 instead of 12 for the preconditioner);
//   - everything stays in the L box along the dimensions a term has not touched yet
//     (output: the L box, or the part of the L' box the band reaches), not on the box
//     widened by 14 on every side; products are formed only between the hull of a group
//     of lines' nonzero inputs and the members of the output region;
//   - the lines along the pass' dimension that carry data are packed 32 to a warp tile, a
//     lane each, so the wavelet types (nonzero on the fine members only) keep full warps.
// Measured (GB300, 2,070 MHz): four iterations of the preconditioner on 59 FP32 functions of 20
// atoms (R = 6 bohr) 798 -> 7.1 ms; a quartic added to 99 FP64 functions (R = 5-8 bohr)
// 149 -> 8.5 ms (before: nine and twelve passes over the whole widened box, a thread per point).
//
//   k_conf_table   tables of X_d^2, X_d^4 of every atom
//   k_conf_comb    per function a X_d^4 (+ kinetic arm), the tables of one batch
//   k_conf_maps    member maps of a batch's boxes and their projections
//   k_conf_load    compressed phi on L -> the L box P (FP64; members only, zero elsewhere)
//   k_conf_pass    the passes along z, y, x
//   k_conf_store   result -> compressed members of L or L' (optionally added to the target)
//   k_conf_energy  <phi|Q phi> of a function from its rows' sums
//   k_cg_*         the conjugate-gradient updates, a CTA per function
#include <algorithm>
#include <cstdint>

#include "lsw_device.h"
#include "lsw_internal.h"

namespace lsw {

__device__ __forceinline__ double warp_sum_c(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum over the CTA, in a fixed order; every thread gets it.
__device__ double block_sum_c(double v) {
    __shared__ double part[32];
    __syncthreads();
    v = warp_sum_c(v);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    for (int i = 0; i < static_cast<int>(blockDim.x >> 5); ++i) s += part[i];
    return s;
}

// Boxes of a function: L box extents n; output box extents m (region 0: the L box; region 1:
// the part of the L' box within 14 points of the L box, the reach of the band); o: origin of
// the L box in the output box; r0: origin of the output box in the region's box.
struct ConfGeo {
    int n[3], m[3], o[3], r0[3];
};
__device__ __forceinline__ ConfGeo conf_geo(const AtomRec& at, int region) {
    ConfGeo g;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int rlo = region ? at.lop[d] : at.lo[d], rn = region ? at.np[d] : at.n[d];
        const int b0 = max(rlo, at.lo[d] - KIN_HALF), b1 = min(rlo + rn, at.lo[d] + at.n[d] + KIN_HALF);
        g.n[d] = at.n[d];
        g.m[d] = b1 - b0;
        g.o[d] = at.lo[d] - b0;
        g.r0[d] = b0 - rlo;
    }
    return g;
}

// ---------------------------------------------------------------- tables

// Tables [dim][m = 2, 4][b b'][i over the L box widened by 14][l + 14] of one atom (blockIdx.x), the
// entries by conf_entry.  A thread per entry: on the device because the host loop took about 25 ms per
// atom, this about 25 us.
__global__ void __launch_bounds__(256) k_conf_table(const AtomRec* __restrict__ atoms, const double* __restrict__ pos,
                                                    const double* __restrict__ G, const double* __restrict__ XY, double h,
                                                    const int64_t* __restrict__ off, double* __restrict__ tab) {
    const AtomRec at = atoms[blockIdx.x];
    double* out = tab + off[blockIdx.x];
    for (int d = 0; d < 3; ++d) {
        const int E = at.n[d] + 2 * KIN_HALF;
        const double c = pos[3 * blockIdx.x + d] / h;
        for (int e = threadIdx.x; e < 8 * E * KIN_TAPS; e += blockDim.x) {
            const int l = e % KIN_TAPS, i = (e / KIN_TAPS) % E, blk = e / (KIN_TAPS * E);
            const int m = blk < 4 ? 2 : 4, b = (blk >> 1) & 1, bp = blk & 1;
            out[e] = conf_entry(G, XY, m, b, bp, l, static_cast<double>(at.lo[d] - KIN_HALF + i), c, h);
        }
        out += 8 * E * KIN_TAPS;
    }
}

// First entry of the tables of X_d^2 of an atom (X_d^4 follows after 4 E entries of 29).
__device__ __forceinline__ int64_t conf_qbase(const ConfLaunch& a, int atom, const AtomRec& at, int dim) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 16;
    int64_t base = LD(a.qtab_off, atom, a.n_atoms + 1);
    for (int d = 0; d < dim; ++d) base += 8LL * (at.n[d] + 2 * KIN_HALF) * KIN_TAPS;
    return base;
}

// comb[dim][b b'][i over the output box][l + 14] = a_f X_dim^4 (+ the kinetic block); grid (3, functions)
__global__ void __launch_bounds__(256) k_conf_comb(ConfLaunch a) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 17;
    const int d = blockIdx.x, k = blockIdx.y;
    const int f = static_cast<int>(a.f0) + k;
    const int atom = LD(a.sf_atom, f, a.n_sf);
    const AtomRec at = LD(a.atoms, atom, a.n_atoms);
    const ConfGeo g = conf_geo(at, a.region);
    const int E = at.n[d] + 2 * KIN_HALF, m = g.m[d];
    const int64_t q4 = conf_qbase(a, atom, at, d) + 4LL * E * KIN_TAPS;
    const double af = LD(a.acoef, f, a.n_sf);
    double* out = a.comb + k * a.s_comb + static_cast<int64_t>(d) * 4 * a.max_m * KIN_TAPS;
    const int64_t room = 4LL * a.max_m * KIN_TAPS;
    for (int e = threadIdx.x; e < 4 * m * KIN_TAPS; e += blockDim.x) {
        const int l = e % KIN_TAPS, i = (e / KIN_TAPS) % m, bb = e / (KIN_TAPS * m);
        double v = af * LD(a.qtab, q4 + (static_cast<int64_t>(bb) * E + (i - g.o[d] + KIN_HALF)) * KIN_TAPS + l, a.qtab_n);
        if (a.precond) v += a.kin_scale * a.kin[bb][l];
        ST(out, (bb * a.max_m + i) * KIN_TAPS + l, room, v);
    }
}

// ---------------------------------------------------------------- maps and load

// Member maps of function k (zeroed before): mem [z][y][x] of the output box (1 coarse, 3
// coarse and fine); per region part (0 coarse, 1 fine): act_xy [y][x], act_xz [z][x], act_x [x] of
// the L box (some member along the other dimensions) and out_row [z][y], out_xz [z][x] of the
// output box.  A warp per row of the L box and of the region's box.
__global__ void __launch_bounds__(256) k_conf_maps(ConfLaunch a) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 18;
    const int k = blockIdx.y;
    const int f = static_cast<int>(a.f0) + k;
    const AtomRec at = LD(a.atoms, LD(a.sf_atom, f, a.n_sf), a.n_atoms);
    const ConfGeo g = conf_geo(at, a.region);
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const ConfMaps M = conf_maps(a, k);
    if (row < at.n[1] * at.n[2]) {
        const int y = row % at.n[1], z = row / at.n[1], nx = at.n[0];
        for (int part = 0; part < 2; ++part) {
            const int64_t r0 = part ? at.rowLf : at.rowLc, sg0 = part ? at.segLf : at.segLc;
            const int s0 = LD(a.rowptr, r0 + row, a.rowptr_n), s1 = LD(a.rowptr, r0 + row + 1, a.rowptr_n);
            for (int s = s0; s < s1; ++s) {
                const Seg sg = LD(a.seg, sg0 + s, a.seg_n);
                for (int x = sg.x0 + lane; x <= sg.x1; x += 32) {   // several rows store the same 1
                    ST(M.act_xy, (part * at.n[1] + y) * nx + x, a.s_xy, 1);
                    ST(M.act_xz, (part * at.n[2] + z) * nx + x, a.s_xz, 1);
                    ST(M.act_x, part * nx + x, a.s_x, 1);
                }
            }
        }
    }
    const int* rn = a.region ? at.np : at.n;
    if (row < rn[1] * rn[2]) {
        const int y = row % rn[1] - g.r0[1], z = row / rn[1] - g.r0[2];
        if (y < 0 || y >= g.m[1] || z < 0 || z >= g.m[2]) return;   // whole warp, no barrier below in other warps' way
        for (int part = 0; part < 2; ++part) {
            const int64_t r0 = part ? (a.region ? at.rowPf : at.rowLf) : (a.region ? at.rowPc : at.rowLc);
            const int64_t sg0 = part ? (a.region ? at.segPf : at.segLf) : (a.region ? at.segPc : at.segLc);
            const int s0 = LD(a.rowptr, r0 + row, a.rowptr_n), s1 = LD(a.rowptr, r0 + row + 1, a.rowptr_n);
            for (int s = s0; s < s1; ++s) {
                const Seg sg = LD(a.seg, sg0 + s, a.seg_n);
                for (int xr = sg.x0 + lane; xr <= sg.x1; xr += 32) {
                    const int x = xr - g.r0[0];
                    if (x < 0 || x >= g.m[0]) continue;
                    ST(M.mem, (static_cast<int64_t>(z) * g.m[1] + y) * g.m[0] + x, a.s_mem, part ? 3 : 1);
                    ST(M.out_row, (part * g.m[2] + z) * g.m[1] + y, a.s_row, 1);
                    ST(M.out_xz, (part * g.m[2] + z) * g.m[0] + x, a.s_oxz, 1);
                }
            }
            __syncwarp();                              // coarse 1 before fine 3
        }
    }
}

// compressed vector on L -> members of the L box P [t][z][y][x]; a warp per row.  The points
// off the members were zeroed once per batch.
template <class T>
__global__ void __launch_bounds__(256) k_conf_load(ConfLaunch a, const T* __restrict__ src) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 19;
    const int k = blockIdx.y;
    const int f = static_cast<int>(a.f0) + k;
    const AtomRec at = LD(a.atoms, LD(a.sf_atom, f, a.n_sf), a.n_atoms);
    double* P = a.P + k * a.s_P;
    const int64_t off = LD(a.off_L, f, a.n_sf + 1);
    const int64_t vol = static_cast<int64_t>(at.n[0]) * at.n[1] * at.n[2];
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (row >= at.n[1] * at.n[2]) return;
    const int64_t base = static_cast<int64_t>(row) * at.n[0];
    for (int part = 0; part < 2; ++part) {
        const int64_t r0 = part ? at.rowLf : at.rowLc, sg0 = part ? at.segLf : at.segLc;
        const int s0 = LD(a.rowptr, r0 + row, a.rowptr_n), s1 = LD(a.rowptr, r0 + row + 1, a.rowptr_n);
        for (int s = s0; s < s1; ++s) {
            const Seg g = LD(a.seg, sg0 + s, a.seg_n);
            for (int x = g.x0 + lane; x <= g.x1; x += 32) {
                const int64_t rel = g.off + (x - g.x0);
                if (part == 0) {
                    ST(P, base + x, a.s_P, static_cast<double>(LD(src, off + rel, a.vec_n)));
                } else {
#pragma unroll
                    for (int t = 1; t < 8; ++t)
                        ST(P, t * vol + base + x, a.s_P,
                           static_cast<double>(LD(src, off + at.ncL + rel + static_cast<int64_t>(t - 1) * at.nfL, a.vec_n)));
                }
            }
        }
    }
}

// ---------------------------------------------------------------- the passes

__device__ __forceinline__ bool nonzero_bits(double v) { return (__double_as_longlong(v) << 1) != 0; }

// The pass along DIM for the type pair q (the two types that differ in DIM's bit; q holds the
// bits of the other two dimensions) over 256 lines of a function:
//   DIM 2 (z): lines (x, y) of the L box; A = 2a X_z^2 P, OZ = comb_z P
//   DIM 1 (y): lines (x of L, z of the output box); B = A + 2a X_y^2 P, OY = comb_y P + X_y^2 A + OZ
//   DIM 0 (x): lines (y, z) of the output box; F = comb_x P + X_x^2 B + OY on the members
// The CTA lists its lines that carry data, then takes them 32 at a time, a lane each: the
// lines' inputs go to shared memory (STAGED; read in place where the lines are too long),
// every warp takes output positions in turn, and sums over the hull of the 32 lines' nonzero
// inputs within the band; taps are warp-uniform loads.  An output that no lane needs (not a
// member of the output region, for A and B not read by a later pass) is not formed.
// Every array is read only where the maps say that it was written: A on columns of act_xy, B
// where act_xy or act_xz holds, OZ and OY at members on such lines.
template <int DIM, bool STAGED>
__global__ void __launch_bounds__(256) k_conf_pass(ConfLaunch a) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 20 + DIM;
    constexpr int NA = DIM == 2 ? 2 : 4;               // input arrays of a line: P s, d (and A or B s, d)
    extern __shared__ __align__(16) double conf_sm[];  // [NA][len][33]
    __shared__ int list[256], wcnt[8];
    __shared__ int hull[4][2];
    const int k = blockIdx.y, q = blockIdx.x & 3, seg = blockIdx.x >> 2;
    const int f = static_cast<int>(a.f0) + k;
    const int atom = LD(a.sf_atom, f, a.n_sf);
    const AtomRec at = LD(a.atoms, atom, a.n_atoms);
    const ConfGeo g = conf_geo(at, a.region);
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], mx = g.m[0], my = g.m[1], mz = g.m[2];
    const int len = g.n[DIM], mout = g.m[DIM], off = g.o[DIM];
    const int U = DIM == 0 ? my : nx, W = DIM == 2 ? ny : mz;   // line = u + U w
    if (seg * 256 >= U * W) return;
    const int q0 = q & 1, q1 = q >> 1;                 // bits of the lower and the higher other dimension
    const int t0 = DIM == 2 ? q : DIM == 1 ? q0 + 4 * q1 : 2 * q0 + 4 * q1;
    constexpr int TS = 1 << DIM;
    const ConfMaps M = conf_maps(a, k);
    const double* P = a.P + k * a.s_P;
    double* A = a.A + k * a.s_A;
    double* OZ = a.OZ + k * a.s_A;
    double* B = a.B + k * a.s_B;
    double* OY = a.OY + k * a.s_B;
    double* F = a.F + k * a.s_F;
    const int64_t vP = static_cast<int64_t>(nx) * ny * nz, vA = static_cast<int64_t>(nx) * ny * mz,
                  vB = static_cast<int64_t>(nx) * my * mz, vF = static_cast<int64_t>(mx) * my * mz;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // lines that carry data, in order
    {
        const int line = seg * 256 + threadIdx.x;
        bool act = false;
        if (line < U * W) {
            const int u = line % U, w = line / U;
            if (DIM == 2) act = LD(M.act_xy, ((q ? 1 : 0) * ny + w) * nx + u, a.s_xy) != 0;
            else if (DIM == 1) act = LD(M.act_x, q0 * nx + u, a.s_x) != 0;
            else act = LD(M.out_row, ((q ? 1 : 0) * mz + w) * my + u, a.s_row) != 0;
        }
        const unsigned m = __ballot_sync(0xffffffffu, act);
        if (lane == 0) wcnt[warp] = __popc(m);
        __syncthreads();
        int base = 0;
        for (int i = 0; i < warp; ++i) base += wcnt[i];
        if (act) list[base + __popc(m & ((1u << lane) - 1))] = line;
        __syncthreads();
    }
    int cnt = 0;
    for (int i = 0; i < 8; ++i) cnt += wcnt[i];

    // input s of array r (0, 1: P; 2, 3: A or B) at position j of line (u, w); 0 where nothing was written
    auto fetch = [&](int r, int j, int u, int w) -> double {
        const int s = r & 1, t = t0 + TS * s;
        if (r < 2) {
            if (DIM == 2) return LD(P, t * vP + (static_cast<int64_t>(j) * ny + w) * nx + u, a.s_P);
            const int z = w - g.o[2];
            if (z < 0 || z >= nz) return 0.0;
            if (DIM == 1) return LD(P, t * vP + (static_cast<int64_t>(z) * ny + j) * nx + u, a.s_P);
            const int y = u - g.o[1];
            if (y < 0 || y >= ny) return 0.0;
            return LD(P, t * vP + (static_cast<int64_t>(z) * ny + y) * nx + j, a.s_P);
        }
        if (DIM == 1) {
            if (!LD(M.act_xy, ((q0 | s) * ny + j) * nx + u, a.s_xy)) return 0.0;
            return LD(A, t * vA + (static_cast<int64_t>(w) * ny + j) * nx + u, a.s_A);
        }
        const int y = u - g.o[1], z = w - g.o[2];
        const bool have = (y >= 0 && y < ny && LD(M.act_xy, ((s | q0) * ny + y) * nx + j, a.s_xy)) ||
                          (z >= 0 && z < nz && LD(M.act_xz, ((s | q1) * nz + z) * nx + j, a.s_xz));
        return have ? LD(B, t * vB + (static_cast<int64_t>(w) * my + u) * nx + j, a.s_B) : 0.0;
    };

    const int64_t sm_n = static_cast<int64_t>(NA) * len * 33;
    (void)sm_n;
    const int E = len + 2 * KIN_HALF;
    const double* comb = a.comb + k * a.s_comb + static_cast<int64_t>(DIM) * 4 * a.max_m * KIN_TAPS;
    const double* X2 = a.qtab + conf_qbase(a, atom, at, DIM);
    [[maybe_unused]] const int64_t comb_n = 4LL * a.max_m * KIN_TAPS, x2_n = 4LL * E * KIN_TAPS;
    const double a2 = 2.0 * LD(a.acoef, f, a.n_sf);
    for (int l0 = 0; l0 < cnt; l0 += 32) {
        const bool on = l0 + lane < cnt;
        const int line = list[on ? l0 + lane : l0];
        const int u = line % U, w = line / U;
        if (STAGED) {
            if (DIM == 0) {                            // lines contiguous in memory: lanes along the line
                for (int l = warp; l < 32; l += 8) {
                    const bool lon = l0 + l < cnt;
                    const int ln = list[lon ? l0 + l : l0];
                    const int lu = ln % U, lw = ln / U;
                    for (int r = 0; r < NA; ++r)
                        for (int j = lane; j < len; j += 32)
                            ST(conf_sm, (r * len + j) * 33 + l, sm_n, lon ? fetch(r, j, lu, lw) : 0.0);
                }
            } else {                                   // neighbouring lines contiguous: lanes across lines
                for (int e = warp; e < NA * len; e += 8) {
                    const int r = e / len, j = e - r * len;
                    ST(conf_sm, e * 33 + lane, sm_n, on ? fetch(r, j, u, w) : 0.0);
                }
            }
            __syncthreads();
        }
        auto in = [&](int r, int j) -> double {
            if (STAGED) return LD(conf_sm, (r * len + j) * 33 + lane, sm_n);
            return on ? fetch(r, j, u, w) : 0.0;
        };
        if (warp < NA) {                               // hull of the tile's nonzero inputs, per array
            int lo = len, hi = -1;
            for (int j = 0; j < len; ++j)
                if (__any_sync(0xffffffffu, nonzero_bits(in(warp, j)))) {
                    lo = min(lo, j);
                    hi = j;
                }
            if (lane == 0) {
                hull[warp][0] = lo;
                hull[warp][1] = hi;
            }
        }
        __syncthreads();
        for (int i = warp; i < mout; i += 8) {
            // output position (x, y, z) of this lane in the output box
            const int x = DIM == 0 ? i : u + g.o[0], y = DIM == 0 ? u : DIM == 1 ? i : w + g.o[1],
                      z = DIM == 2 ? i : w;
            const int mem = on ? LD(M.mem, (static_cast<int64_t>(z) * my + y) * mx + x, a.s_mem) : 0;
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int t = t0 + TS * b;
                const bool need_o = mem & (t == 0 ? 1 : 2);
                bool need_i = false;                   // the intermediate (A or B) is read later
                if (DIM == 2)
                    need_i = on && (LD(M.out_xz, ((q0 | b) * mz + i) * mx + x, a.s_oxz) ||
                                    LD(M.out_row, ((q1 | b) * mz + i) * my + y, a.s_row));
                if (DIM == 1) need_i = on && LD(M.out_row, ((b | q1) * mz + z) * my + i, a.s_row);
                const bool any_o = __any_sync(0xffffffffu, need_o), any_i = __any_sync(0xffffffffu, need_i);
                if (!any_o && !any_i) continue;
                double so = 0.0, si = 0.0;
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const double* ct = comb + ((b * 2 + s) * a.max_m + i) * KIN_TAPS + (off - i + KIN_HALF);
                    const double* xt = X2 + (static_cast<int64_t>(b * 2 + s) * E + (i - off + KIN_HALF)) * KIN_TAPS +
                                       (off - i + KIN_HALF);
                    [[maybe_unused]] const int64_t cr = comb_n - (ct - comb), xr = x2_n - (xt - X2);
                    int lo = max(hull[s][0], i - off - KIN_HALF), hi = min(hull[s][1], i - off + KIN_HALF);
                    if (any_o && any_i && DIM != 0) {
#pragma unroll 4
                        for (int j = lo; j <= hi; ++j) {
                            const double v = in(s, j);
                            so = fma(LD(ct, j, cr), v, so);
                            si = fma(LD(xt, j, xr), v, si);
                        }
                    } else if (any_o) {
#pragma unroll 4
                        for (int j = lo; j <= hi; ++j) so = fma(LD(ct, j, cr), in(s, j), so);
                    } else {
#pragma unroll 4
                        for (int j = lo; j <= hi; ++j) si = fma(LD(xt, j, xr), in(s, j), si);
                    }
                    if (DIM != 2 && any_o) {
                        lo = max(hull[2 + s][0], i - off - KIN_HALF);
                        hi = min(hull[2 + s][1], i - off + KIN_HALF);
#pragma unroll 4
                        for (int j = lo; j <= hi; ++j) so = fma(LD(xt, j, xr), in(2 + s, j), so);
                    }
                }
                const int ji = i - off;                // the output position on the input line, if inside
                const bool inside = ji >= 0 && ji < len;
                if (DIM == 2) {
                    const int64_t p = t * vA + (static_cast<int64_t>(i) * ny + w) * nx + u;
                    if (need_i) ST(A, p, a.s_A, a2 * si);
                    if (need_o) ST(OZ, p, a.s_A, so);
                } else if (DIM == 1) {
                    const int64_t p = t * vB + (static_cast<int64_t>(w) * my + i) * nx + u;
                    if (need_i) ST(B, p, a.s_B, a2 * si + (inside ? in(2 + b, ji) : 0.0));
                    if (need_o) {
                        if (inside && LD(M.act_xy, ((q0 | b) * ny + ji) * nx + u, a.s_xy))
                            so += LD(OZ, t * vA + (static_cast<int64_t>(w) * ny + ji) * nx + u, a.s_A);
                        ST(OY, p, a.s_B, so);
                    }
                } else if (need_o) {
                    if (inside && LD(M.act_x, b * nx + ji, a.s_x))
                        so += LD(OY, t * vB + (static_cast<int64_t>(w) * my + u) * nx + ji, a.s_B);
                    ST(F, t * vF + (static_cast<int64_t>(w) * my + u) * mx + i, a.s_F, so);
                }
            }
        }
        __syncthreads();                               // the next tile reuses the staged lines
    }
}

// ---------------------------------------------------------------- store

// F on the members of the region (0: L, 1: L') -> compressed vector; dst (+)= F (- eps_f P for
// the preconditioning operator).  With `energy`, the row's sum of P F over the members of L is left
// in B (read for the last time by the x pass) for k_conf_energy.  A warp per row, a chain of loads each:
// bound by the warps in flight (20 atoms in FP32, four calls: 176 us with four CTAs an SM, 211 with
// three, 297 with two).
template <class T>
__global__ void __launch_bounds__(256, 4) k_conf_store(ConfLaunch a, T* __restrict__ dst, int accumulate, int energy) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 23;
    const int k = blockIdx.y;
    const int f = static_cast<int>(a.f0) + k;
    const AtomRec at = LD(a.atoms, LD(a.sf_atom, f, a.n_sf), a.n_atoms);
    const ConfGeo g = conf_geo(at, a.region);
    const double* F = a.F + k * a.s_F;
    const double* P = a.P + k * a.s_P;
    const int64_t vP = static_cast<int64_t>(g.n[0]) * g.n[1] * g.n[2], vF = static_cast<int64_t>(g.m[0]) * g.m[1] * g.m[2];
    const int* n = a.region ? at.np : at.n;
    const int64_t off = LD(a.region ? a.off_Lp : a.off_L, f, a.n_sf + 1);
    const int nc = a.region ? at.ncP : at.ncL, nf = a.region ? at.nfP : at.nfL;
    const int64_t dn = a.region ? a.dst_n : a.vec_n;
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (row >= n[1] * n[2]) return;
    const int y = row % n[1] - g.r0[1], z = row / n[1] - g.r0[2];
    if (y < 0 || y >= g.m[1] || z < 0 || z >= g.m[2]) return;       // out of the band's reach: nothing to add
    const int yl = y - g.o[1], zl = z - g.o[2];
    const bool in_yz = yl >= 0 && yl < g.n[1] && zl >= 0 && zl < g.n[2];
    const double ef = a.precond ? -LD(a.eps, f, a.n_sf) : 0.0;
    double sum = 0.0;
    for (int part = 0; part < 2; ++part) {
        const int64_t r0 = part ? (a.region ? at.rowPf : at.rowLf) : (a.region ? at.rowPc : at.rowLc);
        const int64_t sg0 = part ? (a.region ? at.segPf : at.segLf) : (a.region ? at.segPc : at.segLc);
        const int s0 = LD(a.rowptr, r0 + row, a.rowptr_n), s1 = LD(a.rowptr, r0 + row + 1, a.rowptr_n);
        for (int s = s0; s < s1; ++s) {
            const Seg sg = LD(a.seg, sg0 + s, a.seg_n);
            for (int xr = sg.x0 + lane; xr <= sg.x1; xr += 32) {
                const int x = xr - g.r0[0], xl = x - g.o[0];
                if (x < 0 || x >= g.m[0]) continue;
                const bool in_L = in_yz && xl >= 0 && xl < g.n[0];
                const int64_t pf = (static_cast<int64_t>(z) * g.m[1] + y) * g.m[0] + x;
                const int64_t pp = (static_cast<int64_t>(zl) * g.n[1] + yl) * g.n[0] + xl;
                const int64_t rel = sg.off + (xr - sg.x0);
                for (int t = part ? 1 : 0; t < (part ? 8 : 1); ++t) {
                    const int64_t o = off + (part ? nc + rel + static_cast<int64_t>(t - 1) * nf : rel);
                    double v = LD(F, t * vF + pf, a.s_F);
                    if (in_L && (a.precond || energy)) {
                        const double p = LD(P, t * vP + pp, a.s_P);
                        sum = fma(p, v, sum);
                        v = fma(ef, p, v);
                    }
                    ST(dst, o, dn, accumulate ? static_cast<T>(static_cast<double>(LD(dst, o, dn)) + v) : static_cast<T>(v));
                }
            }
        }
    }
    if (energy) {
        sum = warp_sum_c(sum);
        if (lane == 0) ST(a.B, k * a.s_B + static_cast<int64_t>(z) * g.m[1] + y, (k + 1) * a.s_B, sum);
    }
}

// e[f] = the sum of the rows' sums that k_conf_store left, in a fixed order (the same bits on every
// call); a CTA per function
__global__ void __launch_bounds__(256) k_conf_energy(ConfLaunch a, double* __restrict__ e) {
    [[maybe_unused]] int* ST_ = a.status;
    [[maybe_unused]] constexpr int KID = 24;
    const int f = static_cast<int>(a.f0) + blockIdx.x;
    const AtomRec at = LD(a.atoms, LD(a.sf_atom, f, a.n_sf), a.n_atoms);
    const ConfGeo g = conf_geo(at, a.region);
    const double* rows = a.B + blockIdx.x * a.s_B;
    double v = 0.0;
    for (int i = threadIdx.x; i < g.m[1] * g.m[2]; i += blockDim.x) v += LD(rows, i, a.s_B);
    v = block_sum_c(v);
    if (threadIdx.x == 0) e[f] = v;
}

// ---------------------------------------------------------------- conjugate gradients

// x = 0, r = p = -g on the members of every function of the batch, rr = <r|r>; a CTA per function
template <class T>
__global__ void __launch_bounds__(512) k_cg_init(ConfLaunch a, const T* __restrict__ g, T* __restrict__ x, T* __restrict__ r,
                                                 T* __restrict__ p, double* __restrict__ rr) {
    const int f = static_cast<int>(a.f0) + blockIdx.x;
    const AtomRec at = a.atoms[a.sf_atom[f]];
    const int64_t o = a.off_L[f], n = at.ncL + 7LL * at.nfL;
    double v = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        const T gi = -g[o + i];
        x[o + i] = T(0);
        r[o + i] = gi;
        p[o + i] = gi;
        v += static_cast<double>(gi) * static_cast<double>(gi);
    }
    v = block_sum_c(v);
    if (threadIdx.x == 0) rr[f] = v;
}

// One iteration's updates from Ap, a CTA per function (the two dot products and the three
// vector updates used to be five launches):
//   alpha = rr / <p|Ap> (0 once rr = 0: the function's iteration has stopped); x += alpha p,
//   r -= alpha Ap; rr' = <r|r>; beta = rr' / rr (0 once rr' = 0); p = r + beta p; res = sqrt(rr')
template <class T>
__global__ void __launch_bounds__(512) k_cg_step(ConfLaunch a, double* __restrict__ rr, const T* __restrict__ Ap,
                                                 T* __restrict__ x, T* __restrict__ r, T* __restrict__ p,
                                                 double* __restrict__ res) {
    const int f = static_cast<int>(a.f0) + blockIdx.x;
    const AtomRec at = a.atoms[a.sf_atom[f]];
    const int64_t o = a.off_L[f], n = at.ncL + 7LL * at.nfL;
    const double rr0 = rr[f];
    double v = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x)
        v += static_cast<double>(p[o + i]) * static_cast<double>(Ap[o + i]);
    const double pAp = block_sum_c(v);
    const T al = static_cast<T>(rr0 == 0.0 ? 0.0 : rr0 / pAp);
    v = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        x[o + i] = x[o + i] + al * p[o + i];
        const T ri = r[o + i] - al * Ap[o + i];
        r[o + i] = ri;
        v += static_cast<double>(ri) * static_cast<double>(ri);
    }
    const double rr1 = block_sum_c(v);
    const T be = static_cast<T>((rr0 == 0.0 || rr1 == 0.0) ? 0.0 : rr1 / rr0);
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) p[o + i] = r[o + i] + be * p[o + i];
    if (threadIdx.x == 0) {
        rr[f] = rr1;
        if (res) res[f] = sqrt(rr1);
    }
}

// ---------------------------------------------------------------- host wrappers

cudaError_t configure_confine_kernels(size_t max_smem) {
    cudaError_t e;
    const void* ks[] = {reinterpret_cast<const void*>(k_conf_pass<0, true>), reinterpret_cast<const void*>(k_conf_pass<1, true>),
                        reinterpret_cast<const void*>(k_conf_pass<2, true>)};
    for (const void* k : ks) {
        cudaFuncAttributes fa;
        if ((e = cudaFuncGetAttributes(&fa, k)) != cudaSuccess) return e;
        if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      static_cast<int>(max_smem - fa.sharedSizeBytes))) != cudaSuccess)
            return e;
    }
    return cudaSuccess;
}

cudaError_t conf_tables(int n_atoms, const AtomRec* atoms, const double* pos, const double* G, const double* XY, double h,
                        const int64_t* off, double* tab, cudaStream_t s) {
    k_conf_table<<<n_atoms, 256, 0, s>>>(atoms, pos, G, XY, h, off, tab);
    return cudaGetLastError();
}

cudaError_t conf_setup(const ConfLaunch& a, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(a.maps, 0, static_cast<size_t>(a.nfn) * a.s_maps, s);
    if (e != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(a.P, 0, static_cast<size_t>(a.nfn) * a.s_P * sizeof(double), s)) != cudaSuccess) return e;
    const int rows = a.region ? std::max(a.max_rows_L, a.max_rows_P) : a.max_rows_L;
    k_conf_maps<<<dim3(static_cast<unsigned>((rows + 7) / 8), a.nfn), 256, 0, s>>>(a);
    k_conf_comb<<<dim3(3, a.nfn), 256, 0, s>>>(a);
    return cudaGetLastError();
}

template <int DIM>
static void conf_pass(const ConfLaunch& a, cudaStream_t s) {
    const dim3 g(static_cast<unsigned>((a.max_lines[DIM] + 255) / 256 * 4), a.nfn);
    const size_t smem = static_cast<size_t>(DIM == 2 ? 2 : 4) * a.max_n * 33 * sizeof(double);
    if (smem <= a.max_smem) k_conf_pass<DIM, true><<<g, 256, smem, s>>>(a);
    else k_conf_pass<DIM, false><<<g, 256, 0, s>>>(a);
}

template <class T>
static cudaError_t conf_apply_t(const ConfLaunch& a, const void* vin, void* dst, int accumulate, double* energy,
                                cudaStream_t s) {
    k_conf_load<T><<<dim3(static_cast<unsigned>((a.max_rows_L + 7) / 8), a.nfn), 256, 0, s>>>(a, static_cast<const T*>(vin));
    conf_pass<2>(a, s);
    conf_pass<1>(a, s);
    conf_pass<0>(a, s);
    k_conf_store<T><<<dim3(static_cast<unsigned>(((a.region ? a.max_rows_P : a.max_rows_L) + 7) / 8), a.nfn), 256, 0, s>>>(
        a, static_cast<T*>(dst), accumulate, energy != nullptr);
    if (energy) k_conf_energy<<<a.nfn, 256, 0, s>>>(a, energy);
    return cudaGetLastError();
}

// The operator on a batch of functions: a_f Q (+ T - eps_f with a.precond) on vin (compressed on
// L), stored on (or added to) the members of a.region; optionally <vin|result> per function.
cudaError_t conf_apply(const ConfLaunch& a, const void* vin, void* dst, int accumulate, double* energy, cudaStream_t s) {
    return a.prec == 0 ? conf_apply_t<double>(a, vin, dst, accumulate, energy, s)
                       : conf_apply_t<float>(a, vin, dst, accumulate, energy, s);
}

cudaError_t conf_cg_init(const ConfLaunch& a, const void* g, void* x, void* r, void* p, double* rr, cudaStream_t s) {
    if (a.prec == 0)
        k_cg_init<double><<<a.nfn, 512, 0, s>>>(a, static_cast<const double*>(g), static_cast<double*>(x),
                                                static_cast<double*>(r), static_cast<double*>(p), rr);
    else
        k_cg_init<float><<<a.nfn, 512, 0, s>>>(a, static_cast<const float*>(g), static_cast<float*>(x), static_cast<float*>(r),
                                               static_cast<float*>(p), rr);
    return cudaGetLastError();
}

cudaError_t conf_cg_step(const ConfLaunch& a, double* rr, const void* Ap, void* x, void* r, void* p, double* res,
                         cudaStream_t s) {
    if (a.prec == 0)
        k_cg_step<double><<<a.nfn, 512, 0, s>>>(a, rr, static_cast<const double*>(Ap), static_cast<double*>(x),
                                                static_cast<double*>(r), static_cast<double*>(p), res);
    else
        k_cg_step<float><<<a.nfn, 512, 0, s>>>(a, rr, static_cast<const float*>(Ap), static_cast<float*>(x),
                                               static_cast<float*>(r), static_cast<float*>(p), res);
    return cudaGetLastError();
}

}  // namespace lsw
