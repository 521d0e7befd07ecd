// Internal declarations shared by the host code (lsw_host.cpp, lsw_filters.cpp) and
// the CUDA kernels (lsw_kernels.cu).  Not part of the public ABI (include/lsw.h).
#pragma once

#include <cstddef>
#include <cstdint>
#include <string>

#include <cuda_runtime.h>

namespace lsw {

constexpr int D16 = 16;          // filter length 2m, m = 8 (Sec. II.B)
constexpr int H_LO = -7;         // h, g, magic filter indices -7..8
constexpr int KIN_HALF = 14;     // kinetic blocks l = -14..14
constexpr int KIN_TAPS = 2 * KIN_HALF + 1;
constexpr int FWD_LO = -14;      // combined filters (w * h), (w * g): m = -14..16
constexpr int FWD_TAPS = 31;
constexpr int MOVL_P = 5;        // moment overlaps F^p, p = 0..4 (quartic confinement)
constexpr int V_REACH = 14;      // real-space box of a coarse block [lo, hi]: [2lo-14, 2hi+16]
constexpr int ALIGN_ELEMS = 64;  // function offsets in the compressed arrays
constexpr int ZCOLS_F64 = 64;    // real-space columns per block of the z stage (FP64)
constexpr int ZCOLS_F32 = 128;   // (FP32)
constexpr size_t BWD_STATIC_SMEM = 256;               // upper bound of k_bwd_xy's static shared memory
constexpr size_t BWD_TC_STATIC_SMEM = 8 * 1024 + 512; // ... of its tensor-core versions (checked at set-up)
constexpr size_t FWD_STATIC_SMEM = 4 * 1024;          // ... of k_fwd_xy
constexpr size_t CONF_STATIC_SMEM = 2 * 1024;         // ... of k_conf_pass

// Filter tables, FP64 (rounded once from double-double).
struct FilterSet {
    double h[D16], g[D16], moments[D16], magic[D16];
    double kin_r[KIN_TAPS];
    double kin[4][KIN_TAPS];     // hh, hg, gh, gg: <X_0|d2|Y_l>
    double fwd[2][FWD_TAPS];     // (w*h)_m, (w*g)_m
    double movl[5][KIN_TAPS];    // F^p(l) = int x^p phi(x) phi(x - l) dx, p = 0..4
};

// Derive the whole table (lsw_filters.cpp).  Returns false with a message on failure.
bool derive_filters(FilterSet* out, std::string* err);

// A run of members along x inside a box: x0..x1 inclusive (box-local), row = y + ny*z
// (box-local), off = coefficient offset of x0 within its part.
struct Seg {
    int32_t x0, x1, row, off;
};

// Geometry of one atom's locregs as seen by the kernels.
struct AtomRec {
    int32_t lo[3], n[3];         // L box (coarse bounding box of the L members)
    int32_t lop[3], np[3];       // L' box
    int32_t ncL, nfL, ncP, nfP;  // member counts (coarse, fine) of L and L'
    int32_t nsegLc, nsegLf, nsegPc, nsegPf;
    int64_t segLc, segLf, segPc, segPf;  // first index in the global Seg array
    int64_t rowLc, rowLf, rowPc, rowPf;  // first index of the per-row CSR (n_rows + 1)
    int64_t colz;                // first entry of the L' column table (n_x' n_y' ColZ)
};

// Per (x, y) column of an L' box (entry y n_x' + x): the z range of its coarse members and
// the z hull of its fine members, L' box coordinates; -1, -1: none.
struct ColZ {
    int16_t c0, c1, f0, f1;
};

// One support function's real-space block in the density store (Eq. density): the
// values u = M W L phi on the fine points [2 lo - 14, 2 hi + 16] of its L box, stored
// [Z][Y][X] (x fastest) from element `off`.
struct DensFn {
    int64_t off;
    int32_t o[3];                // block origin, as a fine index local to the density grid
    int32_t d[3];                // X, Y, Z = 2 n + 29
};

// Density tiles: DT_X x DT_Y x DT_Z fine points (x fastest), one CTA each.
constexpr int DT_X = 32, DT_Y = 4, DT_Z = 4;
constexpr int DT_THREADS = 256;
constexpr int DT_PP = DT_X * DT_Y * DT_Z / DT_THREADS;   // points per thread
constexpr int DT_MC = 32;                                 // functions per chunk

// One support function inside an H phi batch.
struct FnRec {
    int32_t f, atom;
    int32_t lo[3], n[3], lop[3], np[3];
    int64_t off_phi, off_hphi;
    int64_t ws_D, ws_Bf, ws_Bb, ws_G;    // element offsets inside the batch workspace
    int64_t ws_Gf;                       // element offset of the z-arm column flags (bytes
                                         // [4][n_x n_y]: 1 where the D column pair is nonzero)
};

// The "transposed" layout of the scalar products (App. D) on one GPU: the grid is cut
// into tiles of T^3 coarse points; every function whose region touches a tile gets a
// panel row there holding its coefficients on the tile's points (T^3 scaling values,
// then the 7 wavelet values of each of the tile's fine points, zero where the function
// has no member, padded to a multiple of 4).  Panels of phi on L (the "A" side) and of
// H phi on L' (the "Q" side) turn S_ab and H_ab into small dense products per tile.
struct PanelTile {
    int32_t org[3];              // tile origin (coarse grid)
    int32_t fine0, nfine;        // the tile's fine points: tile_fine[fine0 .. fine0 + nfine)
    int32_t nA, nB;              // functions whose L (A) / L' (Q) touch the tile
    int32_t kp;                  // panel row length
    int64_t listA, listB;        // first entry of the tile's functions in listA / listB
    int64_t pA, pQ;              // element offsets of the tile's panels in its slab's buffers
};
// Per atom: its tile boxes (tiles its L and L' touch) and, per tile of each box, the
// used-tile index and the slot of the atom's first function in that tile's list
// (int2 {tile, slot}, tile = -1 where the region does not touch the tile).
struct PanelAtom {
    int32_t tloA[3], tnA[3];     // tile box of L
    int32_t tloB[3], tnB[3];     // tile box of L'
    int64_t tabA, tabB;          // first entry of the boxes' tables in the tile-table array
    int32_t f0, nsf;             // the atom's functions f0 .. f0 + nsf - 1
};
// One product work item: tile, rows a0 .. a0+na of its A list, columns c0 .. c0+nc of
// the concatenated column list [A list (S_ab); B list (H_ab)].
struct PanelItem {
    int32_t tile, a0, na, c0, nc, pad;
};
// One slab of tiles (consecutive tile-z layers) whose panels fit the panel buffers.
struct PanelSlab {
    int32_t tz0, tz1;            // tile-z layers tz0 .. tz1 - 1
    int64_t u0, u1;              // used tiles
    int64_t i0, i1;              // product items
    int64_t ci0, ci1;            // combination items (tile, A rows, panel entries)
    int64_t s0, s1;              // entries of the slab-atom list (atoms whose L' meets the slab)
    int64_t elemsA, elemsQ;      // panel elements of the slab
    size_t smem_pack;            // dynamic shared memory of the pack kernel (0: tables read from global)
};

// Dynamic shared memory of the FMA backward plane kernel for L extents (nx, ny), L' extents
// (nxp, nyp), element size es and nb outputs per block: byte offsets and sizes.  gstage: room
// for the z-arm plane; lists: as HphiLaunch::lists.
#ifdef __CUDACC__
#define LSW_HD __host__ __device__ __forceinline__
#else
#define LSW_HD inline
#endif
constexpr int BWD_NB_F32 = 8, BWD_NB_F64 = 4;   // outputs per block
struct BwdLayout {
    int RS, PS;                  // row stride (odd: rows land in different banks) and type stride of the D plane
    int nb_y, nb_x;              // blocks of rows and of columns (upper bounds)
    int taskN, taskkN, memN;     // x pass tasks, kinetic y tasks, fine members listed
    uint32_t o_pl, o_mid, o_D, o_task, o_roff, o_blk, o_row, o_mem, bytes;
};
LSW_HD BwdLayout bwd_layout(int nx, int ny, int nxp, int nyp, int es, int nb, bool gstage, bool lists) {
    BwdLayout L;
    const int X = 2 * nx + 29, Y = 2 * ny + 29;
    auto up = [](uint32_t v) { return (v + 15u) & ~15u; };
    auto mx = [](int u, int v) { return u > v ? u : v; };
    L.RS = nx | 1;
    L.PS = ny * L.RS + 1;                              // a zero after each type's rows
    L.nb_y = (nyp + nb - 1) / nb + 1;
    L.nb_x = (nxp + nb - 1) / nb;
    L.taskN = 2 * L.nb_x * nyp;
    L.taskkN = 2 * L.nb_y * (nx < nxp ? nx : nxp);
    L.memN = lists ? nxp * nyp / 3 : 0;
    L.o_pl = 16;                                       // the mbarrier first
    L.o_mid = up(L.o_pl + static_cast<uint32_t>(es) * mx(Y * X + 8, 4 * nyp * nxp));
    const int slot = (nyp * nxp + 15) & ~7;
    L.o_D = up(L.o_mid + static_cast<uint32_t>(es) * (gstage ? mx(2 * nyp * X, 4 * slot) : 2 * nyp * X));
    L.o_task = up(L.o_D + static_cast<uint32_t>(es) * (4 * L.PS));
    L.o_roff = up(L.o_task + 2u * (L.taskN + L.taskkN));
    L.o_blk = L.o_roff + 4u * nyp;
    L.o_row = L.o_blk + 4u * (3 * L.nb_y + 1 + 6 * L.nb_y + 1 + 6 * L.nb_x + 1);
    L.o_mem = L.o_row + 2u * (4 * nyp + 4 * ny + 4 * nx);
    L.bytes = up(L.o_mem + 2u * L.memN);
    return L;
}

// <chi^b_i|(x - R)^m|chi^b'_{i+l}> = (h/2)^m sum_p C(m,p) sum_k X_k (2i + k - 2c)^(m-p) G^p_Y(l, k),
// c = R / h, X, Y = XY[b], XY[b'] (h, g), G[y][p][l + 14][k] = sum_k' Y_k' F^p(2l + k' - k); lt = l + 14.
LSW_HD double conf_entry(const double* G, const double* XY, int m, int b, int bp, int lt, double i, double c, double h) {
    double acc = 0.0, cp = 1.0;                        // cp = C(m, p)
    for (int p = 0; p <= m; ++p) {
        if (p > 0) cp = cp * (m - p + 1) / p;
        const double* Gp = G + ((bp * MOVL_P + p) * KIN_TAPS + lt) * D16;
        double sk = 0.0;
        for (int k = 0; k < D16; ++k) {
            const double z = 2.0 * i + (k + H_LO) - 2.0 * c;
            double zp = 1.0;
            for (int r = 0; r < m - p; ++r) zp *= z;
            sk += XY[b * D16 + k] * zp * Gp[k];
        }
        acc += cp * sk;
    }
    const double h2 = 0.5 * h;
    double hm = 1.0;
    for (int r = 0; r < m; ++r) hm *= h2;
    return hm * acc;
}

// Kernel kinds of the per-launch device trace (lsw_profile / lsw_profile_read).
enum TraceKind : int {
    TK_MEMSET = 0, TK_UNCOMPRESS, TK_FWD_XY, TK_Z, TK_BWD_XY, TK_KINETIC, TK_PACK, TK_HS,
    TK_DENS_U, TK_DENSITY, TK_COUNT
};

// Host-side recorder of CUDA event pairs around launches; NULL = no tracing.
struct Tracer;
void trace_begin(Tracer* tr, int kind, cudaStream_t s);
void trace_end(Tracer* tr, cudaStream_t s);

struct HphiLaunch {
    Tracer* tr;
    int prec;                    // 0 FP64, 1 FP32
    const FnRec* fn;             // device records of this batch
    int nfn;
    int n_sm;                    // of the device
    int max_nz, max_nzp;         // largest L / L' z extents in the batch
    int max_cols;                // largest (2ny+29)(2nx+29) in the batch
    int max_rowsP;               // largest ny'*nz' of L'
    int64_t max_ptsP;            // largest nx'*ny'*nz' of L'
    int max_colsP;               // largest nx'*ny' of L'
    int max_colsL;               // largest nx*ny of L
    int max_rowsL;               // largest ny*nz of L
    int max_segL;                // largest coarse+fine segment count of L
    int max_segP;
    size_t smem_fwd, smem_z, smem_bwd;
    int gstage;                  // 1: the backward plane kernel stages the z-arm plane in shared
                                 // memory (smem_bwd includes it); 0: reads it from global memory
    int lists;                   // 1: room for its list of fine members; 0 (boxes that leave none):
                                 // the members are searched in the segments
    int zcols;                   // columns per CTA of the z stage
    int zsplit;                  // 0: z stage on FMA units; 2 or 3: bfloat16 parts per
                                 // FP32 operand of the tensor-core z stage
    int xy_tc;                   // 1: the x, y passes run on the tensor-core plane kernels too
                                 // (with zsplit parts); 0: on the FMA plane kernels
    size_t smem_ztc;             // dynamic shared memory of the tensor-core z stage
    size_t smem_bwd_tc;          // dynamic shared memory of the tensor-core plane kernel
    size_t smem_fwd_tc;          // dynamic shared memory of the tensor-core forward plane kernel
    size_t smem_kin;             // dynamic shared memory of the kinetic z-arm kernel
    // persistent FMA plane kernels: the batch's items (first function, functions << 11 |
    // plane << 1 | z type; the forward kernel's hold one function), largest first, taken
    // from queue[0] (forward) and queue[1] (backward), which are zeroed before the batch;
    // grid_* CTAs (as many as fit on the GPU).  NULL items: one CTA per (2 planes + z type,
    // function) grid slot.
    const int2* items_fwd;
    const int2* items_bwd;
    int n_items_fwd, n_items_bwd;
    int grid_fwd, grid_bwd;
    int* queue;
    int fwd_list;                // 1: the forward x pass computes only the blocks whose input
                                 // window meets the row's members (the rest of its plane is 0)
    int wait_out;                // 1: the backward kernel's waits count as run out (tests of the failure path)
    const AtomRec* atoms;
    const Seg* seg;
    const int32_t* rowptr;
    const ColZ* colz;            // L' column tables (NULL: the kinetic z arm computes every plane)
    int64_t colz_n;
    const void* phi;
    void* hphi;
    double* e_kin;
    double* e_pot;
    const void* V;
    int64_t vlo[3], vn[3];
    void* ws;                    // batch workspace base
    int64_t ws_D_elems;          // D region size (memset)
    double kin_scale;            // -1 / (2 h^2)
    int* status;
    // extents used by the self-checking build (-DLSW_CHECKED)
    int64_t phi_n, hphi_n, v_n, ws_n, seg_n, rowptr_n;
    int n_atoms;
    // density: real-space store written by the density z stage (NULL otherwise)
    void* U;
    const DensFn* dfn;           // per function (indexed by FnRec::f)
    int64_t U_n;
};

// The density products rho_j = sum_ab K_ab u_a(j) u_b(j) over the tiles of the grid.
struct DensLaunch {
    Tracer* tr;
    int prec;
    const DensFn* fn;            // per function
    const void* U;               // real-space store
    const int64_t* tptr;         // [ntiles + 1]: functions of tile t are tfn[tptr[t] .. tptr[t+1])
    const int32_t* tfn;          // ascending within a tile
    const int32_t* sf_atom;
    const int64_t* row_ptr;      // pattern CSR
    const int32_t* col;
    const double* K;             // density kernel on the pattern
    double* rho;                 // [gz][gy][gx]
    int64_t gn[3];               // grid extents
    int32_t ntile[3];
    int max_m, max_g;            // most functions and atoms of a tile (0: too many for shared memory)
    int* status;
    // extents used by the self-checking build (-DLSW_CHECKED)
    int64_t U_n, tfn_n, nnz, rho_n, fn_n, tptr_n, rowp_n;
};

// Pack: panels of one slab (grid: slab atoms x 2 sides).
struct PackLaunch {
    Tracer* tr;
    int prec;
    const PanelTile* tiles;
    const PanelAtom* patoms;
    const int2* ttab;            // per-atom tile tables
    const int32_t* slab_atoms;   // atoms of this slab
    int n_slab_atoms;
    int tz0, tz1;
    int tile;                    // tile edge T
    int64_t u0;                  // first used tile of the slab
    const int32_t* tile_fine;    // fine points of the tiles: local x | y << 8 | z << 16
    const AtomRec* atoms;
    const Seg* seg;
    const int32_t* rowptr;
    const int64_t* off_L;
    const int64_t* off_Lp;
    const void* phi;
    const void* hphi;            // NULL: pack the A side only
    void* PA;
    void* PQ;
    size_t smem;                 // dynamic shared memory: 0 = region tables read from global
    void* out;                   // unpack (combination): compressed output on L; NULL: pack
    int* status;
    int64_t phi_n, hphi_n, seg_n, rowptr_n, fine_n, ttab_n, PA_n, PQ_n, out_n;
    int n_atoms, n_tiles, n_sf;
};

// Product: S_ab and H_ab contributions of one slab's tiles, added to the CSR values
// (or, for the combination, the output panels of one slab's tiles).
struct PanelHSLaunch {
    Tracer* tr;
    int prec;
    const PanelTile* tiles;
    const PanelItem* items;
    int64_t nitems;
    const int32_t* listA;
    const int32_t* listB;
    const int32_t* sf_atom;
    const int64_t* row_ptr;      // pattern CSR
    const int32_t* col;
    const void* PA;
    const void* PQ;              // combination: the output panels (A layout) in the Q buffer
    double* H;
    double* S;
    const double* M;             // combination: coefficients on the pattern
    int coef_rows;               // combination: functions whose coefficients a CTA holds at a time (a multiple of 32)
    int tc;                      // 1: FP32 products on the tensor cores (split bfloat16)
    int* status;
    int64_t listA_n, listB_n, nnz, PA_n, PQ_n, n_tiles;
    int n_sf;
};

// Fermi operator expansion on the pattern (lsw_foe.cu): shared arguments.
struct FoeLaunch {
    int n;                       // functions (rows)
    int64_t nnz;
    const int64_t* row_ptr;      // pattern CSR (symmetric, with the diagonal)
    const int32_t* col;
    const int64_t* tpos;         // position of the transposed entry of each entry
    const int64_t* diag;         // position of the diagonal entry of each row
    // groups: the functions of an atom, which share their pattern row
    int ng;
    const int32_t* gfirst;       // first function of each group (ng + 1)
    const int32_t* nptr;         // neighbours of a group: ngrp, npos [nptr[g] .. nptr[g + 1])
    const int32_t* ngrp;         // neighbour group
    const int32_t* npos;         // position of its first function in the group's rows
    int64_t nn;                  // neighbour entries
    size_t triple_smem;          // dynamic shared memory of the grouped triple product (0: the rows
                                 // of w do not fit; scratch is used)
    double* scratch;             // triple_ctas dense rows of n values, zero between uses
    int triple_ctas, cheb_ctas;
    int split;                   // CTAs that share a group's neighbours in the Chebyshev step
    int chunk;                   // entries a warp of the Chebyshev step lists at a time (a multiple of 32)
    int* status;
};
inline size_t foe_cheb_smem(int n, int chunk) { return (static_cast<size_t>(n) + 8 * static_cast<size_t>(chunk)) * sizeof(int); }
cudaError_t configure_foe_kernels(size_t max_smem);
cudaError_t foe_prep(const FoeLaunch& a, const double* H, const double* S, double sigma, double tau, double* Ht,
                     double* X, cudaStream_t s);
cudaError_t foe_triple(const FoeLaunch& a, const double* X, const double* A, double* Y, cudaStream_t s);
cudaError_t foe_cheb(const FoeLaunch& a, const double* Htp, const double* Tc, const double* Tp, double alpha, double* Tn,
                     cudaStream_t s);
cudaError_t foe_traces(const FoeLaunch& a, const double* T, int count, double* out, cudaStream_t s);
cudaError_t foe_kernel_sum(const FoeLaunch& a, const double* I, const double* T, const double* c, int m, double* K,
                           cudaStream_t s);
constexpr int FOE_PARTS = 1024;  // partial sums of E_BS
cudaError_t foe_axpy_t(const FoeLaunch& a, double* K, const double* T, double c, cudaStream_t s);
cudaError_t foe_transpose(const FoeLaunch& a, const double* src, double* dst, cudaStream_t s);
cudaError_t foe_ebs(const FoeLaunch& a, const double* K, const double* Ht, const double* S, double sigma, double tau,
                    double* part, double* out, cudaStream_t s);

// Quartic confinement and preconditioning (lsw_confine.cu): one batch of functions
// f0 .. f0 + nfn - 1.  Boxes (FP64, strides s_* in elements per function, x fastest, 8 types
// each): P on the L box n; A, OZ on [z: output box][y, x: L box]; B, OY on [z, y: output box]
// [x: L box]; F on the output box m (region 0: the L box; 1: the L' box within the band's reach).
struct ConfLaunch {
    int prec;
    int region;                  // output region: 0 L, 1 L'
    int precond;                 // 1: + T - eps (Eq. precond)
    int64_t f0;
    int nfn;
    const int32_t* sf_atom;
    const AtomRec* atoms;
    const Seg* seg;
    const int32_t* rowptr;
    const int64_t* off_L;
    const int64_t* off_Lp;
    const double* qtab;          // per atom: [dim][m = 2, 4][b b'][i over the L box widened by 14][l + 14] of X_d^m
    const int64_t* qtab_off;     // first table entry of each atom (n_atoms + 1)
    const double* acoef;         // a_f, the confinement prefactor of each function
    const double* eps;           // eps_f of the preconditioning equation (NULL otherwise)
    double kin[4][KIN_TAPS];     // kinetic blocks hh, hg, gh, gg
    double kin_scale;            // -1 / (2 h^2)
    double *P, *A, *OZ, *B, *OY, *F;
    double* comb;                // per function [dim][b b'][max_m][29]: a_f X_d^4 (+ kinetic)
    unsigned char* maps;         // member maps of a batch (ConfMaps)
    int64_t s_P, s_A, s_B, s_F, s_comb, s_maps;
    int64_t s_mem, s_xy, s_xz, s_x, s_row, s_oxz;   // bytes of one function's maps
    int max_n, max_m;            // largest extents of the L and the output boxes
    int max_lines[3];            // largest number of lines of the passes along x, y, z
    int max_rows_L, max_rows_P;  // largest ny * nz of L and of L' boxes in the batch
    size_t max_smem;             // dynamic shared memory the pass kernels may use
    int* status;
    int64_t qtab_n, seg_n, rowptr_n, vec_n, dst_n;
    int n_sf, n_atoms;
};
// Maps of one function of a batch; the two halves of act_* and out_*: coarse, fine members.
struct ConfMaps {
    unsigned char *mem, *act_xy, *act_xz, *act_x, *out_row, *out_xz;
};
#ifdef __CUDACC__
__device__ __forceinline__ ConfMaps conf_maps(const ConfLaunch& a, int k) {
    ConfMaps m;
    m.mem = a.maps + k * a.s_maps;
    m.act_xy = m.mem + a.s_mem;
    m.act_xz = m.act_xy + a.s_xy;
    m.act_x = m.act_xz + a.s_xz;
    m.out_row = m.act_x + a.s_x;
    m.out_xz = m.out_row + a.s_row;
    return m;
}
#endif
cudaError_t configure_confine_kernels(size_t max_smem);
cudaError_t conf_tables(int n_atoms, const AtomRec* atoms, const double* pos, const double* G, const double* XY, double h,
                        const int64_t* off, double* tab, cudaStream_t s);
cudaError_t conf_setup(const ConfLaunch& a, cudaStream_t s);
cudaError_t conf_apply(const ConfLaunch& a, const void* vin, void* dst, int accumulate, double* energy, cudaStream_t s);
cudaError_t conf_cg_init(const ConfLaunch& a, const void* g, void* x, void* r, void* p, double* rr, cudaStream_t s);
cudaError_t conf_cg_step(const ConfLaunch& a, double* rr, const void* Ap, void* x, void* r, void* p, double* res,
                         cudaStream_t s);

// Fixed device scratch of the allocation-free Hamiltonian entry point (lsw_kernels.cu).
constexpr size_t NOALLOC_SCRATCH_BYTES = static_cast<size_t>(32) << 20;   // 32 MiB
constexpr int NOALLOC_MAX_DEVICES = 64;
constexpr int NOALLOC_MAX_BATCH = 64;      // functions per batch (records kept in the scratch)
cudaError_t noalloc_scratch(int device, void** ptr);
// Batch records of the allocation-free path, built on the device from the system's
// resident records all[f0 .. f0 + nb) with the batch's own workspace offsets.
cudaError_t enqueue_noalloc_records(const FnRec* all, int64_t f0, int nb, int64_t esize, FnRec* out, cudaStream_t s);

// Support-function reuse across geometries (lsw_reformat).
struct ReformatLaunch {
    const FnRec* fn;             // destination records (boxes, offsets); unused ws fields
    int nfn;
    int max_seg;                 // largest coarse+fine segment count of a destination L
    const AtomRec* atoms_dst;
    const AtomRec* atoms_src;
    const Seg* seg_dst;
    const Seg* seg_src;
    const int32_t* rowptr_src;
    const int32_t* shift;        // [n_atoms][3] grid shift of each atom (dst = src + shift)
    const int64_t* off_src;      // source function offsets
    const void* phi_src;
    void* phi_dst;
    int prec;
    int* status;
    int64_t seg_dst_n, seg_src_n, rowptr_src_n, src_n, dst_n;
};
cudaError_t enqueue_reformat(const ReformatLaunch& a, cudaStream_t s);

// Device entry points (lsw_kernels.cu).
cudaError_t upload_filters(const FilterSet& fs, int device);
cudaError_t measure_peaks(int n_sm, double* fp32_tflops, double* fp64_tflops, double* copy_gbs);
cudaError_t configure_kernels(size_t max_smem);
// Resident CTAs per SM of the FMA plane kernels at these dynamic shared-memory sizes.
cudaError_t plane_kernel_blocks(int prec, size_t smem_fwd, size_t smem_bwd, int* fwd, int* bwd);
cudaError_t enqueue_hphi_batch(const HphiLaunch& a, cudaStream_t s);
cudaError_t enqueue_pack(const PackLaunch& a, cudaStream_t s);     // panels of a slab (lsw_panels.cu)
cudaError_t enqueue_panel_hs(const PanelHSLaunch& a, cudaStream_t s);   // S, H from the panels
int combine_rows(int max_functions);   // PanelHSLaunch::coef_rows for tiles of at most that many functions
cudaError_t enqueue_panel_combine(const PanelHSLaunch& a, cudaStream_t s);   // M Phi panels
cudaError_t enqueue_lowdin_coeffs(const int64_t* row_ptr, const int32_t* col, const double* S, double* T, int n_sf,
                                  cudaStream_t s);
cudaError_t configure_panel_kernels(size_t max_smem);
size_t panel_hs_smem(int prec);
cudaError_t enqueue_dens_batch(const HphiLaunch& a, cudaStream_t s);   // real-space values
cudaError_t enqueue_density(const DensLaunch& a, cudaStream_t s);      // pair products
size_t density_smem(int prec, int max_m, int max_g);

// Status word bits set by device-side checks.
enum : int {
    ST_BAD_BOX = 1,
    ST_BAD_SEG = 2,
    ST_BAD_PAIR = 4,
    ST_BAD_INDEX = 8,   // self-checking build: an index fell outside its buffer
    ST_WAIT_TIMEOUT = 16,   // a bounded wait for tensor-core completion ran out
};

// Layout of the device status block (int32 words): [0] status bits, [1] first bad
// kernel id, [2] source line, [3] block, [4..5] index (int64), [6..7] bound (int64).
constexpr int STATUS_WORDS = 8;

}  // namespace lsw
