// Device-side argument blocks and launchers of libfdu (internal).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace fdu {

constexpr int kSell = 32;        // SELL slice width of the divergence tables (one warp)
constexpr int kEdgeBlock = 128;  // threads per block, edge-flux kernels
constexpr int kDivBlock = 128;   // threads per block, divergence kernels

// Precision 64 takes an edge's increments in double words where FP32's exponent
// range holds them.  The kernels that write a state's fluxes (vertex_flux, the
// stage epilogues) check every vertex: density and energy within 2^+-kWideExp
// and a positive pressure, which bounds the momentum, so that squares and
// products of the edge flux stay far from 2^+-126 and no NaN or infinity is there.  wide[i]
// is non-zero when the state of flux buffer i (0..2) failed, wide[3] when a
// ghost of the state that was set did (Dirichlet ghosts keep it).  A stage
// that finds wide[in] or wide[3] set runs in FP64 throughout.  The edge kernels
// clear the slots (clear_wide): the first stage's those of the two intermediate
// states, the third stage's that of the result, so that the flag of a state
// whose step is only partly taken (the adjoint's recomputation) stands.  A batch
// has a group of kWideSlots flags for each of its meshes after the first group,
// which then says whether any mesh's is set: a mesh takes the arithmetic that it
// would take alone.
constexpr int kWideGhost = 3;
constexpr int kWideSlots = 4;
constexpr int kWideExp = 24;
constexpr double kDwMax = 0x1p40;  // largest table entry of the double-word path of precision 64

// Edge-flux inputs (internal ids, SoA over the active edges).
struct EdgeArgs {
    const int32_t *sten;  // [6][ne]  L3 L2 L1 R1 R2 R3
    const void *coef;     // FP64: [kEdgeCoef][ne]; FP32: [6][ne] float4 of values 0..23, or (coef_gaps) [ne]
                          // float4 of stencil gaps; then [ne] float2 (n_x, n_y)
    bool coef_gaps;       // FP32: the block is the compact gaps form (values formed in the kernel)
    const void *w;        // FP64: [nv][4] double; FP32: [nv] float4
    void *r;              // FP64: [ne][4] double; FP32: [ne] float4
    int64_t ne;
    double gm1, eps;      // gamma - 1 and the WENO epsilon (FP64 path)
    double hgm1;          // (gamma - 1) / 2
    float gm1f, epsf;     // the same for the FP32 path
    unsigned long long *fallback;  // edges that fell back to first order (device counter)
    const double *dt_dev; // adaptive stepping: a zero time step here skips the launch
    const double *Q;      // FP64: per-vertex Roe records of the stage state (nullptr = compute per edge)
    // double-word edge flux (precision 48; Q is required there): r receives
    // the increment r_k - F_n(L1_k) as double words, [ne] x two float4
    // (h0, l0, h1, l1), (h2, l2, h3, l3)
    const float4 *coefdw; // [kDwPairs][ne] paired double words of the coefficient block
    float dw_gm1[2];      // gamma - 1 as a double word
    float dw_tenth[2];    // 0.1 as a double word
    float dw_eps[2];      // WENO epsilon = dw_eps * 2^dw_eps_e, dw_eps in [1, 2)
    int dw_eps_e;
    // precision 64 and 48: whether a state left the double words' window
    // (WideFlags), and the buffer slot of the stage state; nullptr: FP64 only
    int *wide;
    int wide_in;
    const int32_t *wcomp; // batch: mesh of each vertex (nullptr: one mesh)
    int n_comp;           // and their number
};


// Divergence of an FP64 state: plain FP64 tables and edge fluxes; double-word
// edge increments with the folded tables (precision 48); or by the wide flags
// either of the two (precision 64).
enum { kDivPlain = 0, kDivDw = 1, kDivGuard = 2 };

// Divergence (+ optional SSP-RK3 stage) inputs.
struct DivArgs {
    int64_t n_real;              // vertices with a residual (internal ids 0..n_real-1)
    const int64_t *slice_voff;   // [nslice+1] start of each slice's vertex entries
    const int64_t *slice_eoff;   // [nslice+1]
    const int32_t *perm;         // [n_real] vertex at each SELL position (nullptr = position i is vertex i)
    const int32_t *vid;          // vertex entries (SELL: entry j of lane l at off + 32 j + l)
    const void *wf, *wg;         // weights of f_j and g_j
    // precision 64 and 48: folded vertex weights, double-word edge weights and
    // centre weights that go with the double-word edge increments
    const double *wf48, *wg48, *cfg48;
    const float2 *we48;
    const int32_t *eid;          // edge entries
    const void *we;              // weights of r_k
    const void *cfg;             // [2][n_real] centre weights: -(sum wf + sum we nx), -(sum wg + sum we ny)
    const void *F;               // vertex fluxes of the stage state: FP64 [nv][8] (f0..3, g0..3); FP32 [nv][2] float4 pairs
    const void *r;               // edge fluxes (double-word edge increments for kDivDw)
    int kind;                    // FP64 state: kDivPlain, kDivDw or kDivGuard
    int *wide;                   // WideFlags (nullptr: not kept), and the slots of the stage's input and output
    int wide_in, wide_out;
    const int32_t *wcomp;        // batch: mesh of each vertex, for the flags
    // residual output (mode 0)
    double *out;                 // [nv][4] FP64
    const int32_t *out_map;      // internal -> output row (nullptr = internal order)
    // RK stage (modes 1..3)
    const double *wn;            // [nv][4] state at the start of the step
    const double *ws;            // [nv][4] stage input state
    double *wout;                // [nv][4] stage output state (may alias ws)
    void *Fout;                  // vertex fluxes of wout (same layout as F)
    double *Qout;                // FP64: Roe records of wout (nullable)
    float4 *w32out;              // FP32 copy of wout (FP32 residual path), or nullptr
    double dt;
    const double *dt_dev;        // if non-null, dt is read here
    double gm1;                  // gamma - 1
    float gm1f;
    const int32_t *comp;         // batched meshes: component of each internal vertex (nullptr = one mesh)
    const double *dt_comp;       // batched meshes: time step of each component
    double pos_alpha;            // stage positivity safeguard (0 = off)
    unsigned long long *limited; // vertices whose stage update the safeguard scaled
};

// ---- Divergence tiles.  A tile is up to kTile consecutive vertices (internal
// order) of one mesh: a batch starts a tile at each of its meshes, so that a
// vertex's entries are summed in the order they have in the mesh alone.
// The distinct vertices and edges of its stencils are listed once (ascending
// ids), a block copies their fluxes into shared memory, and the stencil entries
// name them by 16-bit position in those lists.  Inside a tile the vertices are
// ordered by decreasing stencil size (perm), 32 to a slice; a slice's entries
// are stored in groups of four per lane (four positions, four weights: 8- and
// 16-byte loads), each slice padded to its longest list with weight 0.
constexpr int kTile = 128;
constexpr int kTileMaxV = 1024, kTileMaxE = 2048;  // capacity of a tile's lists
// Source of the tiles: a SELL layout of the divergence tables.
struct TileSource {
    const int32_t *start;  // [ntiles + 1] first vertex of each tile
    const int64_t *slice_voff, *slice_eoff;
    const int32_t *vid, *eid;
    const float *wf, *wg, *we;
};
struct TileTables {
    int64_t ntiles;
    int smem;                    // staging bytes of the largest tile (0: no tiles)
    int32_t *perm;               // [ntiles * kTile] vertex at each position (-1 past the last)
    int32_t *voff, *eoff;        // [ntiles + 1] start of each tile's lists
    int32_t *vlist, *elist;      // vertex and edge ids
    int32_t *gvoff, *geoff;      // [ntiles * kTile / kSell + 1] first entry group of each slice
    ushort4 *vpos, *epos;        // [groups][kSell] positions in the tile's lists
    float4 *wf, *wg, *we;        // [groups][kSell] weights
};
// Sizes of the tiles' lists (nv, ne; -1 where a tile exceeds the capacity) and
// of the slices' entry groups (gv, ge), and the positions' order (T.perm).
void launch_tile_count(const TileSource &S, const TileTables &T, int32_t *nv, int32_t *ne, int32_t *gv, int32_t *ge,
                       cudaStream_t s);
// Lists, positions and weights (the offsets are in place).
void launch_tile_fill(const TileSource &S, const TileTables &T, cudaStream_t s);

// F[v] = (f, g) of w[v]; Q (optional) = Roe records (sqrt rho, sqrt rho u, sqrt rho v, sqrt rho H)
// wide (optional): slot 0 of the WideFlags for vertices below n_real, kWideGhost for the others; wcomp: a batch's meshes
void launch_vertex_flux_f64(const double *w, double *F, int64_t n, double gamma, cudaStream_t s, double *Q = nullptr,
                            int *wide = nullptr, int64_t n_real = 0, const int32_t *wcomp = nullptr);
void launch_vertex_flux_f32(const double *w, float4 *F, float4 *w32, int64_t n, double gamma, cudaStream_t s);
void launch_edge_flux_f64(const EdgeArgs &a, cudaStream_t s);    // FP64 throughout
void launch_edge_flux_guard(const EdgeArgs &a, cudaStream_t s);  // precision 64: double words within the window
void launch_edge_flux_f32(const EdgeArgs &a, cudaStream_t s);
void launch_edge_flux_dw(const EdgeArgs &a, cudaStream_t s);
// Folded divergence tables from the FP64 SELL tables in `a` (n_real, perm,
// slices, ids, wf, wg, we, cfg), the edges' left vertices and normals; *bad |= 1
// where an edge's left vertex is outside a vertex's stencil, |= 2 where a
// weight or coefficient is beyond the double words' window.
void launch_fold_tables(const DivArgs &a, const int32_t *left, const double *nx, const double *ny, double *wf48,
                        double *wg48, float2 *we48, double *cfg48, int *bad, cudaStream_t s);
// coefdw[kDwPairs][ne] = the double words of coef[kEdgeCoef][ne], paired
void launch_coef_dw(const double *coef, float4 *coefdw, int64_t ne, int *bad, cudaStream_t s);
// z = double-word primitive `op` of x (and y), device pointers (accuracy check)
void launch_dw_check(int op, const double *x, const double *y, double *z, int64_t n, cudaStream_t s);
void launch_div_f64(const DivArgs &a, int mode, cudaStream_t s);
void launch_div_f32(const DivArgs &a, int mode, cudaStream_t s);
void launch_div_f32_tiles(const DivArgs &a, const TileTables &t, int mode, cudaStream_t s);
// *bad = min(*bad, first row of w[n][4] with rho <= 0 or a non-finite value)
void launch_check_rows(const double *w, int64_t n, unsigned long long *bad, cudaStream_t s);
// zero (optional): nzero doubles (at most max(n, 256)) that the launch also sets to 0
void launch_permute_rows(const double *in, double *out, const int32_t *map, int64_t n, bool gather, cudaStream_t s,
                         double *zero = nullptr, int nzero = 0);
void launch_ghost_fill(double *w, const double *wsrc, void *F, const void *Fsrc, int fq, double *Q, const double *Qsrc,
                       float4 *w32, const int32_t *donor, int64_t n_real, int64_t n_ghost, cudaStream_t s);
// FMA throughput (TFLOP/s) of `precision` 64 or 32 with sms*8 blocks of 256
// threads; scratch holds sms*8*256 elements of that precision.
double fma_probe_tflops(int precision, int sms, void *scratch, cudaStream_t s);
// y[i] = the kernels' FP64 reciprocal (which = 0) or reciprocal square root
// (which = 1) of x[i] (device pointers; accuracy check)
void launch_recip_check(const double *x, double *y, int64_t n, int which, cudaStream_t s);
// k[24 i + j] = value j of the FP32 edge kernel's NU-WENO5 block formed from gaps g[i]
void launch_weno_coef32_check(const float4 *g, float *k, int64_t n, cudaStream_t s);
// Adaptive step, finalised by the last block of the reduction: dt = min(cfl *
// bound, t_end - t) from the reduced bound in *slot (bit pattern of a positive
// double); tstate = (t, dt, nonphysical); the slot is reset to +inf for the next
// reduction; *nsteps counts steps with dt > 0; *done counts the blocks (0
// between launches).  tstate = nullptr: the reduction alone.
struct DtFinal {
    double *tstate;
    double cfl, t_end;
    unsigned long long *nsteps;
    unsigned int *done;
};
void launch_max_dt(const double *w, const double *hmin, int64_t n, double gamma, unsigned long long *slot,
                   cudaStream_t s, const int32_t *comp = nullptr, const DtFinal &fin = DtFinal{});

// One SSP-RK3 stage (mode 1..3) of a batch as one cooperative launch of
// `blocks` x `threads` (edge fluxes, bounded grid barrier, divergence +
// stage).  The barrier expects `nblocks_expected` arrivals (= blocks in
// normal use) and gives up after `spin_limit` polls, setting *err.
cudaError_t launch_stage_persistent(int prec, int mode, const EdgeArgs &ea, const DivArgs &da, unsigned int *bar_count,
                                    unsigned int *bar_gen, unsigned int nblocks_expected,
                                    unsigned long long spin_limit, int *err, int threads, int blocks,
                                    const TileTables &tiles, cudaStream_t s);
// Co-resident blocks per SM of the persistent stage kernel at `threads`; guard:
// the mesh's precision-64 kernel takes the double-word path (kDivGuard); tiles:
// its FP32 divergence tiles.
int persistent_blocks_per_sm(int prec, int threads, bool guard, const TileTables &tiles);

}  // namespace fdu
