// Stage kernels of the ASE-DFF-CGKS step.  See cgks_device.cuh for the
// mathematics; this file maps it onto the work items of every mesh in a
// descriptor table: a block per tile in the 2-D Steps 1-2, a contiguous run of
// strips per warp in the 2-D flux, grid-stride loops in the other kernels.
//
// Local frame of a direction: dir 0 (faces normal to x): a = i (normal
// index), b = j (tangential); dir 1 (faces normal to y): a = j, b = i.
// Momentum components are ordered normal first in the local frame.
//
// Scratch layouts per mesh and direction (na, nb: cells along / across the
// normal; M Gauss points per face).  Direction 0 as written; direction 1 with
// the two spatial indices swapped, so the global x index is always fastest:
//   FR  [2][3][M][nb+2][na+1][4]      face states: side 0 = left (from cell f-1),
//                                     side 1 = right (from cell f); W, W_n and W_nn,
//                                     one plane per Gauss line, so that the lanes of
//                                     a warp, which cover consecutive faces, read a
//                                     line's points as consecutive 16-byte groups
//   FO  [NO][M][nb][na+1][4], [NO][nb][na+1][4]   stage outputs (local frame; NO = 2
//                                     quantities of each kind in stage 1, 1 in stage 2):
//                                     interface states per point, one plane per quantity
//                                     and line, then the Gauss sums of the fluxes per face.
//                                     1-D: [4][nx+1][4]
//   AT  [nb+2][na+6]                  tangential r5 DFF of each cell (Step 3)
//   TD  [nb+2][na+6][12]              FP32 bulk: the cell's hi (the base of the face
//                                     states) and its tangential differences hi(a, b-1) -
//                                     hi(a, b), hi(a, b+1) - hi(a, b), for the bases of the
//                                     Step 3 segments
//
// FP32-bulk form: a cell average W (FP64) is held in the float planes as
// hi = float(W) and lo = float(W - hi), and every reconstructed quantity that
// is a value (line averages, face states, the equilibrium state, the
// interface states) is carried as an increment over the hi of one cell: the
// line average of cell i as lo_i + (its reconstruction's increment), both
// states of a face, its equilibrium state and its interface states as
// increments over hi of the face's right cell.  Stencil
// data enter as differences (hi_k - hi_i) + (lo_k - lo_i), exact in float
// for neighbouring values, so the FP32 arithmetic only ever rounds small
// increments; the O(1) Euler flux of the base hi is formed in float-float in
// the update and the flux of the increment by difference algebra in the
// flux kernel.  The rounding that remains is relative to the increments.
#pragma once
#include "cgks_device.cuh"

namespace cgks {

__device__ __forceinline__ int vglob(int dir, int v) { return dir == 0 ? v : (v == 1 ? 2 : (v == 2 ? 1 : v)); }

template <int M>
__device__ __forceinline__ void local_dims(const Mesh& g, int dir, int& na, int& nb)
{
    na = dir == 0 ? g.nx : g.ny;
    nb = dir == 0 ? g.ny : g.nx;
}

// cell value in local coordinates; lkind: 0 W, 1 W_n (cell), 2 W_t (cell), 3 W_n line,
// 5 the low part of W (FP32-bulk form)
template <int D, int M, typename T, bool WALLS = true>
__device__ __forceinline__ T lcell(const Mesh& g, const T* S, int dir, int lkind, int v, int l, int a, int b,
                                   double tb)
{
    int kind;
    if (lkind == 0 || lkind == 5) kind = lkind;  // W, or its low part (FP32-bulk form)
    else if (lkind == 1) kind = dir == 0 ? 1 : 2;
    else if (lkind == 2) kind = dir == 0 ? 2 : 1;
    else kind = dir == 0 ? 3 : 4;
    int i = dir == 0 ? a : b, j = dir == 0 ? b : a;
    return cell<D, M, T, WALLS>(g, S, kind, vglob(dir, v), l, i, j, tb);
}

// sigma of normal faces (f, b) and of tangential faces of column a (a, f)
template <int D, bool WALLS = true>
__device__ __forceinline__ double lsigN(const Mesh& g, const double* sx, const double* sy, int dir, int f, int b)
{
    return dir == 0 ? sigx<D, WALLS>(g, sx, f, b) : sigy<WALLS>(g, sy, b, f);
}
template <bool WALLS = true>
__device__ __forceinline__ double lsigT(const Mesh& g, const double* sx, const double* sy, int dir, int a, int f)
{
    return dir == 0 ? sigy<WALLS>(g, sy, a, f) : sigx<2, WALLS>(g, sx, f, a);
}

// Scratch indexing.  Direction 0 keeps the normal index a (= i) fastest,
// direction 1 the tangential index b (= i): in both directions the global x
// index runs fastest, in memory and across threads, so every kernel walks the
// SoA state planes with unit stride.
//   cell_idx: a in [-3, na+2], b in [-1, nb]   (AT, TD)
//   fr_row:   bb = b + 1 in [0, nb+1], f in [0, na]   (FR)
//   pt_idx:   b in [0, nb), f in [0, na]       (FO)
__device__ __forceinline__ long long cell_idx(int dir, int na, int nb, int a, int b)
{
    return dir == 0 ? (long long)(b + 1) * (na + 6) + (a + 3) : (long long)(a + 3) * (nb + 2) + (b + 1);
}
// FR rows are padded to 8 points (128 bytes of FP32), so that the strips of the
// flux kernel start on whole memory sectors: unpadded, it read 1436 MB instead
// of 917 at 1024^2.  Unsigned: 1-D meshes go up to 2^31 - 3 cells
__host__ __device__ __forceinline__ unsigned fr_pitch(int n) { return ((unsigned)n + 7u) & ~7u; }
__device__ __forceinline__ long long fr_row(int dir, int na, int nb, int bb, int f)
{
    return dir == 0 ? (long long)bb * fr_pitch(na + 1) + f : (long long)f * fr_pitch(nb + 2) + bb;
}
__device__ __forceinline__ long long pt_idx(int dir, int na, int nb, int b, int f)
{
    return dir == 0 ? (long long)b * (na + 1) + f : (long long)f * nb + b;
}
// element offsets of a 4-value group: FR (row = fr_row of nrow rows) and FO
// (face = pt_idx, nf faces a plane)
__host__ __device__ __forceinline__ long long fr_nrow(int dir, int na, int nb)
{
    return dir == 0 ? (long long)(nb + 2) * fr_pitch(na + 1) : (long long)(na + 1) * fr_pitch(nb + 2);
}
__device__ __forceinline__ long long fr_off(long long nrow, int M, int side, int nd, int l, long long row)
{
    return (((long long)(side * 3 + nd) * M + l) * nrow + row) * 4;
}
__device__ __forceinline__ long long fo_off(long long nf, int M, int q, int l, long long face)
{
    return ((long long)(q * M + l) * nf + face) * 4;
}

// sums over a face's points, after the NO quantities of the points
__device__ __forceinline__ long long fs_off(long long nf, int M, int NO, int q, long long face)
{
    return ((long long)NO * M * nf + q * nf + face) * 4;
}

__device__ __forceinline__ void flag_bad(const Mesh& g, long long idx)
{
    atomicOr(g.status, STATUS_NONPHYS);
    atomicMin((unsigned long long*)g.bad, (unsigned long long)idx);
}

// Step kernels are launched as programmatic dependents: a kernel's blocks may
// come up while the last blocks of the one before run, and wait here until it
// has completed and its writes are visible; then the next kernel may come up in
// its turn.  The launch latency between kernels, half of a small mesh's step, is
// hidden that way.
__device__ __forceinline__ void grid_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Asynchronous copies from global to shared memory: one value, 4 values
__device__ __forceinline__ void copy_async16(void* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
template <typename R>
__device__ __forceinline__ void copy_async1(R* dst, const R* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(sizeof(R))
                 : "memory");
}
__device__ __forceinline__ void copy_async4(float* dst, const float* src) { copy_async16(dst, src); }
__device__ __forceinline__ void copy_async4(double* dst, const double* src)
{
    copy_async16(dst, src);
    copy_async16(dst + 2, src + 2);
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// -------------------------------------------------------------- Steps 1-2 (2-D)
//
// One launch per direction over tiles of TA x TB cells (a along the face
// normal, b across it) of the range a in [-1, na], b in [-1, nb] whose faces
// the stage evaluates (ghost columns and rows included: Step 3 reads the face
// states of the rows beside the mesh).  A tile goes through shared memory in
// four parts:
//   stage  asynchronous copies of what the tile reads: averages (FP32 bulk: hi
//          and lo) and tangential slopes of the tile and two halo layers each
//          way, line slopes of the tile and its halo along a, and the face sigma;
//          ghost values are resolved here, once each;
//   0      per cell: the DFFs of the tangential and the normal stencil;
//   1      Step 1 per cell, a variable at a time: the tangential reconstruction at the M
//          Gauss lines -> line averages; for the cells whose faces this tile
//          evaluates also AT and TD (Step 3);
//   2      Step 2 (Algorithm 1) per (cell, variable), all M lines: both face
//          states with their derivatives.
// A lane per (cell, variable) needs a quarter of the registers of a lane per
// cell and line, so that more warps hide each other's latencies, and the M lines
// share the cell's differences of averages; 8 cells x 4 variables a warp write
// whole 128-byte groups of FR.  The tile shape is fixed at compile time (index
// arithmetic was a third of the instructions): along x 32 cells with the halo
// (28 + 4 in direction 0, 12 + 4 by 16 in direction 1), and a block's cells fill
// its threads.  FP64 tiles are half as large: the HWENO-AO cells of a front hold
// up their tile, and 100^2 cells leave few (28 x 4 -> 28 x 2: 169 -> 129 us there,
// 551 -> 557 us at 512^2).
//
// Before, a lane took a cell (Step 1) or a cell and line (Step 2) and loaded its
// 60 or 20 stencil values from global memory, resolving ghosts at each; 128
// registers, 16 warps per SM, waiting on those loads and on barriers.  FP32,
// 1024^2, order 9, per launch: 288 -> 163 us (x), 317 -> 175 us (y), now bound by
// issue slots and latency together (87 M warp instructions; the DRAM traffic
// alone would take 80 us); FP64 512^2: 730 -> 558 us, near the FP64 pipe's
// bound; 47 x 33, order 5: 38 -> 12 us, where the ghosts' serial loads had been
// the time.
template <typename R, int DIR>
struct ReconTile {
    static constexpr int TA = DIR == 0 ? 28 : 12, TB = DIR == 0 ? (sizeof(R) == 4 ? 4 : 2) : (sizeof(R) == 4 ? 16 : 8);
    static constexpr int threads = (TA + 4) * TB;
};

template <int M, typename R, int DIR>
struct ReconShared {
    using T = ReconTile<R, DIR>;
    static constexpr bool BULK32 = sizeof(R) == 4;
    static constexpr int TA = T::TA, TB = T::TB, TAH = TA + 4;
    static constexpr int NA = BULK32 ? 12 : 8;  // planes of A: W (hi), W_t, lo
    // plane strides = 8 mod 32, so that lanes of 8 cells x 4 variables touch every bank once
    static constexpr int pad(int n) { return ((n + 23) & ~31) + 8; }
    static constexpr int nc = TAH * TB;                                   // cells with their halo along a
    static constexpr int nA = TAH * (TB + 4);                             // and along b
    static constexpr int sA = pad(nA), sB = pad(nc);                      // plane strides
    static constexpr int nst = TAH * (TB + 5), nsn = (TA + 5) * TB;       // faces across b, along a
    // offsets in bytes
    static constexpr int st = 0, sn = st + nst * 8, A = sn + nsn * 8;     // sigma; averages and slopes
    static constexpr int B = A + NA * sA * (int)sizeof(R);                // line slopes [M * 4][sB]
    static constexpr int la = B + 4 * M * sB * (int)sizeof(R);            // line averages [M * 4][sB]
    static constexpr int at = la + 4 * M * sB * (int)sizeof(R);           // DFFs of S0, S1, r5 [3][nc]: tangential
    static constexpr int an = at + 3 * nc * (int)sizeof(R);               // and normal
    static constexpr int ct = an + 3 * nc * (int)sizeof(R);               // stencil codes: tangential
    static constexpr int cn = ct + nc * 4;                                // and normal
    static constexpr int bytes = cn + nc * 4;
};

// A ghost cell's value into shared memory
template <int M, typename R, bool WALLS>
__device__ __forceinline__ void ghost_into(R* d, const Mesh& g, const R* S, const CellMap& c, int kind, int v, int l)
{
    if (WALLS && (c.state || c.wx || c.wy)) *d = mapped<2, M, R, WALLS>(g, S, c, kind, v, l);
    else if ((c.zx && (kind == 1 || kind == 3)) || (c.zy && (kind == 2 || kind == 4))) *d = (R)0;
    else copy_async1(d, S + value_plane<2, M>(kind, v, l) * g.plane + c.idx);
}

// body(StTag<0>()) .. body(StTag<N - 1>())
template <int N, int K = 0, typename Body>
__device__ __forceinline__ void for_rows(Body&& body)
{
    if constexpr (K < N) {
        body(StTag<K>());
        for_rows<N, K + 1>(body);
    }
}

// (quotient, remainder) by a compile-time extent
template <int N>
__device__ __forceinline__ void split(int t, int& q, int& r) { q = t / N; r = t - q * N; }

template <int M, typename R, bool WALLS, int DIR, bool ONE>
__global__ void __launch_bounds__(ReconTile<R, DIR>::threads, sizeof(R) == 4 ? 768 / ReconTile<R, DIR>::threads : 1)
k_recon(const __grid_constant__ Work w, int stage)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned long long cnt[4];
    using L = ReconShared<M, R, DIR>;
    constexpr bool BULK32 = sizeof(R) == 4;
    constexpr int TA = L::TA, TB = L::TB, TAH = L::TAH, nc = L::nc, sA = L::sA, sB = L::sB;
    constexpr int NT = ReconTile<R, DIR>::threads;
    grid_wait();
    if (threadIdx.x < 4) cnt[threadIdx.x] = 0;
    double* s_st = (double*)(smem_raw + L::st);
    double* s_sn = (double*)(smem_raw + L::sn);
    R* s_A = (R*)(smem_raw + L::A);
    R* s_B = (R*)(smem_raw + L::B);
    R* s_la = (R*)(smem_raw + L::la);
    R* s_at = (R*)(smem_raw + L::at);
    R* s_an = (R*)(smem_raw + L::an);
    int* s_ct = (int*)(smem_raw + L::ct);
    int* s_cn = (int*)(smem_raw + L::cn);
    // shared-memory strides of a and b: the global x index is fastest
    constexpr int aA = DIR == 0 ? 1 : TB + 4, bA = DIR == 0 ? TAH : 1;  // of A
    constexpr int aB = DIR == 0 ? 1 : TB, bB = DIR == 0 ? TAH : 1;      // of B, la and the cell arrays
    constexpr int aT = DIR == 0 ? 1 : TB + 5, bT = DIR == 0 ? TAH : 1;  // of the tangential sigma
    constexpr int aN = DIR == 0 ? 1 : TB, bN = DIR == 0 ? TA + 5 : 1;   // of the normal sigma
    // this thread's cell of the tile and its halo
    const int tc = threadIdx.x;
    int ia, ib;
    if (DIR == 0) split<TAH>(tc, ib, ia); else split<TB>(tc, ia, ib);
    {
        // one tile per block: the tiles along a shock take many times longer, and the
        // hardware deals blocks to SMs as they come free (dealt in fixed strides, a
        // 960 x 240 mesh put most of them on a few SMs: 2.29 instead of 0.9 ms)
        long long ltl;
        const Mesh& g = mesh_of<ONE>(w, blockIdx.x, ltl);
        int na, nb;
        local_dims<M>(g, DIR, na, nb);
        const int nta = (na + 2 + TA - 1) / TA;
        const int lt = (int)ltl;                    // 32-bit tile index (bounded on the host)
        const int a0 = -1 + (lt % nta) * TA, b0 = -1 + (lt / nta) * TB;
        const int a = a0 - 2 + ia, b = b0 + ib;
        const bool on = a <= na + 2 && b <= nb;                  // within the mesh's halo
        const bool core = on && ia >= 2 && ia < TA + 2 && a <= na;  // evaluates its faces
        const R* S = state_planes<R>(g, stage == 1 ? 0 : 1);
        const double tb = WALLS ? stage_time(g, stage) : 0.0;  // inflow ghost states
        const long long P = g.plane;
        // ---- stage
        for (int t = threadIdx.x; t < L::nA; t += NT) {
            int ia, ib;
            if (DIR == 0) split<TAH>(t, ib, ia); else split<TB + 4>(t, ia, ib);
            const int a = a0 - 2 + ia, b = b0 - 2 + ib;
            if (a > na + 2 || b > nb + 2) continue;
            const int i = DIR == 0 ? a : b, j = DIR == 0 ? b : a;
            R* d = s_A + t;
            if ((unsigned)i < (unsigned)g.nx && (unsigned)j < (unsigned)g.ny) {
                const R* p = S + (long long)j * g.nx + i;
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    copy_async1(d + v * sA, p + vglob(DIR, v) * P);
                    copy_async1(d + (4 + v) * sA, p + ((DIR == 0 ? 8 : 4) + vglob(DIR, v)) * P);
                    if (BULK32) copy_async1(d + (8 + v) * sA, p + (12 + 8 * M + vglob(DIR, v)) * P);
                }
            } else {
                const CellMap c = cell_map<WALLS>(g, i, j, tb);
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    ghost_into<M, R, WALLS>(d + v * sA, g, S, c, 0, vglob(DIR, v), 0);
                    ghost_into<M, R, WALLS>(d + (4 + v) * sA, g, S, c, DIR == 0 ? 2 : 1, vglob(DIR, v), 0);
                    if (BULK32) ghost_into<M, R, WALLS>(d + (8 + v) * sA, g, S, c, 5, vglob(DIR, v), 0);
                }
            }
        }
        if (on) {
            const int i = DIR == 0 ? a : b, j = DIR == 0 ? b : a;
            R* d = s_B + tc;
            if ((unsigned)i < (unsigned)g.nx && (unsigned)j < (unsigned)g.ny) {
                const R* p = S + (DIR == 0 ? 12 : 12 + 4 * M) * P + (long long)j * g.nx + i;
#pragma unroll
                for (int l = 0; l < M; ++l)
#pragma unroll
                    for (int v = 0; v < 4; ++v) copy_async1(d + (4 * l + v) * sB, p + (4 * l + vglob(DIR, v)) * P);
            } else {
                const CellMap c = cell_map<WALLS>(g, i, j, tb);
#pragma unroll
                for (int l = 0; l < M; ++l)
#pragma unroll
                    for (int v = 0; v < 4; ++v)
                        ghost_into<M, R, WALLS>(d + (4 * l + v) * sB, g, S, c, DIR == 0 ? 3 : 4, vglob(DIR, v), l);
            }
        }
        {
            // sigma of the DFF (Sec. 3.1): of step n-1 in both stages, or, in stage 2
            // of the stage-lag reading, the face means of stage 1 of this step
            const bool lag_stage = stage == 2 && g.dff_lag;
            const double* SX = lag_stage ? g.sig_xn : g.sig_x;
            const double* SY = lag_stage ? g.sig_yn : g.sig_y;
            for (int t = threadIdx.x; t < L::nst; t += NT) {
                int ia, q;
                if (DIR == 0) split<TAH>(t, q, ia); else split<TB + 5>(t, ia, q);
                const int a = a0 - 2 + ia, f = b0 - 2 + q;  // tangential face f of column a
                if (a > na + 2 || f > nb + 3) continue;
                s_st[t] = lsigT<WALLS>(g, SX, SY, DIR, a, f);
            }
            for (int t = threadIdx.x; t < L::nsn; t += NT) {
                int q, ib;
                if (DIR == 0) split<TA + 5>(t, ib, q); else split<TB>(t, q, ib);
                const int f = a0 - 2 + q, b = b0 + ib;      // normal face f of row b
                if (f > na + 3 || b > nb) continue;
                s_sn[t] = lsigN<2, WALLS>(g, SX, SY, DIR, f, b);
            }
        }
        copy_commit();
        copy_wait<0>();
        __syncthreads();
        // ---- 0: DFFs
        if (on) {
            double s6[6];
#pragma unroll
            for (int q = 0; q < 6; ++q) s6[q] = s_st[ia * aT + (ib + q) * bT];
            const Dff dt = dff_select(g.order, s6, g.thr);
            s_ct[tc] = dt.st;
            if (dt.st < 0) {
                s_at[tc] = (R)dt.a[0]; s_at[nc + tc] = (R)dt.a[1]; s_at[2 * nc + tc] = (R)dt.a[3];
            }
            if (core) {
                // tangential r5 DFF of this cell, reused by Step 3
                ((R*)g.AT[DIR])[cell_idx(DIR, na, nb, a, b)] = (R)dt.a[3];
#pragma unroll
                for (int q = 0; q < 6; ++q) s6[q] = s_sn[(ia - 2 + q) * aN + ib * bN];
                const Dff dn = dff_select(g.order, s6, g.thr);
                s_cn[tc] = dn.st;
                if (dn.st < 0) {
                    s_an[tc] = (R)dn.a[0]; s_an[nc + tc] = (R)dn.a[1]; s_an[2 * nc + tc] = (R)dn.a[3];
                }
                // branch counts of the M lines, aggregated per warp
                const int bi = dn.st < 0 ? 0 : dn.st - ST_R5 + 1;
                const unsigned same = __match_any_sync(__activemask(), bi);
                if ((int)(threadIdx.x & 31) == __ffs(same) - 1)
                    atomicAdd(&cnt[bi], (unsigned long long)(M * __popc(same)));
            }
        }
        __syncthreads();
        const R* gw = MeshR<R>::ao(g);
        const R eps = (R)g.eps;
        // ---- 1: Step 1; a lane per cell, its variables in turn
        if (on) {
            const R ht = (R)(DIR == 0 ? g.dy : g.dx);
            const R* A = s_A + ia * aA + (ib + 2) * bA;
            with_stencil<M>(s_ct[tc], [&](auto tag) {
                constexpr int ST = decltype(tag)::value;
                if constexpr (ST >= 0 && BULK32) {
                    // differences of averages as (hi - hi) + (lo - lo), and the line
                    // average kept as lo + increment (over the cell's hi); two
                    // variables at once
#pragma unroll
                    for (int v = 0; v < 4; v += 2) {
                        const float* A0 = (const float*)A + v * sA;
                        auto at2 = [&](int k) { return make_float2(A0[k], A0[k + sA]); };
                        const float2 h0 = at2(0), l0 = at2(8 * sA);
                        float2 dp[10];
#pragma unroll
                        for (int q = 0; q < 5; ++q) {
                            if (st_tap(ST, q)) {
                                dp[q] = add2(sub2(at2((q - 2) * bA), h0), sub2(at2(8 * sA + (q - 2) * bA), l0));
                            }
                            if (st_tap(ST, 5 + q)) dp[5 + q] = mul2(ht, at2(4 * sA + (q - 2) * bA));
                        }
                        for_rows<M>([&](auto row) {
                            constexpr int l = decltype(row)::value;
                            const float2 r = add2(l0, row_taps<M - 2, ST, 6 + l>(dp));
                            s_la[(4 * l + v) * sB + tc] = r.x;
                            s_la[(4 * l + v + 1) * sB + tc] = r.y;
                        });
                    }
                } else {
#pragma unroll(ST >= 0 ? 4 : 1)
                    for (int v = 0; v < 4; ++v) {
                        const R* Av = A + v * sA;
                        R dp[10], out[M];
#pragma unroll
                        for (int q = 0; q < 5; ++q) {
                            dp[q] = Av[(q - 2) * bA] - Av[0];
                            if (BULK32) dp[q] += Av[8 * sA + (q - 2) * bA] - Av[8 * sA];
                            dp[5 + q] = ht * Av[4 * sA + (q - 2) * bA];
                        }
                        if constexpr (ST >= 0) {
                            const auto& T = c_tab[M - 2];
                            double e[2], o[2], E[2], O[2];
                            sym_data<double>((const double*)dp, e, o, E, O);
#pragma unroll
                            for (int l = 0; l < (M + 1) / 2; ++l) {
                                double p, q;
                                sym_row<ST, double>(T.sym[ST - ST_R5][3 + l], e, o, E, O, p, q);
                                out[l] = (R)(M - 1 - l == l ? p : p + q);
                                if (M - 1 - l != l) out[M - 1 - l] = (R)(p - q);
                            }
                        } else {
                            const R al[4] = {s_at[tc], s_at[nc + tc], s_at[2 * nc + tc], s_at[2 * nc + tc]};
                            recon_ao<R, M>(al, M - 2, 6, dp, out, gw, eps);
                        }
                        const R base = BULK32 ? Av[8 * sA] : Av[0];
#pragma unroll
                        for (int l = 0; l < M; ++l) s_la[(4 * l + v) * sB + tc] = base + out[l];
                    }
                }
            });
            if (BULK32 && core) {
                // hi and its tangential differences: the bases of the face states
                // and of Step 3's segments
                R hi[4], tdm[4], tdp[4];
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    hi[v] = A[v * sA];
                    tdm[v] = A[v * sA - bA] - hi[v];
                    tdp[v] = A[v * sA + bA] - hi[v];
                }
                R* td = (R*)g.TD[DIR] + cell_idx(DIR, na, nb, a, b) * 12;
                st4(td, hi);
                st4(td + 4, tdm);
                st4(td + 8, tdp);
            }
        }
        __syncthreads();
        // ---- 2: Step 2; variable fastest
        {
            const R hn = (R)(DIR == 0 ? g.dx : g.dy);
            const R ih = (R)1 / hn, ih2 = ih * ih;
            const long long nrow = fr_nrow(DIR, na, nb) * 4;  // values of a line's plane
            for (int it = threadIdx.x; it < 4 * TA * TB; it += NT) {
                const int v = it & 3, c = it >> 2;
                int ia, ib;
                if (DIR == 0) split<TA>(c, ib, ia); else split<TB>(c, ia, ib);
                ia += 2;
                const int a = a0 - 2 + ia, b = b0 + ib;
                if (a > na || b > nb) continue;
                const int t = ia * aB + ib * bB;
                // side 0: left state of face a+1 (value at xi = +1/2), side 1: right
                // state of face a (xi = -1/2)
                R* FR = (R*)g.FR[DIR];
                R* fl = FR + fr_row(DIR, na, nb, b + 1, a + 1) * 4 + v;
                R* fr = FR + 3 * M * nrow + fr_row(DIR, na, nb, b + 1, a >= 0 ? a : 0) * 4 + v;
                const bool left = a + 1 <= na, right = a >= 0;
                // value r (0..2 left state and its derivatives, 3..5 right) of line l
                auto put = [&](int r, int l, R x) {
                    if (r < 3) { if (left) fl[(r * M + l) * nrow] = x; }
                    else { if (right) fr[((r - 3) * M + l) * nrow] = x; }
                };
                const R* A = s_A + v * sA + ia * aA + (ib + 2) * bA;
                const R* la = s_la + v * sB + t;
                const R* sl = s_B + v * sB + t;
                // FP32 bulk: line averages are increments over the cells' hi, so a
                // difference of them is (hi - hi) + (la - la), and the face values
                // come out as increments over this cell's hi; the left state of face
                // a+1 over the hi of that face's right cell a+1, like the right
                // state: a face's two states share a base
                R h5[5];
#pragma unroll
                for (int q = 0; q < 5; ++q) h5[q] = BULK32 ? A[(q - 2) * aA] - A[0] : (R)0;
                with_stencil<M>(s_cn[t], [&](auto tag) {
                    constexpr int ST = decltype(tag)::value;
                    if constexpr (ST >= 0 && BULK32) {
                        // two lines at once (the last of an odd number twice)
                        constexpr int NP = (M + 1) / 2;
                        float2 dp[NP][10], qi[NP];
#pragma unroll
                        for (int p = 0; p < NP; ++p) {
                            constexpr int step = 4 * sB;
                            const int l0 = 2 * p, l1 = 2 * p + 1 < M ? 2 * p + 1 : 2 * p;
                            auto two = [&](const R* x, int k) { return make_float2(x[l0 * step + k], x[l1 * step + k]); };
                            qi[p] = two(la, 0);
#pragma unroll
                            for (int q = 0; q < 5; ++q) {
                                if (st_tap(ST, q))
                                    dp[p][q] = add2(make_float2(h5[q], h5[q]), sub2(two(la, (q - 2) * aB), qi[p]));
                                if (st_tap(ST, 5 + q)) dp[p][5 + q] = mul2(hn, two(sl, (q - 2) * aB));
                            }
                        }
                        for_rows<6>([&](auto row) {
                            constexpr int r = decltype(row)::value;
#pragma unroll
                            for (int p = 0; p < NP; ++p) {
                                float2 x = row_taps<M - 2, ST, r>(dp[p]);
                                if (r == 0) x = add2(sub2(qi[p], make_float2(h5[3], h5[3])), x);
                                else if (r == 3) x = add2(qi[p], x);
                                else x = mul2(r % 3 == 1 ? ih : ih2, x);
                                put(r, 2 * p, x.x);
                                if (2 * p + 1 < M) put(r, 2 * p + 1, x.y);
                            }
                        });
                    } else {
#pragma unroll(ST >= 0 ? 2 : 1)
                        for (int l = 0; l < M; ++l) {
                            R qi = la[4 * l * sB], dp[10], out[6];
#pragma unroll
                            for (int q = 0; q < 5; ++q) {
                                dp[q] = h5[q] + (la[4 * l * sB + (q - 2) * aB] - qi);
                                dp[5 + q] = hn * sl[4 * l * sB + (q - 2) * aB];
                            }
                            if constexpr (ST >= 0) {
                                faces_sym<ST>(c_tab[M - 2], dp, out);
                            } else {
                                const R al[4] = {s_an[t], s_an[nc + t], s_an[2 * nc + t], s_an[2 * nc + t]};
                                recon_ao<R, 6>(al, M - 2, 0, dp, out, gw, eps);
                            }
                            put(0, l, (qi - h5[3]) + out[0]);
                            put(1, l, out[1] * ih);
                            put(2, l, out[2] * ih2);
                            put(3, l, qi + out[3]);
                            put(4, l, out[4] * ih);
                            put(5, l, out[5] * ih2);
                        }
                    }
                });
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < 4 && cnt[threadIdx.x] && w.n > 0)
        atomicAdd(&(ONE ? w.m0 : w.mesh[0]).branch[threadIdx.x], cnt[threadIdx.x]);
}

// -------------------------------------------------------------- Step 2 (1-D)
// The reconstruction of a 1-D cell a in [-1, nx] from the cell averages and
// slopes of a-2..a+2: the right state of face a and the left state of face a+1.
// A mesh of 1-D size is bound by latency: the five cells are mapped once and
// their values loaded together, and each stencil sums only its own taps (80
// cells FP64 21.5 -> 11.4 us, 400 cells FP32 24.6 -> 13.2, between two events).
template <typename R, bool WALLS, bool ONE>
__global__ void __launch_bounds__(256) k_normal1(const __grid_constant__ Work w, int stage)
{
    __shared__ unsigned long long cnt[4];
    grid_wait();
    if (threadIdx.x < 4) cnt[threadIdx.x] = 0;
    __syncthreads();
    constexpr int NV = 3;
    constexpr bool BULK32 = sizeof(R) == 4;
    for (long long gi = blockIdx.x * (long long)blockDim.x + threadIdx.x; gi < w.total;
         gi += (long long)gridDim.x * blockDim.x) {
        long long li;
        const Mesh& g = mesh_of<ONE>(w, gi, li);
        const int a = (int)li - 1;
        const int na = g.nx;
        const long long P = g.plane;
        const R* S = state_planes<R>(g, stage == 1 ? 0 : 1);
        // sigma of the DFF: step n-1, or in stage 2 of the stage-lag reading the
        // face means of stage 1 of this step
        const double* SX = (stage == 2 && g.dff_lag) ? g.sig_xn : g.sig_x;
        R h[NV][5], lo[NV][5], sl[NV][5];  // averages (FP32 bulk: hi), low parts, slopes
        double s6[6];
        if (a >= 2 && a + 3 <= na) {
#pragma unroll
            for (int q = 0; q < 6; ++q) s6[q] = SX[a - 2 + q];
        } else {
#pragma unroll
            for (int q = 0; q < 6; ++q) s6[q] = sigx<1, WALLS>(g, SX, a - 2 + q, 0);
        }
        if (a >= 2 && a + 2 < na) {
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    h[v][q] = S[v * P + a - 2 + q];
                    sl[v][q] = S[(3 + v) * P + a - 2 + q];
                    if (BULK32) lo[v][q] = S[(6 + v) * P + a - 2 + q];
                }
        } else {
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                const int i = a - 2 + q;
                if ((i < 0 || i >= na) && g.bc[i < 0 ? 0 : 1] == BC_FIXED) {
                    const double* gh = g.ghost + ((i < 0 ? 0 : 1) * 3 + (i < 0 ? -1 - i : i - na)) * 6;
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        h[v][q] = (R)gh[v];
                        sl[v][q] = (R)gh[3 + v];
                        if (BULK32) lo[v][q] = low_part<R>(gh[v]);
                    }
                } else {
                    const CellMap m = cell_map<WALLS>(g, i, 0, 0.0, false);
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        h[v][q] = mapped<1, 1, R, WALLS>(g, S, m, 0, v, 0);
                        sl[v][q] = mapped<1, 1, R, WALLS>(g, S, m, 1, v, 0);
                        if (BULK32) lo[v][q] = mapped<1, 1, R, WALLS>(g, S, m, 5, v, 0);
                    }
                }
            }
        }
        const Dff dff = dff_select(g.order, s6, g.thr);
        {
            // branch counts, aggregated per warp
            int bi = dff.st < 0 ? 0 : dff.st - ST_R5 + 1;
            unsigned act = __activemask();
            unsigned same = __match_any_sync(act, bi);
            if ((int)(threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(&cnt[bi], (unsigned long long)__popc(same));
        }
        const R hn = (R)g.dx;
        const R ih = (R)1 / hn;
        R sideL[3][4], sideR[3][4];
        with_stencil<4>(dff.st, [&](auto tag) {
            constexpr int ST = decltype(tag)::value;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                // FP32 bulk: differences as (hi - hi) + (lo - lo); the face values
                // come out as increments over this cell's hi
                R dp[10], out[6];
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    dp[q] = h[v][q] - h[v][2];
                    if (BULK32) dp[q] += lo[v][q] - lo[v][2];
                    dp[5 + q] = hn * sl[v][q];
                }
                // the rows at the faces are the same in every order's table
                if constexpr (ST < 0) {
                    const R al[4] = {(R)dff.a[0], (R)dff.a[1], (R)dff.a[2], (R)dff.a[3]};
                    recon_ao<R, 6>(al, 2, 0, dp, out, MeshR<R>::ao(g), (R)g.eps);
                } else if constexpr (BULK32) {
#pragma unroll
                    for (int r = 0; r < 6; ++r) {
                        R s = 0;
#pragma unroll
                        for (int k = 0; k < 10; ++k)
                            if (st_tap(ST, k)) s += Tab<R>::get(2).row[ST][r][k] * dp[k];
                        out[r] = s;
                    }
                } else {
                    faces_sym<ST>(c_tab[2], dp, out);
                }
                // the left state of face a+1 over hi of cell a+1 (a face's states share a base)
                const R qi = BULK32 ? lo[v][2] : h[v][2], shift = BULK32 ? h[v][2] - h[v][3] : (R)0;
                sideL[0][v] = (qi + shift) + out[0]; sideL[1][v] = out[1] * ih; sideL[2][v] = out[2] * ih * ih;
                sideR[0][v] = qi + out[3]; sideR[1][v] = out[4] * ih; sideR[2][v] = out[5] * ih * ih;
            }
        });
#pragma unroll
        for (int nd = 0; nd < 3; ++nd) { sideL[nd][3] = (R)0; sideR[nd][3] = (R)0; }
        R* FR = (R*)g.FR[0];
        const long long nrow = fr_nrow(0, na, 1);
        // side 0: left state of face a+1 (value at xi = +1/2)
        if (a + 1 <= na) {
            const long long row = fr_row(0, na, 1, 1, a + 1);
#pragma unroll
            for (int nd = 0; nd < 3; ++nd) st4(FR + fr_off(nrow, 1, 0, nd, 0, row), sideL[nd]);
        }
        // side 1: right state of face a (value at xi = -1/2)
        if (a >= 0) {
            const long long row = fr_row(0, na, 1, 1, a);
#pragma unroll
            for (int nd = 0; nd < 3; ++nd) st4(FR + fr_off(nrow, 1, 1, nd, 0, row), sideR[nd]);
        }
    }
    __syncthreads();
    if (threadIdx.x < 4 && cnt[threadIdx.x] && w.n > 0)
        atomicAdd(&(ONE ? w.m0 : w.mesh[0]).branch[threadIdx.x], cnt[threadIdx.x]);
}

// -------------------------------------------------------------- Step 3 + flux
//
// One thread per face Gauss point.  1-D: a grid-stride loop over the faces.
// 2-D: each warp marches along the tangential direction b of a strip of faces
// and keeps the face states that Step 3 reads of the segments b-1, b, b+1 in
// its own ring in shared memory, which asynchronous copies fill one step ahead.
// A step is 32 / M faces (dir 0: 32 / M columns f of row b; dir 1: 32 / M
// consecutive b of face row f) and has two parts: Step 3 with a lane per
// (side, face, variable), then the kinetic part with a lane per (face, line).
//
// Why: with every point summing its own 3 M segment points from global memory
// the FP32 kernel waited on those loads (762 us for stage 1 at 1024^2, order 9;
// 582 us when they hit in L1 always), and from shared memory it spent 400
// shared-memory passes a step on them (780 us): a 16-byte load takes four,
// whichever lanes read alike.  A lane per variable reads 4 bytes, one pass for
// a whole segment point of 8 faces, serves all M lines from it with weights from
// constant memory, and sums mirrored points once for mirrored lines.  With the
// ghost bases out of the way (TD) and the face sums (below), FP32 takes 416 + 363
// us for the two stages (start 889 + 770), bound by issue slots: 75% of them used
// by 16 warps per SM, about 920 FP32 instructions of 1450 a point.  FP64, bound by
// its pipe (87% busy), takes 3.28 + 2.99 ms at 512^2 (start 5.96 + 5.51).  The
// steps of a mesh are dealt to the warps in equal contiguous runs: a run has one
// prologue, the rest streams.
template <int M> struct FluxStrip {
    static constexpr int FW = 32 / M;    // faces per step
    static constexpr int RING = 3 * FW;  // ring positions: rows or blocks of rows j, j + 1, j + 2
};

// Values of one warp in shared memory: the ring of W and W_n of both sides; the
// tangential derivatives of the step; two slots of what only the step's own
// points read: W_nn, and the bases of the face (TD of its right cell, FP32
// bulk) with the tangential DFF of its two cells; the step's sigma.
template <int M, typename R>
struct FluxShared {
    static constexpr int FW = FluxStrip<M>::FW, RING = FluxStrip<M>::RING;
    static constexpr bool BULK32 = sizeof(R) == 4;
    static constexpr int ring = 0;                                    // [side][W, W_n][M][RING][4]
    static constexpr int tang = ring + 2 * 2 * M * RING * 4;          // [side][t, tt, nt][M][FW][4]
    static constexpr int nn = tang + 2 * 3 * M * FW * 4;              // [slot][side][M][FW][4]
    static constexpr int td = nn + 2 * 2 * M * FW * 4;                // [slot][FW][12]
    static constexpr int at = td + (BULK32 ? 2 * FW * 12 : 0);        // [slot][side][FW]
    static constexpr int total = at + (2 * 2 * FW + 3) / 4 * 4;
};

// Steps (strips of 32 / M faces) of an nx x ny mesh
__host__ __device__ inline long long flux_steps(int M, int nx, int ny)
{
    const int fw = 32 / M;
    return (long long)((nx + 1 + fw - 1) / fw) * ny + (long long)(ny + 1) * ((nx + fw - 1) / fw);
}

// Step 3 for one (side, face, variable): the derivatives t, tt and nt at the M
// lines of the face, from the 3 M points of segments b-1, b, b+1 (W: value of
// the variable at ring position p of line k is W[(k * RING + p) * 4], Wn the
// normal derivative likewise; q: ring positions of the segments).  Lines l and
// M-1-l mirror each other: first derivatives of the even part of the points and
// second ones of the odd part change sign.  dm, dp (FP32 bulk): the segment
// points' values are increments over hi of the right cells (f, b-1), (f, b),
// (f, b+1); the bases' part comes from their differences (the weights of a
// constant sum to zero).  out[(q * M + l) * FW * 4]: quantity q at line l.
template <int M, typename R>
__device__ __forceinline__ void step3(const R* W, const R* Wn, const int q[3], R dm, R dp, R c1, R c2, R* out)
{
    constexpr int K = 3 * M, H = K / 2, RING = FluxStrip<M>::RING, FW = FluxStrip<M>::FW;
    constexpr bool BULK32 = sizeof(R) == 4;
    const auto& T = Tab<R>::get(M - 2);
    constexpr int NE = (K + 1) / 2;
    // quantity q at line l and its mirror: scale (odd + even), +-scale (odd - even)
    auto put = [&](int q, int l, R scale, R plus, R minus) {
        const R m = scale * minus;  // the part that changes sign
        out[(q * M + l) * FW * 4] = scale * plus + m;
        if (M - 1 - l != l) out[(q * M + M - 1 - l) * FW * 4] = scale * plus - m;
    };
    if constexpr (BULK32) {
        // W and W_n share the first-derivative weights: both at once, with two-wide FMAs
        float2 e[H + 1], o[H];
#pragma unroll
        for (int k = 0; k <= (K % 2 ? H : H - 1); ++k) {
            auto at2 = [&](int j) {
                const int x = ((j % M) * RING + q[j / M]) * 4;
                return make_float2(W[x], Wn[x]);
            };
            const float2 x = at2(k);
            if (k == H) {
                e[k] = x;
            } else {
                const float2 y = at2(K - 1 - k);
                e[k] = add2(x, y);
                o[k] = sub2(x, y);
            }
        }
        const float sb = dm + dp, db = dm - dp;
#pragma unroll
        for (int l = 0; l < (M + 1) / 2; ++l) {
            float2 te = __fmul2_rn(T.sd1w[l][0][0], e[0]), to = __fmul2_rn(T.sd1w[l][1][0], o[0]);
            float se = T.sd2[l][0][0] * e[0].x, so = T.sd2[l][1][0] * o[0].x;
#pragma unroll
            for (int k = 1; k < NE; ++k) {
                te = __ffma2_rn(T.sd1w[l][0][k], e[k], te);
                se += T.sd2[l][0][k] * e[k].x;
                if (k < H) {
                    to = __ffma2_rn(T.sd1w[l][1][k], o[k], to);
                    so += T.sd2[l][1][k] * o[k].x;
                }
            }
            put(0, l, c1, to.x + T.sd1[l][1][6] * db, te.x + T.sd1[l][0][6] * sb);
            put(1, l, c2, se + T.sd2[l][0][6] * sb, so + T.sd2[l][1][6] * db);
            put(2, l, c1, to.y, te.y);
        }
    } else {
        R e[H + 1], o[H];
        auto split = [&](const R* P) {
            R x[K];
#pragma unroll
            for (int s = 0; s < 3; ++s)
#pragma unroll
                for (int k = 0; k < M; ++k) x[s * M + k] = P[(k * RING + q[s]) * 4];
#pragma unroll
            for (int k = 0; k < H; ++k) { e[k] = x[k] + x[K - 1 - k]; o[k] = x[k] - x[K - 1 - k]; }
            e[H] = K % 2 ? x[H] : (R)0;
        };
        auto sum = [&](const R* w, const R* v, int n) {
            R r = w[0] * v[0];
#pragma unroll
            for (int k = 1; k < n; ++k) r += w[k] * v[k];
            return r;
        };
        split(W);
#pragma unroll
        for (int l = 0; l < (M + 1) / 2; ++l) {
            put(0, l, c1, sum(T.sd1[l][1], o, H), sum(T.sd1[l][0], e, NE));
            put(1, l, c2, sum(T.sd2[l][0], e, NE), sum(T.sd2[l][1], o, H));
        }
        split(Wn);
#pragma unroll
        for (int l = 0; l < (M + 1) / 2; ++l) put(2, l, c1, sum(T.sd1[l][1], o, H), sum(T.sd1[l][0], e, NE));
    }
}

// What a face point reads, from a warp's shared memory (2-D).
template <int M, typename R>
struct StripPoint {
    using L = FluxShared<M, R>;
    const R* s;       // the warp's values
    R* FO;
    long long nf;     // faces of the direction
    int slot, own_q;  // slot of the step, ring position of the point's own segment
    int x, l;
    __device__ __forceinline__ void own(int side, int nd, R* v) const
    {
        if (nd < 2) ld4(s + L::ring + (((side * 2 + nd) * M + l) * L::RING + own_q) * 4, v);
        else ld4(s + L::nn + (((slot * 2 + side) * M + l) * L::FW + x) * 4, v);
    }
    __device__ __forceinline__ void base(R* v) const { ld4(s + L::td + (slot * L::FW + x) * 12, v); }
    __device__ __forceinline__ void tangential(int side, int q, R* v) const
    {
        ld4(s + L::tang + (((side * 3 + q) * M + l) * L::FW + x) * 4, v);
    }
    // interface states to global memory; fluxes and sigma are left to the face's sums
    template <int STAGE>
    __device__ __forceinline__ void put(const R o[4][4], long long face, R) const
    {
#pragma unroll
        for (int q = 0; q < (STAGE == 1 ? 2 : 1); ++q) st4(FO + fo_off(nf, M, q, l, face), o[2 + q]);
    }
};

// A face's Gauss sums of its points' fluxes and the mean of their sigma, over
// the M lanes of the face (all lanes of the warp take part).  Each lane ends up
// with a share of the sums and writes it: the update reads one value per face
// where it read M: 1024^2, order 9, FP32, the updates took 307 + 160 us, now 189 +
// 150 (with 24 warps per SM), the fluxes 395 + 354, now 418 +
// 364; at 2048^2, order 5, 905 + 413 -> 518 + 399 and 770 + 703 -> 821 + 721.
__device__ __forceinline__ float swap_lane(float v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }
__device__ __forceinline__ double swap_lane(double v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }

template <int M, int NO, typename R>
__device__ __forceinline__ void face_sums(R (&o)[4][4], R* FS, long long nf, long long face, int l, bool on)
{
    const auto& T = Tab<R>::get(M - 2);
    R w = T.gw[0];  // the lane's weight, mirrored lines alike
    if (M == 3 ? l == 1 : (M == 4 && (l == 1 || l == 2))) w = T.gw[1];
#pragma unroll
    for (int q = 0; q < NO; ++q)
#pragma unroll
        for (int v = 0; v < 4; ++v) o[q][v] *= w;
    if (M == 3) {
        const int base = (threadIdx.x & 31) - l;
#pragma unroll
        for (int q = 0; q < NO; ++q) {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                R s = __shfl_sync(0xffffffffu, o[q][v], base);
                s += __shfl_sync(0xffffffffu, o[q][v], base + 1);
                s += __shfl_sync(0xffffffffu, o[q][v], base + 2);
                o[q][v] = s;
            }
            if (on && l == q) st4(FS + (q * nf + face) * 4, o[q]);
        }
    } else if (NO == 2) {
        // lines l and l ^ M/2 split the two quantities ...
        const bool up = (l & (M / 2)) != 0;
        R s[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const R give = up ? o[0][v] : o[NO - 1][v], keep = up ? o[NO - 1][v] : o[0][v];
            s[v] = keep + swap_lane(give, M / 2);
        }
        R* p = FS + ((up ? nf : 0) + face) * 4;
        if (M == 2) {
            if (on) st4(p, s);
        } else {
            // ... and l and l ^ 1 the variables
            const bool odd = l & 1;
            R r[2];
#pragma unroll
            for (int v = 0; v < 2; ++v) r[v] = (odd ? s[2 + v] : s[v]) + swap_lane(odd ? s[v] : s[2 + v], 1);
            if (on) st2(p + (odd ? 2 : 0), r);
        }
    } else {
        const bool up = (l & (M / 2)) != 0;
        R s[2];
#pragma unroll
        for (int v = 0; v < 2; ++v) s[v] = (up ? o[0][2 + v] : o[0][v]) + swap_lane(up ? o[0][v] : o[0][2 + v], M / 2);
        R* p = FS + face * 4 + (up ? 2 : 0);
        if (M == 2) {
            if (on) st2(p, s);
        } else {
            const bool odd = l & 1;
            const R r = (odd ? s[1] : s[0]) + swap_lane(odd ? s[0] : s[1], 1);
            if (on) p[odd ? 1 : 0] = r;
        }
    }
}

template <int M, typename R>
__device__ __forceinline__ void face_sigma(R sig, double* out, int l, bool on)
{
    double s = (double)sig;
    if (M == 3) {
        const int base = (threadIdx.x & 31) - l;
        s = __shfl_sync(0xffffffffu, s, base) + __shfl_sync(0xffffffffu, s, base + 1) + __shfl_sync(0xffffffffu, s, base + 2);
    } else {
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        if (M == 4) s += __shfl_xor_sync(0xffffffffu, s, 2);
    }
    if (on && l == 0) *out = s / M;
}

// What a 1-D face reads, from global memory.
template <typename R>
struct LinePoint {
    const R* FR;
    long long nrow, row;
    R h[4];
    __device__ __forceinline__ void own(int side, int nd, R* v) const { ld4(FR + fr_off(nrow, 1, side, nd, 0, row), v); }
    __device__ __forceinline__ void base(R* v) const { for (int q = 0; q < 4; ++q) v[q] = h[q]; }
    R* FO;
    double* sx;
    long long nf;
    template <int STAGE>
    __device__ __forceinline__ void put(const R o[4][4], long long face, R sig) const
    {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (STAGE == 1 || q % 2 == 0) st4(FO + (q * nf + face) * 4, o[q]);
        if (STAGE == 1) sx[face] = (double)sig;
    }
};

// One face Gauss point.  Each side's reconstructed data (Step 2 values, Step 3
// tangential derivatives) and the differentials of its half-range moments are
// folded into the kinetic weighting Q0, dQ0 (Eq. 2.7) and the half-range terms
// of Eq. 2.6 as soon as they are formed.  HG = 1 compiles the collision-time
// terms (tau > 0); the tau = 0 instance leaves them out and carries fewer live
// values.  PF = true compiles the first-order fallback at face points whose
// reconstructed state is not physical (a flagged option).  Dt: the step, dt26 =
// Dt^2 / 6.
template <int D, int M, typename R, int STAGE, int HG, bool PF, typename Point>
__device__ __forceinline__ void flux_point(const Mesh& g, int dir, int na, int nb, int f, int b, int l, const Point& in,
                                           R Dt, R dt26, R (&o)[4][4], R& sig)
{
    constexpr int NV = D + 2;
    constexpr int ND = D == 2 ? 5 : 2;  // derivatives: n, nn (, t, tt, nt)
    constexpr bool BULK32 = sizeof(R) == 4;
    // FP32 bulk: the two sides unrolled, so that their independent chains interleave
    constexpr int kSides = BULK32 ? 2 : 1;
    constexpr bool hgks = HG != 0;  // the collision-time terms of Eq. 2.6 (tau > 0)
    const R gm = MeshR<R>::gamma(g), gm1 = gm - (R)1, Kx = MeshR<R>::K(g) + (R)(D - 1);
    {
        // FP32 bulk: hi of the face's right cell f (local frame), the base of
        // both face states
        const R* SF = state_planes<R>(g, STAGE == 1 ? 0 : 1);
        const double tb = PF ? stage_time(g, STAGE) : 0.0;
        R hb1[4] = {0, 0, 0, 0};
        if (BULK32) in.base(hb1);
        // FP32 bulk: whether the jump W_l - W_r is small enough for the kinetic
        // weighting to be taken to first order in it (decided with the left
        // state, below); the first-order term, held in Q0 itself unless the
        // point fallback may still change the states
        bool lin = false;
        R Dl[4] = {0, 0, 0, 0};
        R Q0[4] = {0, 0, 0, 0};
        R dQ[ND][4];
#pragma unroll
        for (int q = 0; q < ND; ++q)
#pragma unroll
            for (int v = 0; v < 4; ++v) dQ[q][v] = 0;
        R T5[4] = {0, 0, 0, 0}, T6[4] = {0, 0, 0, 0}, S1h[4] = {0, 0, 0, 0};
        R pz[2], mn[2], mt[2];
        bool ok = true;
#pragma unroll kSides
        for (int side = 0; side < 2; ++side) {
            // Step 2 data: W, W_n, W_nn (FP32 bulk: W as an increment over hb1);
            // Step 3's tangential derivatives are read when they are folded in
            R d0[4], dn[2][4];
            const int a = side == 0 ? f - 1 : f;  // the reconstructing cell
            in.own(side, 0, d0);
            in.own(side, 1, dn[0]);
            in.own(side, 2, dn[1]);
            // the side's state
            R ws[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) ws[v] = BULK32 ? hb1[v] + d0[v] : d0[v];
            bool fb = false;  // the side fell back to its cell average (all derivatives zero)
            if (PF) {
                // fallback: a side whose point state has rho <= 0 or p <= 0 takes
                // the average of the cell it was reconstructed from, first order;
                // the test is made in FP64 (FP32 bulk: on hi + increment)
                double W4[4];
#pragma unroll
                for (int v = 0; v < 4; ++v) W4[v] = BULK32 ? (double)hb1[v] + (double)d0[v] : (double)d0[v];
                double rho = W4[0];
                double m2 = W4[1] * W4[1] + (D == 2 ? W4[2] * W4[2] : 0.0);
                double p = (g.gamma - 1.0) * (W4[NV - 1] - 0.5 * m2 / rho);
                if (!(rho > 0.0) || !(p > 0.0)) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        // FP32 bulk: the average over hb1, (hi_a - hb1) + lo_a
                        if (BULK32)
                            d0[v] = (side == 0 ? lcell<D, M, R, true>(g, SF, dir, 0, v, 0, a, b, tb) - hb1[v] : (R)0)
                                  + lcell<D, M, R, true>(g, SF, dir, 5, v, 0, a, b, tb);
                        else
                            d0[v] = lcell<D, M, R, true>(g, SF, dir, 0, v, 0, a, b, tb);
                        ws[v] = BULK32 ? hb1[v] + d0[v] : d0[v];
                        dn[0][v] = dn[1][v] = (R)0;
                    }
                    fb = true;
                    lin = false;  // the states changed: weight them directly
                    atomicAdd(g.nfall, 1ull);
                }
            }
            // the side's state variables serve Eq. 3.2 (in the precision the
            // states carry: the face means, stencil sums and branch thresholds
            // that use sigma are FP64), the positivity test and the moments
            const Gas<R, D> Gs = gas_of<R, D>(ws, gm1);
            const R q = recip_sqrt(Gs.th);
            pz[side] = Gs.p; mn[side] = Gs.U * q; mt[side] = Gs.V * q;
            ok &= Gs.rho > (R)0 && Gs.p > (R)0;
            // kinetic weighting (Eq. 2.7): this side's half-range integrals
            const Range<R, hgks ? 5 : 3> Hs = half_range<R, D, hgks ? 5 : 3>(Gs, q, side == 0);
            if (BULK32 && side == 0) {
                // Q0 = W_r + (H(W_l) - H(W_r)), H the u > 0 half-range moments;
                // for a small jump, H(W_l) - H(W_r) = dH/dW (W_l - W_r) to second
                // order: the rounding then stays relative to the jump.  W_l - W_r
                // is the difference of the two increments (a face's states share
                // a base).
                R e1[4], dW[4];
                in.own(1, 0, e1);
                const R sc = fabs(hb1[0]) + fabs(hb1[NV - 1]);
                lin = true;
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    dW[v] = d0[v] - e1[v];
                    lin &= fabs(dW[v]) <= (R)2.5e-4 * sc;
                }
                if (lin) add_dhalf(Gs, Hs, Kx, dW, var_of<R, D>(Gs, gm1, dW), PF ? Dl : Q0);
            }
            R t[4];
            if (!(BULK32 && lin && !PF)) {
                half_moments(Gs, Hs, ws, t);
#pragma unroll
                for (int v = 0; v < NV; ++v) Q0[v] += t[v];
            }
            if (hgks) {
                half_flux(Gs, Hs, ws, Kx, t);
#pragma unroll
                for (int v = 0; v < NV; ++v) T5[v] += t[v];
            }
            // one derivative into the weighted derivative dQ[q], and for q = 0 (n)
            // and 2 (t) the half-range (a_n u + a_t v) terms of Eq. 2.6 without
            // and with the flux's u
            auto fold = [&](int q, const R* dv) {
                const Var<R> h = var_of<R, D>(Gs, gm1, dv);
                add_dhalf(Gs, Hs, Kx, dv, h, dQ[q]);
                if constexpr (hgks) {
                    if (q == 0) {
                        add_dmoments_u<1>(Gs, Hs, Kx, h, S1h);
                        add_dmoments_u<2>(Gs, Hs, Kx, h, T6);
                    }
                    if constexpr (D == 2) {
                        if (q == 2) {
                            add_dmoments_v<0>(Gs, Hs, Kx, h, S1h);
                            add_dmoments_v<1>(Gs, Hs, Kx, h, T6);
                        }
                    }
                }
            };
            fold(0, dn[0]);
            fold(1, dn[1]);
            if constexpr (D == 2) {
                // Step 3's tangential derivatives of this side, t, tt and nt
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    R dv[4];
                    in.tangential(side, q, dv);
                    if (PF && fb) {
#pragma unroll
                        for (int v = 0; v < 4; ++v) dv[v] = (R)0;
                    }
                    fold(2 + q, dv);
                }
            }
        }
        // FP32 bulk: the equilibrium state as an increment qv over hb1
        R qv[4] = {0, 0, 0, 0};
        if (BULK32) {
            if (lin) {
                R e1[4];
                in.own(1, 0, e1);
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    qv[v] = e1[v] + (PF ? Dl[v] : Q0[v]);
                    Q0[v] = hb1[v] + qv[v];
                }
            } else {
#pragma unroll
                for (int v = 0; v < NV; ++v) qv[v] = Q0[v] - hb1[v];
            }
        }
        {
            R dpz = fabs(pz[0] - pz[1]);
            sig = (dpz * recip(pz[0]) + dpz * recip(pz[1])
                           + MeshR<R>::igamma(g) * ((mn[0] - mn[1]) * (mn[0] - mn[1]) + (mt[0] - mt[1]) * (mt[0] - mt[1])));
        }
        // equilibrium state g0 (Eq. 2.8): derivatives in the variables of its
        // Euler Jacobians, S1 = <a_n u + a_t v>, A = -S1, the time derivatives
        // y1, y2 of W_n and W_t, S2 = <A1t u + A2t v>, and <A u>
        const Gas<R, D> G0 = gas_of<R, D>(Q0, gm1);
        ok &= G0.rho > (R)0 && G0.p > (R)0;
        const R igm1 = MeshR<R>::igm1(g), cs2 = gm * G0.th;
        Hat<R> hx[ND];
#pragma unroll
        for (int q = 0; q < ND; ++q) hx[q] = hat_of<R, D>(G0, gm1, dQ[q]);
        const Hat<R> s1 = euler_uv<R, D>(G0, cs2, hx[0], hx[D == 2 ? 2 : 0]);
        Hat<R> y1 = euler_uv<R, D>(G0, cs2, hx[1], hx[D == 2 ? 4 : 0]);
        Hat<R> y2 = {0, 0, 0, 0};
        if (D == 2) y2 = euler_uv<R, D>(G0, cs2, hx[D == 2 ? 4 : 0], hx[D == 2 ? 3 : 0]);
        y1 = {-y1.r, -y1.a, -y1.b, -y1.p};
        y2 = {-y2.r, -y2.a, -y2.b, -y2.p};
        const Hat<R> s2 = euler_uv<R, D>(G0, cs2, y1, y2);
        const Hat<R> ft = euler_u<R, D>(G0, cs2, s1);  // <A u> = -ft
        // flux terms <u> and <A u>; the linear / quadratic fits of Eq. 2.19-2.20
        // and 2.29 reduce to F = <u>, F_t = <A u>, W_t = -S1, W_tt = -S2 at tau = 0
        R F[4], Ft[4], Wt[4], Wtt[4];
        F[0] = Q0[1];
        F[1] = Q0[1] * G0.U + G0.p;
        if (D == 2) F[2] = Q0[1] * G0.V;
        F[NV - 1] = G0.U * (Q0[NV - 1] + G0.p);
        unhat<R, D>(G0, igm1, ft, Ft);
        unhat<R, D>(G0, igm1, s1, Wt);
        unhat<R, D>(G0, igm1, s2, Wtt);
#pragma unroll
        for (int v = 0; v < NV; ++v) { Ft[v] = -Ft[v]; Wt[v] = -Wt[v]; Wtt[v] = -Wtt[v]; }
        // the flux carried out: F itself (FP64), or its increment over the Euler
        // flux of hb1 (FP32 bulk; that flux is added in the update): the Euler
        // flux of Q0 = hb1 + qv taken as a difference
        R Fo[4];
        if (BULK32) euler_flux_delta<D>(hb1, qv, G0.ir, gm1, Fo);
        else {
#pragma unroll
            for (int v = 0; v < 4; ++v) Fo[v] = F[v];
        }
        if (hgks) {
            // inviscid: c1 dt; viscous (Sec. 4): mu / p with p the pressure of
            // the equilibrium state at the face point
            R base = g.tau_mode == 2 ? MeshR<R>::mu(g) / G0.p : MeshR<R>::c1(g) * Dt;
            R tau = base + MeshR<R>::c2(g) * fabs(pz[0] - pz[1]) / (pz[0] + pz[1]) * Dt;
            // collision and non-equilibrium terms of Eq. 2.6, fitted analytically
            R T2[4], T3[4] = {0, 0, 0, 0}, T4[4] = {0, 0, 0, 0};
            unhat<R, D>(G0, igm1, euler_u<R, D>(G0, cs2, s2), T2);  // <Att u> = -T2
            const Range<R, 5> H0 = full_range<R, D, 5>(G0);
            add_dmoments_u<2>(G0, H0, Kx, var_of<R, D>(G0, hx[0]), T3);
            add_dmoments_u<2>(G0, H0, Kx, var_of<R, D>(G0, y1), T4);
            if constexpr (D == 2) {
                add_dmoments_v<1>(G0, H0, Kx, var_of<R, D>(G0, hx[2]), T3);
                add_dmoments_v<1>(G0, H0, Kx, var_of<R, D>(G0, y2), T4);
            }
            R ed = exp(-Dt / tau), eh = exp((R)-0.5 * Dt / tau);
            R h = (R)0.5 * Dt;
            R E0d = tau * ((R)1 - ed), E0h = tau * ((R)1 - eh);
            R E1d = tau * tau * ((R)1 - ed) - tau * Dt * ed, E1h = tau * tau * ((R)1 - eh) - tau * h * eh;
            R f0 = ((R)4 * E0h - E0d) / Dt, g0 = (R)4 * (E0d - (R)2 * E0h) / (Dt * Dt);
            R f1 = ((R)4 * E1h - E1d) / Dt, g1 = (R)4 * (E1d - (R)2 * E1h) / (Dt * Dt);
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const R T3s = T3[v], T4s = T4[v], T2s = -T2[v];
                R T0v = F[v], T1v = Ft[v];
                // F = T0 + (the terms below); FP32 bulk adds them to the increment
                Fo[v] += -f0 * T0v - tau * T1v + (f1 - tau) * T3s + f0 * T5[v] - f1 * T6[v];
                Ft[v] = -g0 * T0v + T1v - tau * T2s + g1 * T3s - tau * T4s + g0 * T5[v] - g1 * T6[v];
                R dS = -Wt[v] - S1h[v];  // S1 - S1h
                Wt[v] += ((R)2 * eh - ed) * dS;
                Wtt[v] += (R)4 * (ed - eh) / Dt * dS;
            }
        }
        // stage outputs: o[0], o[1] fluxes, o[2], o[3] interface states
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            if (v >= NV) { o[0][v] = o[1][v] = o[2][v] = o[3][v] = (R)0; continue; }
            // interface-state values: Q0 itself, or its increment over hb1 (FP32 bulk)
            const R Qv = BULK32 ? qv[v] : Q0[v];
            if (STAGE == 1) {
                o[0][v] = (R)0.5 * Dt * Fo[v] + (R)0.125 * Dt * Dt * Ft[v];
                o[1][v] = Dt * Fo[v] + dt26 * Ft[v];
                o[2][v] = Qv + (R)0.5 * Dt * Wt[v] + (R)0.125 * Dt * Dt * Wtt[v];
                o[3][v] = Qv + Dt * Wt[v] + dt26 * Wtt[v];
            } else {
                o[0][v] = (R)2 * dt26 * Ft[v];
                o[2][v] = (R)2 * dt26 * Wtt[v];
            }
        }
        // finite outputs: 0 * x is 0 for finite x only
        R zero = (R)0;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (STAGE == 1 || q % 2 == 0) {
#pragma unroll
                for (int v = 0; v < NV; ++v) zero += (R)0 * o[q][v];
            }
        const long long face = pt_idx(dir, na, nb, b, f);
        in.template put<STAGE>(o, face, sig);
        if (!ok || !(zero == (R)0)) flag_bad(g, face * M + l);
    }
}

// 1-D: one thread per face.  CAP = 1 asks for at least 4 resident blocks of 128
// threads (<= 128 registers, spilling the rest); CAP = 0 for 4, or 3 with the
// collision-time terms, in FP32 (<= 128, 168 registers) and 1 in FP64.  The
// autotuner times both variants in FP64, where they round alike; the FP32-bulk
// form has the uncapped one only (a capped compilation may contract its FP32
// arithmetic differently, and results must not depend on tuning).
template <typename R, int STAGE, int CAP, int HG, bool PF, bool ONE>
__global__ void __launch_bounds__(128, CAP ? 4 : (sizeof(R) == 4 ? (HG ? 3 : 4) : 1))
k_flux1(const __grid_constant__ Work w)
{
    grid_wait();
    for (long long gi = blockIdx.x * (long long)blockDim.x + threadIdx.x; gi < w.total;
         gi += (long long)gridDim.x * blockDim.x) {
        long long li;
        const Mesh& g = mesh_of<ONE>(w, gi, li);
        const int f = (int)li, na = g.nx;
        const R Dt = MeshR<R>::dt(g);
        LinePoint<R> in;
        in.FR = (const R*)g.FR[0];
        in.nrow = fr_nrow(0, na, 1);
        in.row = fr_row(0, na, 1, 1, f);
        in.FO = (R*)g.FO[0];
        in.sx = g.sig_xn;
        in.nf = na + 1;
        if (sizeof(R) == 4) {
            const R* SF = state_planes<R>(g, STAGE == 1 ? 0 : 1);
            const double tb = stage_time(g, STAGE);
#pragma unroll
            for (int v = 0; v < 3; ++v) in.h[v] = cell<1, 1, R, true>(g, SF, 0, v, 0, f, 0, tb);
            in.h[3] = (R)0;
        }
        R o[4][4], sig;
        flux_point<1, 1, R, STAGE, HG, PF>(g, 0, na, 1, f, 0, 0, in, Dt, Dt * Dt / (R)6, o, sig);
    }
}

// 2-D: warps marching over strips of faces (above).  Dynamic shared memory:
// FluxShared<M, R>::total values of R per warp.  Work offsets count steps.
// FP32: 4 blocks of 128 threads per SM (128 registers).  FP64: a warp's ring takes
// 21-23 KB, so that 8 to 10 warps fit an SM, which its 164-226 registers allow
// (a variant capped at 128 registers only spilled: of 72 tuned fluxes between
// 12^2 and 512^2 cells 3 took it, on small meshes, where the timings scatter).
template <int M, typename R, int STAGE, int HG, bool PF, bool ONE>
__global__ void __launch_bounds__(128, sizeof(R) == 4 ? 4 : 1) k_flux2(const __grid_constant__ Work w)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    grid_wait();
    using L = FluxShared<M, R>;
    constexpr bool BULK32 = sizeof(R) == 4;
    constexpr int FW = L::FW, RING = L::RING;
    const int lane = threadIdx.x & 31, x = lane / M, l = lane - x * M;
    R* sm = (R*)smem_raw + (threadIdx.x >> 5) * L::total;
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
    const long long wid = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    long long t = wid * w.total / nw;
    const long long tend = (wid + 1) * w.total / nw;
    while (t < tend) {
        long long tl;
        __syncwarp();  // the last run's reads are done
        const Mesh& g = mesh_of<ONE>(w, t, tl);
        // the run's direction, strip and steps [k0, kend)
        const int nc0 = (g.nx + 1 + FW - 1) / FW, nc1 = (g.nx + FW - 1) / FW;
        const long long n0 = (long long)nc0 * g.ny;
        const int dir = tl < n0 ? 0 : 1;
        if (dir == 1) tl -= n0;
        int na, nb;
        local_dims<M>(g, dir, na, nb);
        const int nk = dir == 0 ? nb : nc1;
        const int outer = (int)(tl / nk);  // dir 0: strip of faces; dir 1: face row f
        const int k0 = (int)(tl - (long long)outer * nk);
        const int kend = (int)min((long long)nk, k0 + (tend - t));
        t += kend - k0;
        const R Dt = MeshR<R>::dt(g);
        const R dt26 = Dt * Dt / (R)6, iht = (R)1 / (R)(dir == 0 ? g.dy : g.dx);
        const int f = dir == 0 ? outer * FW + x : outer;
        const long long nf = (long long)nb * (na + 1);
        // this lane's sources of the next row (dir 0) or block of rows (dir 1) of
        // face states, advanced by `step` values a row or block; its copies stop at
        // row bb = nb + 1
        const bool mine = lane < FW * M && f <= na;
        const long long plane = M * fr_nrow(dir, na, nb) * 4;  // values of a quantity's M line planes
        const long long step = dir == 0 ? (long long)fr_pitch(na + 1) * 4 : FW * 4;
        int bs = dir == 0 ? k0 : k0 * FW + x;  // row bb of the next states
        const R* ps = (const R*)g.FR[dir] + fr_off(fr_nrow(dir, na, nb), M, 0, 0, l, fr_row(dir, na, nb, bs, mine ? f : 0));
        int slot3 = 0;                          // ring slot of the next states
        auto load_states = [&]() {
            if (mine && bs <= nb + 1) {
                R* dst = sm + L::ring + (l * RING + slot3 * FW + x) * 4;
#pragma unroll
                for (int side = 0; side < 2; ++side)
#pragma unroll
                    for (int nd = 0; nd < 2; ++nd)
                        copy_async4(dst + (side * 2 + nd) * M * RING * 4, ps + (side * 3 + nd) * plane);
            }
            ps += step;
            bs += dir == 0 ? 1 : FW;
            slot3 = slot3 == 2 ? 0 : slot3 + 1;
        };
        // and of what only a step's own points read, for step kn: W_nn, and the
        // face's items dealt to its M lanes: TD of the right cell in three parts,
        // the tangential DFF of its two cells
        int kn = k0;
        const int b0 = dir == 0 ? k0 : k0 * FW + x;
        const R* pn = (const R*)g.FR[dir] + fr_off(fr_nrow(dir, na, nb), M, 0, 2, l, fr_row(dir, na, nb, b0 + 1, mine ? f : 0));
        long long cidx = cell_idx(dir, na, nb, f, b0);
        const long long prev = dir == 0 ? 1 : nb + 2;
        auto load_own = [&]() {
            const int b = dir == 0 ? kn : kn * FW + x;
            if (mine && b < nb) {
                const int slot = kn & 1;
#pragma unroll
                for (int side = 0; side < 2; ++side)
                    copy_async4(sm + L::nn + (((slot * 2 + side) * M + l) * FW + x) * 4, pn + side * 3 * plane);
                if (BULK32)
                    for (int q = l; q < 3; q += M)
                        copy_async4(sm + L::td + (slot * FW + x) * 12 + q * 4, (const R*)g.TD[dir] + cidx * 12 + q * 4);
                if (l == M - 1) {
                    copy_async1(sm + L::at + (slot * 2 + 0) * FW + x, (const R*)g.AT[dir] + cidx - prev);
                    copy_async1(sm + L::at + (slot * 2 + 1) * FW + x, (const R*)g.AT[dir] + cidx);
                }
            }
            pn += step;
            cidx += dir == 0 ? na + 6 : FW;
            ++kn;
        };
        load_states();
        if (dir == 0) load_states();
        load_states();
        load_own();
        copy_commit();
        int r0 = 0;  // ring slot of row or block k
        for (int k = k0; k < kend; ++k) {
            copy_wait<0>();
            __syncwarp();
            const int r1 = r0 == 2 ? 0 : r0 + 1, r2 = r1 == 2 ? 0 : r1 + 1, slot = k & 1;
            // Step 3: items (side, face, variable)
#pragma unroll 1
            for (int it = lane; it < 2 * FW * 4; it += 32) {
                const int v = it & 3, xi = (it >> 2) % FW, side = (it >> 2) / FW;
                int q[3];
                if (dir == 0) {
                    q[0] = r0 * FW + xi; q[1] = r1 * FW + xi; q[2] = r2 * FW + xi;
                } else {
                    q[0] = r0 * FW + xi;
                    q[1] = xi + 1 < FW ? r0 * FW + xi + 1 : r1 * FW;
                    q[2] = xi + 2 < FW ? r0 * FW + xi + 2 : r1 * FW + xi + 2 - FW;
                }
                R dm = (R)0, dp = (R)0;
                if (BULK32) {
                    dm = sm[L::td + (slot * FW + xi) * 12 + 4 + v];
                    dp = sm[L::td + (slot * FW + xi) * 12 + 8 + v];
                }
                // scaled by the tangential r5 DFF of the reconstructing cell
                // (f-1 for the left state, f for the right)
                const R c1 = sm[L::at + (slot * 2 + side) * FW + xi] * iht;
                step3<M, R>(sm + L::ring + side * 2 * M * RING * 4 + v, sm + L::ring + (side * 2 + 1) * M * RING * 4 + v, q,
                            dm, dp, c1, c1 * iht, sm + L::tang + (side * 3 * M * FW + xi) * 4 + v);
            }
            __syncwarp();
            // the next step's copies; ring row k is free now
            if (k + 1 < kend) {
                load_states();
                load_own();
            }
            copy_commit();
            const int b = dir == 0 ? k : k * FW + x;
            const bool point = mine && b < nb;
            const long long face = pt_idx(dir, na, nb, point ? b : 0, point ? f : 0);
            R o[4][4] = {}, sig = (R)0;
            if (point) {
                StripPoint<M, R> in;
                in.s = sm;
                in.FO = (R*)g.FO[dir];
                in.nf = nf;
                in.slot = slot;
                in.own_q = dir == 0 ? r1 * FW + x : (x + 1 < FW ? r0 * FW + x + 1 : r1 * FW);
                in.x = x;
                in.l = l;
                flux_point<2, M, R, STAGE, HG, PF>(g, dir, na, nb, f, b, l, in, Dt, dt26, o, sig);
            }
            __syncwarp();
            constexpr int NO = STAGE == 1 ? 2 : 1;
            face_sums<M, NO>(o, (R*)g.FO[dir] + fs_off(nf, M, NO, 0, 0), nf, face, l, point);
            if (STAGE == 1) face_sigma<M>(sig, (dir == 0 ? g.sig_xn : g.sig_yn) + face, l, point);
            r0 = r1;
        }
    }
}

// -------------------------------------------------------------- update (2-D)
// Stage 1 writes W* (S1) and the accumulator; stage 2 writes state n+1 (S0).
// FP32-bulk form: the float planes (F1 / F0) receive everything the next stage
// reads, the FP64 planes the cell averages of state n+1 (W* lives in F1 only).
template <typename R> __device__ __forceinline__ void swap12(R* v) { const R z = v[1]; v[1] = v[2]; v[2] = z; }

template <int M, typename R, int STAGE, bool ONE>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 3 : 1) k_update2(const __grid_constant__ Work w)
{
    grid_wait();
    constexpr bool BULK32 = sizeof(R) == 4;
    int km = -1;
    for (long long gi = blockIdx.x * (long long)blockDim.x + threadIdx.x; gi < w.total;
         gi += (long long)gridDim.x * blockDim.x) {
        long long c;
        const Mesh& g = mesh_from<ONE>(w, gi, c, km);
        unsigned cu = (unsigned)c, qj = cu / (unsigned)g.nx;  // 32-bit (bounded on the host)
        int i = (int)(cu - qj * (unsigned)g.nx), j = (int)qj;
        const R* FX = (const R*)g.FO[0];
        const R* FY = (const R*)g.FO[1];
        // x-faces: b = j, f = i and i+1; y-faces: b = i, f = j and j+1
        const long long fxl = (long long)j * (g.nx + 1) + i, fyl = (long long)j * g.nx + i;
        const long long nfx = (long long)g.ny * (g.nx + 1), nfy = (long long)g.nx * (g.ny + 1);
        const double idx = g.idx, idy = g.idy;
        const R ridx = MeshR<R>::ih(g, 0), ridy = MeshR<R>::ih(g, 1);
        long long P = g.plane;
        double* out = STAGE == 1 ? g.S1 : g.S0;
        // line-slope part of the accumulator, held in the bulk precision (a float
        // view in the FP32-bulk form: it only ever holds bulk values)
        R* accs = (R*)(g.ACC + 4 * P);
        float* outf = STAGE == 1 ? g.F1 : g.F0;
        const auto& TR = Tab<R>::get(g.oi);
        // Conserved quantities: the Gauss sum over a face's points was formed
        // per face, in the bulk precision, and both cells of a face use it.  The
        // difference of a cell's two face sums is taken in FP64 or, FP32 bulk, in
        // float-float (exactly, by a two-sum), scaled, and subtracted from the
        // FP64 average in FP64: the updates telescope over the mesh and the totals
        // change only by the boundary fluxes and by rounding at FP64's level.
        // Slopes use bulk differences.
        // FP32 bulk, stage 1: the face outputs are increments over hi of each
        // face's right cell (this cell for the left and bottom faces, cells
        // (i+1, j) and (i, j+1) for the others).  Their flux parts add
        // dt/2 (F(hi_R) - F(hi_L)) and dt (...) with the Euler fluxes F of the
        // bases in float-float (each cell forms the same values bitwise, so
        // the update still telescopes), their state parts the difference of
        // the bases' hi.
        R h0[4] = {0, 0, 0, 0}, hxn[4] = {0, 0, 0, 0}, hyn[4] = {0, 0, 0, 0};
        ff Bx[4], By[4];
        if (BULK32 && STAGE == 1) {
            const float* SF = g.F0;
            const double tb = *g.tn;
            const bool nx = i + 1 < g.nx, ny = j + 1 < g.ny;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                h0[v] = (R)SF[v * P + c];
                if (nx) hxn[v] = (R)SF[v * P + c + 1];
                if (ny) hyn[v] = (R)SF[v * P + c + g.nx];
            }
            if (!nx) {
                const CellMap m = cell_map<true>(g, i + 1, j, tb);
#pragma unroll
                for (int v = 0; v < 4; ++v) hxn[v] = (R)mapped<2, M, float, true>(g, SF, m, 0, v, 0);
            }
            if (!ny) {
                const CellMap m = cell_map<true>(g, i, j + 1, tb);
#pragma unroll
                for (int v = 0; v < 4; ++v) hyn[v] = (R)mapped<2, M, float, true>(g, SF, m, 0, v, 0);
            }
            const double gm1d = g.gamma - 1.0;
            const ff gm1 = {(float)gm1d, (float)(gm1d - (double)(float)gm1d)};
            ff f0[4], f1[4];
            float wl[4];
            // x: local frame = global (rho, m_x, m_y, E)
            for (int v = 0; v < 4; ++v) wl[v] = (float)h0[v];
            euler_flux_ff<2>(wl, gm1, f0);
            for (int v = 0; v < 4; ++v) wl[v] = (float)hxn[v];
            euler_flux_ff<2>(wl, gm1, f1);
            for (int v = 0; v < 4; ++v) Bx[v] = ff_add(f1[v], ff_neg(f0[v]));
            // y: local frame (rho, m_y, m_x, E), back to global order
            wl[0] = (float)h0[0]; wl[1] = (float)h0[2]; wl[2] = (float)h0[1]; wl[3] = (float)h0[3];
            euler_flux_ff<2>(wl, gm1, f0);
            wl[0] = (float)hyn[0]; wl[1] = (float)hyn[2]; wl[2] = (float)hyn[1]; wl[3] = (float)hyn[3];
            euler_flux_ff<2>(wl, gm1, f1);
            const int yl[4] = {0, 2, 1, 3};
            for (int v = 0; v < 4; ++v) By[v] = ff_add(f1[yl[v]], ff_neg(f0[yl[v]]));
        }
        // the faces' flux sums (y-faces: local frame (rho, m_y, m_x, E) to global order)
        constexpr int NO = STAGE == 1 ? 2 : 1;
        R gxr[NO][4], gxl[NO][4], gyr[NO][4], gyl[NO][4];
#pragma unroll
        for (int q = 0; q < NO; ++q) {
            ld4(FX + fs_off(nfx, M, NO, q, fxl + 1), gxr[q]);
            ld4(FX + fs_off(nfx, M, NO, q, fxl), gxl[q]);
            ld4(FY + fs_off(nfy, M, NO, q, fyl + g.nx), gyr[q]);
            ld4(FY + fs_off(nfy, M, NO, q, fyl), gyl[q]);
            swap12(gyr[q]);
            swap12(gyl[q]);
        }
        double W0[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) W0[v] = STAGE == 1 ? g.S0[v * P + c] : g.ACC[v * P + c];
        R sx[4] = {0, 0, 0, 0}, sy[4] = {0, 0, 0, 0};
#pragma unroll 1
        for (int l = 0; l < M; ++l) {
            R wl = TR.gw[l];
            R a[4], bq[4], cq[4], dq[4];
            // stage 1: W(dt/2), W0 + dt W_t + dt^2/6 W_tt; stage 2: dt^2/3 W_tt*
#pragma unroll
            for (int q = 0; q < NO; ++q) {
                ld4(FX + fo_off(nfx, M, q, l, fxl + 1), a);
                ld4(FX + fo_off(nfx, M, q, l, fxl), bq);
                ld4(FY + fo_off(nfy, M, q, l, fyl + g.nx), cq);
                ld4(FY + fo_off(nfy, M, q, l, fyl), dq);
                swap12(cq);
                swap12(dq);
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    R dx_ = a[v] - bq[v];
                    R dy_ = cq[v] - dq[v];
                    if (BULK32 && STAGE == 1) {  // interface states over the bases' hi
                        dx_ += hxn[v] - h0[v];
                        dy_ += hyn[v] - h0[v];
                    }
                    if (q == 0) {
                        R lx = dx_ * ridx, ly = dy_ * ridy;
                        if (STAGE == 2) {
                            lx += accs[(4 * l + v) * P + c];
                            ly += accs[(4 * M + 4 * l + v) * P + c];
                        }
                        if (BULK32) {
                            outf[(12 + 4 * l + v) * P + c] = (float)lx;
                            outf[(12 + 4 * M + 4 * l + v) * P + c] = (float)ly;
                        } else {
                            out[(12 + 4 * l + v) * P + c] = (double)lx;
                            out[(12 + 4 * M + 4 * l + v) * P + c] = (double)ly;
                        }
                        sx[v] += wl * lx;
                        sy[v] += wl * ly;
                    } else {  // the line-slope part of the accumulator
                        accs[(4 * l + v) * P + c] = dx_ * ridx;
                        accs[(4 * M + 4 * l + v) * P + c] = dy_ * ridy;
                    }
                }
            }
        }
        bool bad = false;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            double Wn;
            if (BULK32) {
                // float-float: the exact differences of the face sums (two-sums),
                // the bases' flux differences times dt/2 or dt, over dx and dy;
                // one conversion to FP64 per quantity (the FP64 pipe is narrow)
                const ff ix = {g.idxf, g.idxlo}, iy = {g.idyf, g.idylo};
                ff tx = ff_two_sum((float)gxr[0][v], -(float)gxl[0][v]), ty = ff_two_sum((float)gyr[0][v], -(float)gyl[0][v]);
                if (STAGE == 1) {
                    const ff hdt = {0.5f * g.dtf[0], 0.5f * g.dtf[1]}, fdt = {g.dtf[0], g.dtf[1]};
                    tx = ff_add(tx, ff_mul(hdt, Bx[v]));
                    ty = ff_add(ty, ff_mul(hdt, By[v]));
                    ff ax = ff_add(ff_two_sum((float)gxr[NO - 1][v], -(float)gxl[NO - 1][v]), ff_mul(fdt, Bx[v]));
                    ff ay = ff_add(ff_two_sum((float)gyr[NO - 1][v], -(float)gyl[NO - 1][v]), ff_mul(fdt, By[v]));
                    g.ACC[v * P + c] = W0[v] - ff_val(ff_add(ff_mul(ax, ix), ff_mul(ay, iy)));
                }
                // Eq. 2.21, 2.22-2.23: from the FP64 average or its accumulator, in FP64
                Wn = W0[v] - ff_val(ff_add(ff_mul(tx, ix), ff_mul(ty, iy)));
            } else {
                const double dx0 = gxr[0][v] - gxl[0][v], dy0 = gyr[0][v] - gyl[0][v];
                if (STAGE == 1) {
                    const double W = W0[v];
                    Wn = W - dx0 * idx - dy0 * idy;  // Eq. 2.21
                    g.ACC[v * P + c] = W - (double)(gxr[NO - 1][v] - gxl[NO - 1][v]) * idx
                                     - (double)(gyr[NO - 1][v] - gyl[NO - 1][v]) * idy;
                } else {
                    Wn = W0[v] - dx0 * idx - dy0 * idy;  // Eq. 2.22-2.23
                }
            }
            // the FP32-bulk stage 2 reads W* from the float planes only
            if (!BULK32 || STAGE == 2) out[v * P + c] = Wn;
            bad |= !isfinite(Wn);
            if (BULK32) {
                const float hi = (float)Wn;
                outf[v * P + c] = hi;
                outf[(12 + 8 * M + v) * P + c] = (float)(Wn - (double)hi);  // low part
                outf[(4 + v) * P + c] = (float)sx[v];  // cell slopes: Gauss sum of the line slopes
                outf[(8 + v) * P + c] = (float)sy[v];
            } else {
                out[(4 + v) * P + c] = (double)sx[v];
                out[(8 + v) * P + c] = (double)sy[v];
            }
        }
        // the step's face sigma (Eq. 3.1) for the next step
        if (STAGE == 2) {
            g.sig_x[(long long)j * (g.nx + 1) + i] = g.sig_xn[(long long)j * (g.nx + 1) + i];
            if (i == g.nx - 1) g.sig_x[(long long)j * (g.nx + 1) + g.nx] = g.sig_xn[(long long)j * (g.nx + 1) + g.nx];
            g.sig_y[(long long)j * g.nx + i] = g.sig_yn[(long long)j * g.nx + i];
            if (j == g.ny - 1) g.sig_y[(long long)g.ny * g.nx + i] = g.sig_yn[(long long)g.ny * g.nx + i];
        }
        if (bad) flag_bad(g, c);
    }
}

// -------------------------------------------------------------- update (1-D)
template <typename R, int STAGE, bool ONE>
__global__ void __launch_bounds__(256) k_update1(const __grid_constant__ Work w)
{
    grid_wait();
    constexpr bool BULK32 = sizeof(R) == 4;
    for (long long gi = blockIdx.x * (long long)blockDim.x + threadIdx.x; gi < w.total;
         gi += (long long)gridDim.x * blockDim.x) {
        long long il;
        const Mesh& g = mesh_of<ONE>(w, gi, il);
        int i = (int)il;
        const R* FX = (const R*)g.FO[0];
        // q-th output quantity of variable v at face i (left) or i + 1 (right)
        const long long nf = g.nx + 1;
        auto xl = [&](int e) { return FX[fo_off(nf, 1, e >> 2, 0, i) + (e & 3)]; };
        auto xr = [&](int e) { return FX[fo_off(nf, 1, e >> 2, 0, i + 1) + (e & 3)]; };
        const double idx = g.idx;
        long long P = g.plane;
        bool bad = false;
        // FP32 bulk, stage 1: face outputs are increments over hi of the face's
        // right cell (i, and i+1); their flux parts add the float-float Euler
        // fluxes of the bases, their state parts the bases' difference
        double B[3] = {0, 0, 0}, hd[3] = {0, 0, 0};
        if (BULK32 && STAGE == 1) {
            const double tb = *g.tn;
            float h0[3], h1[3];
            for (int v = 0; v < 3; ++v) {
                h0[v] = g.F0[v * P + i];
                h1[v] = cell<1, 1, float, true>(g, g.F0, 0, v, 0, i + 1, 0, tb);
                hd[v] = (double)(h1[v] - h0[v]);
            }
            const double gm1d = g.gamma - 1.0;
            const ff gm1 = {(float)gm1d, (float)(gm1d - (double)(float)gm1d)};
            ff f0[3], f1[3];
            euler_flux_ff<1>(h0, gm1, f0);
            euler_flux_ff<1>(h1, gm1, f1);
            for (int v = 0; v < 3; ++v) B[v] = ff_val(ff_add(f1[v], ff_neg(f0[v])));
        }
        for (int v = 0; v < 3; ++v) {
            double Wn, Sn;
            if (STAGE == 1) {
                double W = g.S0[v * P + i];
                const double dtd = *g.dt;
                Wn = W - (((double)xr(v) - (double)xl(v)) + 0.5 * dtd * B[v]) * idx;
                Sn = (((double)xr(8 + v) - (double)xl(8 + v)) + hd[v]) * idx;
                if (!BULK32) g.S1[v * P + i] = Wn;  // the FP32-bulk stage 2 reads the float planes
                g.ACC[v * P + i] = W - (((double)xr(4 + v) - (double)xl(4 + v)) + dtd * B[v]) * idx;
                g.ACC[(3 + v) * P + i] = (((double)xr(12 + v) - (double)xl(12 + v)) + hd[v]) * idx;
            } else {
                Wn = g.ACC[v * P + i] - ((double)xr(v) - (double)xl(v)) * idx;
                Sn = g.ACC[(3 + v) * P + i] + ((double)xr(8 + v) - (double)xl(8 + v)) * idx;
                g.S0[v * P + i] = Wn;
            }
            if (BULK32) {
                float* outf = STAGE == 1 ? g.F1 : g.F0;
                const float hi = (float)Wn;
                outf[v * P + i] = hi;
                outf[(6 + v) * P + i] = (float)(Wn - (double)hi);  // low part
                outf[(3 + v) * P + i] = (float)Sn;
            } else {
                (STAGE == 1 ? g.S1 : g.S0)[(3 + v) * P + i] = Sn;
            }
            bad |= !isfinite(Wn);
        }
        if (STAGE == 2) {
            g.sig_x[i] = g.sig_xn[i];
            if (i == g.nx - 1) g.sig_x[g.nx] = g.sig_xn[g.nx];
        }
        if (bad) flag_bad(g, i);
    }
}

// -------------------------------------------------------------- FP32-bulk state copies
// to_float: all FP64 planes of state n -> the float planes (after a state is set);
// otherwise the float slope planes -> the FP64 planes (before a state is read
// out; the FP64 cell averages are already current).
template <int D, int M>
__global__ void __launch_bounds__(256) k_convert(const __grid_constant__ Work w, int to_float)
{
    constexpr int NP = D == 2 ? 12 + 8 * M : 6;
    constexpr int NV = D + 2;
    for (long long gi = blockIdx.x * (long long)blockDim.x + threadIdx.x; gi < w.total;
         gi += (long long)gridDim.x * blockDim.x) {
        int k = find_mesh(w, gi);
        const Mesh& g = w.mesh[k];
        long long c = gi - w.off[k];
        long long P = g.plane;
        if (to_float) {
            for (int p = 0; p < NP; ++p) g.F0[p * P + c] = (float)g.S0[p * P + c];
            // low parts of the cell averages, after the other planes
            for (int v = 0; v < NV; ++v) g.F0[(NP + v) * P + c] = low_part<float>(g.S0[v * P + c]);
        } else {
            for (int p = NV; p < NP; ++p) g.S0[p * P + c] = (double)g.F0[p * P + c];
        }
    }
}

// -------------------------------------------------------------- the step size
// The step in flight takes dt from t^n = t, and t moves on.
__device__ __forceinline__ void set_step(const Mesh& g, double dt)
{
    *g.dt = dt;
    g.dtf[0] = (float)dt;
    g.dtf[1] = (float)(dt - (double)(float)dt);
    const double t = *g.t;
    *g.tn = t;
    *g.t = t + dt;
    for (int q = 0; q < 4; ++q) g.branch[q] = 0ull;  // counts cover the latest step
}

// CFL (Sec. 4):
// max over cells of (|U| + a) / h (and 4 nu / h^2 for viscous flow), h =
// min(dx, dy); one atomicMax per block on the
// bit pattern of a positive double (ordered like the value).  The plain form
// evaluates the speeds in FP64 from the FP64 averages; the FP32-bulk form in
// FP32 from its float state planes (the step size is not a conserved
// quantity: its 1e-7 relative rounding only shifts where the steps fall),
// and the maximum is taken in FP64 in both.
//
// MODE 0 leaves the maximum in smax.  A single mesh's step (MODE 1) and the
// step size for the host (MODE 2) are finished by the last block to arrive,
// which saves a launch (and the host two copies): MODE 1 sets the step, MODE 2
// writes the maximum to *out, mapped host memory.
template <int D, typename R, int MODE>
__global__ void __launch_bounds__(256) k_cfl(const __grid_constant__ Work w, double* out)
{
    grid_wait();
    __shared__ double red[8];
    double best = 0.0;
    int kprev = -1, k = -1;
    // a block takes a contiguous run of cells: of a batch, it meets few meshes (in
    // strides of the grid every thread met another mesh at every cell and sent its
    // maximum off by an atomic: 282 us for 2.2 million cells in 24 meshes)
    const long long end = w.total * (blockIdx.x + 1LL) / gridDim.x;
    for (long long gi = w.total * blockIdx.x / gridDim.x + threadIdx.x; gi < end; gi += blockDim.x) {
        long long c;
        const Mesh& g = mesh_from<false>(w, gi, c, k);
        if (k != kprev && kprev >= 0 && best > 0.0)
            atomicMax(w.mesh[kprev].smax, (unsigned long long)__double_as_longlong(best)), best = 0.0;
        kprev = k;
        long long P = g.plane;
        const R* S = state_planes<R>(g, 0);
        const R gm = MeshR<R>::gamma(g);
        R rho = S[c], ir = (R)1 / rho;
        R mu = S[P + c] * ir;
        R mv = D == 2 ? S[2 * P + c] * ir : (R)0;
        R E = S[(D + 1) * P + c];
        R q2 = mu * mu + mv * mv;
        R p = (gm - (R)1) * (E - (R)0.5 * rho * q2);
        R ih = D == 2 ? fmax(MeshR<R>::ih(g, 0), MeshR<R>::ih(g, 1)) : MeshR<R>::ih(g, 0);  // 1 / min(dx, dy)
        R sp = (sqrt(q2) + sqrt(gm * p * ir)) * ih;
        // viscous flow: the diffusive limit dt <= h^2 / (4 nu), nu = mu / rho
        if (g.tau_mode == 2) sp = fmax(sp, (R)4 * MeshR<R>::mu(g) * ir * ih * ih);
        double s = (double)sp;
        if (!(s == s)) s = 1e300;  // a NaN state yields a tiny step and is flagged by the stages
        best = fmax(best, s);
    }
    // single-mesh tables reduce per block; batches flush per mesh change above
    if (w.n == 1) {
        for (int o = 16; o > 0; o >>= 1) best = fmax(best, __shfl_xor_sync(0xffffffffu, best, o));
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = best;
        __syncthreads();
        if (threadIdx.x == 0) {
            double b = 0.0;
            for (int q = 0; q < (int)(blockDim.x >> 5); ++q) b = fmax(b, red[q]);
            const Mesh& g = w.m0;
            if (b > 0.0) atomicMax(g.smax, (unsigned long long)__double_as_longlong(b));
            if (MODE > 0) {
                __threadfence();
                if (atomicAdd(g.done, 1u) == gridDim.x - 1) {
                    __threadfence();
                    const double s = __longlong_as_double((long long)atomicExch(g.smax, 0ull));
                    *g.done = 0u;
                    if (MODE == 1) {
                        set_step(g, s > 0.0 ? g.cfl / s : 0.0);
                    } else {
                        *out = s;
                        __threadfence_system();
                    }
                }
            }
        }
    } else {
        // one atomic per warp where its lanes end in one mesh
        const int k0 = __shfl_sync(0xffffffffu, kprev, 0);
        if (__all_sync(0xffffffffu, kprev == k0)) {
            for (int o = 16; o > 0; o >>= 1) best = fmax(best, __shfl_xor_sync(0xffffffffu, best, o));
            if ((threadIdx.x & 31) != 0) best = 0.0;
        }
        if (kprev >= 0 && best > 0.0) atomicMax(w.mesh[kprev].smax, (unsigned long long)__double_as_longlong(best));
    }
}

// dt = cfl / smax per mesh (or the fixed value); t^n = t, t += dt; reset the
// reduction.  A template, so that only the unit that launches it holds it.
template <int Unused = 0>
__global__ void k_dt(Mesh* meshes, int n, int use_cfl, const double* fixed)
{
    grid_wait();
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        Mesh& g = meshes[k];
        double dt;
        if (use_cfl) {
            double s = __longlong_as_double((long long)*g.smax);
            dt = s > 0.0 ? g.cfl / s : 0.0;
            *g.smax = 0ull;
        } else {
            dt = fixed[k];
        }
        set_step(g, dt);
    }
}

// Initial sigma from the two cell averages adjacent to each face (Eq. 3.2), in
// FP64 and bound by its pipe: a thread takes kSigRows cells of a column, so that
// the cell below is evaluated once, with one reciprocal and one reciprocal
// square root a cell and one division a face (2048^2: 3.06 -> 0.91 ms).
constexpr int kSigRows = 4;

struct Mach { double p, mx, my; };  // pressure, Mach numbers along x and y

template <int D>
__device__ __forceinline__ Mach mach_of(const Mesh& g, int i, int j, double tb)
{
    double W[4];
    if (i >= 0 && i < g.nx && j >= 0 && j < g.ny) {
        const double* p = g.S0 + (long long)j * g.nx + i;
#pragma unroll
        for (int v = 0; v < D + 2; ++v) W[v] = p[v * g.plane];
    } else {
        for (int v = 0; v < D + 2; ++v) W[v] = cell<D, 4, double>(g, g.S0, 0, v, 0, i, j, tb);
    }
    const double ir = 1.0 / W[0], u = W[1] * ir, v = D == 2 ? W[2] * ir : 0.0;
    Mach m;
    m.p = (g.gamma - 1.0) * (W[D + 1] - 0.5 * W[0] * (u * u + v * v));
    const double ic = rsqrt(g.gamma * m.p * ir);
    m.mx = u * ic;
    m.my = v * ic;
    return m;
}
__device__ __forceinline__ double sigma_of(const Mach& l, const Mach& r)
{
    const double dx = l.mx - r.mx, dy = l.my - r.my;
    return fabs(l.p - r.p) * (l.p + r.p) / (l.p * r.p) + dx * dx + dy * dy;
}

template <int D>
__global__ void k_sigma_init(const __grid_constant__ Work w)
{
    for (long long gi = blockIdx.x * (long long)blockDim.x + threadIdx.x; gi < w.total;
         gi += (long long)gridDim.x * blockDim.x) {
        int k = find_mesh(w, gi);
        const Mesh& g = w.mesh[k];
        const unsigned li = (unsigned)(gi - w.off[k]), q = li / (unsigned)g.nx;
        const int i = (int)(li - q * (unsigned)g.nx), j0 = (int)q * kSigRows, j1 = min(j0 + kSigRows, g.ny);
        const double tb = *g.t;  // inflow ghost states at the current time
        Mach below = {};
        if (D == 2) below = mach_of<D>(g, i, j0 - 1, tb);
        for (int j = j0; j < j1; ++j) {
            const Mach c = mach_of<D>(g, i, j, tb);
            g.sig_x[(long long)j * (g.nx + 1) + i] = sigma_of(mach_of<D>(g, i - 1, j, tb), c);
            if (i == g.nx - 1) g.sig_x[(long long)j * (g.nx + 1) + g.nx] = sigma_of(c, mach_of<D>(g, g.nx, j, tb));
            if (D == 2) {
                g.sig_y[(long long)j * g.nx + i] = sigma_of(below, c);
                if (j == g.ny - 1) g.sig_y[(long long)g.ny * g.nx + i] = sigma_of(c, mach_of<D>(g, i, g.ny, tb));
            }
            below = c;
        }
    }
}

// positivity of a state set in (host-side check is done on the device)
template <int D>
__global__ void k_check_state(const __grid_constant__ Work w)
{
    for (long long gi = blockIdx.x * (long long)blockDim.x + threadIdx.x; gi < w.total;
         gi += (long long)gridDim.x * blockDim.x) {
        int k = find_mesh(w, gi);
        const Mesh& g = w.mesh[k];
        long long c = gi - w.off[k];
        long long P = g.plane;
        double rho = g.S0[c], u = g.S0[P + c] / rho, v = D == 2 ? g.S0[2 * P + c] / rho : 0.0;
        double p = (g.gamma - 1.0) * (g.S0[(D + 1) * P + c] - 0.5 * rho * (u * u + v * v));
        if (!(rho > 0.0) || !(p > 0.0)) flag_bad(g, c);
    }
}

} // namespace cgks
