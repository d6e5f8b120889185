// Device code of the ASE-DFF compact gas-kinetic scheme (sm_103a).
//
// One stage of the S2O4 step (Sec. 2.2) runs as four kernels over the work
// items of every mesh in a descriptor table (one mesh, or a batch of uneven
// meshes):
//
//   k_recon   (one launch per direction) Sec. 3.3 Step 1: tangential ASE-DFF
//             reconstruction of every cell (plus a ghost halo), evaluated at the
//             m Gauss lines of the faces -> line averages; Step 2: normal
//             ASE-DFF reconstruction of every (cell, Gauss line) from line
//             averages and line-averaged slopes -> W, W_n, W_nn at the cell's
//             two faces (Algorithm 1).  1-D: k_normal1, Step 2 alone.
//   k_flux1/2 Sec. 3.3 Step 3 (tangential W_t, W_tt, W_nt from the face values
//             of three face segments), Eq. 3.2 (sigma), Step 4 (kinetic
//             weighting, Eq. 2.7-2.8) and the time-integrated flux and
//             interface state of Eq. 2.6, 2.11, 2.12, 2.15 with the linear /
//             quadratic fits of Eq. 2.19-2.20 and 2.29 done analytically per
//             term; emits the per-point quantities the update needs.
//   k_update1/2  Eq. 2.21-2.25, 2.30 and the Gauss-theorem slope update of
//             Sec. 3.3: cell averages, cell slopes and line slopes; the FP64
//             accumulator makes stage 2 need no stage-1 face data; face
//             sigma (Eq. 3.1) for the next step.
//
// Precision: R is the type of the reconstruction and kinetic arithmetic
// (double, or float for the FP32-bulk form).  Cell averages and their
// accumulation, the DFF (the sums of sigma, alpha and the branch tests), the check
// of a state that is set and the point fallback's test are always FP64; a face's
// sigma and the flux kernels' positivity flag are evaluated in R.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "tables.h"

namespace cgks {

enum { BC_PERIODIC = 0, BC_TRANSMISSIVE = 1, BC_FIXED = 2, BC_REFLECTIVE = 3, BC_NOSLIP = 4,
       BC_INFLOW = 5, BC_INFLOW_REFLECTIVE = 6 };
enum { ST_S0 = 0, ST_S1 = 1, ST_S2 = 2, ST_R5 = 3, ST_R7 = 4, ST_R9 = 5 };
enum { STATUS_NONPHYS = 1u };

struct TabF {
    float row[6][10][10];
    float cpoly[4][5][10];
    float bm2[3][3];
    float bm4[5][5];
    float gx[4], gw[4];
    float sd1[2][2][7], sd2[2][2][7];
    // each coefficient twice, for two-wide FMAs: rows of r5, r7, r9, and sd1
    float2 row2[3][10][10], sd1w[2][2][7];
};

static __constant__ CgksTables c_tab[3];  // orders 5, 7, 9 (one copy per translation unit)
static __constant__ TabF c_tabf[3];

template <typename R> struct Tab;
template <> struct Tab<double> {
    __device__ static const CgksTables& get(int oi) { return c_tab[oi]; }
};
template <> struct Tab<float> {
    __device__ static const TabF& get(int oi) { return c_tabf[oi]; }
};

// Per-mesh descriptor (device memory); a batch is an array of these.
struct Mesh {
    int nx, ny, order, oi;          // oi: 0, 1, 2 for orders 5, 7, 9
    int bc[4];
    int tau_mode;
    int dff_lag;                    // 0: sigma of step n-1; 1: stage 2 uses stage 1's
    int pf;                         // first-order fallback at non-physical face points
    double dx, dy, gamma, K, thr, eps, c1, c2, cfl;
    double ao[6];                   // linear weights of HWENO-AO: g0 = g1, g2, g3, g0 / g3, g2 / g3, 1 / g3
    float aof[6];
    double idx, idy;                // 1 / dx, 1 / dy
    double mu;                      // dynamic viscosity (tau_mode 2)
    double x0, y0;                  // lower-left corner
    double bcs[4][2][4];            // inflow ghost states per side: [0] below the split, [1] beyond
    double bcx[4][2];               // split point along the side: bcx[0] + bcx[1] t
    float muf;
    float gf, Kf, c1f, c2f, idxf, idyf;  // FP32-bulk copies (no per-point conversions)
    double igamma, igm1;            // 1 / gamma, 1 / (gamma - 1)
    float igf, igm1f;
    float idxlo, idylo;             // low parts: idx = idxf + idxlo to float-float accuracy
    long long plane;                // nx * ny
    // state: planes of nx*ny doubles.  2-D: W[4] Wx[4] Wy[4] Wxl[m][4] Wyl[m][4];
    // 1-D: W[3] Wx[3]
    double *S0, *S1;                // S0: state n (and n+1), S1: stage-1 state W*
    float *F0, *F1;                 // FP32-bulk form: float copies of all planes of S0 / S1,
                                    // then the low parts float(W - float(W)) of the cell
                                    // averages (the FP64 planes hold the cell averages;
                                    // their slope planes are rebuilt from these on read-out)
    double *ACC;                    // 2-D: W[4] Wxl[m][4] Wyl[m][4]; 1-D: W[3] Wface[3]
    double *sig_x, *sig_y;          // sigma of the previous step [ny][nx+1], [ny+1][nx]
    double *sig_xn, *sig_yn;        // sigma being built this step
    const double* ghost;            // 1-D fixed BC ghost cells
    void *FR[2], *FO[2];            // scratch per direction (R typed)
    void* AT[2];                    // tangential r5 DFF per cell (R typed)
    void* TD[2];                    // FP32 bulk: hi(a, b), hi(a, b-1) - hi(a, b), hi(a, b+1) - hi(a, b)
                                    // of each cell, local frame, [12] floats
    double* dt;                     // device scalar (this mesh's step)
    float* dtf;                     // the same in FP32: [0] float(dt), [1] float(dt - [0])
    double* t;                      // device scalar (simulated time)
    double* tn;                     // device scalar: t^n of the step in flight
    unsigned long long* nfall;      // face-point sides that took the fallback
    unsigned* status;
    long long* bad;
    unsigned long long* smax;       // CFL reduction (bits of a positive double)
    unsigned* done;                 // its blocks that have arrived
    unsigned long long* branch;     // [4] AO, r5, r7, r9 counts
};

// Prefix sums of the work items of every kernel over the meshes of a table,
// and the first mesh's descriptor by value: a launch over one mesh reads its
// descriptor from the kernel parameters (constant-bank operands) instead of
// loading it from the table in every grid-stride iteration.  Kernels take it as
// a __grid_constant__: where a pointer into it escapes (a CellMap's prescribed
// state), the compiler otherwise copies all of it into every thread's local
// memory, 880 bytes (500 x 250 cells between walls, order 5, FP32: a pass of 2602
// instead of 1891 us).
struct Work {
    const Mesh* mesh;
    const long long* off;  // [n+1] prefix of items
    int n;
    long long total;
    Mesh m0;               // mesh[0]
};

__device__ __forceinline__ int find_mesh(const Work& w, long long g)
{
    int lo = 0, hi = w.n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (w.off[mid] <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// The mesh of work item gi and the item's index within it.  ONE: the launch
// covers a single mesh (offset 0), taken from the parameters.
template <bool ONE>
__device__ __forceinline__ const Mesh& mesh_of(const Work& w, long long gi, long long& local)
{
    if (ONE) { local = gi; return w.m0; }
    const int k = find_mesh(w, gi);
    local = gi - w.off[k];
    return w.mesh[k];
}

// The same for a thread whose items only go up: the mesh is searched once and
// then stepped on from.  k: -1 at first.
template <bool ONE>
__device__ __forceinline__ const Mesh& mesh_from(const Work& w, long long gi, long long& local, int& k)
{
    if (ONE) { local = gi; return w.m0; }
    if (k < 0) k = find_mesh(w, gi);
    while (gi >= w.off[k + 1]) ++k;
    local = gi - w.off[k];
    return w.mesh[k];
}

__device__ __forceinline__ int imod(int a, int n) { int r = a % n; return r < 0 ? r + n : r; }

// ------------------------------------------------------------------ ghost cells

// Mesh constants in the bulk precision R.
template <typename R> struct MeshR;
template <> struct MeshR<double> {
    __device__ static double gamma(const Mesh& g) { return g.gamma; }
    __device__ static double K(const Mesh& g) { return g.K; }
    __device__ static double igamma(const Mesh& g) { return g.igamma; }
    __device__ static const double* ao(const Mesh& g) { return g.ao; }
    __device__ static double igm1(const Mesh& g) { return g.igm1; }
    __device__ static double c1(const Mesh& g) { return g.c1; }
    __device__ static double c2(const Mesh& g) { return g.c2; }
    __device__ static double mu(const Mesh& g) { return g.mu; }
    __device__ static double ih(const Mesh& g, int dir) { return dir == 0 ? g.idx : g.idy; }
    __device__ static double dt(const Mesh& g) { return *g.dt; }
};
template <> struct MeshR<float> {
    __device__ static float gamma(const Mesh& g) { return g.gf; }
    __device__ static float K(const Mesh& g) { return g.Kf; }
    __device__ static float igamma(const Mesh& g) { return g.igf; }
    __device__ static const float* ao(const Mesh& g) { return g.aof; }
    __device__ static float igm1(const Mesh& g) { return g.igm1f; }
    __device__ static float c1(const Mesh& g) { return g.c1f; }
    __device__ static float c2(const Mesh& g) { return g.c2f; }
    __device__ static float mu(const Mesh& g) { return g.muf; }
    __device__ static float ih(const Mesh& g, int dir) { return dir == 0 ? g.idxf : g.idyf; }
    __device__ static float dt(const Mesh& g) { return *g.dtf; }
};

// The state planes the bulk arithmetic reads: FP64 planes for R = double,
// the float copies for R = float.  which: 0 state n, 1 stage-1 state.
template <typename R> __device__ __forceinline__ const R* state_planes(const Mesh& g, int which);
template <> __device__ __forceinline__ const double* state_planes<double>(const Mesh& g, int which)
{
    return which == 0 ? g.S0 : g.S1;
}
template <> __device__ __forceinline__ const float* state_planes<float>(const Mesh& g, int which)
{
    return which == 0 ? g.F0 : g.F1;
}

__device__ __forceinline__ bool is_wall(int bc) { return bc == BC_REFLECTIVE || bc == BC_NOSLIP; }
// sides whose ghost faces mirror sigma (a wall along all or part of the side)
__device__ __forceinline__ bool is_mirror(int bc) { return is_wall(bc) || bc == BC_INFLOW_REFLECTIVE; }

// Time at which a stage takes prescribed ghost states: t^n in stage 1, the
// stage-2 state lives at t^n + dt/2.
__device__ __forceinline__ double stage_time(const Mesh& g, int stage)
{
    return stage == 1 ? *g.tn : *g.tn + 0.5 * *g.dt;
}

// Inflow sides: is the centre of ghost row / column k, along side `side`
// (y on the x-sides, x on the y-sides), below the split point at time tb?
__device__ __forceinline__ bool below_split(const Mesh& g, int side, int k, double tb)
{
    double s = side < 2 ? g.y0 + (k + 0.5) * g.dy : g.x0 + (k + 0.5) * g.dx;
    return s < g.bcx[side][0] + g.bcx[side][1] * tb;
}

// Sign of a ghost value mirrored across a wall with normal x (normal = 0) or
// y (normal = 1): reflection maps q to S q(-x), S reversing the normal
// momentum (slip wall) or every momentum component (no-slip wall); a
// derivative along the normal takes one more sign.
template <int D>
__device__ __forceinline__ bool wall_flip(int kind, int v, int normal, int bc)
{
    bool rev = (v == 1 + normal) || (bc == BC_NOSLIP && v >= 1 && v <= D);
    bool dnormal = normal == 0 ? (kind == 1 || kind == 3) : (kind == 2 || kind == 4);
    return rev != dnormal;
}

// The low part of a cell average in the FP32-bulk form: the FP64 average x is
// held as hi = float(x) (the W planes) plus lo = float(x - hi) (the planes
// after all others); FP64 planes need no low part.
template <typename T> __device__ __forceinline__ T low_part(double x) { return (T)(x - (double)(T)x); }
template <> __device__ __forceinline__ double low_part<double>(double) { return 0.0; }

// A prescribed ghost value x (fixed ghost cells, inflow states) as kind asks:
// the value (kind 0), its low part (kind 5), or a zero slope.
template <typename T> __device__ __forceinline__ T prescribed(double x, int kind)
{
    return kind == 0 ? (T)x : (kind == 5 ? low_part<T>(x) : (T)0);
}

// Where the data of cell (i, j) come from.  Ghost rules apply x first, then y: a
// prescribed state, or cell idx with slopes along x / y zeroed and with the
// mirror images at walls normal to x / y (the wall's boundary code, or 0).
struct CellMap {
    long long idx;
    int zx, zy, wx, wy;
    const double* state;  // prescribed state (inflow), or null
};

// tb: the stage's time, read by inflow sides only.  WALLS = false compiles the
// wall and inflow branches out: the stencil kernels have an instance for meshes
// without them.
template <bool WALLS>
__device__ __forceinline__ CellMap cell_map(const Mesh& g, int i, int j, double tb, bool two = true)
{
    CellMap c = {0, 0, 0, 0, 0, nullptr};
    if (i < 0 || i >= g.nx) {
        const int side = i < 0 ? 0 : 1, bc = g.bc[side];
        if (bc == BC_PERIODIC) {
            i = imod(i, g.nx);
        } else if (WALLS && (bc == BC_INFLOW || (bc == BC_INFLOW_REFLECTIVE && below_split(g, side, j, tb)))) {
            // by the row's centre
            c.state = g.bcs[side][below_split(g, side, j, tb) ? 0 : 1];
            return c;
        } else if (WALLS && is_mirror(bc)) {
            // ghost cell -1-k mirrors cell k
            i = i < 0 ? -1 - i : 2 * g.nx - 1 - i;
            c.wx = bc;
        } else {
            i = i < 0 ? 0 : g.nx - 1;
            c.zx = 1;
        }
    }
    if (two && (j < 0 || j >= g.ny)) {
        const int side = j < 0 ? 2 : 3, bc = g.bc[side];
        if (WALLS && (bc == BC_INFLOW || (bc == BC_INFLOW_REFLECTIVE && below_split(g, side, i, tb)))) {
            // by the column's centre (after the x rule)
            c.state = g.bcs[side][below_split(g, side, i, tb) ? 0 : 1];
            return c;
        }
        if (bc == BC_PERIODIC) {
            j = imod(j, g.ny);
        } else if (WALLS && is_mirror(bc)) {
            j = j < 0 ? -1 - j : 2 * g.ny - 1 - j;
            c.wy = bc;
        } else {
            j = j < 0 ? 0 : g.ny - 1;
            c.zy = 1;
        }
    }
    c.idx = (long long)j * g.nx + i;
    return c;
}

// The plane of a value.  kind: 0 W, 1 Wx, 2 Wy, 3 Wx_line, 4 Wy_line (global
// orientation), 5 the low part of W (FP32-bulk float planes only).
template <int D, int M>
__device__ __forceinline__ int value_plane(int kind, int v, int l)
{
    if (D == 1) return kind == 0 ? v : (kind == 5 ? 6 + v : 3 + v);
    switch (kind) {
    case 0: return v;
    case 1: return 4 + v;
    case 2: return 8 + v;
    case 3: return 12 + 4 * l + v;
    case 5: return 12 + 8 * M + v;
    default: return 12 + 4 * M + 4 * l + v;
    }
}

// One value of a mapped cell
template <int D, int M, typename T, bool WALLS>
__device__ __forceinline__ T mapped(const Mesh& g, const T* S, const CellMap& c, int kind, int v, int l)
{
    const bool nx = WALLS && c.wx && wall_flip<D>(kind, v, 0, c.wx), ny = WALLS && c.wy && wall_flip<D>(kind, v, 1, c.wy);
    if (WALLS && c.state) {
        const T val = prescribed<T>(c.state[v], kind);  // zero slopes
        return nx ? -val : val;
    }
    if ((c.zx && (kind == 1 || kind == 3)) || (c.zy && (kind == 2 || kind == 4))) return (T)0;
    // lines across a mirrored side swap ends
    if (WALLS && ((c.wx && kind == 4) != (c.wy && kind == 3))) l = M - 1 - l;
    const T val = S[value_plane<D, M>(kind, v, l) * g.plane + c.idx];
    return nx != ny ? -val : val;
}

// One value of cell (i, j), ghost rules applied
template <int D, int M, typename T, bool WALLS = true>
__device__ __forceinline__ T cell(const Mesh& g, const T* S, int kind, int v, int l, int i, int j, double tb)
{
    if (D == 1 && (i < 0 || i >= g.nx) && g.bc[i < 0 ? 0 : 1] == BC_FIXED) {
        const int side = i < 0 ? 0 : 1, layer = side == 0 ? (-1 - i) : (i - g.nx);
        const double gv = g.ghost[((side * 3 + layer) * 2 + (kind == 0 || kind == 5 ? 0 : 1)) * 3 + v];
        return kind == 5 ? low_part<T>(gv) : (T)gv;
    }
    return mapped<D, M, T, WALLS>(g, S, cell_map<WALLS>(g, i, j, tb, D == 2), kind, v, l);
}

// sigma of x-face f (between cells f-1 and f) in row j; ghost faces: periodic
// wrap, otherwise 0 beyond the boundary face and the nearest row across y.
template <int D, bool WALLS = true>
__device__ __forceinline__ double sigx(const Mesh& g, const double* sx, int f, int j)
{
    if (f < 0 || f > g.nx) {
        int bc = g.bc[f < 0 ? 0 : 1];
        if (bc == BC_PERIODIC) f = imod(f, g.nx);
        else if (WALLS && is_mirror(bc)) f = f < 0 ? -f : 2 * g.nx - f;  // beyond a wall: the mirrored face
        else return 0.0;
    }
    if (D == 2 && (j < 0 || j >= g.ny)) {
        int bc = g.bc[j < 0 ? 2 : 3];
        if (bc == BC_PERIODIC) j = imod(j, g.ny);
        else if (WALLS && is_mirror(bc)) j = j < 0 ? -1 - j : 2 * g.ny - 1 - j;
        else j = j < 0 ? 0 : g.ny - 1;
    }
    return sx[(long long)j * (g.nx + 1) + f];
}

template <bool WALLS = true>
__device__ __forceinline__ double sigy(const Mesh& g, const double* sy, int i, int f)
{
    if (f < 0 || f > g.ny) {
        int bc = g.bc[f < 0 ? 2 : 3];
        if (bc == BC_PERIODIC) f = imod(f, g.ny);
        else if (WALLS && is_mirror(bc)) f = f < 0 ? -f : 2 * g.ny - f;
        else return 0.0;
    }
    if (i < 0 || i >= g.nx) {
        int bc = g.bc[i < 0 ? 0 : 1];
        if (bc == BC_PERIODIC) i = imod(i, g.nx);
        else if (WALLS && is_mirror(bc)) i = i < 0 ? -1 - i : 2 * g.nx - 1 - i;
        else i = i < 0 ? 0 : g.nx - 1;
    }
    return sy[(long long)f * g.nx + i];
}

// 16-byte vector moves of 4 consecutive values (float4, or two double2)
__device__ __forceinline__ void ld4(const float* p, float v[4])
{
    float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void ld4(const double* p, double v[4])
{
    double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void st4(float* p, const float v[4])
{
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st4(double* p, const double v[4])
{
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
    *reinterpret_cast<double2*>(p + 2) = make_double2(v[2], v[3]);
}

__device__ __forceinline__ void ld2(const float* p, float v[2])
{
    const float2 q = *reinterpret_cast<const float2*>(p);
    v[0] = q.x; v[1] = q.y;
}
__device__ __forceinline__ void st2(float* p, const float v[2]) { *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]); }
__device__ __forceinline__ void st2(double* p, const double v[2])
{
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
}
__device__ __forceinline__ void ld2(const double* p, double v[2])
{
    const double2 q = *reinterpret_cast<const double2*>(p);
    v[0] = q.x; v[1] = q.y;
}

// ------------------------------------------------------------------ float-float
// Unevaluated sums hi + lo of two floats (Dekker's double-length arithmetic,
// with Knuth's two-sum and the FMA two-product), about 44 significant bits:
// FP64-level accuracy from FP32 instructions, for the few O(1) quantities of
// the FP32-bulk form whose rounding would otherwise enter every update.  The
// explicit _rn intrinsics keep the compiler from contracting or reassociating.
struct ff { float hi, lo; };

__device__ __forceinline__ ff ff_two_sum(float a, float b)
{
    float s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}
__device__ __forceinline__ ff ff_norm(float hi, float lo)  // |hi| >= |lo|
{
    float s = __fadd_rn(hi, lo);
    return {s, __fsub_rn(lo, __fsub_rn(s, hi))};
}
__device__ __forceinline__ ff ff_add(ff a, ff b)
{
    ff s = ff_two_sum(a.hi, b.hi);
    return ff_norm(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ ff ff_mul(ff a, ff b)
{
    float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, e));
    return ff_norm(p, e);
}
__device__ __forceinline__ ff ff_of(float a) { return {a, 0.0f}; }
// a / b of two floats: the remainder a - q b of the rounded quotient is exact
__device__ __forceinline__ ff ff_div(float a, float b)
{
    float q = __fdiv_rn(a, b);
    return ff_norm(q, __fdiv_rn(__fmaf_rn(-q, b, a), b));
}
__device__ __forceinline__ double ff_val(ff a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ ff ff_neg(ff a) { return {-a.hi, -a.lo}; }

// Euler flux along the local normal of a state given by floats (rho, m_n,
// m_t, E) (2-D, D = 2) or (rho, m, E) (1-D), in float-float: (m_n, m_n u + p,
// m_t u, u (E + p)) with u = m_n / rho, p = (gamma - 1)(E - (m_n u + m_t v) / 2).
// gm1 = gamma - 1 as a float-float.
template <int D>
__device__ __forceinline__ void euler_flux_ff(const float* w, ff gm1, ff* F)
{
    const float rho = w[0], mn = w[1], mt = D == 2 ? w[2] : 0.0f, E = w[D + 1];
    ff u = ff_div(mn, rho);
    ff v = ff_div(mt, rho);
    ff ke = ff_add(ff_mul(ff_of(mn), u), ff_mul(ff_of(mt), v));  // rho |U|^2
    ff p = ff_mul(gm1, ff_add(ff_of(E), ff_mul(ff_of(-0.5f), ke)));
    F[0] = ff_of(mn);
    F[1] = ff_add(ff_mul(ff_of(mn), u), p);
    if (D == 2) F[2] = ff_mul(ff_of(mt), u);
    F[D + 1] = ff_mul(u, ff_add(ff_of(E), p));
}

__device__ __forceinline__ double recip(double x);
__device__ __forceinline__ float recip(float x);

// F(w0 + q) - F(w0) of the Euler flux along the local normal, by algebra in
// which every term is a product with a component of q (no difference of two
// O(1) values), so the result keeps the relative accuracy of q.  w0: the base
// state (floats), q: the increment; same layouts as euler_flux_ff; ir =
// 1 / (w0[0] + q[0]).
template <int D, typename R>
__device__ __forceinline__ void euler_flux_delta(const R* w0, const R* q, R ir, R gm1, R* dF)
{
    const R r0 = w0[0], mn0 = w0[1], mt0 = D == 2 ? w0[2] : (R)0, E0 = w0[D + 1];
    const R dr = q[0], dmn = q[1], dmt = D == 2 ? q[2] : (R)0, dE = q[D + 1];
    const R ir0 = recip(r0);
    const R u0 = mn0 * ir0, v0 = mt0 * ir0;
    const R du = (dmn - u0 * dr) * ir, dv = (dmt - v0 * dr) * ir;  // u - u0, v - v0
    const R u = u0 + du;
    // kinetic energy rho |U|^2 / 2: its change, product by product
    const R dke = (R)0.5 * (dr * (u0 * u0 + v0 * v0) + (r0 + dr) * (du * ((R)2 * u0 + du) + dv * ((R)2 * v0 + dv)));
    const R p0 = gm1 * (E0 - (R)0.5 * r0 * (u0 * u0 + v0 * v0));
    const R dp = gm1 * (dE - dke);
    dF[0] = dmn;
    dF[1] = dmn * u + mn0 * du + dp;             // (m u + p) - (m0 u0 + p0)
    if (D == 2) dF[2] = dmt * u + mt0 * du;      // m_t u - m_t0 u0
    dF[D + 1] = du * (E0 + p0) + u * (dE + dp);  // u H - u0 H0, H = E + p
}

// ------------------------------------------------------------------ ASE-DFF

// Branch and stencil DFFs of one cell from the sigma of the six faces
// i-5/2 .. i+5/2 (Eq. 3.3-3.4).  A stencil's sum covers every face of every
// cell it draws data from; eta = 2 for r9.  Algorithm 1 picks the branch.
struct Dff {
    double a[4];   // alpha of S0, S1, S2, r5
    double alpha;  // alpha of the linear stencil used
    int st;        // linear stencil, or -1 for HWENO-AO
};

__device__ __forceinline__ double dff_alpha(double A, double thr) { return A < thr ? 1.0 : thr / A; }

__device__ __forceinline__ Dff dff_select(int order, const double s[6], double thr)
{
    // The threshold tests come first; a DFF below 1 (a division) is formed
    // only on the HWENO-AO branch, where the sub-stencil DFFs are used.  On
    // every linear branch the chosen stencil's DFF is 1 by construction.
    Dff d;
    double A_r5 = s[1] + s[2] + s[3] + s[4];
    double A_r7 = s[0] + A_r5 + s[5];
    d.a[0] = d.a[1] = d.a[2] = d.a[3] = 1.0;
    d.alpha = 1.0;
    if (A_r5 >= thr) {
        d.st = -1;
        d.a[0] = dff_alpha(s[1] + s[2] + s[3], thr);
        d.a[1] = dff_alpha(s[2] + s[3] + s[4], thr);
        d.a[2] = d.a[3] = d.alpha = thr / A_r5;
    } else if (order == 5 || A_r7 >= thr) {
        d.st = ST_R5;
    } else if (order == 7 || 2.0 * A_r7 >= thr) {
        d.st = ST_R7;
    } else {
        d.st = ST_R9;
    }
    return d;
}

// The taps of dp that sub-stencil k of HWENO-AO uses (S0, S1, S2, r5; the own
// average enters through the differences only)
__host__ __device__ constexpr bool ao_tap(int k, int q)
{
    return k == 0 ? (q == 1 || q == 6)
         : k == 1 ? (q == 3 || q == 8)
         : k == 2 ? (q == 1 || q == 3)
         : (q == 1 || q == 3 || q == 6 || q == 8);
}

// HWENO-AO(5,3) with DFF-scaled sub-polynomials (Eq. 3.11-3.17, 3.19) for
// NOUT consecutive functional rows starting at row0.  Kept out of line: the
// branch is rare, and inlining it in every variable's loop bloats the kernels.
// Only the taps a sub-stencil has are summed (10 of 40 a row), and only the
// entries of the smoothness matrices that are not zero (even x + y); the linear
// weights' ratios gw = (g0, g2, g3, g0 / g3, g2 / g3, 1 / g3) come from the host: a
// few lanes of a shock's cells hold up an FP64 warp for all of this.
template <typename R, int NOUT>
__device__ __noinline__ void recon_ao(const R* al, int oi, int row0, const R* dp, R* out, const R* gw, R eps)
{
    const auto& T = Tab<R>::get(oi);
    R beta[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        constexpr int kDeg[4] = {3, 3, 3, 5};
        R c[5];
#pragma unroll
        for (int n = 1; n < 5; ++n) {
            R s = 0;
            if (n < kDeg[k]) {
#pragma unroll
                for (int q = 0; q < 10; ++q)
                    if (ao_tap(k, q)) s += T.cpoly[k][n][q] * dp[q];
            }
            c[n] = s;
        }
        R b;
        if (k < 3) {
            b = T.bm2[1][1] * (c[1] * c[1]) + T.bm2[2][2] * (c[2] * c[2]);
        } else {
            b = c[1] * (T.bm4[1][1] * c[1] + ((R)2 * T.bm4[1][3]) * c[3]) + c[2] * (T.bm4[2][2] * c[2] + ((R)2 * T.bm4[2][4]) * c[4])
              + T.bm4[3][3] * (c[3] * c[3]) + T.bm4[4][4] * (c[4] * c[4]);
        }
        beta[k] = al[k] * al[k] * b;  // smoothness of the DFF-scaled polynomial
    }
    const R tz = (fabs(beta[3] - beta[0]) + fabs(beta[3] - beta[1]) + fabs(beta[3] - beta[2])) * (R)(1.0 / 3.0);
    R w[4], ws = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const R q = tz / (beta[k] + eps), g = gw[k < 2 ? 0 : k - 1];
        w[k] = g + g * (q * q);
        ws += w[k];
    }
    const R inv = (R)1 / ws;
    R ck[4];
#pragma unroll
    for (int k = 0; k < 3; ++k) ck[k] = (w[k] - w[3] * gw[k < 2 ? 3 : 4]) * inv * al[k];
    ck[3] = w[3] * inv * gw[5] * al[3];
#pragma unroll
    for (int r = 0; r < NOUT; ++r) {
        R s = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            R p = 0;
#pragma unroll
            for (int q = 0; q < 10; ++q)
                if (ao_tap(k, q)) p += T.row[k][row0 + r][q] * dp[q];
            s += ck[k] * p;
        }
        out[r] = s;
    }
}

// The taps of dp = (Qbar_{i-2..i+2} - Qbar_i, h Qx_{i-2..i+2}) that a linear
// stencil of Sec. 3.2 uses: the own average enters only through the
// differences (dp[2] = 0) and the own gradient not at all; r5 spans cells
// i-1..i+1 with the neighbour gradients, r7 cells i-2..i+2 with the gradients
// of i-1 and i+1, r9 cells i-2..i+2 with the four neighbour gradients.
__host__ __device__ constexpr bool st_tap(int st, int k)
{
    return st == ST_R9 ? (k != 2 && k != 7)
         : st == ST_R7 ? (k == 0 || k == 1 || k == 3 || k == 4 || k == 6 || k == 8)
         : (k == 1 || k == 3 || k == 6 || k == 8);
}

// FP32: a linear stencil's functional rows tap by tap, on two data sets at once
// (two lines, or two variables) with two-wide FMAs; Steps 1-2 are bound by issue
// slots.  The order (table OI), the stencil and the row are fixed at compile time.
template <int OI, int ST, int ROW>
__device__ __forceinline__ float2 row_taps(const float2 dp[10])
{
    const auto& c = c_tabf[OI].row2[ST - ST_R5][ROW];
    float2 r = __fmul2_rn(c[1], dp[1]);
#pragma unroll
    for (int k = 0; k < 10; ++k)
        if (k != 1 && st_tap(ST, k)) r = __ffma2_rn(c[k], dp[k], r);
    return r;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float a, float2 b) { return __fmul2_rn(make_float2(a, a), b); }

// FP64: the rows in mirrored pairs: on the sums e and differences o of the averages
// of cells i+j and i-j (relative to cell i's) and the sums E and differences O
// of their slopes, j = 1, 2, a functional at place xi is even + odd with even =
// c0 e1 + c1 e2 + c2 O1 + c3 O2 and odd = c4 o1 + c5 o2 + c6 E1 + c7 E2, and the
// same functional at -xi is +-(even - odd): half the multiplications of both.
// The FP64 pipe bounds its Steps 1-2 (0.73 -> 0.57 ms per direction at 512^2,
// order 9); FP32 keeps the taps, whose rounding is a third smaller (order 9
// density wave on 20^2 to t = 2: 1.35e-8 against 1.99e-8).
template <int ST, typename R>
__device__ __forceinline__ void sym_row(const R c[8], const R e[2], const R o[2], const R E[2], const R O[2], R& even,
                                        R& odd)
{
    constexpr bool a2 = ST != ST_R5, s2 = ST == ST_R9;
    even = c[0] * e[0] + c[2] * O[0];
    odd = c[4] * o[0] + c[6] * E[0];
    if (a2) { even += c[1] * e[1]; odd += c[5] * o[1]; }
    if (s2) { even += c[3] * O[1]; odd += c[7] * E[1]; }
}

template <typename R>
__device__ __forceinline__ void sym_data(const R dp[10], R e[2], R o[2], R E[2], R O[2])
{
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        e[j] = dp[3 + j] + dp[1 - j];
        o[j] = dp[3 + j] - dp[1 - j];
        E[j] = dp[8 + j] + dp[6 - j];
        O[j] = dp[8 + j] - dp[6 - j];
    }
}

// value, first and second derivative at xi = +1/2 (out[0..2]) and -1/2 (out[3..5])
template <int ST>
__device__ __forceinline__ void faces_sym(const CgksTables& T, const double dp[10], double out[6])
{
    double e[2], o[2], E[2], O[2];
    sym_data(dp, e, o, E, O);
#pragma unroll
    for (int nd = 0; nd < 3; ++nd) {
        double p, q;
        sym_row<ST, double>(T.sym[ST - ST_R5][nd], e, o, E, O, p, q);
        out[nd] = p + q;
        out[3 + nd] = nd == 1 ? q - p : p - q;
    }
}
template <int ST>
__device__ __forceinline__ void faces_sym(const CgksTables&, const float*, float*) {}  // FP32 keeps the taps

// Calls body(StTag<st>()) for a stencil code (-1: HWENO-AO); the order bounds
// the linear stencils that occur.  The branch is taken once, outside the loop
// over lines or variables, so that each branch is one straight run of code.
template <int V> struct StTag { static constexpr int value = V; };
template <int M, typename Body>
__device__ __forceinline__ void with_stencil(int st, Body&& body)
{
    if (M == 4 && st == ST_R9) body(StTag<(M == 4 ? ST_R9 : ST_R5)>());
    else if (M >= 3 && st == ST_R7) body(StTag<(M >= 3 ? ST_R7 : ST_R5)>());
    else if (st == ST_R5) body(StTag<ST_R5>());
    else body(StTag<-1>());
}

// ------------------------------------------------------------------ kinetics
//
// Every moment the scheme needs of a micro-slope a (Eq. 2.8) is <a u^p v^q psi>
// with <a psi> = dW prescribed: the change of rho <u^p v^q psi> of the
// Maxwellian along dW.  The moments are known functions of (rho, U, V, theta),
// theta = p / rho = 1 / (2 lambda), so that change is their differential: no
// micro-slope is formed and no Gram matrix built.  Per derivative that is 7
// operations to the variables (d rho, rho dU, rho dV, dp) and about 16 to a
// half-range moment vector, where a slope solve (25) and a 4 x 4 Gram product
// (20) did the same; full-range u- and v-moments are the Euler flux Jacobians,
// which act on those variables in 7 operations each.  Alone that took the FP64
// flux kernel, bound by the FP64 pipe, from 11.46 to 7.2 ms at 512^2, order 9,
// tau = 0 (two stages), and the FP32 one, then bound by load latency, from
// 889 + 770 to 768 + 680 us at 1024^2.

// 1 / x.  FP32: the hardware's approximation r (PTX states 1 ulp for
// rcp.approx) and one step of the Newton-Raphson iteration for 1 / r - x = 0, r + r
// (1 - x r), with the residual in one fused operation (as in Markstein, IBM J.
// Res. Dev. 34, 1990): its error d becomes d^2, so that the result is within 0.5 +
// 2^-21 ulp of 1 / x wherever both are normal numbers.  x = 0, infinite x and x
// whose reciprocal overflows give NaN: no physical density or pressure.  1.0f / x
// in its place: 1024^2, order 9, 9670 against 9514 us for five steps, 2048^2 with
// finite tau 18967 against 18808 for two.
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }
__device__ __forceinline__ float recip(float x)
{
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return __fmaf_rn(r, __fmaf_rn(-x, r, 1.0f), r);
}

// 1 / sqrt(x).  FP32: rsqrtf (2 ulp stated) and one Newton-Raphson step for
// 1 / r^2 - x = 0, r + r (1 - x r^2) / 2: within 1 ulp, of which the rounding of x r is
// half; without it the half-range moments of a shock's two sides carry rsqrtf's error.
__device__ __forceinline__ double recip_sqrt(double x) { return rsqrt(x); }
__device__ __forceinline__ float recip_sqrt(float x)
{
    const float r = rsqrtf(x);
    return __fmaf_rn(0.5f * r, __fmaf_rn(-x * r, r, 1.0f), r);
}

// The state variables of a Maxwellian: density and its reciprocal, velocity,
// pressure, theta, and the specific kinetic energy ek = (U^2 + V^2) / 2.
template <typename R, int D>
struct Gas { R rho, ir, U, V, p, th, ek; };

template <typename R, int D>
__device__ __forceinline__ Gas<R, D> gas_of(const R* W, R gm1)
{
    Gas<R, D> G;
    G.rho = W[0];
    G.ir = recip(G.rho);
    G.U = W[1] * G.ir;
    G.V = D == 2 ? W[2] * G.ir : (R)0;
    G.ek = (R)0.5 * (G.U * G.U + (D == 2 ? G.V * G.V : (R)0));
    G.p = gm1 * (W[D + 1] - G.rho * G.ek);
    G.th = G.p * G.ir;
    return G;
}

// A derivative of the conservative variables at a state, in the variables the
// differentials are short in: r = d rho, a = rho dU, b = rho dV, p = dp.
template <typename R>
struct Hat { R r, a, b, p; };

// the change of the internal energy density along a derivative, e = d(rho E)
template <typename R, int D>
__device__ __forceinline__ R internal(const Gas<R, D>& G, R e, R r, R a, R b)
{
    e -= G.ek * r;
    e -= G.U * a;
    if (D == 2) e -= G.V * b;
    return e;
}

template <typename R, int D>
__device__ __forceinline__ Hat<R> hat_of(const Gas<R, D>& G, R gm1, const R* x)
{
    Hat<R> h;
    h.r = x[0];
    h.a = x[1] - G.U * x[0];
    h.b = D == 2 ? x[2] - G.V * x[0] : (R)0;
    h.p = gm1 * internal(G, x[D + 1], h.r, h.a, h.b);
    return h;
}

// The same with t = rho d theta = dp - theta d rho in the place of dp.
template <typename R>
struct Var { R r, a, b, t; };

template <typename R, int D>
__device__ __forceinline__ Var<R> var_of(const Gas<R, D>& G, R gm1, const R* x)
{
    Var<R> h;
    h.r = x[0];
    h.a = x[1] - G.U * x[0];
    h.b = D == 2 ? x[2] - G.V * x[0] : (R)0;
    h.t = gm1 * internal(G, x[D + 1], h.r, h.a, h.b) - G.th * h.r;
    return h;
}
template <typename R, int D>
__device__ __forceinline__ Var<R> var_of(const Gas<R, D>& G, const Hat<R>& h)
{
    return {h.r, h.a, h.b, h.p - G.th * h.r};
}

// back to conservative variables; igm1 = 1 / (gamma - 1)
template <typename R, int D>
__device__ __forceinline__ void unhat(const Gas<R, D>& G, R igm1, const Hat<R>& h, R* x)
{
    x[0] = h.r;
    x[1] = h.a + G.U * h.r;
    if (D == 2) x[2] = h.b + G.V * h.r;
    R e = igm1 * h.p + G.U * h.a + G.ek * h.r;
    if (D == 2) e += G.V * h.b;
    x[D + 1] = e;
}

// y = F'(W) x + G'(W) z: the Jacobians of the Euler fluxes along u and v (the
// full-range moments <a_x u psi> + <a_z v psi>); c2 = gamma theta
template <typename R, int D>
__device__ __forceinline__ Hat<R> euler_uv(const Gas<R, D>& G, R c2, const Hat<R>& x, const Hat<R>& z)
{
    Hat<R> y;
    y.r = G.U * x.r + x.a;
    y.a = G.U * x.a + x.p;
    y.b = G.U * x.b;
    y.p = G.U * x.p + c2 * x.a;
    if (D == 2) {
        y.r += G.V * z.r + z.b;
        y.a += G.V * z.a;
        y.b += G.V * z.b + z.p;
        y.p += G.V * z.p + c2 * z.b;
    }
    return y;
}
template <typename R, int D>
__device__ __forceinline__ Hat<R> euler_u(const Gas<R, D>& G, R c2, const Hat<R>& x)
{
    return {G.U * x.r + x.a, G.U * x.a + x.p, G.U * x.b, G.U * x.p + c2 * x.a};
}

// Moments m[n] = <u^n> of the normal velocity over u > 0 (s = 1), u < 0 (s = -1)
// or all of it, with their derivatives: d m_n / dU = n m_{n-1} and d m_n / dtheta
// = n (n - 1) / 2 m_{n-2}, where the boundary at u = 0 of a half range gives
// d m_0 / dU = k = s f(0), d m_0 / dtheta = -hk = -k U / (2 theta) and
// d m_1 / dtheta = k / 2, f the normal distribution of mean U and variance theta.
template <typename R, int NM>
struct Range { R m[NM]; R k, hk; };

// erfc(x) / 2 for x >= 0, e = exp(-x^2).  FP64: the scaled function takes the
// exponential that f(0) needs anyway, which then scales m_0 and f(0) alike: where
// they cancel in m_1 and m_2 (x > 1/2) those are as accurate as with erfc(x) or up to a
// quarter better, below they carry 1-3 ulp more; the fields' errors against 64
// bits are the same to 1%, and erfc(x) takes 17597 -> 18145 us at 512^2, order 9 (two
// steps).  FP32: erfcf alone is the shorter.
__device__ __forceinline__ double half_erfc(double x, double e) { return 0.5 * e * erfcx(x); }
__device__ __forceinline__ float half_erfc(float x, float) { return 0.5f * erfcf(x); }

// q = 1 / sqrt(theta)
template <typename R, int D, int NM>
__device__ __forceinline__ Range<R, NM> half_range(const Gas<R, D>& G, R q, bool left)
{
    Range<R, NM> H;
    const R x = (R)0.70710678118654752 * G.U * q;  // U / sqrt(2 theta)
    const R e = exp(-x * x);
    const R c = half_erfc(fabs(x), e);
    H.k = (R)0.39894228040143268 * e * q;          // f(0)
    if (!left) H.k = -H.k;
    H.m[0] = (left ? x < (R)0 : x > (R)0) ? c : (R)1 - c;
    H.m[1] = G.U * H.m[0] + G.th * H.k;
#pragma unroll
    for (int n = 0; n + 2 < NM; ++n) H.m[n + 2] = G.U * H.m[n + 1] + (R)(n + 1) * G.th * H.m[n];
    H.hk = (R)0.5 * G.U * q * q * H.k;
    return H;
}
template <typename R, int D, int NM>
__device__ __forceinline__ Range<R, NM> full_range(const Gas<R, D>& G)
{
    Range<R, NM> H;
    H.m[0] = (R)1;
    H.m[1] = G.U;
#pragma unroll
    for (int n = 0; n + 2 < NM; ++n) H.m[n + 2] = G.U * H.m[n + 1] + (R)(n + 1) * G.th * H.m[n];
    H.k = H.hk = (R)0;
    return H;
}

// rho <psi> of the state W over its half range: m0 W plus what the cut at u = 0
// carries, k (0, p, 0, p U / 2).  W enters with one rounding.
template <typename R, int D, int NM>
__device__ __forceinline__ void half_moments(const Gas<R, D>& G, const Range<R, NM>& H, const R* W, R* out)
{
    const R pk = G.p * H.k;
    out[0] = H.m[0] * W[0];
    out[1] = H.m[0] * W[1] + pk;
    if (D == 2) out[2] = H.m[0] * W[2];
    out[D + 1] = H.m[0] * W[D + 1] + (R)0.5 * G.U * pk;
}
// its half-range Euler flux rho <u psi>
template <typename R, int D, int NM>
__device__ __forceinline__ void half_flux(const Gas<R, D>& G, const Range<R, NM>& H, const R* W, R Kx, R* out)
{
    const R w = H.m[0] * W[1] + G.p * H.k;
    out[0] = w;
    out[1] = G.U * w + G.p * H.m[0];
    if (D == 2) out[2] = G.V * w;
    out[D + 1] = (R)0.5 * G.U * out[1] + ((R)0.5 * (G.V * G.V + Kx * G.th) + G.th) * w;
}

// acc += the differential of half_moments along a derivative x: m0 x plus the
// change of m0 and of the cut's terms
template <typename R, int D, int NM>
__device__ __forceinline__ void add_dhalf(const Gas<R, D>& G, const Range<R, NM>& H, R Kx, const R* x, const Var<R>& h,
                                          R* acc)
{
    const R z = H.k * h.a - H.hk * h.t;  // rho d m0
    const R tk = G.th * H.k;
    acc[0] += H.m[0] * x[0];
    acc[0] += z;
    acc[1] += H.m[0] * x[1];
    acc[1] += tk * h.r;
    acc[1] += ((R)0.5 * H.k) * h.t;
    if (D == 2) {
        acc[2] += H.m[0] * x[2];
        acc[2] += G.V * z;
    }
    R e = acc[D + 1];
    e += H.m[0] * x[D + 1];
    e += ((R)0.5 * (G.V * G.V + Kx * G.th)) * z;
    e += tk * h.a;
    e += ((R)0.5 * G.U * tk) * h.r;
    acc[D + 1] = e;
}

// d(rho m_n) along a derivative, and s times it added to acc
template <int N, typename R, int NM>
__device__ __forceinline__ R dmom(const Range<R, NM>& H, const Var<R>& h)
{
    if (N == 0) return H.m[0] * h.r + H.k * h.a - H.hk * h.t;
    if (N == 1) return H.m[1] * h.r + H.m[0] * h.a + ((R)0.5 * H.k) * h.t;
    return H.m[N] * h.r + ((R)N * H.m[N >= 1 ? N - 1 : 0]) * h.a + ((R)(N * (N - 1) / 2) * H.m[N >= 2 ? N - 2 : 0]) * h.t;
}
template <int N, typename R, int NM>
__device__ __forceinline__ void add_dmom(const Range<R, NM>& H, const Var<R>& h, R& acc)
{
    acc += H.m[N] * h.r;
    acc += ((R)N * H.m[N - 1]) * h.a;
    if (N == 1) acc += ((R)0.5 * H.k) * h.t;
    else acc += ((R)(N * (N - 1) / 2) * H.m[N >= 2 ? N - 2 : 0]) * h.t;
}

// acc += d(rho <u^P psi>) along a derivative, as chains of fused multiply-adds.
// Kx = K + D - 1: the degrees of freedom besides u and the mean tangential
// motion.
template <int P, typename R, int D, int NM>
__device__ __forceinline__ void add_dmoments_u(const Gas<R, D>& G, const Range<R, NM>& H, R Kx, const Var<R>& h, R* acc)
{
    const R g = (R)0.5 * (G.V * G.V + Kx * G.th);
    const R d0 = dmom<P>(H, h);
    acc[0] += d0;
    add_dmom<P + 1>(H, h, acc[1]);
    if (D == 2) {
        acc[2] += G.V * d0;
        acc[2] += H.m[P] * h.b;
    }
    R e = acc[D + 1];
    e += ((R)0.5 * H.m[P + 2]) * h.r;
    e += ((R)(0.5 * (P + 2)) * H.m[P + 1]) * h.a;
    e += (((R)(0.25 * (P + 2) * (P + 1)) + (R)0.5 * Kx) * H.m[P]) * h.t;
    e += g * d0;
    if (D == 2) e += (G.V * H.m[P]) * h.b;
    acc[D + 1] = e;
}

// acc += d(rho <u^P v psi>) along a derivative (2-D)
template <int P, typename R, int NM>
__device__ __forceinline__ void add_dmoments_v(const Gas<R, 2>& G, const Range<R, NM>& H, R Kx, const Var<R>& h, R* acc)
{
    const R g = (R)0.5 * (G.V * G.V + Kx * G.th);
    const R d0 = dmom<P>(H, h), d1 = dmom<P + 1>(H, h);
    const R bm = H.m[P] * h.b, tm = H.m[P] * h.t;
    acc[0] += G.V * d0;
    acc[0] += bm;
    acc[1] += G.V * d1;
    acc[1] += H.m[P + 1] * h.b;
    acc[2] += (G.V * G.V + G.th) * d0;
    acc[2] += ((R)2 * G.V) * bm;
    acc[2] += tm;
    // energy: V times the differential of rho <u^P psi_4>, that moment times dV, and rho <u^P> V theta
    R e = (g + G.th) * d0;
    e += ((R)0.5 * H.m[P + 2]) * h.r;
    e += ((R)(0.5 * (P + 2)) * H.m[P + 1]) * h.a;
    e += ((R)(0.25 * (P + 2) * (P + 1) + 1.0) + (R)0.5 * Kx) * tm;
    e += G.V * bm;
    acc[3] += G.V * e;
    acc[3] += ((R)0.5 * H.m[P + 2] + (g + G.th) * H.m[P]) * h.b;
}

} // namespace cgks
