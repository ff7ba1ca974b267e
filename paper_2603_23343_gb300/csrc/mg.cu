// Geometric multigrid preconditioner and PCG with it (the paper names
// multigrid as future work in its conclusion; Sec. VII's iteration is kept).
//
// Hierarchy (aggregation): coarse cell I owns the 2 x 2 x 2 fine cells
// 2I + {0,1}^3, P copies a coarse value to its eight fine cells, and the
// coarse operator is the Galerkin product P^T A P.  For a seven-point
// operator in face-weight form, (A u)_c = D_c u_c - sum over interior faces
// w_f u_nb, that product is again one: a coarse face carries the sum of the
// four fine face weights across it and the coarse diagonal is the sum of the
// eight fine diagonals minus twice the twelve face weights inside the
// aggregate.  Level 0 is the solver's operator (weights computed per point,
// nothing stored but omega / D of block coefficients); coarser levels store
// w+x, w+y, w+z, D and omega / D per cell, an array each.
// Levels are added while every size is even and stays >= 4 (at most 8
// levels).
//
// V-cycle z = M r (level l, right-hand side f; the coarsest level takes
// kMgCoarseSweeps damped Jacobi sweeps from zero in one CTA):
//   f_{l+1} = P^T (f - A u),  u = omega D^-1 f              (one kernel)
//   e = V-cycle(l + 1)
//   out = u' + omega D^-1 (f - A u'),  u' = u + sigma P e   (one kernel)
// (u is formed from f wherever it is used).  Levels of at most kMgTailCells
// cells, the coarsest with them, run these steps inside one CTA
// (mg_tail_kernel) instead of a launch per step.
// Pre- and post-smoothing are adjoint, so M is symmetric (positive definite
// for omega < 1, 0 < sigma < 2).  omega = 0.9 and sigma = 1.5 took the
// fewest iterations in a sweep of the oracle at 32^3 and 64^3.
//
// PCG with M: pass A of the Jacobi solver (p_k = z_k + beta p_{k-1} on the
// fly, the deferred x update, p.Ap -> alpha), pass R (r -= alpha A p_k, r.r,
// the convergence test and the replacement trigger), and the V-cycle, whose
// last kernel also sums r.z (-> beta); residual replacements store r = b - A x (FP64) and go through
// the V-cycle again.  One CUDA graph with a device-driven loop.
#include <algorithm>
#include <cstring>
#include <vector>

#include "solver.cuh"

namespace gb {

namespace {

constexpr int kMgMaxLevels = 8;
constexpr int kMgMinCoarse = 4;
constexpr float kMgOmega = 0.9f;
constexpr float kMgSigma = 1.5f;
constexpr int kMgCoarseSweeps = 24;
constexpr int64_t kMgMaxCoarsest = 32768;
// Grids up to this size (and ny even, for the row pairs) take the solver's passes A and R on the
// march of the level kernels instead of through the TMA ring.  us per MG-PCG iteration, ring ->
// march, Poisson / block coefficients: 32^3 67 -> 53 / 70 -> 50; 64^3 66 -> 59 / 70 -> 61; 128^3
// 92 -> 91 / 102 -> 98; 160^3 132 -> 132 / 165 -> 153; 192^3 179 -> 187 / 219 -> 224; 256^3 308 ->
// 334 / 410 -> 433.
constexpr int64_t kMgDirectPoints = 5000000;
constexpr int kMgUnroll = 3;  // iterations per turn of the loop (kLoopUnroll)
constexpr int kMgThreads = 256;
constexpr int64_t kMgRunPoints = 1 << 27;  // a run of planes: its offsets fit 32 bits
constexpr int kMgTailThreads = 1024;
constexpr int64_t kMgTailCells = 4096;  // levels this small run inside the one-CTA tail kernel
constexpr int kMgTailCtas = 8;          // the cluster that sweeps a larger coarsest level
static_assert(kMgTailCells / 8 <= kMgTailThreads, "a tail of several levels sweeps a cell a thread");
// coarsest cells a thread keeps the weights of in registers
constexpr int kMgSweepCells = (int)((kMgTailCells + kMgTailThreads - 1) / kMgTailThreads);
// shared memory of the tail; the sweeps' two buffers of every coarsest level of kMgMinCoarse planes or more fit
constexpr size_t kMgTailSmem = 216 * 1024;
constexpr int kMgTailLevels = 3;  // 4096 cells, 512, 64: a coarsest level holds 4^3 cells or more
static_assert(kMgTailSmem >= 2 * 3 * (kMgMaxCoarsest / kMgMinCoarse) * sizeof(float), "sweep buffers");

struct MgLevel {
    int nx, ny, nz;
    float *f;        // right-hand side (level 0: the solver's r)
    float *od;       // omega / D per point (constant level 0 above the tail: unused; coarsest: unused)
    float *w;        // post-smoothed result (level 0: z; coarsest: the sweeps' result)
    const float *wx, *wy, *wz, *D;  // levels >= 1 and a level 0 inside the tail: w+x, w+y, w+z and D per cell
    int64_t m;                      // cells
};

struct MgArgs {
    int L;
    MgLevel lv[kMgMaxLevels];
    int block;     // level 0: block coefficients (ob.weights) or constant (ob.cx, cy, cz)
    OpBlock ob;
    const float4 *tab;  // block coefficients: the solver's per-block face table (the same weights, no divisions)
    float rkbx, rkby, rkbz;  // 1 / the block edges (mg_div)
    const SolveState *st;  // inside a solve: kernels stand down by its flags (NULL outside)
};

// n / d for 0 <= n < 2^22 and d >= 1, with rd = 1/d rounded to FP32:
// (n + 1/2) / d lies at least 1/(2d) from an integer, and the two FP32
// roundings (of rd and of the product) move it by at most
// 2^-23 (n + 1/2) / d < 1/(2d), so truncation gives the exact quotient.
__device__ __forceinline__ int mg_div(int n, float rd) { return (int)(((float)n + 0.5f) * rd); }

// Weights of point (i, j, k) of a level: w[0..5] = faces x-, x+, y-, y+, z-,
// z+ towards interior neighbours (0 across the boundary), and D.
__device__ __forceinline__ void mg_weights_stored(const MgLevel &L, int i, int j, int k, float w[6], float &D) {
    const int64_t c = ((int64_t)k * L.ny + j) * L.nx + i;
    w[1] = L.wx[c];
    w[3] = L.wy[c];
    w[5] = L.wz[c];
    D = L.D[c];
    w[0] = i > 0 ? L.wx[c - 1] : 0.f;
    w[2] = j > 0 ? L.wy[c - L.nx] : 0.f;
    w[4] = k > 0 ? L.wz[c - (int64_t)L.nx * L.ny] : 0.f;
}

__device__ __forceinline__ void mg_weights(const MgArgs &a, int l, int i, int j, int k, float w[6], float &D) {
    const MgLevel &L = a.lv[l];
    if (l == 0) {
        if (a.block) {
            // the face table holds the harmonic means (or the block's k on the domain boundary):
            // bitwise the weights of OpBlock::weights, without their divisions
            const OpBlock &o = a.ob;
            const int bx = mg_div(i, a.rkbx), by = mg_div(j, a.rkby), bz = mg_div(k, a.rkbz);
            const int ix = i - bx * o.kbx, iy = j - by * o.kby, iz = k - bz * o.kbz;
            const float4 *t = a.tab + 2 * (((int64_t)bz * o.nby + by) * o.nbx + bx);
            const float4 t0 = __ldg(t), t1 = __ldg(t + 1);
            const float kc = t0.x;
            w[0] = o.cx * (ix == 0 ? t0.y : kc);
            w[1] = o.cx * (ix == o.kbx - 1 ? t0.z : kc);
            w[2] = o.cy * (iy == 0 ? t0.w : kc);
            w[3] = o.cy * (iy == o.kby - 1 ? t1.x : kc);
            w[4] = o.cz * (iz == 0 ? t1.y : kc);
            w[5] = o.cz * (iz == o.kbz - 1 ? t1.z : kc);
        } else {
            w[0] = w[1] = a.ob.cx;
            w[2] = w[3] = a.ob.cy;
            w[4] = w[5] = a.ob.cz;
        }
        D = ((w[0] + w[1]) + (w[2] + w[3])) + (w[4] + w[5]);
        if (i == 0) w[0] = 0.f;
        if (i == L.nx - 1) w[1] = 0.f;
        if (j == 0) w[2] = 0.f;
        if (j == L.ny - 1) w[3] = 0.f;
        if (k == 0) w[4] = 0.f;
        if (k == L.nz - 1) w[5] = 0.f;
        return;
    }
    mg_weights_stored(L, i, j, k, w, D);
}

__device__ __forceinline__ bool mg_stand_down(const SolveState *st) { return st && (st->done || st->replace); }

// Launch geometry of the Galerkin kernel: a block is bx threads along x times
// by rows along y and marches through zper planes.
struct MgLaunch {
    dim3 grid, block;
    int zper;
};
inline MgLaunch mg_launch(int nx, int ny, int nz) {
    const int bx = std::min(kMgThreads, (nx + 31) / 32 * 32);
    const int by = std::max(1, std::min(kMgThreads / bx, ny));
    const int64_t gxy = (int64_t)((nx + bx - 1) / bx) * ((ny + by - 1) / by);
    const int64_t want = (int64_t)device_sm_count() * 16;
    const int gz = (int)std::max<int64_t>(1, std::min<int64_t>(nz, (want + gxy - 1) / gxy));
    const int zper = (nz + gz - 1) / gz;
    return MgLaunch{dim3((unsigned)((nx + bx - 1) / bx), (unsigned)((ny + by - 1) / by), (unsigned)((nz + zper - 1) / zper)),
                    dim3((unsigned)bx, (unsigned)by), zper};
}

// ------------------------------------------------- level kernels --
//
// A level above the tail takes two kernels: the restriction (with the
// pre-smoothing u = (omega / D) f formed from f at every use, so u is neither
// stored nor read back) and the post-smoothing.  Both are bound by memory if
// the instructions per point stay near 30, so a thread keeps what it can:
//   - V neighbouring points of a row (V = 4; 2 where nx % 4 == 2), marching
//     along z with the planes before and after in registers;
//   - lanes 0..15 of a warp hold 16 such segments of row 2J, lanes 16..31
//     those of row 2J + 1: the x neighbours and the row inside the pair come
//     by shuffle, only the one row outside the pair is loaded;
//   - segments are numbered along the plane (row pair times segments of a
//     row), so rows of any length fill the warps;
//   - level-0 block weights are read from the face table once per block of
//     planes, the stored weights of coarser levels are arrays per face
//     direction read as vectors.
// Loads of the plane after next are issued before the current plane is
// computed, at two or three CTAs per SM: the registers hold what is in flight.
// The work is split evenly over the CTAs the device holds (mg_runs).  Block
// coefficients at 256^3 (ncu): pre-smoothing and restriction 30 + 68 us in two
// kernels -> 44 us, post-smoothing 115 -> 51 us (and no pass of 20 us for r.z
// after it); the stored 128^3 level 64 -> 27 us both ways.

// V consecutive floats (V * 4 byte aligned) -> registers
template <int V>
__device__ __forceinline__ void ldv(const float *p, float v[V]) {
    if constexpr (V == 4) {
        const float4 t = __ldg(reinterpret_cast<const float4 *>(p));
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else {
        const float2 t = __ldg(reinterpret_cast<const float2 *>(p));
        v[0] = t.x; v[1] = t.y;
    }
}

// What one launch of a level kernel reads of the hierarchy: a launch's
// parameters are read through a cold constant cache, a line at a time.
struct MgStep {
    const SolveState *st;
    MgLevel L;
    float *c;  // the coarse level's f (restriction) or w (post-smoothing)
    OpBlock ob;
    const float4 *tab;
    float rkbx, rkby, rkbz;
};

// Kind of weights a level kernel is compiled for.  W_TABV: block
// coefficients whose block edge along x is a multiple of V, so that the V
// points of a thread lie in one block.
enum MgWeights { W_CONST0 = 1, W_TABV = 2, W_TAB0 = 3, W_STORED = 4 };

// CTAs per SM the register count is held to: the constant weights leave room for three.
constexpr int mg_min_blocks(int wk) { return wk == W_CONST0 ? 3 : 2; }

// A thread's segment: V points from i0 of row j = 2J + hi.
template <int V>
struct MgSeg {
    int i0, j;
    bool hi, live, el, er, eo;  // eo: the row outside the pair exists; el / er: x neighbours to be loaded
    bool xl0, xr0;              // the row starts / ends here
    unsigned c;                 // flat index at plane 0
    int dro;                    // offset of the row outside the pair
    __device__ __forceinline__ MgSeg(const MgLevel &L, unsigned wseg) {  // the warp's 16 segments per row: 16 wseg ..
        const int lane = threadIdx.x & 31, q = L.nx / V, np = q * (L.ny / 2);
        int p = (int)wseg * 16 + (lane & 15);
        live = p < np;
        p = min(p, np - 1);
        const int J = p / q;
        hi = lane >= 16;
        i0 = (p - J * q) * V;
        j = 2 * J + (hi ? 1 : 0);
        xl0 = i0 == 0;
        xr0 = i0 + V >= L.nx;
        el = (lane & 15) == 0 && !xl0;
        er = (lane & 15) == 15 && !xr0;
        eo = hi ? j + 1 < L.ny : j > 0;
        dro = hi ? L.nx : -L.nx;
        c = (unsigned)j * L.nx + i0;
    }
};

// The weights of a segment's points at the current plane: w[m][0..5] = x-,
// x+, the row inside the pair, the row outside it, z-, z+.  Values outside
// the grid are read as 0, so boundary weights need not be cleared.
template <int V, int WK>
struct MgCol {
    float wc, wxl, wxr, win, wout, wz, wzl, wzh;      // W_TABV (wc, win, wout, wz also W_CONST0)
    float px[WK == W_TAB0 ? V : 1][8];                // W_TAB0: the same per point
    float sx[V], sxl, si[V], so[V], szm[V], sz[V], sD[V];  // W_STORED
    int iz;

    __device__ __forceinline__ void table(const MgStep &a, int i, int j, int k, bool hi, float t[8], bool last_of_seg) {
        const OpBlock &o = a.ob;
        const int bx = mg_div(i, a.rkbx), by = mg_div(j, a.rkby), bz = mg_div(k, a.rkbz);
        const int ix = i - bx * o.kbx, iy = j - by * o.kby;
        const float4 *tb = a.tab + 2 * (((int64_t)bz * o.nby + by) * o.nbx + bx);
        const float4 t0 = __ldg(tb), t1 = __ldg(tb + 1);
        const float kc = t0.x;
        t[0] = o.cx * kc;
        t[1] = o.cx * (ix == 0 ? t0.y : kc);
        t[2] = o.cx * (ix + (last_of_seg ? V - 1 : 0) == o.kbx - 1 ? t0.z : kc);
        const float ylo = o.cy * (iy == 0 ? t0.w : kc), yhi = o.cy * (iy == o.kby - 1 ? t1.x : kc);
        t[3] = hi ? ylo : yhi;
        t[4] = hi ? yhi : ylo;
        t[5] = o.cz * kc;
        t[6] = o.cz * t1.y;
        t[7] = o.cz * t1.z;
    }
    __device__ __forceinline__ void block_at(const MgStep &a, const MgSeg<V> &s, int k) {
        if constexpr (WK == W_TABV) {
            float t[8];
            table(a, s.i0, s.j, k, s.hi, t, true);
            wc = t[0]; wxl = t[1]; wxr = t[2]; win = t[3]; wout = t[4]; wz = t[5]; wzl = t[6]; wzh = t[7];
        } else if constexpr (WK == W_TAB0) {
#pragma unroll
            for (int m = 0; m < V; ++m) table(a, s.i0 + m, s.j, k, s.hi, px[m], false);
        }
    }
    // the weights of the planes from k on
    __device__ __forceinline__ void start(const MgStep &a, const MgLevel &L, const MgSeg<V> &s, int k) {
        if constexpr (WK == W_CONST0) {
            wc = a.ob.cx;
            win = wout = a.ob.cy;
            wz = a.ob.cz;
        } else if constexpr (WK == W_STORED) {
#pragma unroll
            for (int m = 0; m < V; ++m) sz[m] = 0.f;
            if (k > 0) ldv<V>(L.wz + s.c + (int64_t)(k - 1) * L.nx * L.ny, sz);
        } else {
            iz = k - mg_div(k, a.rkbz) * a.ob.kbz - 1;
            block_at(a, s, k);
        }
    }
    // plane k (called for consecutive k from start's)
    __device__ __forceinline__ void plane(const MgStep &a, const MgLevel &L, const MgSeg<V> &s, int64_t cb, unsigned c, int k) {
        if constexpr (WK == W_TABV || WK == W_TAB0) {
            if (++iz == a.ob.kbz) {
                iz = 0;
                block_at(a, s, k);
            }
        } else if constexpr (WK == W_STORED) {
            float y[V], yo[V];
#pragma unroll
            for (int m = 0; m < V; ++m) {
                szm[m] = sz[m];
                yo[m] = 0.f;
            }
            ldv<V>(L.wx + cb + c, sx);
            ldv<V>(L.wy + cb + c, y);
            ldv<V>(L.wz + cb + c, sz);
            ldv<V>(L.D + cb + c, sD);
            if (!s.hi && s.eo) ldv<V>(L.wy + cb + (c - L.nx), yo);
            const float xl = s.el ? __ldg(L.wx + cb + (c - 1)) : 0.f;
            const float xs = __shfl_up_sync(0xffffffffu, sx[V - 1], 1);
            sxl = s.xl0 ? 0.f : s.el ? xl : xs;
#pragma unroll
            for (int m = 0; m < V; ++m) {
                const float yp = __shfl_xor_sync(0xffffffffu, y[m], 16);
                si[m] = s.hi ? yp : y[m];
                so[m] = s.hi ? y[m] : yo[m];
            }
        }
    }
    __device__ __forceinline__ void get(const MgStep &a, int m, float w[6], float &D) const {
        if constexpr (WK == W_CONST0) {
            w[0] = w[1] = wc;
            w[2] = win;
            w[3] = wout;
            w[4] = w[5] = wz;
            D = ((w[0] + w[1]) + (w[2] + w[3])) + (w[4] + w[5]);
        } else if constexpr (WK == W_TABV) {
            w[0] = m == 0 ? wxl : wc;
            w[1] = m == V - 1 ? wxr : wc;
            w[2] = win;
            w[3] = wout;
            w[4] = iz == 0 ? wzl : wz;
            w[5] = iz == a.ob.kbz - 1 ? wzh : wz;
            D = ((w[0] + w[1]) + (w[2] + w[3])) + (w[4] + w[5]);
        } else if constexpr (WK == W_TAB0) {
            w[0] = px[m][1];
            w[1] = px[m][2];
            w[2] = px[m][3];
            w[3] = px[m][4];
            w[4] = iz == 0 ? px[m][6] : px[m][5];
            w[5] = iz == a.ob.kbz - 1 ? px[m][7] : px[m][5];
            D = ((w[0] + w[1]) + (w[2] + w[3])) + (w[4] + w[5]);
        } else {
            w[0] = m == 0 ? sxl : sx[m > 0 ? m - 1 : 0];
            w[1] = sx[m];
            w[2] = si[m];
            w[3] = so[m];
            w[4] = szm[m];
            w[5] = sz[m];
            D = sD[m];
        }
    }
};

// The march all these kernels make: for the planes [k0, k1) of a segment, the
// iterate v at the segment and its neighbours (0 outside the grid), and
// body(k, c, A v, v, f, o) per plane.  What a plane reads is loaded one plane
// ahead (its own row two ahead: the z neighbour).
//   I_U     v = (omega / D) f, o = omega / D     (restriction)
//   I_POST  v = (omega / D) f + sigma P e        (post-smoothing)
//   I_P     v = f + beta o, o = p_{k-1}          (pass A)
//   I_V     v = f                                (pass R)
// The solver's passes form A v from the differences w (v - v_nb), whose
// rounding is relative to A v's terms, the V-cycle as D v - sum w v_nb.
enum MgIter { I_U, I_POST, I_P, I_V };
template <int V, int WK, int IT, typename Body>
__device__ __forceinline__ void mg_march(const MgStep &a, const float *f, const float *od, float beta, bool first,
                                         const MgSeg<V> &s, int k0, int k1, Body body) {
    constexpr bool POST = IT == I_POST, HAS_O = IT == I_P || (IT != I_V && WK != W_CONST0);
    const MgLevel &L = a.L;
    const float *e = a.c;
    // offsets from plane kb on: 32 bits (a run of planes is kept below 2^29 points), shared by all arrays
    const int kb = max(k0 - 1, 0) & ~1;
    const unsigned sz = (unsigned)L.nx * L.ny;
    const int cnx = L.nx / 2;
    const unsigned csz = (unsigned)cnx * (L.ny / 2);
    f += (int64_t)kb * sz;
    if (HAS_O) od += (int64_t)kb * sz;
    if (POST) e += (int64_t)(kb / 2) * csz;
    const float wd = kMgOmega / (((a.ob.cx + a.ob.cx) + (a.ob.cy + a.ob.cy)) + (a.ob.cz + a.ob.cz));  // W_CONST0
    struct Raw {
        float f[V], o[V], e[V / 2];
    };
    // the V values at flat index c, whose parents start at flat index pc
    auto fetch = [&](Raw &r, unsigned c, unsigned pc) {
        ldv<V>(f + c, r.f);
        if constexpr (HAS_O) {
            ldv<V>(od + c, r.o);
        } else {
#pragma unroll
            for (int m = 0; m < V; ++m) r.o[m] = wd;
        }
        if constexpr (POST) {
            if constexpr (V == 4) {
                const float2 t = __ldg(reinterpret_cast<const float2 *>(e + pc));
                r.e[0] = t.x;
                r.e[1] = t.y;
            } else {
                r.e[0] = __ldg(e + pc);
            }
        }
    };
    auto form = [&](float fv, float o, float ev) {
        if constexpr (IT == I_V) return fv;
        else if constexpr (IT == I_P) return first ? fv : fmaf(beta, o, fv);  // no p_{k-1} to read in the first iteration
        else return POST ? fmaf(kMgSigma, ev, fv * o) : fv * o;
    };
    auto iterate = [&](const Raw &r, float v[V]) {
#pragma unroll
        for (int m = 0; m < V; ++m) v[m] = form(r.f[m], r.o[m], r.e[m >> 1]);
    };
    // flat index of the parents of this row at plane k, of the row outside the pair, of the edge point
    auto par = [&](int k) { return (unsigned)((k - kb) >> 1) * csz; };
    const int p0 = (s.j >> 1) * cnx + (s.i0 >> 1), po = p0 + (s.hi ? cnx : -cnx);
    const bool ed = s.el || s.er;  // the point beside the segment that no lane of the half holds
    const int de = s.el ? -1 : V, pe = (s.j >> 1) * cnx + ((s.i0 + de) >> 1);
    struct Edge {
        float f = 0.f, o = 0.f, e = 0.f;
    };
    auto edge = [&](Edge &g, unsigned c, int k) {
        if (!ed) return;
        g.f = __ldg(f + c + de);
        g.o = HAS_O ? __ldg(od + c + de) : wd;
        if constexpr (POST) g.e = __ldg(e + par(k) + pe);
    };
    MgCol<V, WK> col;
    col.start(a, L, s, k0);
    unsigned c = s.c + (unsigned)(k0 - kb) * sz;
    Raw rc, rn, ro;
    Edge g;
    float vm[V], vc[V];
    const int klast = min(k1, L.nz - 1);  // the last plane read
    fetch(rc, c, par(k0) + p0);
    if (s.eo) fetch(ro, c + s.dro, par(k0) + po);
    edge(g, c, k0);
    if (k0 + 1 <= klast) fetch(rn, c + sz, par(k0 + 1) + p0);
#pragma unroll
    for (int m = 0; m < V; ++m) vm[m] = 0.f;
    if (k0 > 0) {
        Raw rm;
        fetch(rm, c - sz, par(k0 - 1) + p0);
        iterate(rm, vm);
    }
    iterate(rc, vc);
    const int64_t cb = (int64_t)kb * sz;
#pragma unroll 1
    for (int k = k0; k < k1; ++k, c += sz) {
        Raw r2, ron;
        Edge gn;
        if (k + 2 <= klast) fetch(r2, c + 2 * sz, par(k + 2) + p0);
        if (k + 1 < k1) {
            if (s.eo) fetch(ron, c + sz + s.dro, par(k + 1) + po);
            edge(gn, c + sz, k + 1);
        }
        col.plane(a, L, s, cb, c, k);
        float vn[V], vo[V], vi[V];
#pragma unroll
        for (int m = 0; m < V; ++m) vn[m] = vo[m] = 0.f;
        if (k + 1 < L.nz) iterate(rn, vn);
        if (s.eo) iterate(ro, vo);
        const float ve = form(g.f, g.o, g.e);
#pragma unroll
        for (int m = 0; m < V; ++m) vi[m] = __shfl_xor_sync(0xffffffffu, vc[m], 16);
        const float xls = __shfl_up_sync(0xffffffffu, vc[V - 1], 1), xrs = __shfl_down_sync(0xffffffffu, vc[0], 1);
        const float xl = s.xl0 ? 0.f : s.el ? ve : xls, xr = s.xr0 ? 0.f : s.er ? ve : xrs;
        float av[V];
#pragma unroll
        for (int m = 0; m < V; ++m) {
            float w[6], D;
            col.get(a, m, w, D);
            const float xm = m == 0 ? xl : vc[m > 0 ? m - 1 : 0], xp = m == V - 1 ? xr : vc[m < V - 1 ? m + 1 : 0];
            if constexpr (IT == I_P || IT == I_V) {
                float q = w[0] * (vc[m] - xm);
                q = fmaf(w[1], vc[m] - xp, q);
                q = fmaf(w[2], vc[m] - vi[m], q);
                q = fmaf(w[3], vc[m] - vo[m], q);
                q = fmaf(w[4], vc[m] - vm[m], q);
                av[m] = fmaf(w[5], vc[m] - vn[m], q);
            } else {
                float off = w[0] * xm;
                off = fmaf(w[1], xp, off);
                off = fmaf(w[2], vi[m], off);
                off = fmaf(w[3], vo[m], off);
                off = fmaf(w[4], vm[m], off);
                off = fmaf(w[5], vn[m], off);
                av[m] = fmaf(D, vc[m], -off);
            }
        }
        body(k, cb, c, av, vc, rc.f, rc.o);
#pragma unroll
        for (int m = 0; m < V; ++m) {
            vm[m] = vc[m];
            vc[m] = vn[m];
        }
        rc = rn;
        rn = r2;
        ro = ron;
        g = gn;
    }
}

// The level kernels' work: blocks of kMgThreads / 2 segments times planes
// (coarse ones for the restriction), `planes` per block of segments, split
// evenly over the grid's CTAs as runs of planes; fn(block of segments, planes
// [k0, k1)) per run.
template <typename F>
__device__ __forceinline__ void mg_runs(const MgLevel &L, int seg, int planes, F fn) {
    const int64_t np = (int64_t)(L.nx / seg) * (L.ny / 2), units = (np + kMgThreads / 2 - 1) / (kMgThreads / 2) * planes;
    int64_t u = units * blockIdx.x / gridDim.x;
    const int64_t u1 = units * (blockIdx.x + 1) / gridDim.x;
    unsigned blk = (unsigned)(u / planes);
    int k = (int)(u - (int64_t)blk * planes);
    while (u < u1) {
        const int n = (int)min(min((int64_t)(planes - k), u1 - u), kMgRunPoints / ((int64_t)L.nx * L.ny) + 1);
        fn(blk * (kMgThreads / 32) + (threadIdx.x >> 5), k, k + n);
        u += n;
        k += n;
        if (k == planes) {
            k = 0;
            ++blk;
        }
    }
}

// One warp's restriction of the coarse planes [K0, K1) of its segments.
template <int V, int WK>
__device__ __forceinline__ void mg_restrict_warp(const MgStep &a, unsigned wseg, int K0, int K1) {
    const int cnx = a.L.nx / 2;
    const int64_t csz = (int64_t)cnx * (a.L.ny / 2);
    const MgSeg<V> s(a.L, wseg);
    float sum[V / 2];
    float *fc = a.c + (int64_t)(s.j >> 1) * cnx + (s.i0 >> 1);
    mg_march<V, WK, I_U>(a, a.L.f, a.L.od, 0.f, false, s, 2 * K0, 2 * K1,
                                 [&](int k, int64_t, unsigned, const float *av, const float *, const float *f, const float *) {
                                     float r[V / 2];
#pragma unroll
                                     for (int m = 0; m < V / 2; ++m) {
                                         r[m] = (f[2 * m] - av[2 * m]) + (f[2 * m + 1] - av[2 * m + 1]);
                                         r[m] += __shfl_xor_sync(0xffffffffu, r[m], 16);
                                     }
                                     if (!(k & 1)) {
#pragma unroll
                                         for (int m = 0; m < V / 2; ++m) sum[m] = r[m];
                                         return;
                                     }
                                     if (!s.live || s.hi) return;
                                     float *o = fc + (k >> 1) * csz;
                                     if constexpr (V == 4)
                                         *reinterpret_cast<float2 *>(o) = make_float2(sum[0] + r[0], sum[1] + r[1]);
                                     else
                                         o[0] = sum[0] + r[0];
                                 });
}

// One warp's post-smoothing of the planes [k0, k1) of its segments; DOT: its
// points' f.out go into acc, compensated, for a thread may hold hundreds of
// terms (215 at 256^3, more on larger grids).
template <int V, int WK, bool DOT>
__device__ __forceinline__ void mg_post_warp(const MgStep &a, unsigned wseg, int k0, int k1, KahanF &acc) {
    const MgSeg<V> s(a.L, wseg);
    float *out = a.L.w;
    mg_march<V, WK, I_POST>(a, a.L.f, a.L.od, 0.f, false, s, k0, k1,
                                [&](int, int64_t cb, unsigned c, const float *av, const float *v, const float *f, const float *o) {
                                    float r[V];
#pragma unroll
                                    for (int m = 0; m < V; ++m) r[m] = fmaf(o[m], f[m] - av[m], v[m]);
                                    if (!s.live) return;
                                    if constexpr (V == 4) {
                                        *reinterpret_cast<float4 *>(out + cb + c) = make_float4(r[0], r[1], r[2], r[3]);
                                    } else {
                                        *reinterpret_cast<float2 *>(out + cb + c) = make_float2(r[0], r[1]);
                                    }
                                    if constexpr (DOT) {
                                        float t = f[0] * r[0];
#pragma unroll
                                        for (int m = 1; m < V; ++m) t = fmaf(f[m], r[m], t);
                                        acc.add(t);
                                    }
                                });
}

// f_{l+1} = P^T (f - A u), u = (omega / D) f; 
template <int V, int WK>
__global__ void __launch_bounds__(kMgThreads, mg_min_blocks(WK)) mg_restrict_kernel(const MgStep a) {
    if (mg_stand_down(a.st)) return;
    mg_runs(a.L, V, a.L.nz / 2, [&](unsigned wseg, int K0, int K1) { mg_restrict_warp<V, WK>(a, wseg, K0, K1); });
}

// The scalars a V-cycle inside a solve ends with: r.z -> beta (the first time
// only r.z), breakdown, the loop condition.
struct MgDot {
    SolveState *st;
    double *partials;
    int init;
    cudaGraphConditionalHandle cond;
    int use_cond;
};
__device__ __forceinline__ void mg_rz_finish(const MgDot &d, double rz) {
    SolveState *st = d.st;
    if (!isfinite(rz) || !(rz > 0.0)) {
        st->done = 1;
        st->status = GBPCG_BREAKDOWN;
    } else {
        if (!d.init) st->beta = rz / st->rzm;
        st->rz = rz;
        st->rzm = rz;
    }
    if (d.use_cond) cudaGraphSetConditional(d.cond, st->done ? 0u : 1u);
}

// out = u' + omega D^-1 (f - A u'), u' = u + sigma P e with e the level-(l+1)
// result.  DOT (level 0 inside a solve): also f.out, r.z of the solver,
// instead of a pass of its own over both vectors.
template <int V, int WK, bool DOT>
__global__ void __launch_bounds__(kMgThreads, mg_min_blocks(WK)) mg_post_kernel(const MgStep a, const MgDot d) {
    if (mg_stand_down(a.st)) return;
    KahanF sum;
    mg_runs(a.L, V, a.L.nz, [&](unsigned wseg, int k0, int k1) { mg_post_warp<V, WK, DOT>(a, wseg, k0, k1, sum); });
    if constexpr (DOT) {
        const float acc[1] = {(float)sum.value()};
        double part[1], tot[1];
        block_sum<1, kMgThreads>(acc, part);
        if (grid_sum_last<1, kMgThreads>(part, d.partials, &d.st->ticket[1], tot) && threadIdx.x == 0)
            mg_rz_finish(d, tot[0]);
    }
}

// The solver's passes A and R on the same march, for grids on which the
// passes' TMA ring is a chain of planes in a few CTAs (kMgDirectPoints).
//   A: p_k = z + beta p_{k-1} (p_out), d += alpha_{k-1} p_{k-1}, p.Ap -> alpha
//   R: r -= alpha A p_k, r.r -> convergence test and replacement trigger
struct MgPass {
    float *p0, *p1, *d, *r;
    SolveState *st;
    double *partials;
    cudaGraphConditionalHandle cond, cond_rep;
    int use_cond;
};
template <int WK, bool A>
__global__ void __launch_bounds__(kMgThreads, mg_min_blocks(WK)) mg_pass_kernel(const MgStep a, const MgPass d) {
    SolveState *st = d.st;
    if (mg_stand_down(st)) return;
    const int it = st->it;
    const float alpha = (float)st->alpha, beta = (float)st->beta;  // A: alpha_{k-1}
    const bool pending = st->pending != 0;
    float *pk = it & 1 ? d.p1 : d.p0;
    const float *pp = it & 1 ? d.p0 : d.p1;
    float acc[1] = {0.f};
    mg_runs(a.L, 4, a.L.nz, [&](unsigned wseg, int k0, int k1) {
        const MgSeg<4> s(a.L, wseg);
        if constexpr (A) {
            mg_march<4, WK, I_P>(a, a.L.f, pp, beta, it == 0, s, k0, k1,
                                 [&](int, int64_t cb, unsigned c, const float *av, const float *v, const float *, const float *o) {
                                     if (!s.live) return;
                                     *reinterpret_cast<float4 *>(pk + cb + c) = make_float4(v[0], v[1], v[2], v[3]);
#pragma unroll
                                     for (int m = 0; m < 4; ++m) acc[0] = fmaf(v[m], av[m], acc[0]);
                                     if (!pending) return;
                                     float4 *dp = reinterpret_cast<float4 *>(d.d + cb + c);
                                     const float4 t = *dp;
                                     *dp = make_float4(fmaf(alpha, o[0], t.x), fmaf(alpha, o[1], t.y),
                                                       fmaf(alpha, o[2], t.z), fmaf(alpha, o[3], t.w));
                                 });
        } else {
            mg_march<4, WK, I_V>(a, pk, nullptr, 0.f, false, s, k0, k1,
                                 [&](int, int64_t cb, unsigned c, const float *av, const float *, const float *, const float *) {
                                     if (!s.live) return;
                                     float4 *rp = reinterpret_cast<float4 *>(d.r + cb + c);
                                     const float4 t = *rp;
                                     const float r[4] = {fmaf(-alpha, av[0], t.x), fmaf(-alpha, av[1], t.y),
                                                         fmaf(-alpha, av[2], t.z), fmaf(-alpha, av[3], t.w)};
                                     *rp = make_float4(r[0], r[1], r[2], r[3]);
#pragma unroll
                                     for (int m = 0; m < 4; ++m) acc[0] = fmaf(r[m], r[m], acc[0]);
                                 });
        }
    });
    double part[1], tot[1];
    block_sum<1, kMgThreads>(acc, part);
    if (!grid_sum_last<1, kMgThreads>(part, d.partials, &st->ticket[A ? K_PASSA : K_PASSR], tot) || threadIdx.x != 0)
        return;
    if constexpr (A) passa_finish(st, tot[0], false);
    else passr_finish(st, it, tot[0], false);
    if (d.use_cond) {
        cudaGraphSetConditional(d.cond, st->done ? 0u : 1u);
        cudaGraphSetConditional(d.cond_rep, st->replace ? 1u : 0u);
    }
}

// ------------------------------------------------------------ the tail --
//
// The levels of at most kMgTailCells cells in one launch of one CTA: on such
// levels a launch costs more than its work.  Weights and omega / D of all of
// them lie in one block of memory and are brought into shared memory by one
// copy; the vectors stay there.  A pass over a level in one SM is bound by
// its shared-memory reads, so the passes run over flat indices, two cells a
// thread, without decoding (i, j, k): halo planes of zeros around u and the
// zero weights of boundary faces make every neighbour read harmless.  Only
// the transfers between levels decode, one coarse cell a thread.  The launch's
// parameters are kept to a line or two of the constant cache, which is cold:
// as an array of levels they took 11000 cycles to read, a miss after another.
// 16^3 and below: 36 us with the levels in global memory -> 11.5 us (ncu;
// 15700 cycles: copies 4000, 16^3 7800, 8^3 900, 24 sweeps 2970).

struct MgTail {
    const SolveState *st;
    const float *wts;   // per level w+x, w+y, w+z, D, omega / D (m values each)
    const float *f;     // the first level's right-hand side
    float *w;           // and its result
    int nl;             // levels before the coarsest
    int nx, ny, nz;     // the first level's size
    int nwts;           // floats of wts
};

// What sweeps a coarsest level that is the whole tail: one CTA, or above
// kMgTailCells cells a cluster, its halo planes exchanged through distributed
// shared memory (31^3 cells, the coarsest level of 248^3: 700 us in one CTA with
// the vectors in global memory -> 35 us).
struct MgSweep {
    int ppc, na;  // planes per CTA, sweeping CTAs
    unsigned ctas;
    size_t smem;  // 0: in global memory
};

__device__ __forceinline__ void cluster_barrier() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// (i, j, k) of flat cell c of a level (32-bit: the tail's levels are small)
__device__ __forceinline__ void mg_cell(int nx, int ny, int c, int &i, int &j, int &k) {
    const int t = c / nx;
    i = c - t * nx;
    k = t / ny;
    j = t - k * ny;
}

// n floats into shared memory by the CTA (dst 16-byte aligned); wait with mg_copy_wait
__device__ __forceinline__ void mg_copy(float *dst, const float *src, int n) {
    const uint32_t d = smem_u32(dst);
    const int n4 = (reinterpret_cast<uintptr_t>(src) & 15) == 0 ? n & ~3 : 0;
    for (int i = threadIdx.x * 4; i < n4; i += kMgTailThreads * 4)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 4u * i), "l"(src + i) : "memory");
    for (int i = n4 + threadIdx.x; i < n; i += kMgTailThreads)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d + 4u * i), "l"(src + i) : "memory");
}
__device__ __forceinline__ void mg_copy_wait() {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
}

// A level of the tail in shared memory: offsets in floats.  u has a plane of
// zeros on either side (so what a weight array's neighbour read finds before
// its first element only has to be finite); g is the residual on the way down
// and the result on the way up.
struct MgSm {
    int nx, ny, pl, m;
    int u, wx, wy, wz, D, od, f, g;
};
__host__ __device__ inline int mg_round4(int n) { return (n + 3) & ~3; }
// the coarsest level: wx, wy, wz, D, f, g and the sweeps' two buffers in u
__host__ __device__ inline MgSm mg_sm_level(int nx, int ny, int nz, bool coarsest, int &wat, int &at) {
    MgSm s;
    s.nx = nx;
    s.ny = ny;
    s.pl = nx * ny;
    s.m = s.pl * nz;
    s.wx = wat;
    s.wy = s.wx + s.m;
    s.wz = s.wy + s.m;
    s.D = s.wz + s.m;
    s.od = s.D + s.m;
    wat += 5 * s.m;
    s.u = at + mg_round4(s.pl);
    at = s.u + mg_round4(s.m) + (coarsest ? 2 * mg_round4(s.pl) + s.m + s.pl : s.pl);
    at = mg_round4(at);
    s.f = at;
    s.g = at + mg_round4(s.m);
    at = s.g + mg_round4(s.m);
    return s;
}

// (f - A u) (UP: u + omega D^-1 (f - A u)) of a level into out
template <bool UP>
__device__ __forceinline__ void mg_sm_residual(const float *sm, const MgSm &s, float *out) {
    auto ld2 = [&](int o) { return *reinterpret_cast<const float2 *>(sm + o); };
    const int nx = s.nx, pl = s.pl;
    for (int c = 2 * threadIdx.x; c < s.m; c += 2 * kMgTailThreads) {
        const float2 u = ld2(s.u + c), ym = ld2(s.u + c - nx), yp = ld2(s.u + c + nx), zm = ld2(s.u + c - pl),
                     zp = ld2(s.u + c + pl), x = ld2(s.wx + c), y0 = ld2(s.wy + c - nx), y1 = ld2(s.wy + c),
                     z0 = ld2(s.wz + c - pl), z1 = ld2(s.wz + c), D = ld2(s.D + c), f = ld2(s.f + c);
        const float ul = sm[s.u + c - 1], ur = sm[s.u + c + 2], xl = sm[s.wx + c - 1];
        float a = fmaf(x.x, u.y, xl * ul), b = fmaf(x.y, ur, x.x * u.x);
        a = fmaf(y0.x, ym.x, a);
        b = fmaf(y0.y, ym.y, b);
        a = fmaf(y1.x, yp.x, a);
        b = fmaf(y1.y, yp.y, b);
        a = fmaf(z0.x, zm.x, a);
        b = fmaf(z0.y, zm.y, b);
        a = fmaf(z1.x, zp.x, a);
        b = fmaf(z1.y, zp.y, b);
        a = f.x - fmaf(D.x, u.x, -a);
        b = f.y - fmaf(D.y, u.y, -b);
        if (UP) {
            const float2 o = ld2(s.od + c);
            a = fmaf(o.x, a, u.x);
            b = fmaf(o.y, b, u.y);
        }
        out[c] = a;
        out[c + 1] = b;
    }
}

// fn(coarse cell, flat index of its first fine cell) for every coarse cell of a level
template <typename F>
__device__ __forceinline__ void mg_sm_coarse(const MgSm &s, F fn) {
    const int cnx = s.nx / 2, cny = s.ny / 2, cm = s.m / 8;
    for (int cc = threadIdx.x; cc < cm; cc += kMgTailThreads) {
        int I, J, K;
        mg_cell(cnx, cny, cc, I, J, K);
        fn(cc, (2 * K * s.ny + 2 * J) * s.nx + 2 * I);
    }
}

// The coarsest level of a tail of several levels (at most a cell a thread):
// kMgCoarseSweeps damped Jacobi sweeps from zero, into g.  Only the warps with
// cells take part; the buffers' halo planes are zero.
__device__ __forceinline__ void mg_sm_sweeps(float *sm, const MgSm &s) {
    const int c = threadIdx.x, nthr = (s.m + 31) / 32 * 32, nx = s.nx, pl = s.pl;
    if (c >= nthr) return;  // the caller's barrier follows
    const int stride = mg_round4(s.m) + 2 * mg_round4(pl) - (mg_round4(pl) - pl);
    const bool on = c < s.m;
    const int q = on ? c : 0;
    const float w0 = sm[s.wx + q - 1], w1 = sm[s.wx + q], w2 = sm[s.wy + q - nx], w3 = sm[s.wy + q],
                w4 = sm[s.wz + q - pl], w5 = sm[s.wz + q], D = sm[s.D + q], f = sm[s.f + q], o = kMgOmega / D;
    float *b0 = sm + s.u + q, *b1 = b0 + stride;
    auto sync = [&] {
        __syncwarp();
        asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");
    };
    float v = o * f;
    if (on) *b0 = v;
    sync();
    auto sweep = [&](const float *p) {
        const float a = fmaf(w2, p[-nx], w0 * p[-1]), b = fmaf(w3, p[nx], w1 * p[1]), d = fmaf(w5, p[pl], w4 * p[-pl]);
        v = fmaf(o, f - fmaf(D, v, -((a + b) + d)), v);
    };
    for (int t = 1; t + 1 < kMgCoarseSweeps; t += 2) {
        sweep(b0);
        if (on) *b1 = v;
        sync();
        sweep(b1);
        if (on) *b0 = v;
        sync();
    }
    if (kMgCoarseSweeps % 2 == 0) sweep(b0);
    if (on) sm[s.g + c] = v;
}

// coarsest level: kMgCoarseSweeps damped Jacobi sweeps from zero; the result
// lands in L.w.  CTA `rank` of t.na sweeps t.ppc planes, kept twice in
// shared memory with a halo plane on either side; a CTA writes its first and
// last plane into the neighbours' halos as it computes them.  Weights of up
// to NC cells a thread stay in registers (NC = 0: they are read each sweep).
template <int NC>
__device__ __forceinline__ void mg_sweeps(const MgArgs &a, const MgSweep &t, int rank, float *sm) {
    const MgLevel L = a.lv[a.L - 1];
    const bool lvl0 = a.L == 1;
    const int nx = L.nx, pl = L.nx * L.ny, ppc = t.ppc, na = t.na;
    const int k0 = rank * ppc, planes = max(0, min(L.nz - k0, ppc)), n = planes * pl;
    const int stride = (ppc + 2) * pl;
    const uint32_t sbase = smem_u32(sm);
    // one CTA: only the warps with cells take part
    const int nthr = min((n + 31) / 32 * 32, kMgTailThreads);
    auto sync = [&] {
        __syncwarp();
        if (na > 1) cluster_barrier();
        else asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");
    };
    auto remote = [&](int r, int which, int idx) {
        uint32_t ra;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(sbase + 4u * (uint32_t)(which * stride + idx)), "r"(r));
        return ra;
    };
    auto put = [&](int which, int c, float v) {
        sm[which * stride + pl + c] = v;
        if (na == 1) return;
        if (c < pl && rank > 0)  // the halo after the previous CTA's (full) planes
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote(rank - 1, which, (ppc + 1) * pl + c)), "f"(v) : "memory");
        if (c >= n - pl && rank + 1 < na)
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote(rank + 1, which, c - (n - pl))), "f"(v) : "memory");
    };
    for (int q = threadIdx.x; q < 2 * stride; q += kMgTailThreads) sm[q] = 0.f;
    if (na > 1) cluster_barrier();
    else __syncthreads();
    if (na == 1 && (int)threadIdx.x >= nthr) return;  // the caller's barrier follows
    constexpr int NR = NC > 0 ? NC : 1;
    float w[NR][6], D[NR], o[NR], f[NR];
    auto load = [&](int c, float (&ww)[6], float &DD, float &oo, float &ff) {
        int i, j, k;
        mg_cell(nx, L.ny, c, i, j, k);
        if (lvl0) mg_weights(a, 0, i, j, k + k0, ww, DD);
        else mg_weights_stored(L, i, j, k + k0, ww, DD);
        ff = L.f[k0 * pl + c];
        oo = kMgOmega / DD;
    };
    auto point = [&](const float *s, int c, const float (&ww)[6], float DD, float oo, float ff) {
        const float *p = s + pl + c;
        float off = ww[0] * p[-1];
        off = fmaf(ww[1], p[1], off);
        off = fmaf(ww[2], p[-nx], off);
        off = fmaf(ww[3], p[nx], off);
        off = fmaf(ww[4], p[-pl], off);
        off = fmaf(ww[5], p[pl], off);
        return fmaf(oo, ff - fmaf(DD, p[0], -off), p[0]);
    };
    float *res = L.w + k0 * pl;
    auto cells = [&](auto fn) {
        if constexpr (NC > 0) {
#pragma unroll
            for (int m = 0; m < NC; ++m) {
                const int c = threadIdx.x + m * kMgTailThreads;
                if (c < n) fn(m, c);
            }
        } else {
            for (int c = threadIdx.x; c < n; c += kMgTailThreads) fn(0, c);
        }
    };
    cells([&](int m, int c) {
        load(c, w[m], D[m], o[m], f[m]);
        put(0, c, o[m] * f[m]);
    });
    sync();
    for (int sweep = 1; sweep < kMgCoarseSweeps - 1; ++sweep) {
        const float *src = sm + ((sweep - 1) & 1) * stride;
        cells([&](int m, int c) {
            if constexpr (NC == 0) load(c, w[0], D[0], o[0], f[0]);
            put(sweep & 1, c, point(src, c, w[m], D[m], o[m], f[m]));
        });
        sync();
    }
    cells([&](int m, int c) {
        if constexpr (NC == 0) load(c, w[0], D[0], o[0], f[0]);
        res[c] = point(sm + (kMgCoarseSweeps & 1) * stride, c, w[m], D[m], o[m], f[m]);
    });
}
static_assert(kMgCoarseSweeps >= 2, "first and last sweep");

// The same sweeps by one CTA in global memory (od and w of the coarsest level
// in turn): a grid of one level whose planes are too large for the shared
// memory (nz < 4).
__device__ __forceinline__ void mg_sweeps_flat(const MgArgs &a) {
    const int l = a.L - 1;
    const MgLevel &L = a.lv[l];
    const int n = (int)L.m, sy = L.nx, sz = L.nx * L.ny;
    float *src = kMgCoarseSweeps % 2 ? L.w : L.od, *dst = kMgCoarseSweeps % 2 ? L.od : L.w;
    for (int sweep = 0; sweep < kMgCoarseSweeps; ++sweep) {
        float *out = sweep == 0 ? src : dst;
        for (int c = threadIdx.x; c < n; c += kMgTailThreads) {
            int i, j, k;
            mg_cell(L.nx, L.ny, c, i, j, k);
            float w[6], D;
            mg_weights(a, l, i, j, k, w, D);
            const float o = kMgOmega / D;
            if (sweep == 0) {
                out[c] = o * L.f[c];
                continue;
            }
            float off = 0.f;
            if (i > 0) off = fmaf(w[0], src[c - 1], off);
            if (i + 1 < L.nx) off = fmaf(w[1], src[c + 1], off);
            if (j > 0) off = fmaf(w[2], src[c - sy], off);
            if (j + 1 < L.ny) off = fmaf(w[3], src[c + sy], off);
            if (k > 0) off = fmaf(w[4], src[c - sz], off);
            if (k + 1 < L.nz) off = fmaf(w[5], src[c + sz], off);
            out[c] = fmaf(o, L.f[c] - fmaf(D, src[c], -off), src[c]);
        }
        __syncthreads();
        if (sweep > 0) {
            float *tmp = src;
            src = dst;
            dst = tmp;
        }
    }
}

__global__ void __launch_bounds__(kMgTailThreads) mg_sweep_kernel(const MgArgs a, const MgSweep t) {
    extern __shared__ __align__(16) float mg_sm[];
    if (mg_stand_down(a.st)) return;  // the same for the whole cluster
    if (t.smem == 0) {                // one CTA
        mg_sweeps_flat(a);
        return;
    }
    const int n = t.ppc * a.lv[a.L - 1].nx * a.lv[a.L - 1].ny, rank = (int)blockIdx.x;
    if (n <= kMgTailThreads) mg_sweeps<1>(a, t, rank, mg_sm);
    else if (n <= kMgSweepCells * kMgTailThreads) mg_sweeps<kMgSweepCells>(a, t, rank, mg_sm);
    else mg_sweeps<0>(a, t, rank, mg_sm);
    if (t.na > 1) cluster_barrier();  // no CTA leaves while its halos can still be written
}

__global__ void __launch_bounds__(kMgTailThreads) mg_tail_kernel(const MgTail t) {
    extern __shared__ __align__(16) float mg_sm[];
    if (mg_stand_down(t.st)) return;
    const int tid = threadIdx.x;
    if (tid < 4) mg_sm[tid] = 0.f;  // before the weights: finite
    mg_copy(mg_sm + 4, t.wts, t.nwts);
    MgSm lv[kMgTailLevels];
    int wat = 4, at = 4 + mg_round4(t.nwts);
#pragma unroll
    for (int q = 0; q < kMgTailLevels; ++q)
        if (q <= t.nl) {
            lv[q] = mg_sm_level(t.nx >> q, t.ny >> q, t.nz >> q, q == t.nl, wat, at);
            const MgSm &s = lv[q];
            // zeros around u (the coarsest: its two buffers)
            if (q < t.nl) {
                for (int i = tid; i < s.pl; i += kMgTailThreads) mg_sm[s.u - s.pl + i] = mg_sm[s.u + s.m + i] = 0.f;
            } else {
                for (int i = s.u - s.pl + tid; i < s.f; i += kMgTailThreads) mg_sm[i] = 0.f;
            }
        }
    mg_copy(mg_sm + lv[0].f, t.f, lv[0].m);
    mg_copy_wait();
    for (int c = tid; c < lv[0].m; c += kMgTailThreads) mg_sm[lv[0].u + c] = mg_sm[lv[0].f + c] * mg_sm[lv[0].od + c];
    __syncthreads();
#pragma unroll
    for (int q = 0; q + 1 < kMgTailLevels; ++q)
        if (q < t.nl) {
            const MgSm &s = lv[q], &C = lv[q + 1];
            const bool next = q + 1 < t.nl;
            mg_sm_residual<false>(mg_sm, s, mg_sm + s.g);
            __syncthreads();
            mg_sm_coarse(s, [&](int cc, int c) {
                const float *g = mg_sm + s.g + c;
                const float a0 = g[0] + g[1], a1 = g[s.nx] + g[s.nx + 1];
                const float b0 = g[s.pl] + g[s.pl + 1], b1 = g[s.pl + s.nx] + g[s.pl + s.nx + 1];
                const float r = (a0 + a1) + (b0 + b1);
                mg_sm[C.f + cc] = r;
                if (next) mg_sm[C.u + cc] = r * mg_sm[C.od + cc];
            });
            __syncthreads();
        }
#pragma unroll
    for (int q = 1; q < kMgTailLevels; ++q)
        if (q == t.nl) mg_sm_sweeps(mg_sm, lv[q]);
    __syncthreads();
#pragma unroll
    for (int q = kMgTailLevels - 2; q >= 0; --q)
        if (q < t.nl) {
            const MgSm &s = lv[q];
            const int e = lv[q + 1].g;
            mg_sm_coarse(s, [&](int cc, int c) {
                float *u = mg_sm + s.u + c;
                const float v = mg_sm[e + cc];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    float *p = u + (r & 1) * s.nx + (r >> 1) * s.pl;
                    p[0] = fmaf(kMgSigma, v, p[0]);
                    p[1] = fmaf(kMgSigma, v, p[1]);
                }
            });
            __syncthreads();
            if (q > 0) {
                mg_sm_residual<true>(mg_sm, s, mg_sm + s.g);
                __syncthreads();
            } else {
                mg_sm_residual<true>(mg_sm, s, t.w);
            }
        }
}

// Level 0 inside the tail: its weights in the coarse levels' stored form
__global__ void __launch_bounds__(kMgThreads) mg_store0_kernel(const MgArgs a, float *W) {
    const MgLevel &L = a.lv[0];
    for (int c = blockIdx.x * kMgThreads + threadIdx.x; c < (int)L.m; c += gridDim.x * kMgThreads) {
        int i, j, k;
        mg_cell(L.nx, L.ny, c, i, j, k);
        float w[6], D;
        mg_weights(a, 0, i, j, k, w, D);
        W[c] = w[1];
        W[c + L.m] = w[3];
        W[c + 2 * L.m] = w[5];
        W[c + 3 * L.m] = D;
    }
}

// Galerkin coarsening of level l into level l + 1 (one thread per coarse
// cell), and omega / D of level l's points into its od (NULL: not used)
__global__ void __launch_bounds__(kMgThreads) mg_galerkin_kernel(const MgArgs a, int l, float *Wc, float *od, int zper) {
    const MgLevel &L = a.lv[l], &C = a.lv[l + 1];
    const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
    if (I >= C.nx || J >= C.ny) return;
    const int K0 = blockIdx.z * zper, K1 = min(C.nz, K0 + zper);
    for (int K = K0; K < K1; ++K) {
        float sx = 0.f, sy = 0.f, sz = 0.f, sD = 0.f, inner = 0.f;
        for (int dz = 0; dz < 2; ++dz)
            for (int dy = 0; dy < 2; ++dy) {
                float o[2];
#pragma unroll
                for (int dx = 0; dx < 2; ++dx) {
                    float w[6], D;
                    mg_weights(a, l, 2 * I + dx, 2 * J + dy, 2 * K + dz, w, D);
                    o[dx] = kMgOmega / D;
                    sD += D;
                    if (dx == 1) sx += w[1]; else inner += w[1];
                    if (dy == 1) sy += w[3]; else inner += w[3];
                    if (dz == 1) sz += w[5]; else inner += w[5];
                }
                if (od)
                    *reinterpret_cast<float2 *>(od + ((int64_t)(2 * K + dz) * L.ny + 2 * J + dy) * L.nx + 2 * I) =
                        make_float2(o[0], o[1]);
            }
        const int64_t c = ((int64_t)K * C.ny + J) * C.nx + I;
        Wc[c] = sx;
        Wc[c + C.m] = sy;
        Wc[c + 2 * C.m] = sz;
        Wc[c + 3 * C.m] = sD - 2.0f * inner;
    }
}

// r.z in a pass of its own, where the tail holds the whole hierarchy
__global__ void __launch_bounds__(kMgThreads)
    mg_rz_kernel(int64_t n, const float *__restrict__ r, const float *__restrict__ z, const MgDot d) {
    if (mg_stand_down(d.st)) return;
    float acc[1] = {0.f};
    for (int64_t i = (int64_t)blockIdx.x * kMgThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kMgThreads)
        acc[0] = fmaf(r[i], z[i], acc[0]);
    double part[1], tot[1];
    block_sum<1, kMgThreads>(acc, part);
    if (!grid_sum_last<1, kMgThreads>(part, d.partials, &d.st->ticket[1], tot) || threadIdx.x != 0) return;
    mg_rz_finish(d, tot[0]);
}

// ---------------------------------------------------------- host side --

struct MgGeom {
    int L;
    int nx[kMgMaxLevels], ny[kMgMaxLevels], nz[kMgMaxLevels];
};

MgGeom mg_geom(const gbpcg_grid &g) {
    MgGeom m;
    m.L = 1;
    m.nx[0] = g.nx; m.ny[0] = g.ny; m.nz[0] = g.nz;
    while (m.L < kMgMaxLevels) {
        const int l = m.L - 1;
        const int a = m.nx[l], b = m.ny[l], c = m.nz[l];
        if (a % 2 || b % 2 || c % 2 || a / 2 < kMgMinCoarse || b / 2 < kMgMinCoarse || c / 2 < kMgMinCoarse) break;
        m.nx[m.L] = a / 2; m.ny[m.L] = b / 2; m.nz[m.L] = c / 2;
        ++m.L;
    }
    return m;
}

// workspace pieces beyond the Jacobi solver's: r, per coarse level f and w, the
// block of all levels' weights and omega / D (level by level, w+x, w+y, w+z, D,
// omega / D; level 0 only where it is inside the tail), and omega / D of a
// level 0 above the tail
struct MgLayout {
    WsLayout base;
    size_t r, od0, f[kMgMaxLevels], w[kMgMaxLevels], wts[kMgMaxLevels];
    size_t total;
};

MgLayout mg_layout(const gbpcg_grid &g, int io) {
    const size_t n = (size_t)g.nx * g.ny * g.nz;
    MgLayout M;
    M.base = ws_layout_n(n, GBPCG_F32, io, false, block_count(g));
    size_t o = M.base.total;
    M.r = o; o += round256(n * 4);
    M.od0 = o;
    if ((int64_t)n > kMgTailCells) o += round256(n * 4);
    const MgGeom G = mg_geom(g);
    auto cells = [&](int l) { return (size_t)G.nx[l] * G.ny[l] * G.nz[l]; };
    for (int l = 1; l < G.L; ++l) {
        M.f[l] = o; o += round256(cells(l) * 4);
        M.w[l] = o; o += round256(cells(l) * 4);
    }
    for (int l = (int64_t)n > kMgTailCells ? 1 : 0; l < G.L; ++l) {
        M.wts[l] = o;
        o += cells(l) * 20;  // every level but the coarsest holds a multiple of 8 cells: 16-byte arrays
    }
    M.total = round256(o);
    return M;
}

MgArgs mg_args(const gbpcg_grid &g, char *ws, const MgLayout &M, float *f0, float *z, const SolveState *st) {
    const MgGeom G = mg_geom(g);
    MgArgs a;
    memset(&a, 0, sizeof(a));
    a.L = G.L;
    for (int l = 0; l < G.L; ++l) {
        MgLevel &L = a.lv[l];
        L.nx = G.nx[l]; L.ny = G.ny[l]; L.nz = G.nz[l];
        L.m = (int64_t)L.nx * L.ny * L.nz;
        L.f = l == 0 ? f0 : reinterpret_cast<float *>(ws + M.f[l]);
        L.w = l == 0 ? z : reinterpret_cast<float *>(ws + M.w[l]);
        if (l > 0 || L.m <= kMgTailCells) {
            L.wx = reinterpret_cast<const float *>(ws + M.wts[l]);
            L.wy = L.wx + L.m;
            L.wz = L.wy + L.m;
            L.D = L.wz + L.m;
            L.od = const_cast<float *>(L.D + L.m);
        } else {
            L.od = reinterpret_cast<float *>(ws + M.od0);
        }
    }
    a.block = g.k_block ? 1 : 0;
    a.tab = g.k_block ? reinterpret_cast<const float4 *>(ws + M.base.tab) : nullptr;
    if (g.k_block) {
        a.rkbx = 1.0f / (float)g.kbx;
        a.rkby = 1.0f / (float)g.kby;
        a.rkbz = 1.0f / (float)g.kbz;
    }
    if (g.k_block) {
        a.ob = make_op_block(g);
    } else {
        memset(&a.ob, 0, sizeof(a.ob));
        auto c = [](int m) { double h = 1.0 / (m + 1); return (float)(1.0 / (h * h)); };
        a.ob.cx = c(g.nx); a.ob.cy = c(g.ny); a.ob.cz = c(g.nz);
    }
    a.st = st;
    return a;
}

unsigned mg_grid(int64_t n) {
    return (unsigned)std::max<int64_t>(
        1, std::min<int64_t>((n + kMgThreads - 1) / kMgThreads, (int64_t)device_sm_count() * 8));
}

// the first level of the tail
int mg_l0(const MgArgs &a) {
    int l0 = a.L - 1;
    while (l0 > 0 && a.lv[l0 - 1].m <= kMgTailCells) --l0;
    return l0;
}

// whether level 0's omega / D is kept per point (constant coefficients above the tail: one number)
bool mg_od0(const MgArgs &a) { return a.block || mg_l0(a) == 0; }

// the coarse operators (once per solve)
cudaError_t mg_setup(const MgArgs &a, cudaStream_t s) {
    if (a.L > 1 && mg_l0(a) == 0)
        mg_store0_kernel<<<mg_grid(a.lv[0].m), kMgThreads, 0, s>>>(a, const_cast<float *>(a.lv[0].wx));
    for (int l = 0; l + 1 < a.L; ++l) {
        const MgLevel &C = a.lv[l + 1];
        const MgLaunch g = mg_launch(C.nx, C.ny, C.nz);
        mg_galerkin_kernel<<<g.grid, g.block, 0, s>>>(a, l, const_cast<float *>(C.wx),
                                                      l > 0 || mg_od0(a) ? a.lv[l].od : nullptr, g.zper);
    }
    return cudaGetLastError();
}

// CTAs of a level kernel: what the device holds at once, and no more than its
// units of work (mg_runs).
template <int V, int WK, int KIND = 0, typename K>
unsigned mg_level_grid(K kernel, const MgLevel &L, int planes) {  // an instance, and so a static, per kernel
    static const int per_sm = [kernel] {
        int n = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, kMgThreads, 0);
        return std::max(1, n);
    }();
    const int64_t np = (int64_t)(L.nx / V) * (L.ny / 2);
    const int64_t units = (np + kMgThreads / 2 - 1) / (kMgThreads / 2) * planes;
    return (unsigned)std::min<int64_t>(std::min<int64_t>(units, kMaxPassBlocks), (int64_t)device_sm_count() * per_sm);
}

// f(V, WK) for a level's row length and kind of weights
template <typename F>
void mg_dispatch(const MgArgs &a, int l, F f) {
    using V4 = std::integral_constant<int, 4>;
    using V2 = std::integral_constant<int, 2>;
    if (l > 0) {
        using Stored = std::integral_constant<int, W_STORED>;
        if (a.lv[l].nx % 4 == 0) f(V4{}, Stored{});
        else f(V2{}, Stored{});
    } else if (!a.block) {
        f(V4{}, std::integral_constant<int, W_CONST0>{});
    } else if (a.ob.kbx % 4 == 0) {
        f(V4{}, std::integral_constant<int, W_TABV>{});
    } else {
        f(V4{}, std::integral_constant<int, W_TAB0>{});
    }
}
MgStep mg_step(const MgArgs &a, int l, float *c) {
    return MgStep{a.st, a.lv[l], c, a.ob, a.tab, a.rkbx, a.rkby, a.rkbz};
}

// z = M f0 (a.lv[0].f -> a.lv[0].w); dot: also r.z and what follows from it
cudaError_t mg_vcycle(const MgArgs &a, cudaStream_t s, const MgDot *dot) {
    const int l0 = mg_l0(a), lc = a.L - 1;
    for (int l = 0; l < l0; ++l)
        mg_dispatch(a, l, [&](auto v, auto wk) {
            const unsigned g = mg_level_grid<v(), wk()>(mg_restrict_kernel<v(), wk()>, a.lv[l], a.lv[l + 1].nz);
            mg_restrict_kernel<v(), wk()><<<g, kMgThreads, 0, s>>>(mg_step(a, l, a.lv[l + 1].f));
        });
    if (l0 < lc) {
        const MgLevel &L = a.lv[l0];
        MgTail t{a.st, L.wx, L.f, L.w, lc - l0, L.nx, L.ny, L.nz, 0};
        int wat = 4, at = 0;
        for (int q = 0; q <= t.nl; ++q) t.nwts += 5 * (int)a.lv[l0 + q].m;
        at = 4 + mg_round4(t.nwts);
        for (int q = 0; q <= t.nl; ++q) (void)mg_sm_level(L.nx >> q, L.ny >> q, L.nz >> q, q == t.nl, wat, at);
        const size_t smem = (size_t)at * sizeof(float);
        if (cudaError_t e = cudaFuncSetAttribute(mg_tail_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMgTailSmem))
            return e;
        mg_tail_kernel<<<1, kMgTailThreads, smem, s>>>(t);
    } else {
        const MgLevel &C = a.lv[lc];
        const bool large = C.m > kMgTailCells;
        MgSweep t;
        t.ppc = large ? (C.nz + kMgTailCtas - 1) / kMgTailCtas : C.nz;
        t.na = (C.nz + t.ppc - 1) / t.ppc;
        t.ctas = large ? kMgTailCtas : 1;
        t.smem = (size_t)2 * (t.ppc + 2) * C.nx * C.ny * sizeof(float);
        if (t.smem > kMgTailSmem) {  // only a single level with nz < 4
            t.smem = 0;
            t.ctas = 1;
        }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(t.ctas);
        cfg.blockDim = dim3(kMgTailThreads);
        cfg.dynamicSmemBytes = t.smem;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = t.ctas;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaError_t e = cudaFuncSetAttribute(mg_sweep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMgTailSmem);
        if (!e) e = cudaLaunchKernelEx(&cfg, mg_sweep_kernel, a, t);
        if (e) return e;
    }
    MgDot none;
    memset(&none, 0, sizeof(none));
    for (int l = l0 - 1; l >= 0; --l)
        mg_dispatch(a, l, [&](auto v, auto wk) {
            if constexpr (wk() != W_STORED) {
                if (dot) {
                    const unsigned g = mg_level_grid<v(), wk(), 1>(mg_post_kernel<v(), wk(), true>, a.lv[l], a.lv[l].nz);
                    mg_post_kernel<v(), wk(), true><<<g, kMgThreads, 0, s>>>(mg_step(a, l, a.lv[l + 1].w), *dot);
                    return;
                }
            }
            const unsigned g = mg_level_grid<v(), wk(), 2>(mg_post_kernel<v(), wk(), false>, a.lv[l], a.lv[l].nz);
            mg_post_kernel<v(), wk(), false><<<g, kMgThreads, 0, s>>>(mg_step(a, l, a.lv[l + 1].w), none);
        });
    if (dot && l0 == 0) mg_rz_kernel<<<mg_grid(a.lv[0].m), kMgThreads, 0, s>>>(a.lv[0].m, a.lv[0].f, a.lv[0].w, *dot);
    return cudaGetLastError();
}

int check_mg_grid(const gbpcg_grid *g) {
    if (int rc = check_grid(g)) return rc;
    const MgGeom G = mg_geom(*g);
    const int l = G.L - 1;
    if ((int64_t)G.nx[l] * G.ny[l] * G.nz[l] > kMgMaxCoarsest)
        return fail_arg("multigrid: the grid does not coarsen below 32768 cells (each size must be even, "
                        "down to >= 4, often enough)");
    if (g->nx % 4) return fail_arg("multigrid solves need nx a multiple of 4 (16-byte rows)");
    if (g->ny > 65535 || g->nz > 65535) return fail_arg("multigrid: ny and nz must be at most 65535");
    return GBPCG_OK;
}

// One MG-PCG solve recorded as a graph: the Jacobi solver's plan for pass A,
// the replacement and the finalize, plus pass R, the V-cycle and r.z.
template <typename Op>
struct MgSolve {
    SolvePlan<Op, true, double, float> sp;
    PassMaps mr;
    PassArgs ar;
    MgArgs mg;
    float *r, *z;
    bool direct;  // passes A and R on the march

    cudaError_t launch_r(cudaStream_t s) {
        return GB_CFG_DISPATCH(sp.cfg_b, float, K_PASSR, true, Op, K::launch(mr, ar, sp.op, sp.gb.grid(), s));
    }
    // pass A (or R) on the march
    template <bool A>
    cudaError_t launch_direct(cudaStream_t s) {
        const MgLevel &L = mg.lv[0];
        MgStep t = mg_step(mg, 0, nullptr);
        t.L.f = z;
        const MgPass d{sp.p0, sp.p1, sp.d, r, sp.st, sp.partials, sp.cond_loop, sp.cond_rep, sp.use_cond};
        mg_dispatch(mg, 0, [&](auto, auto wk) {
            if constexpr (wk() != W_STORED) {
                const unsigned g = mg_level_grid<4, wk(), A ? 3 : 4>(mg_pass_kernel<wk(), A>, L, L.nz);
                mg_pass_kernel<wk(), A><<<g, kMgThreads, 0, s>>>(t, d);
            }
        });
        return cudaGetLastError();
    }
    // the V-cycle and r.z
    cudaError_t launch_m(cudaStream_t s, int init) {
        const MgDot d{sp.st, sp.partials, init, sp.cond_loop, sp.use_cond};
        return mg_vcycle(mg, s, &d);
    }

    int capture(cudaGraph_t *out) {
        cudaStream_t cs = nullptr, bs = nullptr, rs = nullptr;
        GB_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        cudaError_t e = cudaStreamCreateWithFlags(&bs, cudaStreamNonBlocking);
        if (!e) e = cudaStreamCreateWithFlags(&rs, cudaStreamNonBlocking);
        auto add_cond = [&](cudaStream_t st, cudaGraphConditionalHandle h, cudaGraphConditionalNodeType type,
                            cudaGraph_t *body_out) -> cudaError_t {
            cudaStreamCaptureStatus cst;
            cudaGraph_t cap = nullptr;
            const cudaGraphNode_t *deps = nullptr;
            size_t ndeps = 0;
            cudaError_t e2 = cudaStreamGetCaptureInfo(st, &cst, nullptr, &cap, &deps, nullptr, &ndeps);
            if (e2) return e2;
            cudaGraphNodeParams cp = {cudaGraphNodeTypeConditional};
            cp.conditional.handle = h;
            cp.conditional.type = type;
            cp.conditional.size = 1;
            cudaGraphNode_t node;
            e2 = cudaGraphAddNode(&node, cap, deps, nullptr, ndeps, &cp);
            if (e2) return e2;
            *body_out = cp.conditional.phGraph_out[0];
            return cudaStreamUpdateCaptureDependencies(st, &node, nullptr, 1, cudaStreamSetCaptureDependencies);
        };
        cudaGraph_t graph = nullptr;
        bool cap_main = false, cap_b = false, cap_r = false;
        do {
            if (e) break;
            e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
            if (e) break;
            cap_main = true;
            cudaStreamCaptureStatus cst;
            cudaGraph_t cap = nullptr;
            e = cudaStreamGetCaptureInfo(cs, &cst, nullptr, &cap, nullptr, nullptr, nullptr);
            if (e) break;
            cudaGraphConditionalHandle cond;
            e = cudaGraphConditionalHandleCreate(&cond, cap, 1, cudaGraphCondAssignDefault);
            if (e) break;
            sp.set_cond(cond, 0, 1);
            ar.cond = cond;
            ar.use_cond = 1;
            e = sp.launch_setup(cs);  // reset, max |b|, r0 = b - A x0 stored as r
            if (e) break;
            e = mg_setup(mg, cs);
            if (e) break;
            e = launch_m(cs, 1);
            if (e) break;
            cudaGraph_t body = nullptr;
            e = add_cond(cs, cond, cudaGraphCondTypeWhile, &body);
            if (e) break;
            cudaGraphConditionalHandle rep;
            e = cudaGraphConditionalHandleCreate(&rep, body, 0, cudaGraphCondAssignDefault);
            if (e) break;
            sp.set_cond(cond, rep, 1);
            ar.cond_replace = rep;
            e = cudaStreamBeginCaptureToGraph(bs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
            if (e) break;
            cap_b = true;
            for (int u = 0; u < kMgUnroll && !e; ++u) {
                e = direct ? launch_direct<true>(bs) : sp.launch_a(bs);
                if (!e) e = direct ? launch_direct<false>(bs) : launch_r(bs);
                if (!e) e = launch_m(bs, 0);
            }
            if (e) break;
            cudaGraph_t rbody = nullptr;
            e = add_cond(bs, rep, cudaGraphCondTypeIf, &rbody);
            if (e) break;
            e = cudaStreamBeginCaptureToGraph(rs, rbody, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
            if (e) break;
            cap_r = true;
            e = sp.launch_replace(rs);  // flush, r = b - A x (FP64) stored as r
            if (!e) e = launch_m(rs, 0);
            if (e) break;
            cudaGraph_t tmp = nullptr;
            e = cudaStreamEndCapture(rs, &tmp);
            cap_r = false;
            if (e) break;
            e = cudaStreamEndCapture(bs, &tmp);
            cap_b = false;
            if (e) break;
            e = sp.launch_final(cs);
            if (e) break;
            e = cudaStreamEndCapture(cs, &graph);
            cap_main = false;
        } while (0);
        cudaGraph_t tmp = nullptr;
        if (cap_r) cudaStreamEndCapture(rs, &tmp);
        if (cap_b) cudaStreamEndCapture(bs, &tmp);
        if (cap_main) {
            cudaStreamEndCapture(cs, &tmp);
            if (tmp) cudaGraphDestroy(tmp);
        }
        if (rs) cudaStreamDestroy(rs);
        if (bs) cudaStreamDestroy(bs);
        cudaStreamDestroy(cs);
        if (e) {
            if (graph) cudaGraphDestroy(graph);
            cudaGetLastError();
            return fail_cuda(e, "multigrid solve graph capture");
        }
        *out = graph;
        return GBPCG_OK;
    }
};

template <typename Op>
int mg_solve_op(const gbpcg_grid &g, const Op &op, const double *b, double *x, const gbpcg_opts &o, char *ws,
                const MgLayout &M, gbpcg_result *res, cudaStream_t s) {
    MgSolve<Op> P;
    int ca = 0, cb = 0;
    {
        const int narrow = g.nx <= 32 ? CFG_32x16 : g.nx <= 64 ? CFG_64x16 : -1;
        ca = narrow >= 0 ? narrow : (g.nx > 192 && g.nx <= 256) ? CFG_256x4 : CFG_128x8;
        cb = narrow >= 0 ? narrow : CFG_128x8;
    }
    if (int rc = P.sp.init(g, op, ca, cb, b, x, ws, M.base, o.tol, o.maxit, 1.0, nullptr)) return rc;
    P.r = reinterpret_cast<float *>(ws + M.r);
    P.z = P.sp.z;
    // the FP64 residuals store r itself, in the r vector
    P.sp.ra.store_r = 1;
    P.sp.ra.z = P.r;
    // pass R: halo p_k (as pass B), centre and output r
    P.mr = P.sp.mb;
    if (make_pass_map<float>(&P.mr.c0, cb, false, P.r, g.nx, g.ny, g.nz)) return GBPCG_ERR_CUDA;
    P.ar = P.sp.ab;
    P.ar.c0 = P.r;
    P.ar.o0[0] = P.ar.o0[1] = P.r;
    P.ar.o1 = P.r;
    (void)GB_CFG_DISPATCH(cb, float, K_PASSR, true, Op, K::prepare());
    P.mg = mg_args(g, ws, M, P.r, P.z, P.sp.st);
    P.direct = g.ny % 2 == 0 && P.mg.lv[0].m <= kMgDirectPoints;
    cudaGraph_t graph = nullptr;
    if (int rc = P.capture(&graph)) return rc;
    cudaGraphExec_t exec = nullptr;
    cudaError_t e = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e) return fail_cuda(e, "multigrid graph instantiate");
    struct ExecGuard { cudaGraphExec_t g; ~ExecGuard() { cudaGraphExecDestroy(g); } } eg{exec};
    cudaGraphUpload(exec, s);
    cudaEvent_t e0, e1;
    GB_CUDA(cudaEventCreate(&e0));
    GB_CUDA(cudaEventCreate(&e1));
    GB_CUDA(cudaEventRecord(e0, s));
    GB_CUDA(cudaGraphLaunch(exec, s));
    GB_CUDA(cudaEventRecord(e1, s));
    SolveState hs;
    GB_CUDA(cudaMemcpyAsync(&hs, P.sp.st, sizeof(hs), cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    res->iters = hs.it;
    res->status = hs.status;
    res->rel_res_recursive = hs.bb > 0 ? sqrt(hs.rr / hs.bb) : 0.0;
    res->rel_res_true = hs.bb_true > 0 ? sqrt(hs.rr_true / hs.bb_true) : 0.0;
    res->time_ms = ms;
    res->replacements = hs.n_replace;
    res->pass_launches[0] = P.mg.L;  // levels of the hierarchy
    if (hs.status == GBPCG_TIMEOUT) set_error("a bounded device wait timed out during the solve");
    return hs.status;
}

}  // namespace

}  // namespace gb

using namespace gb;

extern "C" {

int gbpcg_mg_workspace_size(const gbpcg_grid *grid, size_t *bytes) {
    clear_error();
    if (int rc = check_mg_grid(grid)) return rc;
    if (!bytes) return fail_arg("bytes is NULL");
    *bytes = mg_layout(*grid, GBPCG_F64).total;
    return GBPCG_OK;
}

int gbpcg_mg_vcycle(const gbpcg_grid *grid, const float *r, float *z, void *workspace, size_t workspace_bytes,
                    int32_t *levels, gbpcg_stream stream) {
    clear_error();
    if (int rc = check_mg_grid(grid)) return rc;
    if (!r || !z || r == z) return fail_arg("r and z must be distinct device arrays");
    const MgLayout M = mg_layout(*grid, GBPCG_F64);
    if (!workspace || workspace_bytes < M.total || (reinterpret_cast<uintptr_t>(workspace) & 255u))
        return fail_arg("workspace: gbpcg_mg_workspace_size() bytes, 256-byte aligned");
    if ((reinterpret_cast<uintptr_t>(r) | reinterpret_cast<uintptr_t>(z)) & (sizeof(float) - 1))
        return fail_arg("r and z must be aligned to their element size");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    char *ws = static_cast<char *>(workspace);
    MgArgs a = mg_args(*grid, ws, M, const_cast<float *>(r), z, nullptr);
    // the level kernels take 16-byte vectors of r and z: others go through the solver's r and z in the workspace
    const size_t bytes = (size_t)a.lv[0].m * sizeof(float);
    if (mg_l0(a) > 0 && (reinterpret_cast<uintptr_t>(r) & 15u)) {
        a.lv[0].f = reinterpret_cast<float *>(ws + M.r);
        GB_CUDA(cudaMemcpyAsync(a.lv[0].f, r, bytes, cudaMemcpyDeviceToDevice, s));
    }
    if (mg_l0(a) > 0 && (reinterpret_cast<uintptr_t>(z) & 15u)) a.lv[0].w = reinterpret_cast<float *>(ws + M.base.z);
    if (grid->k_block) {  // the per-block face table the level-0 weights come from
        const int nbx = (grid->nx + grid->kbx - 1) / grid->kbx, nby = (grid->ny + grid->kby - 1) / grid->kby,
                  nbz = (grid->nz + grid->kbz - 1) / grid->kbz;
        const int64_t nb = (int64_t)nbx * nby * nbz;
        const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((nb + 255) / 256, 4096));
        build_face_table<<<blocks, 256, 0, s>>>(grid->k_block, nbx, nby, nbz, const_cast<float4 *>(a.tab));
    }
    GB_CUDA(mg_setup(a, s));
    GB_CUDA(mg_vcycle(a, s, nullptr));
    if (a.lv[0].w != z) GB_CUDA(cudaMemcpyAsync(z, a.lv[0].w, bytes, cudaMemcpyDeviceToDevice, s));
    if (levels) *levels = a.L;
    return GBPCG_OK;
}

int gbpcg_mg_pcg_solve(const gbpcg_grid *grid, const double *b, double *x, const gbpcg_opts *opts,
                       gbpcg_result *result, gbpcg_stream stream) {
    NvtxRange range("gbpcg_mg_pcg_solve");
    clear_error();
    if (int rc = check_mg_grid(grid)) return rc;
    if (!opts || !b || !x || !result) return fail_arg("NULL argument");
    if (!(opts->tol >= 0.0) || opts->maxit < 0) return fail_arg("tol must be >= 0 and maxit >= 0");
    if (opts->precond != GBPCG_PRECOND_MG || opts->io_dtype != GBPCG_F64 || opts->storage != GBPCG_F32 || opts->flags)
        return fail_arg("multigrid solves take precond MG, FP64 b and x, FP32 vectors, no flags");
    if ((reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(x)) & 15u)
        return fail_arg("b and x must be 16-byte aligned");
    const MgLayout M = mg_layout(*grid, GBPCG_F64);
    if (!opts->workspace || opts->workspace_bytes < M.total || (reinterpret_cast<uintptr_t>(opts->workspace) & 255u))
        return fail_arg("workspace: gbpcg_mg_workspace_size() bytes, 256-byte aligned");
    memset(result, 0, sizeof(*result));
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    char *ws = static_cast<char *>(opts->workspace);
    const gbpcg_grid &g = *grid;
    if (g.k_block)
        return mg_solve_op(g, make_op_table(g, 1.0f, reinterpret_cast<const float4 *>(ws + M.base.tab)), b, x, *opts,
                           ws, M, result, s);
    return mg_solve_op(g, make_op_const(g.nx, g.ny, g.nz), b, x, *opts, ws, M, result, s);
}

}  // extern "C"
