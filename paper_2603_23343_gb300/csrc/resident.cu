// Jacobi-PCG (Sec. VII) with the whole problem on chip: one cooperative launch
// per solve, every iteration vector in registers and shared memory.
//
// The grid is cut into bricks, one per CTA (one CTA of 512 threads per SM).
// A CTA keeps its brick's p in shared memory with a one-point halo, its
// residual r (and, in small bricks, q = A p and the correction vector d) in
// registers; what crosses SMs in an iteration is two sums and the r values on
// brick faces:
//
//   p = r + beta p           own points; halo points from the neighbours' r
//   q = u A p, sum p.q       -> grid sum -> alpha      (u: a power of two, ResProb::unit)
//   d += u alpha p, r -= alpha q, sum r.r; face values of r to L2
//                            -> grid sum -> beta, convergence, replacement
//
// A grid sum is one hop: every CTA publishes its partial sum together with
// the sum's number in one 16-byte store and reads every other CTA's, all add
// them in the same order, so all take the same decisions and no CTA waits
// for a broadcast; the face values travel, and d is updated, while the second
// sum does.  The set-up, the FP64 residual replacements and the final true
// residual run in the same launch, with the arithmetic of solver.cuh.
//
// What bounds it: the two grid sums (about 2 us each between 150 CTAs, in
// which the SMs idle) and, in large bricks, the stencil sweeps' shared-memory
// reads and instruction latency at 16 warps per SM.  Measured per iteration
// (GB300, FP64 b and x; the streaming passes of engine.cuh before): 32^3
// 5.5 us (38), 64^3 6.2, 128^3 9.9, 512 x 112 x 64 19.4 (34.7), 160^3 22.5
// (45).  The passes pay two launches with a serial march through the planes
// per iteration and 32 bytes per point of L2 or HBM traffic; here neither is
// left.  The rule: a problem that fits the chip (find_plan: r in registers
// and p in shared memory) runs here, every other one in the passes.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <list>
#include <mutex>
#include <vector>

#include "resident.cuh"

namespace gb {

namespace {

constexpr int kMaxWarps = kResThreads / 32;
constexpr int kSlotsPerLane = (kResMaxCtas + 31) / 32;
// A poll is an L2 round trip, about 0.7 us: under a second for the waits between CTAs that are in the
// same problem, which are never apart by more than part of an iteration.
constexpr uint32_t kSumPolls = 1u << 20;
constexpr unsigned kResLaunchSums = 16;  // of a host-driven launch: at most two at the start, two per iteration, four after
constexpr int kProgressEvery = 32;  // iterations of a batch's problem between two steps of its progress word

__device__ __forceinline__ void st_slot(ulonglong2 *p, unsigned long long v, unsigned long long tag) {
    asm volatile("{\n .reg .b128 t;\n mov.b128 t, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], t;\n}\n" ::"l"(p),
                 "l"(v), "l"(tag)
                 : "memory");
}
__device__ __forceinline__ void ld_slot(const ulonglong2 *p, unsigned long long &v, unsigned long long &tag) {
    asm volatile("{\n .reg .b128 t;\n ld.relaxed.gpu.global.b128 t, [%2];\n mov.b128 {%0, %1}, t;\n}\n"
                 : "=l"(v), "=l"(tag)
                 : "l"(p)
                 : "memory");
}

__device__ __forceinline__ void st_flag(unsigned *p, unsigned v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned ld_flag(const unsigned *p) {
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void lds4(const float *p, float (&v)[4]) {
    const float4 t = *reinterpret_cast<const float4 *>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void sts4(float *p, const float (&v)[4]) {
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}

// A sum as an unevaluated pair of floats, s + e: each addition's rounding error goes into e (Knuth's
// two-sum), so the pair is good to about 2^-47.  The loop's sums run on these because an FP64 operation
// costs tens of cycles on GB300 and about twenty of them in a row would sit between the two halves of
// every iteration (32^3: 11.2 us per iteration with FP64 sums and divisions).
struct Pair {
    float s, e;
};
__device__ __forceinline__ Pair pair_add(Pair a, Pair b) {
    Pair r;
    r.s = a.s + b.s;
    const float t = r.s - a.s;
    r.e = (a.e + b.e) + ((a.s - (r.s - t)) + (b.s - t));
    return r;
}
__device__ __forceinline__ Pair pair_xor(Pair a, int o) {
    return pair_add(a, Pair{__shfl_xor_sync(0xffffffffu, a.s, o), __shfl_xor_sync(0xffffffffu, a.e, o)});
}
__device__ __forceinline__ double pair_value(Pair a) { return (double)a.s + (double)a.e; }
__device__ __forceinline__ Pair pair_of(double v) {
    const float s = (float)v;
    return Pair{s, (float)(v - (double)s)};
}
// a / b to FP32 for 1e-36 < b < 1e36: one Newton step on the approximate quotient, the remainder of
// the whole pair taken exactly by FMAs (an IEEE division here cost 250 cycles of the chain)
__device__ __forceinline__ float pair_div(Pair a, Pair b) {
    const float rb = rcp_approx(b.s);
    const float q = a.s * rb;
    const float r = fmaf(-q, b.s, a.s) + fmaf(-q, b.e, a.e);
    return fmaf(r, rb, q);
}
__device__ __forceinline__ bool pair_plain(Pair a) { return a.s > 1e-36f && a.s < 1e36f; }
__device__ __forceinline__ unsigned long long pair_bits(Pair a) {
    return ((unsigned long long)__float_as_uint(a.e) << 32) | __float_as_uint(a.s);
}
__device__ __forceinline__ Pair pair_from(unsigned long long b) {
    return Pair{__uint_as_float((unsigned)b), __uint_as_float((unsigned)(b >> 32))};
}

// Loads and stores of single lanes under a predicate: branches around them would cost every warp a
// divergence and a reconvergence per vector.  (A barrier always lies between them and the accesses
// they depend on.)  PIN keeps the loads around them in program order: in the shallow builds the
// compiler otherwise gathers a whole run's loads in front (128^3: 3.71 against 4.26 ms), in the deep
// one the registers decide (512 x 112 x 64: 16.0 against 15.2 ms).
template <bool PIN>
__device__ __forceinline__ void lds_if(float &v, const float *p, bool on) {
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q ld.shared.f32 %0, [%1];\n}\n"
                 : "+f"(v)
                 : "r"(smem_u32(p)), "r"((unsigned)on));
    if (PIN) asm volatile("" ::: "memory");
}
template <bool PIN>
__device__ __forceinline__ void stg4_if(float *p, const float (&v)[4], unsigned on) {
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %5, 0;\n @q st.global.cg.v4.f32 [%0], {%1, %2, %3, %4};\n}\n" ::"l"(p),
                 "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "r"(on));
    if (PIN) asm volatile("" ::: "memory");
}

struct Shared {
    SolveState st;
    double red[kMaxWarps][3];
    float redf[kMaxWarps];
    Pair rr;            // r.r of the current residual
    float alpha, beta;
    float dalpha;       // alpha of d: times ResProb::unit
    float slow_below;   // ||r||^2 at or below this: the FP64 tests of passb_finish decide (fast_range)
    float slow_base;    // the same while r.r is a plain pair
    int timeout;
};

struct AddOp {
    static __device__ __forceinline__ double id() { return 0.0; }
    static __device__ __forceinline__ double op(double a, double b) { return a + b; }
};
struct MaxOp {  // of non-negative doubles
    static __device__ __forceinline__ double id() { return 0.0; }
    static __device__ __forceinline__ double op(double a, double b) { return a > b ? a : b; }
};

// Combines the CTAs' NV values (valid in lane 0 of every warp) over the
// problem's G CTAs and runs finish(total) in thread 0 of each CTA; false in
// every thread once a wait has run out.  FENCE: global stores made before the
// call by any thread of any of the CTAs are visible to all after it.
template <int NV, bool FENCE, typename Op, typename F>
__device__ __forceinline__ bool grid_reduce(Shared &sh, const ResProb &P, int rank, unsigned &seq,
                                            const double (&wv)[NV > 0 ? NV : 1], F &&finish) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int N = NV > 0 ? NV : 1;
    if (lane == 0) {
#pragma unroll
        for (int v = 0; v < N; ++v) sh.red[warp][v] = wv[v];
    }
    seq += 1;
    __syncthreads();
    if (warp == 0) {
        double t[N];
#pragma unroll
        for (int v = 0; v < N; ++v) t[v] = lane < (int)blockDim.x / 32 ? sh.red[lane][v] : Op::id();
#pragma unroll
        for (int o = 8; o > 0; o >>= 1)
#pragma unroll
            for (int v = 0; v < N; ++v) t[v] = Op::op(t[v], __shfl_xor_sync(0xffffffffu, t[v], o));
        bool ok = true;
        if (P.G > 1) {
            // two buffers: a CTA writes sum s + 2 only after sum s + 1 has every contribution, by
            // which time every CTA has read all of sum s
            ulonglong2 *slots = P.slots + (size_t)(seq & 1u) * (kResMaxCtas * kResSlotVals);
            if (lane == 0) {
                if (FENCE) __threadfence();
#pragma unroll
                for (int v = 0; v < N; ++v)
                    st_slot(slots + rank * kResSlotVals + v, (unsigned long long)__double_as_longlong(t[v]), seq);
            }
            double val[kSlotsPerLane][N];
            uint32_t polls = 0;
            for (;;) {
                bool all = true;
#pragma unroll
                for (int m = 0; m < kSlotsPerLane; ++m) {
                    const int j = lane + 32 * m;
                    if (j < P.G) {
#pragma unroll
                        for (int v = 0; v < N; ++v) {
                            unsigned long long bits, tag;
                            ld_slot(slots + j * kResSlotVals + v, bits, tag);
                            val[m][v] = __longlong_as_double((long long)bits);
                            all = all && tag == seq;
                        }
                    } else {
#pragma unroll
                        for (int v = 0; v < N; ++v) val[m][v] = Op::id();
                    }
                }
                if (__all_sync(0xffffffffu, all)) break;
                if (++polls > kSumPolls) {
                    ok = false;
                    break;
                }
            }
            if (FENCE) __threadfence();
#pragma unroll
            for (int v = 0; v < N; ++v) {
                double s = val[0][v];
#pragma unroll
                for (int m = 1; m < kSlotsPerLane; ++m) s = Op::op(s, val[m][v]);
                t[v] = s;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int v = 0; v < N; ++v) t[v] = Op::op(t[v], __shfl_xor_sync(0xffffffffu, t[v], o));
        }
        if (lane == 0) {
            if (ok) {
                finish(t);
            } else {
                sh.timeout = 1;
                sh.st.done = 1;
                sh.st.status = GBPCG_TIMEOUT;
                sh.st.timeout = 1;
            }
        }
    }
    __syncthreads();
    return sh.timeout == 0;
}

// Where brick `rank` lies.
struct Brick {
    int ix, iy, iz, x0, y0, z0;
    int nxl, nyl, nzl;  // its points inside the grid
    __device__ __forceinline__ Brick(const ResProb &P, int rank) {
        ix = rank % P.sx;
        iy = rank / P.sx % P.sy;
        iz = rank / (P.sx * P.sy);
        x0 = ix * P.bx4 * 4;
        y0 = iy * P.by;
        z0 = iz * P.bz;
        nxl = min(4 * P.bx4, P.nx - x0);
        nyl = min(P.by, P.ny - y0);
        nzl = min(P.bz, P.nz - z0);
    }
    // point e of the brick (x fastest) as grid coordinates
    __device__ __forceinline__ void point(int e, int &i, int &j, int &k) const {
        const int row = e / nxl, lz = row / nyl;
        i = x0 + e - row * nxl;
        j = y0 + row - lz * nyl;
        k = z0 + lz;
    }
};

// The set-up, the FP64 residuals and the final x are functions of their own, so that their
// registers and instructions stay out of the iteration's.

// max |b| into S.rhs_bits; false if a wait ran out.
template <typename X>
__device__ __noinline__ bool res_rhs_max(const ResProb &P, int rank, Shared &sh, unsigned &seq) {
    const Brick B(P, rank);
    const X *b = static_cast<const X *>(P.b);
    unsigned long long mu = 0;
    const int npts = B.nxl * B.nyl * B.nzl;
    for (int e = threadIdx.x; e < npts; e += blockDim.x) {
        int i, j, k;
        B.point(e, i, j, k);
        const double v = (double)__ldg(b + ((int64_t)k * P.ny + j) * P.nx + i);
        const unsigned long long u = (unsigned long long)__double_as_longlong(v) & ~(1ull << 63);
        mu = u > mu ? u : mu;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(0xffffffffu, mu, o);
        mu = t > mu ? t : mu;
    }
    // bit patterns of non-negative doubles order like the doubles; a NaN (above infinity) becomes
    // infinity, which the combining maximum keeps: either leaves the scale at 1 (rhs_scale)
    const unsigned long long inf = 0x7ff0000000000000ull;
    const double part[1] = {__longlong_as_double((long long)(mu > inf ? inf : mu))};
    return grid_reduce<1, false, MaxOp>(sh, P, rank, seq, part, [&](const double (&tot)[1]) {
        sh.st.rhs_bits = (unsigned long long)__double_as_longlong(tot[0]);
    });
}

// r = b - A x in FP64 over the brick (the arithmetic of res64_rows, solver.cuh), stored in padded
// rows, from which registers and neighbours take it; sums and decisions of res64_finish.
template <int MODE, typename X>
__device__ __noinline__ bool res_residual(const ResProb &P, int rank, Shared &sh, unsigned &seq) {
    constexpr int NV = res64_nv<MODE>();
    const Brick B(P, rank);
    const X *x = static_cast<const X *>(P.x);
    const X *b = static_cast<const X *>(P.b);
    SolveState &S = sh.st;
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    float fs = 1.0f;
    double unscale = 1.0;
    if (MODE != RES_INIT) {
        const double bb = S.bb;
        if (bb > 0.0 && isfinite(bb)) {
            int e = 0;
            frexp(sqrt(bb / ((double)nx * ny * nz)), &e);
            e = max(-100, min(100, e));
            fs = __int_as_float((127 - e) << 23);
            unscale = ldexp(1.0, 2 * e);
        }
    }
    const double w[6] = {P.cx, P.cx, P.cy, P.cy, P.cz, P.cz};
    const double s_rhs = rhs_scale(S.rhs_bits);
    double s0 = 0.0, s2 = 0.0;
    KahanF k0;
    const int npts = B.nxl * B.nyl * B.nzl;
    for (int e = threadIdx.x; e < npts; e += blockDim.x) {
        int i, j, k;
        B.point(e, i, j, k);
        const int64_t g = ((int64_t)k * ny + j) * nx + i;
        const double ax = apply64<false>(load_nbr64<X, true>(x, g, i, j, k, nx, ny, nz), w);
        const double bl = (double)__ldg(b + g);
        const double r = s_rhs != 1.0 ? s_rhs * (bl - ax) : bl - ax;
        const float rf = (float)r, rs = rf * fs;
        if (MODE != RES_TRUE) {
            float *zp = P.zg + ((int64_t)k * ny + j) * P.nxp + i;
            *zp = rf;
            if (i == nx - 1)
                for (int c = nx; c < P.nxp; ++c) *++zp = 0.0f;
        }
        if (MODE == RES_INIT) {
            const double bv = s_rhs != 1.0 ? s_rhs * bl : bl;
            s0 = fma(r, r, s0);
            s2 = fma(bv, bv, s2);
        } else {
            k0.add(rs * rs);
        }
    }
    if (MODE != RES_INIT) s0 = k0.value();
    // r.z is r.r here (no preconditioner: see resident_solve)
    double part[NV];
    part[0] = warp_sum(s0);
    if (NV > 1) part[NV > 1 ? 1 : 0] = part[0];
    if (NV > 2) part[NV > 2 ? 2 : 0] = warp_sum(s2);
    return grid_reduce<NV, true, AddOp>(sh, P, rank, seq, part, [&](const double (&tot)[NV]) {
        res64_finish<MODE>(&S, tot, unscale);
    });
}

// Every CTA's stores before it are visible to all after it.
__device__ __noinline__ bool res_barrier(const ResProb &P, int rank, Shared &sh, unsigned &seq) {
    const double none[1] = {0.0};
    return grid_reduce<0, true, AddOp>(sh, P, rank, seq, none, [&](const double (&)[1]) {});
}

// b = 0: x = 0 over the brick.
template <typename X>
__device__ __noinline__ void res_zero_x(const ResProb &P, int rank) {
    const Brick B(P, rank);
    X *x = static_cast<X *>(P.x);
    const int npts = B.nxl * B.nyl * B.nzl;
    for (int e = threadIdx.x; e < npts; e += blockDim.x) {
        int i, j, k;
        B.point(e, i, j, k);
        x[((int64_t)k * P.ny + j) * P.nx + i] = X(0);
    }
}

// Zeroes p and lists the halo: {shared-memory offset (-1 outside the grid), padded global index},
// the y and z faces' vectors first, then the x faces' points.
__device__ __noinline__ void res_setup(const ResProb &P, int rank, float *ps, int psize, int2 *tab) {
    const Brick B(P, rank);
    const int bx4 = P.bx4, by = P.by, bz = P.bz, pitch = 4 * bx4 + 4, plane = pitch * (by + 2);
    const bool xlo = B.ix > 0, xhi = B.ix < P.sx - 1, ylo = B.iy > 0, yhi = B.iy < P.sy - 1, zlo = B.iz > 0,
               zhi = B.iz < P.sz - 1;
    const int nvz = by * bx4, nvy = bz * bx4, nsx = by * bz;
    const int cz = (int)zlo + (int)zhi, cy = (int)ylo + (int)yhi, cx = (int)xlo + (int)xhi;
    const int nvec = cz * nvz + cy * nvy, nhalo = nvec + cx * nsx;
    for (int e = threadIdx.x; e < nhalo; e += blockDim.x) {
        int lx, ly, lz;
        if (e < cz * nvz) {
            const int f = e / nvz, r = e - f * nvz;
            lz = (f == 0 && zlo) ? -1 : bz;
            ly = r / bx4;
            lx = 4 * (r - ly * bx4);
        } else if (e < nvec) {
            const int e1 = e - cz * nvz, f = e1 / nvy, r = e1 - f * nvy;
            ly = (f == 0 && ylo) ? -1 : by;
            lz = r / bx4;
            lx = 4 * (r - lz * bx4);
        } else {
            const int e1 = e - nvec, f = e1 / nsx, r = e1 - f * nsx;
            lx = (f == 0 && xlo) ? -1 : 4 * bx4;
            lz = r / by;
            ly = r - lz * by;
        }
        const bool in = B.x0 + lx < P.nx && B.y0 + ly < P.ny && B.z0 + lz < P.nz;
        tab[e] = make_int2(in ? (lz + 1) * plane + (ly + 1) * pitch + 4 + lx : -1,
                           ((B.z0 + lz) * P.ny + B.y0 + ly) * P.nxp + B.x0 + lx);
    }
    for (int e = threadIdx.x; e < psize; e += blockDim.x) ps[e] = 0.0f;
}

// The grid-wide value of one FP32 sum whose per-warp parts are in sh.redf (after a barrier): run by
// warp 0 of every CTA, the total in every lane; false if a wait ran out.  Up to 32 CTAs each reads
// the others' slots; beyond that the slots every CTA polls become a hot spot and each CTA writes
// its part into every CTA's own inbox instead (one round over G CTAs, measured: G = 16 0.63 against
// 0.84 us, G = 64 1.54 against 1.07, G = 152 2.76 against 1.56).
__device__ __forceinline__ bool grid_sum_pair(const Shared &sh, const ResProb &P, int rank, unsigned seq, Pair &t) {
    const int lane = threadIdx.x & 31;
    __syncwarp();  // lanes left apart by the code before would take every shuffle one by one
    t = Pair{(lane & 15) < (int)blockDim.x / 32 ? sh.redf[lane & 15] : 0.0f, 0.0f};
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) t = pair_xor(t, o);
    if (P.G == 1) return true;
    const int G = P.G;
    const ulonglong2 *from;
    if (P.inbox) {
        ulonglong2 *box = P.inbox + (seq & 1u) * (unsigned)(G * G);
        ulonglong2 *to = box + (unsigned)(lane * G + rank);
        const unsigned long long bits = pair_bits(t);
#pragma unroll
        for (int m = 0; m < kSlotsPerLane; ++m)
            if (lane + 32 * m < G) st_slot(to + (unsigned)(32 * m * G), bits, seq);
        from = box + (unsigned)(rank * G);
    } else {
        ulonglong2 *slots = P.slots + (size_t)(seq & 1u) * (kResMaxCtas * kResSlotVals);
        if (lane == 0) st_slot(slots + rank, pair_bits(t), seq);
        from = slots;
    }
    // Every pass re-reads only what has not arrived: a pass over all slots under the load of the other
    // CTAs' passes takes about 1.9 us, one over the stragglers' 0.4.
    unsigned long long bits[kSlotsPerLane];
    unsigned missing = 0;
#pragma unroll
    for (int m = 0; m < kSlotsPerLane; ++m) {
        bits[m] = 0;
        if (lane + 32 * m < G) missing |= 1u << m;
    }
    bool ok = true;
    for (uint32_t polls = 0;; ++polls) {
        unsigned long long tag[kSlotsPerLane];
#pragma unroll
        for (int m = 0; m < kSlotsPerLane; ++m)
            if (missing >> m & 1u) ld_slot(from + lane + 32 * m, bits[m], tag[m]);
#pragma unroll
        for (int m = 0; m < kSlotsPerLane; ++m)
            if ((missing >> m & 1u) && tag[m] == seq) missing &= ~(1u << m);
        if (__all_sync(0xffffffffu, missing == 0)) break;
        if (polls >= kSumPolls) {
            ok = false;
            break;
        }
    }
    t = pair_from(bits[0]);
#pragma unroll
    for (int m = 1; m < kSlotsPerLane; ++m) t = pair_add(t, pair_from(bits[m]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t = pair_xor(t, o);
    return ok;
}

// The same sum in FP64, where the pairs' total is beyond their range: one thread of each CTA, for the
// same seq, through the slots behind those the pairs use.
__device__ __forceinline__ bool grid_sum_wide(const Shared &sh, const ResProb &P, int rank, unsigned seq, double &v) {
    v = 0.0;
    for (int w = 0; w < (int)blockDim.x / 32; ++w) v += (double)sh.redf[w];
    if (P.G == 1) return true;
    ulonglong2 *slots = P.slots + (size_t)(seq & 1u) * (kResMaxCtas * kResSlotVals) + (kResSlotVals - 1) * kResMaxCtas;
    st_slot(slots + rank, (unsigned long long)__double_as_longlong(v), seq);
    v = 0.0;
    for (int j = 0; j < P.G; ++j) {
        unsigned long long bits, tag;
        uint32_t polls = 0;
        do ld_slot(slots + j, bits, tag);
        while (tag != seq && ++polls <= kSumPolls);
        if (tag != seq) return false;
        v += __longlong_as_double((long long)bits);
    }
    return true;
}

// Where r.r is no plain pair (it is then {0, 0}, and S.rz holds it), no half iteration is fast.
__device__ __forceinline__ void fast_range(Shared &sh) {
    sh.slow_below = pair_plain(sh.rr) ? sh.slow_base : INFINITY;
    if (!pair_plain(sh.rr)) sh.rr = Pair{0.0f, 0.0f};
}

// The loop's scalars after an FP64 finish: FP32 pairs (r.r is S.rz where it is no plain pair), and the
// bound above which no FP64 test of passb_finish can trigger.  Thread 0.
__device__ __forceinline__ void loop_scalars(Shared &sh, bool saved_pair) {
    SolveState &S = sh.st;
    sh.rr = saved_pair ? pair_from((unsigned long long)__double_as_longlong(S.rzm)) : pair_of(S.rr);
    sh.beta = S.it == 0 ? 0.0f : (float)S.beta;
    const float t = __double2float_ru(fmax(S.tol2 * S.bb, kReplaceDrop2 * S.rr_rep));
    sh.slow_base = fmaxf(t * 1.00001f, 1e-36f);
    fast_range(sh);
}

// The FP64 finish of a half iteration (thread 0), where the fast tests do not settle it.
__device__ __noinline__ void res_finish(Shared &sh, const ResProb &P, int half, double v) {
    SolveState &S = sh.st;
    if (pair_plain(sh.rr)) S.rz = pair_value(sh.rr);
    if (half == 0) {
        passa_finish(&S, v, false);
        sh.alpha = (float)S.alpha;
        sh.dalpha = sh.alpha * P.unit;
    } else {
        passb_finish(&S, S.it, v, v, false);
        S.pending = 0;            // (d is up to date already)
        sh.beta = (float)S.beta;  // (a replacement sets its own)
    }
}

// The same where the sum is beyond the pairs' range.
__device__ __noinline__ void res_finish_wide(Shared &sh, const ResProb &P, int rank, unsigned seq, int half) {
    double v;
    if (!grid_sum_wide(sh, P, rank, seq, v)) {
        sh.timeout = 1;
        return;
    }
    res_finish(sh, P, half, v);
    if (half) {
        sh.rr = Pair{0.0f, 0.0f};
        fast_range(sh);
    }
}

// One CTA's part of the solve of problem P (brick number `rank`).  With constant coefficients D is
// one number, and the iterates of Jacobi-PCG are those of plain CG with every z and p multiplied by
// D: the loop keeps r instead of z, and r.z becomes r.r.
//   NT    threads of the CTA
//   MAXD  most vectors of four points per thread, one per plane; their r lives in registers
//   QREG  so does q = A p between the two halves of an iteration; else A p is taken twice
//   DREG  so many planes of d do too, updated with p one iteration late; the others: add_d
//   X     type of b and x
//   BATCH the launch holds other problems: their waits count from the last step of P.progress (batch_meet)
template <int NT, int MAXD, bool QREG, int DREG, bool BATCH, typename X>
__device__ __forceinline__ void resident_solve(const ResProb &P, int rank, unsigned char *smem, Shared &sh) {
    const int tid = threadIdx.x, lane = tid & 31;
    const int bx4 = P.bx4, by = P.by, D = P.depth;
    // p: rows of 4 + 4 bx4 floats; x = -1 sits before a row's first point, x = 4 bx4 in the gap
    // before the next row; one halo row and plane on either side
    const int pitch = 4 * bx4 + 4, plane = pitch * (by + 2);
    float *ps = reinterpret_cast<float *>(smem);
    const int psize = plane * (P.bz + 2) + 4;
    float4 *dsm = reinterpret_cast<float4 *>(ps + psize);
    int2 *tab = reinterpret_cast<int2 *>(dsm + P.dplanes * NT);

    // this thread's points: vector i in plane i of a run of D planes
    const bool act = tid < P.cols * P.zseg;
    const int col = act ? tid % P.cols : 0, zs = act ? tid / P.cols * D : 0;
    const int x4 = col % bx4, y = col / bx4;
    float *p0 = ps + (zs + 1) * plane + (y + 1) * pitch + 4 + 4 * x4;
    const bool needl = lane == 0 || x4 == 0, needr = lane == 31 || x4 == bx4 - 1;
    const int gplane = P.ny * P.nxp;  // padded rows
    int g0, xv, nvec, nhalo;
    unsigned valid = 0;  // bit i: vector i has points inside the grid
    unsigned faces = 0;  // bit i: vector i lies on a face some neighbour reads
    bool ragged;         // this brick has vectors reaching past the end of a row
    {
        const Brick B(P, rank);
        g0 = ((B.z0 + zs) * P.ny + B.y0 + y) * P.nxp + B.x0 + 4 * x4;
        xv = act ? max(0, min(4, B.nxl - 4 * x4)) : 0;  // points of a vector inside the grid
        ragged = B.nxl & 3;
        const bool xlo = B.ix > 0, xhi = B.ix < P.sx - 1, ylo = B.iy > 0, yhi = B.iy < P.sy - 1, zlo = B.iz > 0,
                   zhi = B.iz < P.sz - 1;
        for (int i = 0; i < D; ++i) {
            if (!xv || y >= B.nyl || zs + i >= B.nzl) continue;
            valid |= 1u << i;
            if ((x4 == 0 && xlo) || (x4 == bx4 - 1 && xhi) || (y == 0 && ylo) || (y == by - 1 && yhi) ||
                (zs + i == 0 && zlo) || (zs + i == P.bz - 1 && zhi))
                faces |= 1u << i;
        }
        nvec = ((int)zlo + (int)zhi) * by * bx4 + ((int)ylo + (int)yhi) * P.bz * bx4;
        nhalo = nvec + ((int)xlo + (int)xhi) * by * P.bz;
    }
    if (tid == 0) sh.timeout = 0;
    res_setup(P, rank, ps, psize, tab);

    SolveState &S = sh.st;
    unsigned seq = P.seq0;
    float rr_[MAXD][4], qr[QREG ? MAXD : 1][4], dr[DREG ? DREG : 1][4];
    bool pending = false;  // the planes of d in registers lack the last alpha p
    auto clear_d = [&]() {
#pragma unroll
        for (int i = 0; i < DREG; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) dr[i][j] = 0.0f;
    };
    clear_d();
    // The other planes of d are touched once per iteration, while the second grid sum is under way, by the
    // warps that have nothing else to do then (the first takes the sum, the second watches the
    // neighbours' flags; their vectors are shared out among the others).  Planes below dtop lie in shared
    // memory, the rest in L2, both thread by thread.
    const int nact = P.cols * P.zseg, dtop = DREG + P.dplanes;
    float4 *dg = P.dlin + (size_t)rank * nact * D;
    bool fresh = !P.resume;  // d is zero, whatever the arrays hold
    // d += alpha p of thread t's vectors in planes i, i + step, ..., four at a time
    auto add_d = [&](int t, const float *pp, int i0, int step, float alpha) {
        for (int i = i0; i < D; i += 4 * step) {
            float4 o[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = i + u * step;
                o[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (k < D && !fresh) o[u] = k < dtop ? dsm[(k - DREG) * NT + t] : __ldcg(dg + k * nact + t);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = i + u * step;
                if (k < D) {
                    float v[4];
                    lds4(pp + k * plane, v);
                    const float4 d = make_float4(fmaf(alpha, v[0], o[u].x), fmaf(alpha, v[1], o[u].y),
                                                 fmaf(alpha, v[2], o[u].z), fmaf(alpha, v[3], o[u].w));
                    if (k < dtop) dsm[(k - DREG) * NT + t] = d;
                    else __stcg(dg + k * nact + t, d);
                }
            }
        }
    };
    // where thread t's p begins in shared memory
    auto p_of = [&](int t) {
        const int c = t % P.cols;
        return (t / P.cols * D + 1) * plane + (c / bx4 + 1) * pitch + 4 + 4 * (c % bx4);
    };
    const int ow0 = DREG == MAXD ? 0 : p_of(lane), ow1 = DREG == MAXD ? 0 : p_of(lane + 32);
    // A point past the grid's end keeps r = 0, hence p = d = 0.
    // r of this thread's points from the padded global array
    auto load_r = [&]() {
#pragma unroll
        for (int i = 0; i < MAXD; ++i) {
            float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
            if (valid >> i & 1u) t = __ldcg(reinterpret_cast<const float4 *>(P.zg + g0 + i * gplane));
            rr_[i][0] = t.x; rr_[i][1] = t.y; rr_[i][2] = t.z; rr_[i][3] = t.w;
        }
    };
    // x += d / s
    auto flush = [&]() {
        if (fresh) return;
        fresh = true;
        const float a = pending ? sh.dalpha : 0.0f;
        pending = false;
        const double inv_s = 1.0 / rhs_scale(S.rhs_bits);
        const X is = (X)inv_s;
        const Brick B(P, rank);
        X *xp = static_cast<X *>(P.x) + ((int64_t)(B.z0 + zs) * P.ny + B.y0 + y) * P.nx + B.x0 + 4 * x4;
        auto add_x = [&](int i, const float (&dv)[4]) {
            if (!(valid >> i & 1u)) return;
            X *xi = xp + (int64_t)i * P.nx * P.ny;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j < xv) {
                    const X xo = __ldcg(xi + j);
                    xi[j] = inv_s == 1.0 ? xo + (X)dv[j] : xo + (X)dv[j] * is;
                }
        };
#pragma unroll
        for (int i = 0; i < DREG; ++i)
            if (i < D) {
                float v[4];
                lds4(p0 + i * plane, v);
#pragma unroll
                for (int j = 0; j < 4; ++j) v[j] = fmaf(a, v[j], dr[i][j]);
                add_x(i, v);
            }
        clear_d();
#pragma unroll 1
        for (int i = DREG; i < D; ++i) {
            if (!act) break;
            const float4 t = i < dtop ? dsm[(i - DREG) * NT + tid] : __ldcg(dg + i * nact + tid);
            const float v[4] = {t.x, t.y, t.z, t.w};
            add_x(i, v);
        }
    };
    // the first kHaloRegs halo entries of each thread of the warps but the first (r on the neighbours' faces)
    constexpr int kHaloRegs = 4, kHN = NT - 32;
    float4 hz[kHaloRegs];
    auto halo_load = [&](int e) {
        float4 h = make_float4(0.f, 0.f, 0.f, 0.f);
        if (e < nhalo) {
            const int2 t = tab[e];
            if (t.x >= 0) {
                if (e < nvec) h = __ldcg(reinterpret_cast<const float4 *>(P.zg + t.y));
                else h.x = __ldcg(P.zg + t.y);
            }
        }
        return h;
    };
    auto load_halo = [&]() {
        if (tid >= 32) {
#pragma unroll
            for (int u = 0; u < kHaloRegs; ++u) hz[u] = halo_load(tid - 32 + u * kHN);
        }
    };
    // p on one halo entry: r + beta p
    auto halo_p = [&](int e, float4 h, float beta) {
        if (e >= nhalo) return;
        const int2 t = tab[e];
        if (t.x < 0) return;
        if (e < nvec) {
            float v[4];
            lds4(ps + t.x, v);
            v[0] = fmaf(beta, v[0], h.x);
            v[1] = fmaf(beta, v[1], h.y);
            v[2] = fmaf(beta, v[2], h.z);
            v[3] = fmaf(beta, v[3], h.w);
            sts4(ps + t.x, v);
        } else {
            ps[t.x] = fmaf(beta, ps[t.x], h.x);
        }
    };

    bool alive = true;
    if (P.resume) {
        // continue a solve whose state an earlier launch saved
        if (tid == 0) S = *P.st;
        __syncthreads();
        for (int i = 0; i < D; ++i)
            if (valid >> i & 1u)
                *reinterpret_cast<float4 *>(p0 + i * plane) =
                    __ldcg(reinterpret_cast<const float4 *>(P.pg + g0 + i * gplane));
        fresh = S.it == S.pending;  // no update since the last flush (saved below)
#pragma unroll
        for (int i = 0; i < DREG; ++i)
            if (i < D && act) {
                const float4 t = __ldcg(dg + i * nact + tid);
                dr[i][0] = t.x; dr[i][1] = t.y; dr[i][2] = t.z; dr[i][3] = t.w;
            }
        if (act && !fresh)
            for (int i = DREG; i < min(dtop, D); ++i) dsm[(i - DREG) * NT + tid] = __ldcg(dg + i * nact + tid);
        for (int e = tid; e < nhalo; e += NT) {
            const int2 t = tab[e];
            if (t.x < 0) continue;
            if (e < nvec) *reinterpret_cast<float4 *>(ps + t.x) = __ldcg(reinterpret_cast<const float4 *>(P.pg + t.y));
            else ps[t.x] = __ldcg(P.pg + t.y);
        }
    } else {
        if (tid == 0) {
            memset(&S, 0, sizeof(S));
            S.tol2 = P.tol * P.tol;
            S.maxit = P.maxit;
            S.status = GBPCG_NOT_CONVERGED;
        }
        __syncthreads();
        alive = res_rhs_max<X>(P, rank, sh, seq);
        if (alive) alive = res_residual<RES_INIT, X>(P, rank, sh, seq);
    }
    if (tid == 0) loop_scalars(sh, P.resume);
    __syncthreads();
    load_r();
    if (alive && !S.done) load_halo();

    const float cx = P.op.cx, cy = P.op.cy, cz = P.op.cz, dgl = P.op.d;
    int left = P.iters;
    while (alive && !S.done && left-- > 0) {
        // ---- p_k = r_k + beta p_{k-1}: own points, then the halo from the neighbours' r ----
        {
            const float beta = sh.beta, dalpha = pending ? sh.dalpha : 0.0f;
            pending = false;
            int pl = plane;
            asm volatile("" : "+r"(pl));
            if (act) {
#pragma unroll
                for (int i = 0; i < MAXD; ++i)
                    if (i < D) {
                        float v[4];
                        lds4(p0 + i * pl, v);
                        if (i < DREG) {
                            const int k = i < DREG ? i : 0;
#pragma unroll
                            for (int j = 0; j < 4; ++j) dr[k][j] = fmaf(dalpha, v[j], dr[k][j]);
                        }
#pragma unroll
                        for (int j = 0; j < 4; ++j) v[j] = fmaf(beta, v[j], rr_[i][j]);
                        sts4(p0 + i * pl, v);
                    }
            }
            if (tid >= 32) {
#pragma unroll
                for (int u = 0; u < kHaloRegs; ++u) halo_p(tid - 32 + u * kHN, hz[u], beta);
                for (int e = tid - 32 + kHaloRegs * kHN; e < nhalo; e += kHN) halo_p(e, halo_load(e), beta);
            }
            __syncthreads();
        }
        // First half: q = A p, alpha = r.r / p.q.  Second half: d += alpha p, r -= alpha q, and beta
        // from r.r.  One copy of the code around them serves both.
        int half;
#pragma unroll 1
        for (half = 0; half < 2; ++half) {
            const float alpha = sh.alpha;
            float acc = 0.0f;
            // opaque copies: hoisted out of the loop, the addresses of every plane would take the registers
            int pl = plane, gpl = gplane;
            asm volatile("" : "+r"(pl), "+r"(gpl));
            auto update = [&](int i, const float (&q)[4]) {
                const float a = valid >> i & 1u ? -alpha : 0.0f;  // past the grid's end r stays 0
#pragma unroll
                for (int j = 0; j < 4; ++j) rr_[i][j] = fmaf(a, q[j], rr_[i][j]);
                if (ragged) {
#pragma unroll
                    for (int j = 1; j < 4; ++j) rr_[i][j] = j < xv ? rr_[i][j] : 0.0f;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) acc = fmaf(rr_[i][j], rr_[i][j], acc);
                stg4_if<QREG>(P.zg + (g0 + i * gpl), rr_[i], faces & (1u << i));
            };
            if (QREG && half == 1) {
#pragma unroll
                for (int i = 0; i < MAXD; ++i)
                    if (i < D) update(i, qr[QREG ? i : 0]);
            } else {
                float zm[4], c[4], zp[4], lo[4], hi[4], q[4];
                lds4(p0 - pl, zm);
                lds4(p0, c);
#pragma unroll
                for (int i = 0; i < MAXD; ++i) {
                    if (i < D) {
                        const float *pc = p0 + i * pl;
                        lds4(pc + pl, zp);
                        lds4(pc - pitch, lo);
                        lds4(pc + pitch, hi);
                        // the x neighbours come from the lanes beside this one, at row and warp ends from
                        // shared memory (scalar loads a vector apart would conflict four ways)
                        float xl = __shfl_up_sync(0xffffffffu, c[3], 1);
                        float xr = __shfl_down_sync(0xffffffffu, c[0], 1);
                        lds_if<QREG>(xl, pc - 1, needl);
                        lds_if<QREG>(xr, pc + 4, needr);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float xs = (j ? c[j - 1] : xl) + (j < 3 ? c[j + 1] : xr);
                            q[j] = fmaf(dgl, c[j], -fmaf(cx, xs, fmaf(cy, lo[j] + hi[j], cz * (zm[j] + zp[j]))));
                        }
                        if (QREG || half == 0) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                acc = fmaf(c[j], q[j], acc);
                                if (QREG) qr[QREG ? i : 0][j] = q[j];
                            }
                        } else {
                            update(i, q);
                        }
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            zm[j] = c[j];
                            c[j] = zp[j];
                        }
                    }
                }
            }
            acc = warp_sum(act ? acc : 0.0f);
            if (lane == 0) sh.redf[tid >> 5] = acc;
            seq += 1;
            __syncthreads();
            if (tid < 32) {
                Pair t;
                const bool ok = grid_sum_pair(sh, P, rank, seq, t);
                if (lane == 0) {
                    const Pair rr = sh.rr;
                    if (!ok) {
                        sh.timeout = 1;
                    } else if (half == 0 && pair_plain(t) && rr.s != 0.0f) {
                        const float a = pair_div(rr, t);
                        sh.alpha = a;
                        sh.dalpha = a * P.unit;
                    } else if (half == 1 && t.s > sh.slow_below && pair_plain(t) && S.it + 1 < S.maxit) {
                        sh.beta = pair_div(t, sh.rr);
                        sh.rr = t;
                        S.it += 1;
                    } else if (!pair_plain(t)) {
                        res_finish_wide(sh, P, rank, seq, half);
                    } else {
                        res_finish(sh, P, half, pair_value(t));
                        if (half) {
                            sh.rr = t;
                            sh.slow_below = sh.slow_base;
                        }
                    }
                    if (BATCH && half == 1 && rank == 0 && S.it % kProgressEvery == 0) atomicAdd(P.progress, 1u);
                }
            } else if (half == 1) {
                // Meanwhile the other warps take d += alpha p and fetch the neighbours' faces: each CTA
                // raises its flag once its own face values (stored before the barrier above) are visible.
                if (DREG < MAXD && D > DREG && tid >= 64) {
                    const float dalpha = sh.dalpha;
                    if (act) add_d(tid, p0, DREG, 1, dalpha);
                    const int nd = D - DREG;
                    for (int k = (tid >> 5) - 2; k < 2 * nd; k += NT / 32 - 2) {
                        const int t = k < nd ? lane : lane + 32;
                        if (t < nact) add_d(t, ps + (k < nd ? ow0 : ow1), DREG + (k < nd ? k : k - nd), D, dalpha);
                    }
                }
                if (tid < 64 && P.G > 1) {
                    if (lane == 0) {
                        __threadfence();
                        st_flag(P.flags + rank * kResFlagStride, seq);
                    }
                    const int sxy = P.sx * P.sy;
                    const int ix = rank % P.sx, iy = rank / P.sx % P.sy, iz = rank / sxy;
                    const int nb = lane == 0 ? (ix > 0 ? rank - 1 : -1)
                                 : lane == 1 ? (ix < P.sx - 1 ? rank + 1 : -1)
                                 : lane == 2 ? (iy > 0 ? rank - P.sx : -1)
                                 : lane == 3 ? (iy < P.sy - 1 ? rank + P.sx : -1)
                                 : lane == 4 ? (iz > 0 ? rank - sxy : -1)
                                 : lane == 5 ? (iz < P.sz - 1 ? rank + sxy : -1) : -1;
                    uint32_t polls = 0;
                    while (!__all_sync(0xffffffffu, nb < 0 || ld_flag(P.flags + nb * kResFlagStride) == seq)) {
                        if (++polls > kSumPolls) {
                            sh.timeout = 1;
                            break;
                        }
                    }
                    __threadfence();
                }
                if (P.G > 1) {
                    asm volatile("bar.sync 1, %0;" ::"n"(NT - 32) : "memory");  // the warps but the first
                    load_halo();
                }
            }
            __syncthreads();
            if (sh.timeout || S.done) break;
        }
        if (sh.timeout || half == 0) break;  // (half 0: no alpha)
        fresh = false;
        pending = true;
        if (S.replace) {
            flush();
            alive = res_barrier(P, rank, sh, seq);
            if (!alive) break;
            alive = res_residual<RES_REPLACE, X>(P, rank, sh, seq);
            if (!alive || S.done) break;
            load_r();
            load_halo();
            if (tid == 0) loop_scalars(sh, false);
            __syncthreads();
        }
    }
    __syncthreads();
    if (tid == 0) {
        if (sh.timeout) {
            S.done = 1;
            S.status = GBPCG_TIMEOUT;
            S.timeout = 1;
        }
        // what the fast steps kept as pairs (a finish that ended the loop has set its own values)
        if (!S.done) {
            if (pair_plain(sh.rr)) S.rr = S.rz = pair_value(sh.rr);
            S.beta = (double)sh.beta;
        }
        S.rzm = __longlong_as_double((long long)pair_bits(sh.rr));
        S.pending = fresh ? S.it : -1;  // for a resumed solve; no update of d is ever pending here
    }
    alive = alive && sh.timeout == 0;
    __syncthreads();

    if (P.save && alive) {
        const float a = pending ? sh.dalpha : 0.0f;
#pragma unroll
        for (int i = 0; i < DREG; ++i)
            if (i < D && act) {
                float v[4];
                lds4(p0 + i * plane, v);
                dg[i * nact + tid] = make_float4(fmaf(a, v[0], dr[i][0]), fmaf(a, v[1], dr[i][1]),
                                                 fmaf(a, v[2], dr[i][2]), fmaf(a, v[3], dr[i][3]));
            }
        if (act && !fresh)
            for (int i = DREG; i < min(dtop, D); ++i) dg[i * nact + tid] = dsm[(i - DREG) * NT + tid];
#pragma unroll
        for (int i = 0; i < MAXD; ++i)
            if (valid >> i & 1u) {  // whole vectors: the rows are padded, and the points past the end hold zero
                *reinterpret_cast<float4 *>(P.zg + g0 + i * gplane) =
                    make_float4(rr_[i][0], rr_[i][1], rr_[i][2], rr_[i][3]);
                *reinterpret_cast<float4 *>(P.pg + g0 + i * gplane) = *reinterpret_cast<const float4 *>(p0 + i * plane);
            }
    }
    if (P.final_x && alive) {
        if (S.zero_x) res_zero_x<X>(P, rank);
        else if (!S.true_known) flush();  // after a confirming replacement d is zero already
        if (!S.true_known) {
            alive = res_barrier(P, rank, sh, seq);
            if (alive) res_residual<RES_TRUE, X>(P, rank, sh, seq);
        }
    }
    __syncthreads();
    // rank 0 has seen every sum of the solve, so every CTA's part of x is complete when it reports
    if (rank == 0 && tid == 0) *P.st = S;
    __syncthreads();
}

template <int NT, int MAXD, bool QREG, int DREG, typename X>
__global__ void __launch_bounds__(NT, 1) resident_kernel(const __grid_constant__ ResProb one) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ Shared sh;
    resident_solve<NT, MAXD, QREG, DREG, false, X>(one, (int)blockIdx.x, smem, sh);
}

// Many problems: CTA c works through list[first[c]] .. list[first[c + 1] - 1], each entry a problem
// (low half) and a brick of it (high half).  Every CTA takes its problems in the same common order,
// so the CTAs of the first unfinished problem all reach it and no two problems wait for one another.
// Two CTAs of half the threads share an SM: one computes while the other waits for its grid sums.  (With
// GBPCG_FLAG_BATCH_GRAPH, one CTA with the threads and bricks of a standalone solve.)
struct ResSchedule {
    uint32_t first[2 * kResMaxCtas + 1];
};

// Waits until every CTA of problem P has come to it; false if one never does.  A CTA that is early waits
// here for as long as its partners' earlier problems take, so the limit is on the polls since any problem
// of the launch last took kProgressEvery iterations (or began): two loads each, one to two seconds.
__device__ __forceinline__ bool batch_meet(const ResProb &P, int rank, Shared &sh) {
    if (threadIdx.x == 0) {
        sh.timeout = 0;
        if (P.G > 1) {
            atomicAdd(P.arrived, 1u);
            unsigned seen = ld_flag(P.progress);
            for (uint32_t polls = 0; ld_flag(P.arrived) < (unsigned)P.G;) {
                const unsigned now = ld_flag(P.progress);
                polls = now == seen ? polls + 1 : 0;
                seen = now;
                if (polls > kSumPolls) {
                    sh.timeout = 1;
                    break;
                }
            }
        }
        if (rank == 0 && !sh.timeout) atomicAdd(P.progress, 1u);
    }
    __syncthreads();
    return sh.timeout == 0;
}

template <int NT, int MAXD, bool QREG, int DREG, typename X>
__global__ void __launch_bounds__(NT, NT == kResThreads ? 1 : 2)
    resident_batch_kernel(const ResProb *probs, const uint32_t *list, const __grid_constant__ ResSchedule sched) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ Shared sh;
    __shared__ ResProb P;
    for (uint32_t k = sched.first[blockIdx.x]; k < sched.first[blockIdx.x + 1]; ++k) {
        const uint32_t a = list[k];
        const int *src = reinterpret_cast<const int *>(probs + (a & 0xffffu));
        for (int i = threadIdx.x; i < (int)(sizeof(ResProb) / 4); i += NT) reinterpret_cast<int *>(&P)[i] = src[i];
        __syncthreads();
        // after a wait that ran out the problems left over keep done = 0
        if (!batch_meet(P, (int)(a >> 16), sh)) break;
        resident_solve<NT, MAXD, QREG, DREG, true, X>(P, (int)(a >> 16), smem, sh);
        if (sh.timeout) break;
        __syncthreads();
    }
}

// Three builds, by vectors per thread: up to 4, where r, q and d stay in registers; up to 7, where r
// and q do; and up to 14, where r does and A p is taken twice.  A batch runs the second for all its
// problems.
constexpr int kBuildDepth[] = {4, 7, 14}, kBuildDregs[] = {4, 0, 0}, kBuilds = 3;
constexpr int kBatchBuild = 1, kBatchThreads = 256;

// What a plan may use: a CTA's threads and shared memory (less the static part).
struct ResLimits {
    int threads, max_ctas, first_build, last_build;
    size_t smem;
    bool operator==(const ResLimits &o) const {
        return threads == o.threads && max_ctas == o.max_ctas && first_build == o.first_build &&
               last_build == o.last_build && smem == o.smem;
    }
};

size_t plan_smem(const ResPlan &p) {
    const size_t pitch = 4 * p.bx4 + 4, plane = pitch * (p.by + 2);
    const size_t halo = 2 * ((size_t)p.by * p.bx4 + (size_t)p.bz * p.bx4 + (size_t)p.by * p.bz);
    return (plane * (p.bz + 2) + 4) * 4 + halo * 8;  // and p.dplanes planes of d
}

constexpr size_t kResMaxSmem = 227 * 1024 - 2048, kBatchMaxSmem = 112 * 1024;

// Estimated SM cycles of an iteration: the sweeps and updates per warp and vector, the halo exchange,
// and the two grid sums (fitted to clock readings inside the kernel).
double plan_cycles(const ResPlan &p) {
    const double warps = std::ceil((double)p.cols * p.zseg / 32.0);
    const double halo = 2.0 * ((double)p.by * p.bx4 * (p.sz > 1) + (double)p.bz * p.bx4 * (p.sy > 1)) +
                        2.0 * p.by * p.bz * (p.sx > 1);
    const double per_vec = p.build == 0 ? 46.0 : p.build == 1 ? 50.0 : 120.0;
    const double sum = p.G == 1 ? 0.0 : p.G <= 16 ? 1000.0 + 20.0 * p.G : 1500.0 + 11.0 * p.G;
    return 4500.0 + 2.0 * sum + std::max(warps * per_vec, 350.0) * p.depth + 0.5 * halo;
}

// Points of all bricks, those outside the grid included.
int64_t plan_volume(const ResPlan &p) { return (int64_t)p.G * p.cols * p.zseg * p.depth * 4; }

bool make_plan(int nx, int ny, int nz, const ResLimits &lim, ResPlan *best) {
    const int nx4 = (nx + 3) / 4, max_ctas = lim.max_ctas;
    best->G = 0;
    for (int build = lim.first_build; build <= lim.last_build; ++build) {
        for (int sx = 1; sx <= max_ctas && sx <= nx4; ++sx) {
            const int bx4 = (nx4 + sx - 1) / sx;
            if (bx4 > lim.threads || (nx4 + bx4 - 1) / bx4 != sx) continue;
            for (int sy = 1; sx * sy <= max_ctas && sy <= ny; ++sy) {
                const int by = (ny + sy - 1) / sy, cols = bx4 * by;
                if (cols > lim.threads || (ny + by - 1) / by != sy) continue;
                for (int sz = 1; sx * sy * sz <= max_ctas && sz <= nz; ++sz) {
                    const int want = (nz + sz - 1) / sz;
                    if ((nz + want - 1) / want != sz) continue;
                    ResPlan p;
                    p.build = build;
                    p.sx = sx; p.sy = sy; p.bx4 = bx4; p.by = by; p.cols = cols;
                    const int most = std::min(lim.threads / cols, want);
                    p.depth = (want + most - 1) / most;
                    if (p.depth > kBuildDepth[build]) continue;
                    p.zseg = (want + p.depth - 1) / p.depth;
                    p.bz = p.zseg * p.depth;
                    p.sz = (nz + p.bz - 1) / p.bz;
                    p.G = sx * sy * p.sz;
                    p.smem = plan_smem(p);
                    if (p.smem > lim.smem) continue;
                    const size_t dplane = (size_t)lim.threads * sizeof(float4);
                    p.dplanes = (int)std::min<size_t>(std::max(0, p.depth - kBuildDregs[build]), (lim.smem - p.smem) / dplane);
                    p.smem += p.dplanes * dplane;
                    // r and p in padded rows and d by bricks share the workspace's four vectors
                    if (2 * (int64_t)nx4 * 4 * ny * nz + plan_volume(p) > 4 * (int64_t)nx * ny * nz) continue;
                    p.cycles = plan_cycles(p);
                    if (!best->G || p.cycles < best->cycles) *best = p;
                }
            }
        }
    }
    return best->G > 0;
}

// Plans kept per shape and CTA limit (a few hundred bytes each; the search takes tens of
// microseconds, a small solve a few hundred).
struct KeptPlan {
    int nx, ny, nz;
    ResLimits lim;
    bool ok;
    ResPlan plan;
};
std::mutex g_plan_mu;
std::list<KeptPlan> g_plans;  // most recently used first
constexpr size_t kPlansKept = 256;

template <typename X>
void *resident_fn(int build) {
    switch (build) {
        case 0: return reinterpret_cast<void *>(&resident_kernel<kResThreads, kBuildDepth[0], true, kBuildDregs[0], X>);
        case 1: return reinterpret_cast<void *>(&resident_kernel<kResThreads, kBuildDepth[1], true, kBuildDregs[1], X>);
        default: return reinterpret_cast<void *>(&resident_kernel<kResThreads, kBuildDepth[2], false, kBuildDregs[2], X>);
    }
}

// Raises a kernel's shared-memory limit on the current device.
cudaError_t allow_smem(void *fn, size_t bytes) {
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

constexpr int kResInboxAbove = 32;  // CTAs (grid_sum_pair)
size_t inbox_bytes(int G) { return (size_t)2 * G * G * sizeof(ulonglong2); }

ResProb make_prob(const SolveCall &c, const ResPlan &p) {
    const gbpcg_grid &g = *c.g;
    ResProb r;
    memset(&r, 0, sizeof(r));
    r.nx = g.nx; r.ny = g.ny; r.nz = g.nz; r.nxp = (g.nx + 3) & ~3;
    r.sx = p.sx; r.sy = p.sy; r.sz = p.sz; r.bx4 = p.bx4; r.by = p.by; r.bz = p.bz;
    r.zseg = p.zseg; r.depth = p.depth; r.dplanes = p.dplanes; r.cols = p.cols; r.G = p.G;
    // the operator times a power of two (exact) that brings its diagonal below 1: p.q then has r.r's
    // magnitude, and the FP32 sums the range they have in the passes
    r.op = make_op_const(g.nx, g.ny, g.nz);
    int e = 0;
    (void)std::frexp(r.op.d, &e);
    r.unit = std::ldexp(1.0f, -e);
    for (float *c : {&r.op.cx, &r.op.cy, &r.op.cz, &r.op.d}) *c *= r.unit;
    r.maxit = c.maxit; r.iters = 0x7fffffff;
    r.final_x = 1;
    auto cc = [](int m) { double h = 1.0 / (m + 1); return 1.0 / (h * h); };
    r.cx = cc(g.nx); r.cy = cc(g.ny); r.cz = cc(g.nz);
    r.tol = c.tol;
    r.b = c.b; r.x = c.x;
    // the workspace's vectors z, p0, p1, d hold r in padded rows; p likewise (a host-driven loop) or the
    // inboxes of the grid sums; and, at their end, d by bricks (make_plan has seen to the room)
    const size_t padded = (size_t)r.nxp * g.ny * g.nz;
    r.zg = reinterpret_cast<float *>(c.ws + c.L.z);
    r.pg = r.zg + padded;
    r.dlin = reinterpret_cast<float4 *>(r.pg + padded);
    r.st = reinterpret_cast<SolveState *>(c.ws + c.L.state);
    r.slots = reinterpret_cast<ulonglong2 *>(c.ws + c.L.partials);
    r.flags = reinterpret_cast<unsigned *>(r.slots + 2 * kResMaxCtas * kResSlotVals);
    r.arrived = r.flags + kResMaxCtas * kResFlagStride;
    if (p.G > kResInboxAbove && inbox_bytes(p.G) <= padded * 4) r.inbox = reinterpret_cast<ulonglong2 *>(r.pg);
    return r;
}

// A cooperative launch, or kResNoRoom where this context may not use the SMs it asks for (a context
// limited to part of the GPU): nothing has run then, and the caller streams the problem instead.
int cooperative(const cudaLaunchConfig_t &lc, void *fn, void **kargs) {
    const cudaError_t e = cudaLaunchKernelExC(&lc, fn, kargs);
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        cudaGetLastError();
        return kResNoRoom;
    }
    GB_CUDA(e);
    return GBPCG_OK;
}

void *single_fn(const ResPlan &p, int io) {
    return io == GBPCG_F64 ? resident_fn<double>(p.build) : resident_fn<float>(p.build);
}

// One launch (after allow_smem).
int launch_one(const ResProb &r, const ResPlan &p, int io, cudaStream_t s) {
    void *fn = single_fn(p, io);
    ResProb arg = r;
    void *kargs[] = {&arg};
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)p.G);
    lc.blockDim = dim3(kResThreads);
    lc.dynamicSmemBytes = p.smem;
    lc.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cooperative(lc, fn, kargs);
}

// Plan of a shape, from the kept ones if it is there; false if it does not fit.
bool find_plan(int nx, int ny, int nz, const ResLimits &lim, ResPlan *plan) {
    // padded rows need nx >= 8 (make_prob); indices into them are 32-bit
    if (nx < 8 || lim.max_ctas < 1 ||
        (int64_t)nx * ny * nz > (int64_t)lim.max_ctas * lim.threads * 4 * kBuildDepth[lim.last_build])
        return false;
    std::lock_guard<std::mutex> lk(g_plan_mu);
    for (auto it = g_plans.begin(); it != g_plans.end(); ++it)
        if (it->nx == nx && it->ny == ny && it->nz == nz && it->lim == lim) {
            g_plans.splice(g_plans.begin(), g_plans, it);
            *plan = g_plans.front().plan;
            return g_plans.front().ok;
        }
    KeptPlan k{nx, ny, nz, lim, false, {}};
    k.ok = make_plan(nx, ny, nz, lim, &k.plan);
    g_plans.push_front(k);
    if (g_plans.size() > kPlansKept) g_plans.pop_back();
    *plan = k.plan;
    return k.ok;
}

}  // namespace

bool resident_fits(const gbpcg_grid &g, ResPlan *plan) {
    const ResLimits lim{kResThreads, std::min(device_sm_count(), kResMaxCtas), 0, kBuilds - 1, kResMaxSmem};
    return !g.k_block && find_plan(g.nx, g.ny, g.nz, lim, plan);
}

int resident_launch(const SolveCall &c, const ResPlan &plan, cudaStream_t s, SolveState *st) {
    ResProb r = make_prob(c, plan);
    // the state block and the slots behind it (the first part of the partial sums)
    GB_CUDA(cudaMemsetAsync(c.ws + c.L.state, 0, c.L.partials + kResSlotBytes - c.L.state, s));
    if (st) r.st = st;
    if (r.inbox) GB_CUDA(cudaMemsetAsync(r.inbox, 0, inbox_bytes(r.G), s));
    GB_CUDA(allow_smem(single_fn(plan, c.io), kResMaxSmem));
    return launch_one(r, plan, c.io, s);
}

int resident_host_loop(const SolveCall &c, const ResPlan &plan, cudaStream_t s) {
    ResProb r = make_prob(c, plan);
    r.inbox = nullptr;  // p is kept there between launches; the sums are the same either way
    r.final_x = 0;
    r.save = 1;
    r.iters = 0;
    int done = 0;
    // what a launch does besides its iteration is most of the loop: the slots are cleared once, and each
    // launch numbers its sums from where the one before cannot have come to
    GB_CUDA(allow_smem(single_fn(plan, c.io), kResMaxSmem));
    GB_CUDA(cudaMemsetAsync(r.slots, 0, kResSlotBytes, s));
    for (int i = 0;; ++i, r.seq0 += kResLaunchSums) {
        if (int rc = launch_one(r, plan, c.io, s)) return rc;
        GB_CUDA(cudaMemcpyAsync(&done, &r.st->done, sizeof(int), cudaMemcpyDeviceToHost, s));
        GB_CUDA(cudaStreamSynchronize(s));
        if (done || i >= c.maxit) break;
        r.resume = 1;
        r.iters = 1;
    }
    r.resume = 1;
    r.iters = 0;
    r.save = 0;
    r.final_x = 1;
    r.seq0 += kResLaunchSums;
    return launch_one(r, plan, c.io, s);
}

// --------------------------------------------------------------- batches --

namespace {

ResLimits batch_limits(int max_ctas) {
    return ResLimits{kBatchThreads, max_ctas, kBatchBuild, kBatchBuild, kBatchMaxSmem};
}

// Iterations to expect of a solve, up to a factor common to all (for the schedule only): the square
// root of the operator's condition number.
double expected_iters(const gbpcg_grid &g) {
    auto sq = [](int n) { return (double)(n + 1) * (n + 1); };
    return std::sqrt(sq(g.nx) + sq(g.ny) + sq(g.nz));
}

}  // namespace

// Which way a batch goes is decided by estimates of the two, measured with grids of 32 to 160 points per
// axis on GB300.  On chip: a problem alone takes its plan's cycles; in the shared launch an iteration of
// any takes about 14 us and G of the 2 x 152 CTAs.  Streaming kernel: 175 G points per second once the
// GPU is full, a quarter of a microsecond per iteration for its scalar steps, and a problem's own
// iterations follow one another at 32 us and its points (one problem of 64^3: 31 us, 128^3 42, 192^3 73,
// 256^3 126).  So many large grids stream (24 of 48 to 160 points per axis: 65.6 against 78.8 ms
// on chip), a few large or many small ones do not (3: 14.2 against 7.0 ms; 200 of 32^3: 8.2 against 5.4;
// 64 of 64^3: 22.6 against 19.9; 16 of 128^3: 63.3 against 57.0).  Problems that do not fit stream either
// way, and others beside them fill the gaps a long one leaves (160^3, 32^3, 64^3, 192^3 and 48^3: 42.0 ms
// all streamed, 48.0 with the four on chip; 200^3 and 32 of 32^3: 48.9 against 46.6).
constexpr int64_t kBatchPoints = 400000;  // larger ones leave too little of the chip to others
constexpr double kSmMhz = 1900.0, kSharedUs = 14.0, kStreamedPerUs = 175e3, kStreamedStepUs = 0.25, kStreamedUs = 32.0;
constexpr double kMixMargin = 0.95;  // of the estimates, where part of the batch streams in any case

ResidentChoice resident_choice(int n, const gbpcg_grid *grids) {
    ResidentChoice r;
    const double ctas = 2.0 * std::min(device_sm_count(), kResMaxCtas);
    bool aligned = true;  // the streaming kernel's condition on every grid
    double alone = 0.0, shared = 0.0, shared_one = 0.0;
    double streamed = 0.0, streamed_one = 0.0, rest = 0.0, rest_one = 0.0;  // of all problems, of those that do not fit
    for (int i = 0; i < n; ++i) {
        const gbpcg_grid &g = grids[i];
        const int64_t pts = (int64_t)g.nx * g.ny * g.nz;
        const double it = expected_iters(g);
        aligned = aligned && !g.k_block && g.nx % 4 == 0;
        const double sum = it * (pts / kStreamedPerUs + kStreamedStepUs), one = it * (kStreamedUs + pts / kStreamedPerUs);
        streamed += sum;
        streamed_one = std::max(streamed_one, one);
        ResPlan p, q;
        if (!resident_fits(g, &p)) {
            r.rest.push_back(i);
            rest += sum;
            rest_one = std::max(rest_one, one);
        } else if (pts <= kBatchPoints && find_plan(g.nx, g.ny, g.nz, batch_limits((int)(ctas / 2)), &q)) {
            r.in_batch.push_back(i);
            shared += kSharedUs * it * std::ceil((double)pts / (4 * kBatchThreads * kBuildDepth[kBatchBuild])) / ctas;
            shared_one = std::max(shared_one, kSharedUs * it);
        } else {
            r.alone.push_back(i);
            alone += it * p.cycles / kSmMhz;
        }
    }
    if (r.in_batch.size() == 1) {  // nothing to share the chip with
        r.alone.push_back(r.in_batch[0]);
        r.in_batch.clear();
    }
    const double on_chip = alone + std::max(shared, shared_one) + std::max(rest, rest_one);
    if (aligned && (r.rest.empty() ? 1.0 : kMixMargin) * on_chip > std::max(streamed, streamed_one)) {
        r = ResidentChoice{};
        for (int i = 0; i < n; ++i) r.rest.push_back(i);
    }
    return r;
}

namespace {

// A problem of a shared launch, by its number among the calls.
struct Placed {
    int i;
    ResPlan p;
    double cycles;  // estimated, of the whole solve
};

// Each problem in turn, the longest first, on the CTAs that are free first; the end of the last one.
double place(std::vector<Placed> &probs, int ctas, std::vector<uint32_t> *list, ResSchedule *sched) {
    std::sort(probs.begin(), probs.end(), [](const Placed &a, const Placed &b) {
        return a.cycles != b.cycles ? a.cycles > b.cycles : a.i < b.i;
    });
    std::vector<std::vector<uint32_t>> lists(ctas);
    std::vector<double> free_at(ctas, 0.0);
    std::vector<int> by(ctas);
    double end = 0.0;
    for (const Placed &o : probs) {
        for (int c = 0; c < ctas; ++c) by[c] = c;
        std::partial_sort(by.begin(), by.begin() + o.p.G, by.end(), [&](int a, int b) {
            return free_at[a] != free_at[b] ? free_at[a] < free_at[b] : a < b;
        });
        const double t = free_at[by[o.p.G - 1]] + o.cycles;
        for (int r = 0; r < o.p.G; ++r) {
            free_at[by[r]] = t;
            lists[by[r]].push_back((uint32_t)o.i | (uint32_t)r << 16);
        }
        end = std::max(end, t);
    }
    list->clear();
    for (int c = 0; c < ctas; ++c) {
        sched->first[c] = (uint32_t)list->size();
        list->insert(list->end(), lists[c].begin(), lists[c].end());
    }
    sched->first[ctas] = (uint32_t)list->size();
    return end;
}

size_t tables_bytes(size_t n, size_t entries) {
    return round256(256 + n * sizeof(ResProb) + entries * sizeof(uint32_t));
}

// One launch of `fn` over `ctas` CTAs of `threads`, working through `list`.  The tables (tables_bytes):
// the progress word, the problems by their numbers (n of them), the list.
int launch_placed(void *fn, int threads, int ctas, size_t smem_limit, const std::vector<Placed> &placed, int n,
                  const std::vector<uint32_t> &list, const ResSchedule &sched, const SolveCall *calls,
                  SolveState *states, char *tables, cudaStream_t s) {
    std::vector<ResProb> probs(n);
    memset(static_cast<void *>(probs.data()), 0, (size_t)n * sizeof(ResProb));
    size_t smem = 0;
    char *progress = tables, *dprobs = progress + 256, *dlist = dprobs + (size_t)n * sizeof(ResProb);
    for (const Placed &o : placed) {
        ResProb &r = probs[o.i];
        r = make_prob(calls[o.i], o.p);
        r.st = states + o.i;
        r.progress = reinterpret_cast<unsigned *>(progress);
        smem = std::max(smem, o.p.smem);
        GB_CUDA(cudaMemsetAsync(r.slots, 0, kResSlotBytes, s));
        if (r.inbox) GB_CUDA(cudaMemsetAsync(r.inbox, 0, inbox_bytes(o.p.G), s));
    }
    GB_CUDA(cudaMemsetAsync(progress, 0, 256, s));
    // copies from pageable memory have left it when the calls return
    GB_CUDA(cudaMemcpyAsync(dprobs, probs.data(), (size_t)n * sizeof(ResProb), cudaMemcpyHostToDevice, s));
    GB_CUDA(cudaMemcpyAsync(dlist, list.data(), list.size() * sizeof(uint32_t), cudaMemcpyHostToDevice, s));
    GB_CUDA(allow_smem(fn, smem_limit));
    const ResProb *ap = reinterpret_cast<const ResProb *>(dprobs);
    const uint32_t *al = reinterpret_cast<const uint32_t *>(dlist);
    ResSchedule arg = sched;
    void *kargs[] = {&ap, &al, &arg};
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)ctas);
    lc.blockDim = dim3((unsigned)threads);
    lc.dynamicSmemBytes = smem;
    lc.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cooperative(lc, fn, kargs);
}

template <typename X>
void *batch_fn(int build) {
    switch (build) {
        case 0: return reinterpret_cast<void *>(&resident_batch_kernel<kResThreads, kBuildDepth[0], true, kBuildDregs[0], X>);
        case 1: return reinterpret_cast<void *>(&resident_batch_kernel<kResThreads, kBuildDepth[1], true, kBuildDregs[1], X>);
        default: return reinterpret_cast<void *>(&resident_batch_kernel<kResThreads, kBuildDepth[2], false, kBuildDregs[2], X>);
    }
}

}  // namespace

int resident_batch_launch(int n, const SolveCall *calls, SolveState *states, char *tables, size_t table_bytes, int io,
                          cudaStream_t s) {
    const int sms = device_sm_count(), group = std::min(sms, kResMaxCtas), ctas = std::min(2 * sms, 2 * kResMaxCtas);
    // Plans of each problem for a falling number of CTAs.  Fewer CTAs per problem waste less on the grid
    // sums, more finish the longest ones sooner: of a few trade-offs (the most CTA time a problem may
    // take over its cheapest plan) the one whose schedule ends first is taken.
    std::vector<std::vector<Placed>> options(n);
    for (int i = 0; i < n; ++i) {
        const gbpcg_grid &g = *calls[i].g;
        const double it = expected_iters(g);
        for (int m = group;;) {
            ResPlan p;
            if (!find_plan(g.nx, g.ny, g.nz, batch_limits(m), &p)) break;
            options[i].push_back({i, p, p.cycles * it});
            if (p.G <= 1) break;
            m = std::min(p.G - 1, p.G * 3 / 4);
        }
        if (options[i].empty()) return fail_arg("a problem of the batch does not fit the on-chip solver");
    }
    std::vector<Placed> best;
    std::vector<uint32_t> best_list, list;
    ResSchedule best_sched, sched;
    double best_end = 1e300;
    for (double slack : {1.0, 1.1, 1.25, 1.5, 2.0, 3.0}) {
        std::vector<Placed> pick(n);
        for (int i = 0; i < n; ++i) {
            double least = 1e300;
            for (const Placed &o : options[i]) least = std::min(least, o.cycles * o.p.G);
            const Placed *b = nullptr;
            for (const Placed &o : options[i])
                if (o.cycles * o.p.G <= slack * least && (!b || o.cycles < b->cycles)) b = &o;
            pick[i] = *b;
        }
        const double end = place(pick, ctas, &list, &sched);
        if (end < best_end) {
            best_end = end;
            best = pick;
            best_list = list;
            best_sched = sched;
        }
        if (n > 8 * ctas) break;  // many problems: the schedule is even whatever the trade-off
    }
    if (tables_bytes(n, best_list.size()) > table_bytes) return kResNoRoom;
    GB_CUDA(cudaMemsetAsync(states, 0, (size_t)n * sizeof(SolveState), s));
    void *fn = io == GBPCG_F64
                   ? reinterpret_cast<void *>(
                         &resident_batch_kernel<kBatchThreads, kBuildDepth[kBatchBuild], true, kBuildDregs[kBatchBuild], double>)
                   : reinterpret_cast<void *>(
                         &resident_batch_kernel<kBatchThreads, kBuildDepth[kBatchBuild], true, kBuildDregs[kBatchBuild], float>);
    return launch_placed(fn, kBatchThreads, ctas, kBatchMaxSmem, best, n, best_list, best_sched, calls, states, tables, s);
}

int resident_standalone_launch(int n, const SolveCall *calls, SolveState *states, char *tables, size_t table_bytes,
                               int io, cudaStream_t s) {
    const int ctas = std::min(device_sm_count(), kResMaxCtas);
    std::vector<Placed> placed[kBuilds];
    std::vector<uint32_t> list[kBuilds];
    ResSchedule sched[kBuilds];
    for (int i = 0; i < n; ++i) {
        ResPlan p;
        if (!resident_fits(*calls[i].g, &p)) return fail_arg("a problem of the batch does not fit the on-chip solver");
        placed[p.build].push_back({i, p, p.cycles * expected_iters(*calls[i].g)});
    }
    size_t need = 0;
    for (int b = 0; b < kBuilds; ++b) {
        if (placed[b].empty()) continue;
        place(placed[b], ctas, &list[b], &sched[b]);
        need += tables_bytes(n, list[b].size());
    }
    if (need > table_bytes) return kResNoRoom;
    GB_CUDA(cudaMemsetAsync(states, 0, (size_t)n * sizeof(SolveState), s));
    for (int b = 0, launched = 0; b < kBuilds; ++b) {
        if (placed[b].empty()) continue;
        void *fn = io == GBPCG_F64 ? batch_fn<double>(b) : batch_fn<float>(b);
        const int rc = launch_placed(fn, kResThreads, ctas, kResMaxSmem, placed[b], n, list[b], sched[b], calls, states,
                                     tables, s);
        if (rc == kResNoRoom && launched) return fail_cuda(cudaErrorCooperativeLaunchTooLarge, "batch launch");
        if (rc) return rc;
        launched = 1;
        tables += tables_bytes(n, list[b].size());
    }
    return GBPCG_OK;
}

}  // namespace gb
