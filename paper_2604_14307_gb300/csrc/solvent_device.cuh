// Device functions of the solvent passes (Sec. II.A of arXiv 2604.14307): draws,
// binning, streaming, cell records, the SRD rule and the run-merged binning of a
// thread's four particles.  Shared by the passes of kernels_solvent.cu and of the
// angular-momentum-conserving variants (kernels_angular.cu); the draws and the binning
// rule also by the sites (kernels_bodies.cu).
#pragma once

#include "mpcd_internal.cuh"

namespace mpcd {

// (x + 1/2) 2^-32 from all 32 bits, relative error <= 2^-24 (never 0; 1 only
// when x rounds up to 2^32)
__device__ __forceinline__ float u01f(uint32_t x)
{
    return __fmaf_rn(__uint2float_rn(x), 2.3283064365386962890625e-10f, 1.16415321826934814453125e-10f);
}

// -2 ln u for u = (x + 1/2) 2^-32 with full relative precision also near u = 1,
// where 1 - u = (~x + 1/2) 2^-32 is formed exactly from the integer complement
__device__ __forceinline__ float neg2log(uint32_t x)
{
    return (x & 0x80000000u) ? -2.0f * log1pf(-u01f(~x)) : -2.0f * __logf(u01f(x));
}

// three standard normals from one Philox block (Box-Muller); the angles are
// shifted by pi into [-pi, pi) where the fast sine/cosine are accurate
__device__ __forceinline__ void normals3(uint4 w, float n[3])
{
    const float r1 = sqrtf(neg2log(w.x));
    const float r2 = sqrtf(neg2log(w.z));
    float s1, c1;
    __sincosf(6.283185307179586f * (u01f(w.y) - 0.5f), &s1, &c1);
    n[0] = -r1 * c1;
    n[1] = -r1 * s1;
    n[2] = -r2 * __cosf(6.283185307179586f * (u01f(w.w) - 0.5f));
}
__device__ __forceinline__ void normals3(uint4 w, double n[3])
{
    double r1 = sqrt(-2.0 * log(u01d(w.x)));
    double r2 = sqrt(-2.0 * log(u01d(w.z)));
    double s1, c1;
    sincospi(2.0 * u01d(w.y), &s1, &c1);
    n[0] = r1 * c1;
    n[1] = r1 * s1;
    n[2] = r2 * cospi(2.0 * u01d(w.w));
}

// binning rule: X = floor(x 2^20) (box edges below 2048 cells keep it within int32),
// cell = floor((X - S) / 2^20) mod L
__device__ __forceinline__ int lattice_X(float x) { return __float2int_rd(x * 1048576.0f); }
__device__ __forceinline__ int lattice_X(double x) { return lattice_floor(x); }
__device__ __forceinline__ int axis_cell(int X, int S, int L)
{
    int c = (X - S) >> 20;
    c += (c < 0) ? L : 0;
    c -= (c >= L) ? L : 0;
    return ((unsigned)c < (unsigned)L) ? c : 0;   // only a non-finite position gets here; it is flagged
}
template <typename Real> __device__ __forceinline__ int cell_axis(Real x, int S, int L)
{
    return axis_cell(lattice_X(x), S, L);
}
// The same rule in float32 without a conversion instruction (the solvent
// passes).  With S an integer, floor((floor(x 2^20) - S) / 2^20) =
// floor(x - s) for s = S 2^-20, which float32 holds exactly.  x - s rounded
// toward -inf has the floor of the exact difference (the rounding is monotone
// and keeps integers), and floor_magic reads that floor off the mantissa
// (|x - s| < 2^11 here).
// For x in [0, L) and |s| <= 1/2 the floor lies in [-1, L]: the top is wrapped
// by one select and -1 by an unsigned minimum with L - 1, which also keeps a
// non-finite position's cell inside the box (such a position is flagged).
__device__ __forceinline__ int cell_axis_f(float x, float s, int L)
{
    int c = floor_magic_int(floor_magic(__fsub_rd(x, s)));
    c = c == L ? 0 : c;
    return (int)min((unsigned)c, (unsigned)(L - 1));
}
// grid shift of one axis in the form the binning of a precision takes
template <typename Real> struct ShiftT { typedef int32_t type; };
template <> struct ShiftT<float> { typedef float type; };
__device__ __forceinline__ int32_t shift_as(int32_t S, int32_t) { return S; }
__device__ __forceinline__ float shift_as(int32_t S, float)
{
    return __fmul_rn(__int2float_rn(S), 9.5367431640625e-07f);   // S 2^-20, exact for |S| <= 2^19
}
__device__ __forceinline__ int cell_bin(float x, float s, int L) { return cell_axis_f(x, s, L); }
__device__ __forceinline__ int cell_bin(double x, int32_t S, int L) { return cell_axis(x, S, L); }

// streaming x + v dt with periodic wrap, unfused (same rounding as the oracle)
__device__ __forceinline__ float drift(float x, float v, float dt, float L, int &bad)
{
    float y = __fadd_rn(x, __fmul_rn(v, dt));
    if (y >= L) y = __fsub_rn(y, L);
    else if (y < 0.0f) { y = __fadd_rn(y, L); if (y >= L) y = 0.0f; }
    bad |= !(y >= 0.0f && y < L);
    return y;
}
__device__ __forceinline__ double drift(double x, double v, double dt, double L, int &bad)
{
    return wrap_box(__dadd_rn(x, __dmul_rn(v, dt)), L, bad);
}
// Streaming under a constant force (the solvent's share of the balancing
// force of the sedimentation protocol): v += a dt/2, x += v dt, v += a dt/2,
// exact for a constant force; with no force the plain drift.
__device__ __forceinline__ float kick(float v, float h) { return __fadd_rn(v, h); }
__device__ __forceinline__ double kick(double v, double h) { return __dadd_rn(v, h); }

__device__ __forceinline__ void ld4(const float *p, float (&o)[4])
{
    float4 t = __ldcs(reinterpret_cast<const float4 *>(p));
    o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
}
__device__ __forceinline__ void ld4(const double *p, double (&o)[4])
{
    double2 a = __ldcs(reinterpret_cast<const double2 *>(p));
    double2 b = __ldcs(reinterpret_cast<const double2 *>(p) + 1);
    o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
}
__device__ __forceinline__ void st4(float *p, const float (&o)[4])
{
    __stcs(reinterpret_cast<float4 *>(p), make_float4(o[0], o[1], o[2], o[3]));
}
__device__ __forceinline__ void st4(double *p, const double (&o)[4])
{
    __stcs(reinterpret_cast<double2 *>(p), make_double2(o[0], o[1]));
    __stcs(reinterpret_cast<double2 *>(p) + 1, make_double2(o[2], o[3]));
}

// collision parameters of one cell
template <typename Real> struct CellParams { Real ux, uy, uz, kappa, ax, ay, az; };

// 32 bytes by one 256-bit load instead of two of 128 bits: the gathers of a
// warp go to up to 32 lines, and each instruction looks all of them up (80 M
// particles, SRD: 1470 -> 1456 us a pass; MPCD-AT, 9 M: 344 -> 332).  A
// record is 32-byte aligned: 32 or 64 bytes each, from a base at such a boundary.
__device__ __forceinline__ CellParams<float> load_params(const void *params, int64_t c)
{
    CellParams<float> o;
    float pad;
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(o.ux), "=f"(o.uy), "=f"(o.uz), "=f"(o.kappa), "=f"(o.ax), "=f"(o.ay), "=f"(o.az), "=f"(pad)
                 : "l"(reinterpret_cast<const float *>(params) + 8 * c));
    return o;
}
__device__ __forceinline__ CellParams<double> load_params_d(const void *params, int64_t c)
{
    const double *p = reinterpret_cast<const double *>(params) + 8 * c;
    CellParams<double> o;
    double pad;
    asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
                 : "=d"(o.ux), "=d"(o.uy), "=d"(o.uz), "=d"(o.kappa) : "l"(p));
    asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
                 : "=d"(o.ax), "=d"(o.ay), "=d"(o.az), "=d"(pad) : "l"(p + 4));
    return o;
}
template <typename Real> __device__ __forceinline__ CellParams<Real> get_params(const void *pr, int64_t c);
template <> __device__ __forceinline__ CellParams<float> get_params<float>(const void *pr, int64_t c)
{
    return load_params(pr, c);
}
template <> __device__ __forceinline__ CellParams<double> get_params<double>(const void *pr, int64_t c)
{
    return load_params_d(pr, c);
}

template <typename Real> struct Consts;
template <> struct Consts<float> {
    __device__ static float kT(const StepArgs &a) { return a.kTf; }
    __device__ static float dt(const StepArgs &a) { return a.dtf; }
    __device__ static float m(const StepArgs &a) { return a.m_solvent_f; }
    __device__ static float ca(const StepArgs &a) { return a.cos_af; }
    __device__ static float sa(const StepArgs &a) { return a.sin_af; }
    __device__ static float ah(const StepArgs &a, int k) { return a.ahf[k]; }
};
template <> struct Consts<double> {
    __device__ static double kT(const StepArgs &a) { return a.kT; }
    __device__ static double dt(const StepArgs &a) { return a.dt; }
    __device__ static double m(const StepArgs &a) { return a.m_solvent; }
    __device__ static double ca(const StepArgs &a) { return a.cos_a; }
    __device__ static double sa(const StepArgs &a) { return a.sin_a; }
    __device__ static double ah(const StepArgs &a, int k) { return a.ah[k]; }
};

// SRD: v' = u + kappa R(n, alpha)(v - u)  (Rodrigues)
template <typename Real>
__device__ __forceinline__ void srd_rotate(const CellParams<Real> &p, Real ca, Real sa, Real &vx,
                                           Real &vy, Real &vz)
{
    Real wx = vx - p.ux, wy = vy - p.uy, wz = vz - p.uz;
    Real nd = p.ax * wx + p.ay * wy + p.az * wz;
    Real cx = p.ay * wz - p.az * wy, cy = p.az * wx - p.ax * wz, cz = p.ax * wy - p.ay * wx;
    Real t = nd * (Real(1) - ca);
    vx = p.ux + p.kappa * (wx * ca + cx * sa + p.ax * t);
    vy = p.uy + p.kappa * (wy * ca + cy * sa + p.ay * t);
    vz = p.uz + p.kappa * (wz * ca + cz * sa + p.az * t);
}

// word count of the cell sums (FP64 form; Words32: the FP32 form's)
template <typename Real, int RULE> struct NWords;
template <> struct NWords<double, 0> { static constexpr int n = 6; };
template <> struct NWords<double, 1> { static constexpr int n = 8; };
template <typename Real> struct SumWord { typedef double type; };
template <> struct SumWord<float> { typedef long long type; };

// FP64 form: contributions of one particle (mass m, velocity v, AT noise xi)
// to the double sum arrays N, M, m v (3), m v.v (SRD) or m xi (3) (AT)
template <int RULE>
__device__ __forceinline__ void terms64(double m, double vx, double vy, double vz, const double *xi, double *w)
{
    w[0] = 1.0;
    w[1] = m;
    w[2] = m * vx;
    w[3] = m * vy;
    w[4] = m * vz;
    if (RULE == 0) {
        w[5] = m * (vx * vx + vy * vy + vz * vz);
    } else {
        w[5] = m * xi[0];
        w[6] = m * xi[1];
        w[7] = m * xi[2];
    }
}

__device__ __forceinline__ void red_add(long long *p, long long v)
{
    atomicAdd(reinterpret_cast<unsigned long long *>(p), (unsigned long long)v);
}
__device__ __forceinline__ void red_add(double *p, double v) { atomicAdd(p, v); }

// The MPCD-AT normals of a thread's 4 consecutive particles (slots from `slot`) at
// `step`: those that the binning for this collision drew and kept, or drawn
// here (after a re-sort).  The four Philox blocks are independent: a lane past
// the tile end draws for id 0, so that their dependent rounds interleave.  A
// draw is about 150 instructions, a quarter of the pass, which reading 12 bytes
// replaces (9 M particles: a step 542 -> 503 us; FP64, 0.3 M: 328 -> 241).
template <typename Real>
__device__ __forceinline__ void at_normals4(const StepArgs &a, const DevReplica &rr, int64_t step,
                                            const uint32_t (&tg)[4], int nv, int64_t slot, Real (&n)[4][3])
{
    if (a.noise_in) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            Real o[4] = {Real(0), Real(0), Real(0), Real(0)};
            if (nv > 0) ld4(reinterpret_cast<const Real *>(a.noise[k]) + slot, o);
#pragma unroll
            for (int j = 0; j < 4; ++j) n[j][k] = o[j];
        }
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) normals3(draw(rr, step, tg[j], TAG_AT, 0u), n[j]);
    }
}

// y in one of the exchange slabs (the test of the exchange itself)
__device__ __forceinline__ bool in_slab(const StepArgs &a, float y)
{
    return (y >= a.rn_yf[0] && y < a.rn_yf[1]) || (y >= a.rn_yf[2] && y < a.rn_yf[3]);
}
__device__ __forceinline__ bool in_slab(const StepArgs &a, double y)
{
    return (y >= a.rn_y[0] && y < a.rn_y[1]) || (y >= a.rn_y[2] && y < a.rn_y[3]);
}

// Binning of a thread's 4 consecutive particles: cell under the shift S,
// per-particle fixed-point (P32) or double (P64) terms, runs of equal cells
// merged in registers, then one atomic per word and run.
template <typename Real, int RULE, bool COLLIDE, typename W, typename SH>
__device__ __forceinline__ void bin4(const StepArgs &a, const Real (&x)[4], const Real (&y)[4], const Real (&z)[4],
                                     const Real (&vx)[4], const Real (&vy)[4], const Real (&vz)[4],
                                     const uint32_t (&tg)[4], int nv, const SH *S, int L0, int L1, int L2,
                                     int base, const DevReplica &rr, int64_t step, Real m, Real sc, W *sums,
                                     int64_t C, int64_t slot)
{
    int cc[4];
    Real xi[4][3];
    if (a.slab_mark) {   // the exchange reads the marked blocks of slots only
        bool in = false;
#pragma unroll
        for (int j = 0; j < 4; ++j) in = in || (j < nv && in_slab(a, y[j]));
        if (in) a.slab_mark[slot / RN_MARK] = 1;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        cc[j] = base + cell_bin(x[j], S[0], L0) + L0 * (cell_bin(y[j], S[1], L1) + L1 * cell_bin(z[j], S[2], L2));
        xi[j][0] = xi[j][1] = xi[j][2] = Real(0);
        // for every slot, so that the four draws interleave; runs past nv are dropped
        if (RULE == 1) normals3(draw(rr, step + (COLLIDE ? 1 : 0), tg[j], TAG_AT, 0u), xi[j]);
    }
    if (RULE == 1) {
        if (nv > 0)   // kept for the collision that this binning is for
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const Real o[4] = {xi[0][k], xi[1][k], xi[2][k], xi[3][k]};
                st4(reinterpret_cast<Real *>(a.noise[k]) + slot, o);
            }
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int k = 0; k < 3; ++k) xi[j][k] *= sc;
    }
    if constexpr (sizeof(Real) == 4) {
        // forward run merging: one running total, flushed when the cell changes
        constexpr int NW = Words32<RULE>::n;
        long long acc[MAX_WORDS32];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            long long w[MAX_WORDS32];
            record_terms<RULE>(m, vx[j], vy[j], vz[j], xi[j], false, w);
            if (j > 0 && j < nv && cc[j] == cc[j - 1]) {
#pragma unroll
                for (int k = 0; k < NW; ++k) acc[k] += w[k];
            } else {
                if (j > 0 && j - 1 < nv)
#pragma unroll
                    for (int k = 0; k < NW; ++k) red_add(sums + k * C + cc[j - 1], acc[k]);
#pragma unroll
                for (int k = 0; k < NW; ++k) acc[k] = w[k];
            }
        }
        if (nv == 4)
#pragma unroll
            for (int k = 0; k < NW; ++k) red_add(sums + k * C + cc[3], acc[k]);
    } else {
        constexpr int NW = RULE == 0 ? 6 : 8;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j >= nv) break;
            double w[NW];
            terms64<RULE>(m, vx[j], vy[j], vz[j], xi[j], w);
#pragma unroll
            for (int k = 0; k < NW; ++k) red_add(sums + k * C + cc[j], w[k]);
        }
    }
}

}  // namespace mpcd
