// d2q9.cuh -- device-side building blocks of the SmrtLBM kernels (sm_103a).
//
// Lattice constants, storage formats, kernel parameters, the boundary
// resolution of a pulled population and the per-node collision operators.
// Everything here is GPU-side code of this library; it shares nothing with the
// CPU oracle.
//
// Storage: every precision stores the offset g_a = f_a - w_a of each population
// (w_a the D2Q9 weight), which keeps the stored numbers small (|g| ~ |u| w) and
// so gains relative precision in every format; rho = 1 + sum g.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "internal.h"

namespace smrt {

// ---- D2Q9 velocity set in the paper's order (listing below Eq. lb.srt) -------
// a: 0 (0,0), 1 (1,0), 2 (0,1), 3 (-1,0), 4 (0,-1), 5 (1,1), 6 (-1,1), 7 (-1,-1), 8 (1,-1)
__host__ __device__ constexpr int ex(int a)
{
    return (a == 1 || a == 5 || a == 8) ? 1 : ((a == 3 || a == 6 || a == 7) ? -1 : 0);
}
__host__ __device__ constexpr int ey(int a)
{
    return (a == 2 || a == 5 || a == 6) ? 1 : ((a == 4 || a == 7 || a == 8) ? -1 : 0);
}
// reversed link: 1<->3, 2<->4, 5<->7, 6<->8
__host__ __device__ constexpr int opp(int a)
{
    return a == 0 ? 0 : (a <= 4 ? ((a + 1) % 4) + 1 : ((a - 3) % 4) + 5);
}
// weights below Eq. (feq-full)
template <class C>
__host__ __device__ constexpr C wgt(int a)
{
    return a == 0 ? C(4) / C(9) : (a <= 4 ? C(1) / C(9) : C(1) / C(36));
}
static_assert(opp(1) == 3 && opp(3) == 1 && opp(2) == 4 && opp(4) == 2, "opp");
static_assert(opp(5) == 7 && opp(7) == 5 && opp(6) == 8 && opp(8) == 6, "opp");
static_assert(ex(opp(6)) == -ex(6) && ey(opp(6)) == -ey(6), "opp");

// ---- launches that follow one another -------------------------------------------
// An update kernel may be launched before the one in front of it has quite ended (programmatic dependent launch):
// its blocks come up while their predecessor's last ones drain, and wait for it to be complete, with its writes
// visible, before they touch the state.  What the predecessor writes is therefore not constant over the kernel's
// lifetime: such a kernel must not take it as a __restrict__ parameter, which would allow non-coherent loads and
// loads moved in front of the wait.  What overlaps is launch latency alone, 0.5-2 us per launch (us per update,
// before -> after: 64^2 f64 3.8 -> 3.3, 256^2 f64 10.3 -> 8.8, 256^2 f32 in place 6.2 -> 4.1, 1021 x 509 f32
// 6.2 -> 5.4, 1024^2 f32 10.3 -> 9.7).  Letting the successor up as soon as all blocks have started
// (griddepcontrol.launch_dependents) was worse: its waiting blocks crowd the running ones (256^2 f64 20.7).
__device__ __forceinline__ void follow_predecessor()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <class... P, class... A>
inline cudaError_t launch_following(void (*kernel)(P...), unsigned blocks, unsigned threads, size_t shared,
                                    cudaStream_t s, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = shared;
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, P(args)...);
    if (e != cudaSuccess) cudaGetLastError();        // told here: not to be found again by the next launch
    return e;
}

// ---- storage formats ----------------------------------------------------------
// R: the raw stored type; C: the arithmetic type.
template <int PREC> struct Prec;
template <> struct Prec<SMRT_PREC_F64> {
    using R = double;
    using C = double;
    static constexpr bool kExactWeights = true;
    static __device__ __forceinline__ C to_c(R r) { return r; }
    static __device__ __forceinline__ R to_r(C c) { return c; }
};
template <> struct Prec<SMRT_PREC_F32> {
    using R = float;
    using C = float;
    static constexpr bool kExactWeights = true;
    static __device__ __forceinline__ C to_c(R r) { return r; }
    static __device__ __forceinline__ R to_r(C c) { return c; }
};
// Stochastic rounding (to_r_sr): c goes to one of its two neighbours in the storage format, the
// farther one with probability equal to the distance from the nearer one (in units of their
// spacing), so that the expected stored value is c itself.  r supplies 16 uniform bits.
// BF16 keeps the upper 16 bits of the float: adding r to the lower 16 and truncating is exactly
// that.  IEEE half keeps 10 of float's 23 mantissa bits where it is normal (|c| >= 2^-14): add 13 of
// the bits below them and truncate; below that its spacing is fixed at 2^-24, so a uniform fraction
// of 2^-24 is added before truncating.  Truncation is toward zero on the magnitude, so the rounding
// is symmetric in the sign.  The fraction is made in the FP32 pipe: 2^23 + r is an OR, and the product
// r 2^-40 is exact, so one multiply-add rounds as the separate addition would.  (Converting r as an
// integer took the quarter-rate conversion unit once per population: without it 8192^2 in place went
// from 129.8k to 134.6k MLUPS, three updates per pass from 124.7k to 136.0k.)
// to_r2_sr rounds two values into one packed word (a below b), the same bits as two calls of to_r_sr.
template <> struct Prec<SMRT_PREC_F16> {
    using R = unsigned short;
    using C = float;
    static constexpr bool kExactWeights = false;
    static __device__ __forceinline__ C to_c(R r) { return __half2float(__ushort_as_half(r)); }
    static __device__ __forceinline__ R to_r(C c) { return __half_as_ushort(__float2half_rn(c)); }
    // c and its dither: truncating this to half is the stochastic rounding of c
    static __device__ __forceinline__ float dithered(C c, uint32_t r)
    {
        const float yn = __uint_as_float(__float_as_uint(c) + (r & 0x1FFFu));
        const float u = __uint_as_float(0x4B000000u | (r & 0xFFFFu)) - 8388608.0f;
        const float ys = fmaf(u, copysignf(0x1p-40f, c), c);
        return fabsf(c) >= 6.103515625e-05f ? yn : ys;
    }
    static __device__ __forceinline__ R to_r_sr(C c, uint32_t r)
    {
        return __half_as_ushort(__float2half_rz(dithered(c, r)));
    }
    static __device__ __forceinline__ uint32_t to_r2_sr(C a, C b, uint32_t ra, uint32_t rb)
    {
        uint32_t d;
        asm("cvt.rz.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(dithered(b, rb)), "f"(dithered(a, ra)));
        return d;
    }
};
template <> struct Prec<SMRT_PREC_BF16> {
    using R = unsigned short;
    using C = float;
    static constexpr bool kExactWeights = false;
    static __device__ __forceinline__ C to_c(R r) { return __bfloat162float(__ushort_as_bfloat16(r)); }
    static __device__ __forceinline__ R to_r(C c) { return __bfloat16_as_ushort(__float2bfloat16_rn(c)); }
    static __device__ __forceinline__ R to_r_sr(C c, uint32_t r)
    {
        return (R)((__float_as_uint(c) + (r & 0xFFFFu)) >> 16);
    }
    static __device__ __forceinline__ uint32_t to_r2_sr(C a, C b, uint32_t ra, uint32_t rb)
    {
        return __byte_perm(__float_as_uint(a) + (ra & 0xFFFFu), __float_as_uint(b) + (rb & 0xFFFFu), 0x7632);
    }
};

// Counter-based random bits of the stochastic rounding: a 32-bit mix of the node's linear index and
// the step's salt (two multiply-xorshift rounds), and from it 16 bits per population by an odd
// multiplier per population (the upper half of the product).  Keyed by (node, population, time), so
// every layout and every code path that stores f*_a(x, t) draws the same bits.
__device__ __forceinline__ uint32_t sr_node_hash(uint32_t node, uint32_t salt)
{
    uint32_t h = node * 0x9E3779B1u + salt;
    h ^= h >> 16;
    h *= 0x7FEB352Du;
    h ^= h >> 15;
    h *= 0x846CA68Bu;
    h ^= h >> 16;
    return h;
}
__device__ __forceinline__ uint32_t sr_pop_bits(uint32_t h, int a)
{
    const uint32_t m = a == 0 ? 0x9E3779B1u : a == 1 ? 0x85EBCA77u : a == 2 ? 0xC2B2AE3Du : a == 3 ? 0x27D4EB2Fu
                     : a == 4 ? 0x165667B1u : a == 5 ? 0xD3A2646Du : a == 6 ? 0xFD7046C5u : a == 7 ? 0xB55A4F09u
                     : 0x2545F491u;
    return (h * m) >> 16;
}
// The salt of the step that starts from time t (host side).
inline uint32_t sr_salt(long long t)
{
    uint64_t x = (uint64_t)t * 0x9E3779B97F4A7C15ull + 0x632BE59BD9B4E019ull;
    x ^= x >> 31;
    x *= 0xBF58476D1CE4E5B9ull;
    x ^= x >> 29;
    return (uint32_t)(x >> 16);
}

// ---- kernel parameters --------------------------------------------------------
enum { SIDE_LEFT = 0, SIDE_RIGHT = 1, SIDE_BOTTOM = 2, SIDE_TOP = 3 };

template <class C>
struct Params {
    int nx, ny;
    int pitch;          // elements per stored row (>= nx, 128-byte multiple)
    long long plane;    // elements per population plane (pitch * ny)
    int periodic_x;     // left/right periodic
    int periodic_y;     // bottom/top periodic
    C omega;            // 1 / tau
    C omega_s;          // 1 / tau_s (two-relaxation-time form)
    C a4;               // (1 - 1/tau) / 4, SmrtLBM
    C trt4;             // (1/tau_s - 1/tau) / 4, two-relaxation-time form
    C keep, keep_s;     // 1 - 1/tau, 1 - 1/tau_s       (the double collision)
    C deq, deq_s;       // 1/4 - a4 = 1/(4 tau), 1/4 - tau_s trt4 = tau_s/(4 tau)   (the double collision)
    C corr[4][9];       // moving-wall term 6 w_a (e_a . u_w(side)) added to a wall-pulled offset
    int *flag;          // divergence flag (bit 0)
    uint32_t salt;      // stochastic rounding: the salt of this launch's time step
};

template <class C>
inline Params<C> make_params(const HostParams &h)
{
    Params<C> p;
    p.nx = h.nx;
    p.ny = h.ny;
    p.pitch = h.pitch;
    p.plane = h.plane;
    p.periodic_x = ((h.bc & 3u) == SMRT_BC_PERIODIC);
    p.periodic_y = (((h.bc >> 4) & 3u) == SMRT_BC_PERIODIC);
    p.omega = C(1.0 / h.tau);
    p.omega_s = C(1.0 / h.tau_s);
    p.a4 = C((1.0 - 1.0 / h.tau) / 4.0);
    p.trt4 = C((1.0 / h.tau_s - 1.0 / h.tau) / 4.0);
    p.keep = C(1.0 - 1.0 / h.tau);
    p.keep_s = C(1.0 - 1.0 / h.tau_s);
    p.deq = C(0.25 / h.tau);
    p.deq_s = C(0.25 * h.tau_s / h.tau);
    for (int s = 0; s < 4; ++s) {
        unsigned kind = (h.bc >> (2 * s)) & 3u;
        double wx = 0.0, wy = 0.0;
        if (kind == SMRT_BC_MOVING) {
            if (s == SIDE_BOTTOM || s == SIDE_TOP) wx = h.u_lid;
            else wy = h.u_lid;
        }
        for (int a = 0; a < 9; ++a)
            p.corr[s][a] = C(6.0 * wgt<double>(a) * (ex(a) * wx + ey(a) * wy));
    }
    p.flag = h.flag;
    p.salt = sr_salt(h.t);
    return p;
}

// ---- boundary resolution --------------------------------------------------------
// Where a canonical population f_a(i, j) is found in storage.  `side` >= 0 marks a
// wall link (the pull source lies behind a wall on that side) whose stored value
// needs the moving-wall term p.corr[side][a] added.
struct Loc {
    int plane, j, i, side;
};

// Resolve the node (i + di, j + dj): wraps periodic axes; returns the wall side
// crossed (bottom/top take precedence over left/right), or -1 if inside.
template <class C>
__device__ __forceinline__ int resolve(const Params<C> &p, int &i, int &j)
{
    int wy = -1, wx = -1;
    if (j < 0) {
        if (p.periodic_y) j += p.ny; else wy = SIDE_BOTTOM;
    } else if (j >= p.ny) {
        if (p.periodic_y) j -= p.ny; else wy = SIDE_TOP;
    }
    if (i < 0) {
        if (p.periodic_x) i += p.nx; else wx = SIDE_LEFT;
    } else if (i >= p.nx) {
        if (p.periodic_x) i -= p.nx; else wx = SIDE_RIGHT;
    }
    return wy >= 0 ? wy : wx;
}

// Location of canonical f_a(i, j) under each storage mode:
//  AB      : f_a(x) = B_a(x - e_a)                    wall: B_{abar}(x) + corr
//  AA even : f_a(x) = F_a(x)                          wall: F_a(x) + corr
//  AA odd  : f_a(x) = F_{abar}(x - e_a)               wall: F_a(x) + corr
template <int MODE, class C>
__device__ __forceinline__ Loc pull_loc(const Params<C> &p, int a, int i, int j)
{
    int si = i - ex(a), sj = j - ey(a);
    int side = resolve(p, si, sj);
    Loc L;
    L.side = side;
    if (side >= 0) {
        L.plane = (MODE == MODE_AB) ? opp(a) : a;
        L.j = j;
        L.i = i;
    } else if (MODE == MODE_AA_EVEN) {
        L.plane = a;
        L.j = j;
        L.i = i;
    } else {
        L.plane = (MODE == MODE_AB) ? a : opp(a);
        L.j = sj;
        L.i = si;
    }
    return L;
}

// Where the post-collision f*_a(i, j) is written by a step of each mode:
//  AB      : B'_a(x)
//  AA even : F_{abar}(x)
//  AA odd  : F_a(x + e_a), or F_{abar}(x) when x + e_a lies behind a wall
template <int MODE, class C>
__device__ __forceinline__ Loc push_loc(const Params<C> &p, int a, int i, int j)
{
    Loc L;
    L.side = -1;
    if (MODE == MODE_AB) {
        L.plane = a; L.j = j; L.i = i;
    } else if (MODE == MODE_AA_EVEN) {
        L.plane = opp(a); L.j = j; L.i = i;
    } else {
        int ti = i + ex(a), tj = j + ey(a);
        int side = resolve(p, ti, tj);
        if (side >= 0) {
            L.plane = opp(a); L.j = j; L.i = i;
        } else {
            L.plane = a; L.j = tj; L.i = ti;
        }
    }
    return L;
}

__device__ __forceinline__ size_t at(long long plane_elems, int pitch, int plane, int j, int i)
{
    return (size_t)plane * (size_t)plane_elems + (size_t)j * (size_t)pitch + (size_t)i;
}

// ---- collision ------------------------------------------------------------------
// x * w for the D2Q9 weight w (4/9, 1/9 or 1/36), with the product rounded as if the
// weight were exact.  In float, w rounds to fl(w) = w (1 + 7.45e-9) for all three
// weights; a plain product would scale the equilibrium's mass and momentum by that
// factor at every collision (sum_a w_a = 1 and sum_a w_a e_a e_a = 1/3 hold for
// fl(w) only up to it).  The update then pushes the flow along itself by 7.45e-9 of
// its momentum per step, a coherent bias that grows linearly in time.  The split
// w = hi + lo (hi = fl(w), lo = fl(w - hi)) and one fused multiply-add remove it.
// Doubles keep the plain product: there the same bias is about 1e-17 per step.  So do the 16-bit
// storage formats (EXACT = false): rounding a stored offset to 11 or 8 significant bits moves it by
// 1e-4 to 1e-3 of itself each step, which buries the 7e-9, while the two extra operations per
// population cost their near-ALU-bound kernels several per cent.
template <class C, bool EXACT = true>
struct WeightMul {
    template <int A>
    static __device__ __forceinline__ C mul(C x) { return wgt<C>(A) * x; }
};
template <>
struct WeightMul<float, true> {
    template <int A>
    static __device__ __forceinline__ float mul(float x)
    {
        constexpr double w = wgt<double>(A);
        constexpr float hi = (float)w;
        constexpr float lo = (float)(w - (double)hi);
        return fmaf(hi, x, lo * x);
    }
};

// In:  g[a] = f_a - w_a (canonical offsets at one node).
// Out: g[a] = f*_a - w_a (post-collision offsets).
// Returns false when rho is not a positive finite number (divergence).
//
// Moments (Eq. fea-0):   rho = 1 + sum g,  j = sum e_a g_a,  u = j / rho.
// Equilibrium offsets (Eq. feq-full), written with rho u = j so that the momentum of
// the equilibrium is j itself rather than rho (j / rho) rounded twice:
//   f^eq_a - w_a = w_a [ (rho - 1) + 3 e.j + 9/2 (e.j)(e.u) - 3/2 j.u ].
// SmrtLBM (Eq. SmrtLBM-1): with n_k = f_k - f^eq_k the indicator sum is
//   C1 = (-n1 + n2 - n3 + n4)/4 for a in 1..4 and C2 = (-n5 + n6 - n7 + n8)/4 for
//   a in 5..8, so with Pxx = n1 - n2 + n3 - n4 = -4 C1 and Pxy = n5 - n6 + n7 - n8 = -4 C2
//   f*_a = f^eq_a + (-1)^a (1 - 1/tau) C = f^eq_a + s_a (1 - 1/tau)/4 P,
//   s = (+,-,+,-) over a = 1..4 (P = Pxx) and over a = 5..8 (P = Pxy), f*_0 = f^eq_0.
// SRT (Eq. lb.srt): f*_a = f_a - (f_a - f^eq_a) / tau.
// Two-tau (Eq. SmrtLBM-lb.1.5): f*_a = f_a - (f_a - f^eq_a)/tau_s + s_a (1/tau_s - 1/tau)/4 P.
//
// Double: this GPU starts a warp's double operation every 64 clocks per SM sub-partition, so their number is
// the kernel's time.  With the even and odd parts of each opposite pair, K = j.u, D = jx ux - jy uy and
// jx uy, the equilibrium is
//   f^eq_0 - w_0 = 4/9 drho - 2/3 K,   axes: drho/9 + K/12 +- D/4 +- j/3,   diagonals: drho/36 + K/12 +- jx uy/4
//   +- (jx +- jy)/12,
// and its P^eq are D and jx uy themselves, so the collision needs 52 operations (SmrtLBM) where the
// populations one by one took 75: 4096^2 2.31 -> 1.62 ms per update, 10.4 G updates/s.  1/rho is the hardware's approximation
// (20 bits) and one step of Halley's iteration, within one unit in the last place of the division; the
// check of rho works on its upper word.
__device__ __forceinline__ double recip_d(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

template <int KIND, bool EXACT = true>
__device__ __forceinline__ bool collide(const Params<double> &p, double g[9])
{
    const double s13 = g[1] + g[3], s24 = g[2] + g[4], s57 = g[5] + g[7], s68 = g[6] + g[8];
    const double d13 = g[1] - g[3], d24 = g[2] - g[4], d57 = g[5] - g[7], d68 = g[6] - g[8];
    double drho = g[0] + ((s13 + s24) + (s57 + s68));
    const double rho = 1.0 + drho;
    double jx = d13 + (d57 - d68), jy = d24 + (d57 + d68);
    const double inv = recip_d(rho);
    const double ux = jx * inv, uy = jy * inv;
    const int hi = __double2hiint(rho);
    const bool ok = (unsigned)hi < 0x7ff00000u && (hi | __double2loint(rho)) != 0;
    if (KIND != SMRT_COLLISION_SMRT) {          // the equilibrium's share of f*
        const double o = KIND == SMRT_COLLISION_SRT ? p.omega : p.omega_s;
        drho *= o;
        jx *= o;
        jy *= o;
    }
    const double xx = jx * ux, yy = jy * uy, xy = jx * uy;
    const double K = xx + yy, D = xx - yy, k12 = K * (1.0 / 12.0);
    double n, m;                                 // what P adds to the axes and the diagonals
    if (KIND == SMRT_COLLISION_SMRT) {
        n = fma(p.a4, s13 - s24, p.deq * D);
        m = fma(p.a4, s57 - s68, p.deq * xy);
    } else if (KIND == SMRT_COLLISION_SRT) {
        n = 0.25 * D;
        m = 0.25 * xy;
    } else {
        n = fma(p.trt4, s13 - s24, p.deq_s * D);
        m = fma(p.trt4, s57 - s68, p.deq_s * xy);
    }
    const double a = fma(drho, 1.0 / 9.0, k12), b = fma(drho, 1.0 / 36.0, k12);
    const double ax = a + n, ay = a - n, bp = b + m, bm = b - m;
    const double jp = jx + jy, jm = jx - jy;
    const double q0 = fma(drho, 4.0 / 9.0, K * (-2.0 / 3.0));
    const double q1 = fma(jx, 1.0 / 3.0, ax), q3 = fma(jx, -1.0 / 3.0, ax);
    const double q2 = fma(jy, 1.0 / 3.0, ay), q4 = fma(jy, -1.0 / 3.0, ay);
    const double q5 = fma(jp, 1.0 / 12.0, bp), q7 = fma(jp, -1.0 / 12.0, bp);
    const double q8 = fma(jm, 1.0 / 12.0, bm), q6 = fma(jm, -1.0 / 12.0, bm);
    const double q[9] = {q0, q1, q2, q3, q4, q5, q6, q7, q8};
    #pragma unroll
    for (int k = 0; k < 9; ++k)
        g[k] = KIND == SMRT_COLLISION_SMRT ? q[k] : fma(KIND == SMRT_COLLISION_SRT ? p.keep : p.keep_s, g[k], q[k]);
    return ok;
}

// ---- float arithmetic, one or two nodes at a time ----------------------------------
// F2 holds the values of two nodes in a register pair; its operations are the packed add, sub, mul
// and fma of this architecture: one instruction rounds both halves like the scalar one, so a node
// gets the same bits either way at half the issue slots (the FMA rate is the same).
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 f2(float lo, float hi)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float f2_lo(F2 x)
{
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(x.v));
    return lo;
}
__device__ __forceinline__ float f2_hi(F2 x)
{
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(x.v));
    return hi;
}
__device__ __forceinline__ F2 vadd(F2 a, F2 b)
{
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 vsub(F2 a, F2 b)
{
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 vmul(F2 a, F2 b)
{
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 vfma(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
template <class V> __device__ __forceinline__ V vset(float c);
template <> __device__ __forceinline__ F2 vset<F2>(float c) { return f2(c, c); }

// Four nodes, two by two: written so that the two halves' operations alternate.
struct F4 {
    F2 a, b;
};
__device__ __forceinline__ F4 vadd(F4 x, F4 y) { return {vadd(x.a, y.a), vadd(x.b, y.b)}; }
__device__ __forceinline__ F4 vsub(F4 x, F4 y) { return {vsub(x.a, y.a), vsub(x.b, y.b)}; }
__device__ __forceinline__ F4 vmul(F4 x, F4 y) { return {vmul(x.a, y.a), vmul(x.b, y.b)}; }
__device__ __forceinline__ F4 vfma(F4 x, F4 y, F4 z) { return {vfma(x.a, y.a, z.a), vfma(x.b, y.b, z.b)}; }
__device__ __forceinline__ F4 vsub(F2 x, F4 y) { return {vsub(x, y.a), vsub(x, y.b)}; }
__device__ __forceinline__ F4 vmul(F2 x, F4 y) { return {vmul(x, y.a), vmul(x, y.b)}; }
__device__ __forceinline__ F4 vfma(F2 x, F4 y, F4 z) { return {vfma(x, y.a, z.a), vfma(x, y.b, z.b)}; }

// 1 / rho from -rho, correctly rounded wherever rho and 1 / rho are normal: the hardware's
// approximation, good to one unit in the last place, and one Newton step with an exact residual,
// which Markstein (1990) shows to round correctly (compared with the division for every float with
// an exponent from 2^-126 to 2^125: equal).  The division's own sequence has a branch per node, for the
// other operands, that keeps the nodes of a thread from overlapping.  Where rho is zero, infinite or
// NaN the node has diverged and the result is NaN.
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ F2 vrecip_neg(F2 nrho, F2 one)
{
    const F2 r = f2(rcp_approx(-f2_lo(nrho)), rcp_approx(-f2_hi(nrho)));
    return vfma(r, vfma(nrho, r, one), r);
}

__device__ __forceinline__ F4 vrecip_neg(F4 nrho, F2 one)
{
    const F4 r = {f2(rcp_approx(-f2_lo(nrho.a)), rcp_approx(-f2_hi(nrho.a))),
                  f2(rcp_approx(-f2_lo(nrho.b)), rcp_approx(-f2_hi(nrho.b)))};
    const F4 e = {vfma(nrho.a, r.a, one), vfma(nrho.b, r.b, one)};
    return vfma(r, e, r);
}

// The constants of collide_v are kernel arguments, so that the packed
// instructions take them from there and need no register pair (nor the moves that fill one) for each.
struct CollideConsts {
    F2 m1, p1, m15, c45, p3, m3;          // -1, 1, -3/2, 9/2, 3, -3
    F2 hi[3], lo[3], mhi[3];              // the weights of the rest, axis and diagonal populations: w = hi + lo, and -hi
    F2 r, s, t;                          // relaxation: -1/tau (SRT) or -1/tau_s (two-tau); +-(the P factor)
};
inline void cc_set(F2 &v, float c)
{
    union { float f[2]; unsigned long long u; } w = {{c, c}};
    v.v = w.u;
}
template <int KIND>
inline CollideConsts collide_consts(const Params<float> &p)
{
    CollideConsts k;
    cc_set(k.m1, -1.0f);
    cc_set(k.p1, 1.0f);
    cc_set(k.m15, -1.5f);
    cc_set(k.c45, 4.5f);
    cc_set(k.p3, 3.0f);
    cc_set(k.m3, -3.0f);
    for (int x = 0; x < 3; ++x) {
        const double w = wgt<double>(x == 0 ? 0 : x == 1 ? 1 : 5);
        const float hi = (float)w;
        cc_set(k.hi[x], hi);
        cc_set(k.lo[x], (float)(w - (double)hi));
        cc_set(k.mhi[x], -hi);
    }
    const float f = KIND == SMRT_COLLISION_SMRT ? p.a4 : p.trt4;
    cc_set(k.r, KIND == SMRT_COLLISION_SRT ? -p.omega : -p.omega_s);
    cc_set(k.s, f);
    cc_set(k.t, -f);
    return k;
}

template <bool SPLIT>
__device__ __forceinline__ F2 vfma_last(int dir, F2 a, F2 b, F2 c)
{
    if (SPLIT && ex(dir) != 0)
        return f2(__fmaf_rn(f2_lo(a), f2_lo(b), f2_lo(c)), __fmaf_rn(f2_hi(a), f2_hi(b), f2_hi(c)));
    return vfma(a, b, c);
}

template <bool SPLIT>
__device__ __forceinline__ F4 vfma_last(int dir, F2 a, F4 b, F4 c)
{
    return {vfma_last<SPLIT>(dir, a, b.a, c.a), vfma_last<SPLIT>(dir, a, b.b, c.b)};
}
// The collision of float populations on F4, every operation rounded as written.  Returns -rho.
// EXACT: the weight products are those of WeightMul<float, true>; otherwise they are plain, and fused
// with the operation that follows.  SPLIT: the last operation of the populations that move along x works
// on each half by itself: its caller regroups the halves for the shift, and a scalar result lands in
// either half of a register pair without a move.
template <int KIND, bool EXACT, bool SPLIT>
__device__ __forceinline__ F4 collide_v(const CollideConsts &k, F4 g[9])
{
    using V = F4;
    const V drho = vadd(vadd(vadd(vadd(g[0], g[1]), vadd(g[2], g[3])),
                             vadd(vadd(g[4], g[5]), vadd(g[6], g[7]))), g[8]);
    const V nrho = vsub(k.m1, drho);
    const V jx = vadd(vadd(vsub(g[1], g[3]), vsub(g[5], g[6])), vsub(g[8], g[7]));
    const V jy = vsub(vadd(vsub(g[2], g[4]), vadd(g[5], g[6])), vadd(g[7], g[8]));
    const V inv = vrecip_neg(nrho, k.p1);
    const V ux = vmul(jx, inv), uy = vmul(jy, inv);
    const V base = vfma(k.m15, vfma(jx, ux, vmul(jy, uy)), drho);
    const V jp = vadd(jx, jy), jm = vsub(jx, jy);
    const V up = vadd(ux, uy), um = vsub(ux, uy);
    const V axx = vfma(vmul(k.c45, jx), ux, base), ayy = vfma(vmul(k.c45, jy), uy, base);
    const V app = vfma(vmul(k.c45, jp), up, base), amm = vfma(vmul(k.c45, jm), um, base);
    // q_a = w_a x_a
    const V x[9] = {base, vfma(k.p3, jx, axx), vfma(k.p3, jy, ayy), vfma(k.m3, jx, axx), vfma(k.m3, jy, ayy),
                    vfma(k.p3, jp, app), vfma(k.m3, jm, amm), vfma(k.m3, jp, app), vfma(k.p3, jm, amm)};
    V q[9], n[9];
    #pragma unroll
    for (int a = 0; a < 9; ++a) {
        const int w = a == 0 ? 0 : a < 5 ? 1 : 2;
        if (EXACT) {
            q[a] = vfma(k.hi[w], x[a], vmul(k.lo[w], x[a]));
            n[a] = vsub(g[a], q[a]);
        } else {
            n[a] = vfma(k.mhi[w], x[a], g[a]);
        }
    }
    if (KIND == SMRT_COLLISION_SRT) {
        #pragma unroll
        for (int a = 0; a < 9; ++a) g[a] = vfma_last<SPLIT>(a, k.r, n[a], g[a]);
        return nrho;
    }
    const V pxx = vsub(vadd(n[1], n[3]), vadd(n[2], n[4]));
    const V pxy = vsub(vadd(n[5], n[7]), vadd(n[6], n[8]));
    if (KIND == SMRT_COLLISION_SMRT) {
        if (EXACT) {
            g[0] = q[0];
            #pragma unroll
            for (int a = 1; a < 9; ++a) g[a] = vfma_last<SPLIT>(a, (a & 1) ? k.s : k.t, a < 5 ? pxx : pxy, q[a]);
        } else {
            const V txx = vmul(k.s, pxx), txy = vmul(k.s, pxy), sxx = vmul(k.t, pxx), sxy = vmul(k.t, pxy);
            g[0] = vmul(k.hi[0], x[0]);
            #pragma unroll
            for (int a = 1; a < 9; ++a)
                g[a] = vfma_last<SPLIT>(a, k.hi[a < 5 ? 1 : 2], x[a],
                                        a < 5 ? ((a & 1) ? txx : sxx) : ((a & 1) ? txy : sxy));
        }
    } else {
        g[0] = vfma(k.r, n[0], g[0]);
        #pragma unroll
        for (int a = 1; a < 9; ++a) g[a] = vfma_last<SPLIT>(a, (a & 1) ? k.s : k.t, a < 5 ? pxx : pxy, vfma(k.r, n[a], g[a]));
    }
    return nrho;
}

// One node by plain expressions, which the compiler contracts to the operations of collide_v (compared bit for
// bit): for the kernels bound by memory, where this form measured 2-4 % faster in 16-bit storage.
template <int KIND, bool EXACT = true>
__device__ __forceinline__ bool collide(const Params<float> &p, float g[9])
{
    using C = float;
    using M = WeightMul<C, EXACT>;
    const C drho = ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7])) + g[8];
    const C rho = C(1) + drho;
    const C jx = (g[1] - g[3]) + (g[5] - g[6]) + (g[8] - g[7]);
    const C jy = (g[2] - g[4]) + (g[5] + g[6]) - (g[7] + g[8]);
    const C inv = C(1) / rho;
    const C ux = jx * inv, uy = jy * inv;
    const bool ok = (rho > C(0)) && (rho < C(INFINITY));

    const C base = drho - C(1.5) * (jx * ux + jy * uy);
    const C jp = jx + jy, jm = jx - jy;
    const C up = ux + uy, um = ux - uy;
    const C axx = base + C(4.5) * jx * ux, bxx = C(3) * jx;
    const C ayy = base + C(4.5) * jy * uy, byy = C(3) * jy;
    const C app = base + C(4.5) * jp * up, bpp = C(3) * jp;
    const C amm = base + C(4.5) * jm * um, bmm = C(3) * jm;
    C q[9];
    q[0] = M::template mul<0>(base);
    q[1] = M::template mul<1>(axx + bxx);
    q[3] = M::template mul<3>(axx - bxx);
    q[2] = M::template mul<2>(ayy + byy);
    q[4] = M::template mul<4>(ayy - byy);
    q[5] = M::template mul<5>(app + bpp);
    q[7] = M::template mul<7>(app - bpp);
    q[8] = M::template mul<8>(amm + bmm);
    q[6] = M::template mul<6>(amm - bmm);

    if (KIND == SMRT_COLLISION_SRT) {
        #pragma unroll
        for (int a = 0; a < 9; ++a) g[a] = g[a] - p.omega * (g[a] - q[a]);
        return ok;
    }
    const C pxx = ((g[1] - q[1]) + (g[3] - q[3])) - ((g[2] - q[2]) + (g[4] - q[4]));
    const C pxy = ((g[5] - q[5]) + (g[7] - q[7])) - ((g[6] - q[6]) + (g[8] - q[8]));
    if (KIND == SMRT_COLLISION_SMRT) {
        const C txx = p.a4 * pxx, txy = p.a4 * pxy;
        g[0] = q[0];
        g[1] = q[1] + txx;
        g[3] = q[3] + txx;
        g[2] = q[2] - txx;
        g[4] = q[4] - txx;
        g[5] = q[5] + txy;
        g[7] = q[7] + txy;
        g[6] = q[6] - txy;
        g[8] = q[8] - txy;
    } else {
        const C txx = p.trt4 * pxx, txy = p.trt4 * pxy;
        #pragma unroll
        for (int a = 0; a < 9; ++a) g[a] = g[a] - p.omega_s * (g[a] - q[a]);
        g[1] += txx;
        g[3] += txx;
        g[2] -= txx;
        g[4] -= txx;
        g[5] += txy;
        g[7] += txy;
        g[6] -= txy;
        g[8] -= txy;
    }
    return ok;
}

} // namespace smrt
