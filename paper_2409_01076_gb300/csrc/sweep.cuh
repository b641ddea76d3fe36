// sweep.cuh -- T updates of the two-buffer layout in one pass over memory (float arithmetic: the 32-
// and 16-bit storage formats).
//
// One update moves 9 reads and 9 writes per node, and step_kernel does that at the copy bandwidth, so
// the only way past it is to move the state less often.  A warp owns a strip of 32 x 4 columns (120 of
// them its own, 4 on either side shared with its neighbours) and a segment of rows, and walks it from
// the row below to the row above.  For each row every lane pulls and collides its four nodes (update 1)
// and rounds f* as the step would store it; update 2 of the row before it follows at once from
// registers, update 3 of the row before that, and only the last one's result goes to memory.  Between
// two updates a warp keeps 9 values per node: of the row before the one just collided the populations
// that arrive along x (0, 1, 3), of that row and the one before those that arrive from below (2, 5, 6);
// those that arrive from above (4, 7, 8) come from the row just collided; the shifts along x are warp
// shuffles.  The same operations on the same values as T calls of step_kernel, hence the same bits; the
// shared rows and columns are computed more than once: (rows + T - 1) / rows x 128 / 120 collisions per
// node and update.  The raw populations of the next row are loaded while the current row collides.
//
// With the memory traffic divided by T the kernel is bound by instruction issue, so nodes are collided
// two at a time (F2), and an item is one 32-thread block, which makes every row address uniform.
#pragma once

#include "d2q9.cuh"

namespace smrt {

constexpr int kSwOwn = 120;          // own columns of a strip; the first and last between walls own their outer 4 too
constexpr int kSwBlocks = 15;        // resident per SM (f32, T = 3: 15 KB of shared memory, 136 registers)
constexpr int kSwSeamBlocks = 12;    // 168 registers for the element picking at the seam
constexpr int kSwHalo = 4;           // shared columns on either side: T <= 4, and 16-byte vectors stay aligned

// Four neighbouring stored values, as in memory.
template <class R> struct Raw4;
template <> struct alignas(16) Raw4<float> {
    float x, y, z, w;
    __device__ __forceinline__ void load(const float *p)
    {
        const float4 v = *reinterpret_cast<const float4 *>(p);
        x = v.x; y = v.y; z = v.z; w = v.w;
    }
    __device__ __forceinline__ void set(const float e[4]) { x = e[0]; y = e[1]; z = e[2]; w = e[3]; }
    __device__ __forceinline__ void store(float *p) const { *reinterpret_cast<float4 *>(p) = make_float4(x, y, z, w); }
    // element k of the result is element k - 1 / k + 1, the outer one from the neighbour lane
    __device__ __forceinline__ Raw4 up() const { return {__shfl_up_sync(0xffffffffu, w, 1), x, y, z}; }
    __device__ __forceinline__ Raw4 down() const { return {y, z, w, __shfl_down_sync(0xffffffffu, x, 1)}; }
    template <int PREC> __device__ __forceinline__ void get(F2 &a, F2 &b) const { a = f2(x, y); b = f2(z, w); }
    template <int PREC> __device__ __forceinline__ void round(F2 a, F2 b)
    {
        x = f2_lo(a); y = f2_hi(a); z = f2_lo(b); w = f2_hi(b);
    }
    __device__ __forceinline__ float at(int k) const { return k == 0 ? x : k == 1 ? y : k == 2 ? z : w; }
    __device__ __forceinline__ void put(int k, float v)
    {
        if (k == 0) x = v;
        if (k == 1) y = v;
        if (k == 2) z = v;
        if (k == 3) w = v;
    }
    __device__ __forceinline__ void zero() { x = y = z = w = 0.0f; }
};
template <> struct alignas(8) Raw4<unsigned short> {
    unsigned x, y;
    __device__ __forceinline__ void load(const unsigned short *p)
    {
        const uint2 v = *reinterpret_cast<const uint2 *>(p);
        x = v.x; y = v.y;
    }
    __device__ __forceinline__ void set(const unsigned short e[4])
    {
        x = (unsigned)e[0] | ((unsigned)e[1] << 16);
        y = (unsigned)e[2] | ((unsigned)e[3] << 16);
    }
    __device__ __forceinline__ void store(unsigned short *p) const { *reinterpret_cast<uint2 *>(p) = make_uint2(x, y); }
    __device__ __forceinline__ Raw4 up() const
    {
        return {__byte_perm(__shfl_up_sync(0xffffffffu, y, 1), x, 0x5432), __byte_perm(x, y, 0x5432)};
    }
    __device__ __forceinline__ Raw4 down() const
    {
        return {__byte_perm(x, y, 0x5432), __byte_perm(y, __shfl_down_sync(0xffffffffu, x, 1), 0x5432)};
    }
    template <int PREC> static __device__ __forceinline__ F2 wide(unsigned v)
    {
        return f2(Prec<PREC>::to_c((unsigned short)v), Prec<PREC>::to_c((unsigned short)(v >> 16)));
    }
    template <int PREC> __device__ __forceinline__ void get(F2 &a, F2 &b) const { a = wide<PREC>(x); b = wide<PREC>(y); }
    template <int PREC> static __device__ __forceinline__ unsigned narrow(F2 v)
    {
        if constexpr (PREC == SMRT_PREC_F16) {
            const __half2 h = __floats2half2_rn(f2_lo(v), f2_hi(v));
            return *reinterpret_cast<const unsigned *>(&h);
        } else {
            const __nv_bfloat162 h = __floats2bfloat162_rn(f2_lo(v), f2_hi(v));
            return *reinterpret_cast<const unsigned *>(&h);
        }
    }
    template <int PREC> __device__ __forceinline__ void round(F2 a, F2 b) { x = narrow<PREC>(a); y = narrow<PREC>(b); }
    __device__ __forceinline__ unsigned short at(int k) const { return (unsigned short)((k < 2 ? x : y) >> (16 * (k & 1))); }
    __device__ __forceinline__ void put(int k, unsigned short v)
    {
        unsigned &h = k < 2 ? x : y;
        h = (k & 1) ? (h & 0xffffu) | ((unsigned)v << 16) : (h & 0xffff0000u) | v;
    }
    __device__ __forceinline__ void zero() { x = y = 0u; }
};

template <int T>
struct SweepSalts {
    uint32_t s[T];
};

// A warp's shared memory.  Every lane reads only what it wrote itself, so no barrier is needed.
//   seam   (behind the struct, only with a periodic x axis and nx % 4 != 0) the second vectors of `row`
//   row    the raw populations that the next row pulls, copied there while the current row collides
//   here   between update m and m + 1: of the row that update m collided last, what stays in the row
//          (0; 1 from c - 1; 3 from c + 1)
//   below  of that row and of the one before it, what goes up (2; 5 from c - 1; 6 from c + 1)
//   wall   of that row, f* of the x-wall nodes (3 7 6 of the left one, 1 8 5 of the right one)
template <class R, int T>
struct SweepShared {
    Raw4<R> row[9][32];
    Raw4<R> here[T - 1][3][32];
    Raw4<R> below[T - 1][2][3][32];
    R wall[T - 1][3][2];
};

template <class R>
__device__ __forceinline__ void copy_row4(Raw4<R> *smem, const R *gmem)
{
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    if (sizeof(R) == 4) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(gmem) : "memory");
}

template <bool B>
struct Bool {
    static constexpr bool value = B;
};

// Strips that cover nx columns.
inline int sweep_strips(int nx, bool periodic_x)
{
    return periodic_x ? (nx + kSwOwn - 1) / kSwOwn : (nx <= 128 ? 1 : (nx - 2 * kSwHalo + kSwOwn - 1) / kSwOwn);
}

// Rows per segment of `count` lattices swept together.  The rows that two segments share are computed
// twice, so long segments do less work, but few warps per SM sub-partition (608 of them) are bound by the
// latency of one warp's walk.  Measured (f32, T = 3, 64^2 to 8192^2): a row of one update takes a warp
// max(0.685, 0.35 + 0.30 w) us with w warps per sub-partition, w also standing for the waves beyond the 4
// resident; the minimum of (rows + T - 1) x that is within 4 % of the best of a sweep over rows at every
// size.  (1024^2: 6 rows, 12.3 us per single update -> 10.9; 4096^2: 20, 178 -> 88; 8192^2: 64, 694 -> 290.)
inline int sweep_rows(const int *strips, const int *ny, int count, int T)
{
    int best = 1;
    double least = 1e300;
    for (int rows = 1; rows <= 64; ++rows) {
        double items = 0.0;
        for (int k = 0; k < count; ++k) items += (double)strips[k] * ((ny[k] + rows - 1) / rows);
        const double one = 0.35 + 0.30 * items / 608.0;
        const double cost = (rows + T - 1) * (one > 0.685 ? one : 0.685);
        if (cost < least) {
            least = cost;
            best = rows;
        }
    }
    return best;
}

// T updates of the rows [r0, r1) of one strip, by one warp (blockDim.x == 32).  Needs nx >= 8 and
// ny >= 8.  salt.s[m] is the stochastic-rounding salt of update m.
// SEAM: a periodic x axis with nx % 4 != 0.
template <int PREC, int KIND, bool SR, int T, bool SEAM>
__device__ __forceinline__ void sweep(const typename Prec<PREC>::R *__restrict__ src,
                                      typename Prec<PREC>::R *__restrict__ dst,
                                      const Params<typename Prec<PREC>::C> &p, const CollideConsts &cc,
                                      const SweepSalts<T> &salt, int strip, int r0, int r1,
                                      SweepShared<typename Prec<PREC>::R, T> &sm,
                                      Raw4<typename Prec<PREC>::R> *seam)
{
    static_assert(T >= 2 && T <= kSwHalo, "shared columns");
    using P = Prec<PREC>;
    using R = typename P::R;
    using Row = Raw4<R>;
    const int lane = threadIdx.x;
    const bool wall_x = !p.periodic_x, wall_y = !p.periodic_y;
    const int x0 = strip * kSwOwn - (wall_x ? 0 : kSwHalo);          // the warp's first column, and the lane's:
    const int c4 = x0 + 4 * lane;                                    // either may lie outside
    const bool own = (lane >= 1 || (wall_x && x0 == 0)) && (lane <= kSwOwn / 4 || (wall_x && x0 + 128 >= p.nx)) &&
                     c4 < p.nx;
    const int ny = p.ny;

    // Column to load from.  Behind a wall the values are not used (any stored column will do); on a
    // periodic axis the columns wrap.  A lane whose four columns are not one aligned vector there (nx not
    // a multiple of 4, by the seam) loads the two vectors that hold them, at lc and lw, and picks its
    // elements when it reads: n1 of them from the first, behind its first `o`, then the second's.
    int lc = max(0, min(c4, p.pitch - 4)), lw = 0, n1 = 4, o = 0;
    if (!wall_x) {
        lc = c4 < 0 ? c4 + p.nx : c4 % p.nx;
        o = SEAM ? lc & 3 : 0;
        if (SEAM && o != 0) {
            lc -= o;
            lw = min(lc + 4, p.pitch - 4);
            n1 = 4 - o;
        } else if (SEAM && lc + 4 > p.nx) {
            n1 = p.nx - lc;
        }
    }
    const bool vec = !SEAM || n1 == 4;
    const bool all_vec = !SEAM || __all_sync(0xffffffffu, vec);
    // x-wall nodes: at most one per lane (nx >= 8)
    const bool edge_strip = wall_x && (x0 == 0 || x0 + 128 >= p.nx);
    const bool at_left = wall_x && c4 == 0, at_right = wall_x && c4 < p.nx && c4 + 4 >= p.nx;
    const int kx = at_right ? (p.nx - 1) & 3 : 0;                    // that node's place in its lane
    const R *col = src + lc;

    auto wrap_row = [&](int r) { return r < 0 ? r + ny : (r >= ny ? r - ny : r); };
    auto at_floor = [&](int r) { return wall_y && r == 0; };
    auto at_top = [&](int r) { return wall_y && r == ny - 1; };
    auto load_row = [&](int r) {                                     // the populations that row r pulls
        const int rw = wrap_row(r);
        const R *mid = col + (size_t)rw * (size_t)p.pitch;
        const R *below = col + (size_t)wrap_row(rw - 1) * (size_t)p.pitch;
        const R *above = col + (size_t)wrap_row(rw + 1) * (size_t)p.pitch;
        const bool b = at_floor(rw), t = at_top(rw);
        #pragma unroll
        for (int a = 0; a < 9; ++a) {
            const R *q = (ey(a) == 0 ? mid : ey(a) > 0 ? (b ? mid : below) : (t ? mid : above)) +
                         (size_t)((ey(a) > 0 && b) || (ey(a) < 0 && t) ? opp(a) : a) * (size_t)p.plane;
            copy_row4<R>(&sm.row[a][lane], q);
            if (!vec) copy_row4<R>(&seam[a * 32 + lane], q + (lw - lc));
        }
    };
    unsigned worst[4] = {0u, 0u, 0u, 0u};                            // of -rho by column, in an order that ends with the diverged ones

    // Collides the pulled row j (its populations shifted, wall pulls unshifted and without the moving-wall
    // term; e: the x-wall node's bounce-back values) and rounds f* to the storage format.
    auto collide_row = [&](auto last, Row f[9], const R e[3], int j, uint32_t s) {
        F2 g[2][9];
        #pragma unroll
        for (int a = 0; a < 9; ++a) f[a].template get<PREC>(g[0][a], g[1][a]);
        const bool b = at_floor(j), t = at_top(j);
        if (b || t) {
            #pragma unroll
            for (int a = 1; a < 9; ++a)
                if ((ey(a) > 0 && b) || (ey(a) < 0 && t)) {
                    const F2 w = vset<F2>(p.corr[ey(a) > 0 ? SIDE_BOTTOM : SIDE_TOP][a]);
                    g[0][a] = vadd(g[0][a], w);
                    g[1][a] = vadd(g[1][a], w);
                }
        }
        if (edge_strip && (at_left || at_right)) {
            #pragma unroll
            for (int a = 1; a < 9; ++a) {
                if (ex(a) == 0) continue;
                // the order of `wall` (SweepShared); a link through the bottom or top wall is that wall's
                const bool here = (ex(a) > 0 ? at_left : at_right) && !((ey(a) > 0 && b) || (ey(a) < 0 && t));
                const int x = ey(a) == 0 ? 0 : ey(a) > 0 ? 1 : 2;
                if (here) {
                    const float v = __fadd_rn(P::to_c(e[x]), p.corr[ex(a) > 0 ? SIDE_LEFT : SIDE_RIGHT][a]);
                    #pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (kx == 2 * h) g[h][a] = f2(v, f2_hi(g[h][a]));
                        if (kx == 2 * h + 1) g[h][a] = f2(f2_lo(g[h][a]), v);
                    }
                }
            }
        }
        F4 v[9];
        #pragma unroll
        for (int a = 0; a < 9; ++a) v[a] = {g[0][a], g[1][a]};
        const F4 nr = collide_v<KIND, P::kExactWeights, !decltype(last)::value && sizeof(R) == 4>(cc, v);
        #pragma unroll
        for (int a = 0; a < 9; ++a) { g[0][a] = v[a].a; g[1][a] = v[a].b; }
        #pragma unroll
        for (int h = 0; h < 2; ++h) {
            const F2 nrho = h ? nr.b : nr.a;
            worst[2 * h] = max(worst[2 * h], __float_as_uint(f2_lo(nrho)) - 0x80000001u);
            worst[2 * h + 1] = max(worst[2 * h + 1], __float_as_uint(f2_hi(nrho)) - 0x80000001u);
        }
        if constexpr (SR) {
            uint32_t nh[4];
            #pragma unroll
            for (int k = 0; k < 4; ++k) {
                int i = c4 + k;
                if (!wall_x) i = i < 0 ? i + p.nx : (i >= p.nx ? i - p.nx : i);
                nh[k] = sr_node_hash((uint32_t)wrap_row(j) * (uint32_t)p.nx + (uint32_t)i, s);
            }
            #pragma unroll
            for (int a = 0; a < 9; ++a) {
                f[a].x = P::to_r2_sr(f2_lo(g[0][a]), f2_hi(g[0][a]), sr_pop_bits(nh[0], a), sr_pop_bits(nh[1], a));
                f[a].y = P::to_r2_sr(f2_lo(g[1][a]), f2_hi(g[1][a]), sr_pop_bits(nh[2], a), sr_pop_bits(nh[3], a));
            }
        } else {
            #pragma unroll
            for (int a = 0; a < 9; ++a) f[a].template round<PREC>(g[0][a], g[1][a]);
        }
    };

    // update m collides the rows [r0 - (T - 1 - m), r1 + (T - 1 - m)) that the lattice has
    const int first = wall_y ? max(r0 - (T - 1), 0) : r0 - (T - 1);
    const int last = r1 + T - 2;                                     // with T - 1 rows of lag: row r1 - 1 stored
    const int last_load = wall_y ? min(last, ny - 1) : last;
    load_row(first);
    #pragma unroll 1
    for (int r = first; r <= last; ++r) {
        Row f[9];
        if (r <= last_load) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            const bool b = at_floor(wrap_row(r)), t = at_top(wrap_row(r));
            #pragma unroll
            for (int a = 0; a < 9; ++a) {
                f[a] = sm.row[a][lane];
                if (!all_vec) {
                    const R *x = reinterpret_cast<const R *>(&sm.row[a][lane]) + o;
                    const R *y = reinterpret_cast<const R *>(&seam[a * 32 + lane]) - n1;
                    R v[4];
                    #pragma unroll
                    for (int k = 0; k < 4; ++k) v[k] = (k < n1 ? x : y)[k];
                    f[a].set(v);
                }
                if (ex(a) != 0 && !((ey(a) > 0 && b) || (ey(a) < 0 && t))) f[a] = ex(a) > 0 ? f[a].up() : f[a].down();
            }
            R e[3] = {0, 0, 0};                                      // f*_{abar} of the x-wall node
            if (edge_strip && (at_left || at_right)) {
                const R *q = src + (size_t)wrap_row(r) * (size_t)p.pitch + (at_left ? 0 : p.nx - 1);
                e[0] = q[(size_t)(at_left ? 3 : 1) * (size_t)p.plane];
                e[1] = q[(size_t)(at_left ? 7 : 8) * (size_t)p.plane];
                e[2] = q[(size_t)(at_left ? 6 : 5) * (size_t)p.plane];
            }
            if (r < last_load) load_row(r + 1);                      // row r is in registers
            collide_row(Bool<false>(), f, e, r, salt.s[0]);
        }
        #pragma unroll
        for (int m = 1; m < T; ++m) {
            const int j = r - m;                                     // the row of update m; f: row j + 1 after update m - 1
            if (wall_y && j >= ny) continue;
            const bool node_row = !(wall_y && j + 1 >= ny);          // row j + 1 exists
            const bool wanted = j >= (wall_y ? max(r0 - (T - 1 - m), 0) : r0 - (T - 1 - m));
            const int par = (j + 1) & 1;
            Row (&here)[3][32] = sm.here[m - 1];
            Row (&below)[2][3][32] = sm.below[m - 1];
            R (&wall)[3][2] = sm.wall[m - 1];
            R e[3] = {0, 0, 0};                                      // of row j
            if (edge_strip && (at_left || at_right)) {
                #pragma unroll
                for (int x = 0; x < 3; ++x) e[x] = wall[x][at_right];
            }
            Row g[9];
            if (node_row) {
                g[4] = f[4];
                g[7] = f[7].down();
                g[8] = f[8].up();
            } else {                                                 // below the top wall: its own 2, 5, 6 come back
                g[4] = below[par ^ 1][0][lane];
                g[7] = below[par ^ 1][1][lane].down();
                g[8] = below[par ^ 1][2][lane].up();
                if (at_left) g[8].put(0, e[2]);                      // (shifted out at the outermost lanes)
                if (at_right) g[7].put(kx, e[2]);
            }
            g[0] = here[0][lane]; g[1] = here[1][lane]; g[3] = here[2][lane];
            g[2] = below[par][0][lane]; g[5] = below[par][1][lane]; g[6] = below[par][2][lane];
            if (node_row) {
                // row j + 1 takes the place of row j
                if (at_floor(j + 1)) {                               // below row 0: its own 4, 7, 8 come back
                    below[par ^ 1][0][lane] = f[4];
                    below[par ^ 1][1][lane] = f[7];
                    below[par ^ 1][2][lane] = f[8];
                }
                below[par][0][lane] = f[2];
                below[par][1][lane] = f[5].up();
                below[par][2][lane] = f[6].down();
                here[0][lane] = f[0];
                here[1][lane] = f[1].up();
                here[2][lane] = f[3].down();
                if (edge_strip && (at_left || at_right)) {
                    wall[0][at_right] = at_right ? f[1].at(kx) : f[3].at(0);
                    wall[1][at_right] = at_right ? f[8].at(kx) : f[7].at(0);
                    wall[2][at_right] = at_right ? f[5].at(kx) : f[6].at(0);
                }
            }
            if (!wanted) break;
            if (m < T - 1) {
                collide_row(Bool<false>(), g, e, j, salt.s[m]);
                #pragma unroll
                for (int a = 0; a < 9; ++a) f[a] = g[a];
            } else {
                collide_row(Bool<true>(), g, e, j, salt.s[m]);
                if (own) {
                    R *q = dst + (size_t)j * (size_t)p.pitch + c4;   // past nx: the row's padding
                    #pragma unroll
                    for (int a = 0; a < 9; ++a) g[a].store(q + (size_t)a * (size_t)p.plane);
                }
            }
        }
    }
    // rho <= 0 or not finite in an own column at any of the updates
    bool bad = false;
    #pragma unroll
    for (int k = 0; k < 4; ++k) bad = bad || (worst[k] >= 0x7f7fffffu && c4 + k < p.nx);
    if (bad && own) atomicOr(p.flag, 1);
}

// One item (segment, strip) per block, strips fastest: concurrent blocks share the rows between their
// segments and the columns between their strips in L2.
template <int PREC, int KIND, bool SR, int T, bool SEAM>
__global__ void __launch_bounds__(32, SEAM ? kSwSeamBlocks : kSwBlocks)
sweep_kernel(const typename Prec<PREC>::R *src, typename Prec<PREC>::R *dst,
             const Params<typename Prec<PREC>::C> p, const CollideConsts cc, const SweepSalts<T> salt, int strips,
             int rows)
{
    extern __shared__ __align__(16) unsigned char sweep_smem[];
    using Shared = SweepShared<typename Prec<PREC>::R, T>;
    Shared &sm = *reinterpret_cast<Shared *>(sweep_smem);
    Raw4<typename Prec<PREC>::R> *seam = reinterpret_cast<Raw4<typename Prec<PREC>::R> *>(sweep_smem + sizeof(Shared));
    const int seg = blockIdx.x / strips, strip = blockIdx.x - seg * strips;
    const int r0 = seg * rows;
    follow_predecessor();
    sweep<PREC, KIND, SR, T, SEAM>(src, dst, p, cc, salt, strip, r0, min(r0 + rows, p.ny), sm, seam);
}

} // namespace smrt
