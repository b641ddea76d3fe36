// tile.cuh -- several updates of a small lattice in one launch, two-buffer layout, every storage format.
//
// A launch costs about 4 us from the host and 2 us more until its first blocks run and its last ones end,
// and a 64^2 lattice of single-node threads fills 128 of the 608 SM sub-partitions once: one update is all
// latency.  Here a block owns a W x H tile and computes it for T updates in shared memory: update m pulls
// and collides the tile and T - 1 - m rings of nodes around it, so neighbouring tiles repeat each other's
// rings and no block waits for another.  The rings are affordable because most of the chip would idle;
// tile_plan says where that ends.  One node per thread: a warp's double operation takes the same 64 clocks
// for one lane as for 32, and a wave of the next warps hides the float ones' latency.
// Between updates f* is kept as the storage format rounds it; the same operations on the same values as T
// calls of step_kernel, hence the same bits.
#pragma once

#include "d2q9.cuh"

namespace smrt {

constexpr int kTileMaxT = 8;

struct TileSalts {
    uint32_t s[kTileMaxT];
};

template <int PREC, int KIND, bool SR>
__global__ void __launch_bounds__(512)
tile_kernel(const typename Prec<PREC>::R *src, typename Prec<PREC>::R *dst,
            const Params<typename Prec<PREC>::C> p, const TileSalts salt, int W, int H, int T, int tiles_x)
{
    using P = Prec<PREC>;
    using R = typename P::R;
    using C = typename P::C;
    extern __shared__ __align__(16) unsigned char tile_smem[];
    // two copies of the region (tile and T - 1 rings), population by population
    const int RW = W + 2 * (T - 1), RH = H + 2 * (T - 1), area = RW * RH;
    R *cur = reinterpret_cast<R *>(tile_smem), *nxt = cur + 9 * area;
    const int ty = blockIdx.x / tiles_x, x0 = (blockIdx.x - ty * tiles_x) * W, y0 = ty * H;
    const bool wall_x = !p.periodic_x, wall_y = !p.periodic_y;
    bool bad = false;
    follow_predecessor();
    for (int m = 0; m < T; ++m) {
        // nodes of this update: T - 1 - m rings, as far as the lattice has them
        const int ring = T - 1 - m;
        const int xa = wall_x ? max(x0 - ring, 0) : x0 - ring, ya = wall_y ? max(y0 - ring, 0) : y0 - ring;
        const int xe = min(x0 + W, p.nx), ye = min(y0 + H, p.ny);
        const int xb = wall_x ? min(xe + ring, p.nx) : xe + ring, yb = wall_y ? min(ye + ring, p.ny) : ye + ring;
        const int w = xb - xa, count = w * (yb - ya);
        const unsigned magic = ((1u << 20) + w - 1) / w;             // n / w for n < 4096, w < 64
        for (int n = threadIdx.x; n < count; n += blockDim.x) {
            const int row = (int)(((unsigned)n * magic) >> 20);
            const int i = xa + n - row * w, j = ya + row;            // may lie beyond a periodic side
            const int iw = i < 0 ? i + p.nx : (i >= p.nx ? i - p.nx : i), jw = j < 0 ? j + p.ny : (j >= p.ny ? j - p.ny : j);
            const int at0 = (j - y0 + T - 1) * RW + (i - x0 + T - 1);
            C g[9];
            if (m == 0) {
                #pragma unroll
                for (int a = 0; a < 9; ++a) {
                    const Loc L = pull_loc<MODE_AB>(p, a, iw, jw);
                    C v = P::to_c(src[at(p.plane, p.pitch, L.plane, L.j, L.i)]);
                    if (L.side >= 0) v += p.corr[L.side][a];
                    g[a] = v;
                }
            } else {
                #pragma unroll
                for (int a = 0; a < 9; ++a) {
                    const int side = (wall_y && ey(a) > 0 && j == 0)             ? SIDE_BOTTOM
                                     : (wall_y && ey(a) < 0 && j == p.ny - 1)    ? SIDE_TOP
                                     : (wall_x && ex(a) > 0 && i == 0)           ? SIDE_LEFT
                                     : (wall_x && ex(a) < 0 && i == p.nx - 1)    ? SIDE_RIGHT
                                                                                 : -1;
                    C v = P::to_c(cur[side >= 0 ? opp(a) * area + at0 : a * area + at0 - ey(a) * RW - ex(a)]);
                    if (side >= 0) v += p.corr[side][a];
                    g[a] = v;
                }
            }
            if (!collide<KIND, P::kExactWeights>(p, g)) bad = true;
            const uint32_t nh = SR ? sr_node_hash((uint32_t)jw * (uint32_t)p.nx + (uint32_t)iw, salt.s[m]) : 0u;
            #pragma unroll
            for (int a = 0; a < 9; ++a) {
                R v;
                if constexpr (SR) v = P::to_r_sr(g[a], sr_pop_bits(nh, a));
                else v = P::to_r(g[a]);
                if (m == T - 1) dst[at(p.plane, p.pitch, a, j, i)] = v;
                else nxt[a * area + at0] = v;
            }
        }
        __syncthreads();
        R *t = cur;
        cur = nxt;
        nxt = t;
    }
    if (bad) atomicOr(p.flag, 1);
}

} // namespace smrt
