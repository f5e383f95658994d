// tclbm_resident.cuh -- many time steps of one small lattice in one launch, its state
// resident in shared memory (sm_103a).
//
// A lattice of a few hundred thousand nodes or less fits in the shared memory of the
// chip, and a launch per step costs it more than the step: the launch-to-launch chain of a
// one-wave grid is about 2.4 of the 3.2 us that a 256 x 128 step takes on 2-D tiles.  Here
// one CTA per SM owns a tile of nodes for all the steps of the call.  Its populations
// live in a frame in shared memory (the tile and a ring of R halo cells around it, two
// copies), and after each step the CTA publishes the cells near its edge on a board in
// global memory, from which its neighbours fill their halo cells.
//
// Every 16-byte word of the board carries three populations and the number of the step
// they belong to, written and read as one 128-bit access, so a reader that finds the
// number it waits for has the data as well: no flag, no fence and no grid-wide barrier,
// one L2 round trip between neighbours per step.  The board has two copies by parity of
// the step: a CTA publishes step s + 2 only after it has read step s + 1 of every
// neighbour, which that neighbour published after reading step s of this one.  The launch
// is cooperative (all CTAs resident), waits are bounded by the global timer, and step
// numbers only grow over the life of a lattice, so what an earlier launch left on the
// board never matches.
//
// A run of an even number of steps ends in the copy it started from, as that many launches
// would (work that a caller captured earlier reads that copy).  Updating in place is safe:
// only a tile and the tiles around it read its nodes from the source copy, all before the
// first publication, and a CTA stores its last state after it has read publications of every
// tile around it.
//
// What bounds it: the exchange (a store through L2 to a neighbour's read, 1 to 1.5 us) and
// the dependent chain of one node update (about 1 us at one or two warps per scheduler).
// Measured (GB300, us per step in runs of 200 against one launch per step): thermal with the
// correction term 8 x 64 2.1 / 2.8, 128 x 64 2.4 / 2.9, 4096 x 4 2.6 / 3.9, 256 x 128 2.94 / 3.15
// (periodic 2.81 / 2.79), 300 x 150 3.3 / 4.2; without it 128 x 128 1.9 / 2.8, 400 x 400 5.4 / 6.1;
// athermal 64 x 64 1.6 / 2.6, 256 x 256 2.1 / 3.1, 512 x 512 5.9 / 8.2.
// With the correction term tiles of more nodes than threads lose (512 x 256: 7.1 / 5.9).
//
// The arithmetic is that of the one-step kernels, node for node.
#pragma once

#include "tclbm_device.cuh"

namespace tclbm {

enum { RES_ATHERMAL = 0, RES_THERMAL = 1, RES_CORR = 2 };

// Tiles of a resident launch: gx x gy of nearly equal size.
struct ResPlan {
    int gx, gy, threads, multi;
};

// Words all CTAs read from the board per step above which they poll with one lane per warp.
// Measured (all lanes / one lane, us per step): 64 x 32 with 12,600 words 2.35 / 2.33, the
// 4096 x 4 shock tube with 29,000 words 2.59 / 2.75, 128 x 64 with 48,000 words 2.53 / 2.55,
// 256 x 128 with 122,000 words 3.49 / 2.94 (periodic 3.57 / 2.78).
constexpr long long kResQuietWords = 40000;

// (With the correction term tiles of more nodes than threads lose, see above.)
template <int KIND, bool MULTI>
struct ResShape {
    static_assert(KIND != RES_CORR || !MULTI, "one node per thread with the correction term");
    static constexpr int R = KIND == RES_CORR ? 2 : 1;           // halo cells on each side
    static constexpr int NP = KIND == RES_ATHERMAL ? 9 : 18;     // populations per node
    static constexpr int CELLS = !MULTI ? 640 : (KIND == RES_ATHERMAL ? 2944 : 1472);  // cells of a frame
    static constexpr int W = NP / 3;                             // board words per node
    static constexpr int PHI = KIND == RES_CORR ? 2 * CELLS : 0;  // u (1 - theta), both components
    static constexpr size_t SMEM = sizeof(float) * (2 * NP * CELLS + PHI);
    static constexpr int THREADS = 512;
};

__device__ __forceinline__ void board_st(uint4* d, float a, float b, float c, unsigned tag) {
    asm volatile(
        "{\n\t.reg .b64 lo, hi;\n\t.reg .b128 v;\n\t"
        "mov.b64 lo, {%1, %2};\n\tmov.b64 hi, {%3, %4};\n\tmov.b128 v, {lo, hi};\n\t"
        "st.relaxed.gpu.global.b128 [%0], v;\n\t}" ::"l"(d),
        "r"(__float_as_uint(a)), "r"(__float_as_uint(b)), "r"(__float_as_uint(c)), "r"(tag)
        : "memory");
}
__device__ __forceinline__ unsigned board_ld(const uint4* s, float& a, float& b, float& c) {
    unsigned x, y, z, w;
    asm volatile(
        "{\n\t.reg .b64 lo, hi;\n\t.reg .b128 v;\n\t"
        "ld.relaxed.gpu.global.b128 v, [%4];\n\t"
        "mov.b128 {lo, hi}, v;\n\tmov.b64 {%0, %1}, lo;\n\tmov.b64 {%2, %3}, hi;\n\t}"
        : "=r"(x), "=r"(y), "=r"(z), "=r"(w)
        : "l"(s)
        : "memory");
    a = __uint_as_float(x);
    b = __uint_as_float(y);
    c = __uint_as_float(z);
    return w;
}

__device__ __forceinline__ long long res_timer_ns() {
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The value a store of v in format ST and a load give back.
template <class ST>
__device__ __forceinline__ float stored(float v) {
    ST s;
    Store<ST>::st(&s, v);
    return Store<ST>::ld_smem(&s);
}

// Node values as store_node() would leave them in memory.
template <class ST, int NP>
__device__ __forceinline__ void round_node(const DevParams& p, int x, int y, uint32_t step, float* v) {
    if (sizeof(ST) == 2 && p.rounding) {
        const uint32_t seed = sr_bits((uint32_t)(y * p.nx + x), 0u, step);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            if (2 * k >= NP) break;
            const float hi = 2 * k + 1 < NP ? v[2 * k + 1] : 0.0f;
            const uint32_t d = cvt_rs_pair<ST>(hi, v[2 * k], sr_pair_bits(seed, (uint32_t)k));
            const unsigned short lo16 = (unsigned short)d, hi16 = (unsigned short)(d >> 16);
            v[2 * k] = Store<ST>::ld_smem(reinterpret_cast<const ST*>(&lo16));
            if (2 * k + 1 < NP) v[2 * k + 1] = Store<ST>::ld_smem(reinterpret_cast<const ST*>(&hi16));
        }
    } else if (sizeof(ST) == 2) {
#pragma unroll
        for (int q = 0; q < NP; ++q) v[q] = stored<ST>(v[q]);
    }
}

// Streamed populations of the node at frame index i (rows FX apart).
template <int KIND, int CELLS>
__device__ __forceinline__ void res_pull(const float* fr, int i, int FX, float* f, float* h) {
    const float *c = fr + i, *up = c + FX, *dn = c - FX;
    const float* const r[9] = {c, c - 1, dn, c + 1, up, dn - 1, dn + 1, up + 1, up - 1};
#pragma unroll
    for (int q = 0; q < 9; ++q) f[q] = r[q][q * CELLS];
    if (KIND != RES_ATHERMAL) {
#pragma unroll
        for (int q = 0; q < 9; ++q) h[q] = r[q][(9 + q) * CELLS];
    }
}

// A node a thread works on: its place, what its wall (if any) needs, and what is its own.
struct ResNode {
    int lx, ly, x, y;  // in the tile, in the lattice
    int i;             // frame index
    int side, in;      // wall side (-1: none) and the frame step to the interior neighbour
    int one_x, one_y;  // one-sided derivative: +1 at the lower wall, -1 at the upper, 0 none
};

// n >= 2 steps of the lattice from `src` to `dst`, which may be the same copy.  MULTI: more
// nodes than threads.
template <class ST, int KIND, bool MULTI, bool FAST>
__global__ void __launch_bounds__(512, 1) tclbm_resident(const __grid_constant__ DevParams p, const ST* src,
                                                         ST* dst, uint4* __restrict__ board, int gx, int gy,
                                                         int n, unsigned tag0, int* __restrict__ err) {
    using S = ResShape<KIND, MULTI>;
    constexpr int R = S::R, NP = S::NP, CELLS = S::CELLS, W = S::W, ITEMS = 4;
    constexpr bool THERMAL = KIND != RES_ATHERMAL, CORR = KIND == RES_CORR;
    extern __shared__ float smem_res[];
    __shared__ int halo_node[512], halo_cell[512];  // board node and frame cell of each halo cell read
    __shared__ int halo_count;
    float* const frame = smem_res;                    // [2][NP][CELLS]
    float* const phx = smem_res + 2 * NP * CELLS;     // [CELLS], frame indices
    float* const phy = phx + CELLS;
    if (*(volatile int*)err) return;
    const int tid = threadIdx.x, T = blockDim.x;
    const int nx = p.nx, ny = p.ny;
    const int bx = blockIdx.x % gx, by = blockIdx.x / gx;
    const int x0 = (int)((long long)bx * nx / gx), y0 = (int)((long long)by * ny / gy);
    const int bw = (int)((long long)(bx + 1) * nx / gx) - x0, bh = (int)((long long)(by + 1) * ny / gy) - y0;
    const int FX = bw + 2 * R, FY = bh + 2 * R;
    // an axis with one tile and periodic wrap: its halo cells are this tile's own cells
    const bool selfx = gx == 1 && p.xper, selfy = gy == 1 && p.yper, self = selfx || selfy;
    const long long N = (long long)nx * ny;

    // the frame from the source copy, and the list of halo cells to read from the board
    if (tid == 0) halo_count = 0;
    __syncthreads();
    for (int c = tid; c < FX * FY; c += T) {
        const int fx = c % FX - R, fy = c / FX - R;
        int x = x0 + fx, y = y0 + fy;
        bool valid = true;
        if (p.xper) x = ((x % nx) + nx) % nx; else valid = x >= 0 && x < nx;
        if (p.yper) y = ((y % ny) + ny) % ny; else valid = valid && y >= 0 && y < ny;
#pragma unroll
        for (int q = 0; q < NP; ++q)
            // (an ordinary load, not the read-only path: dst may be src)
            frame[q * CELLS + c] = valid ? Store<ST>::ld_smem(src + q * p.plane + ((long long)y * p.pitch + x)) : 0.0f;
        if (!valid)  // past a wall: never written again, and replaced by the wall scheme where it is pulled
#pragma unroll
            for (int q = 0; q < NP; ++q) frame[(NP + q) * CELLS + c] = 0.0f;
        const bool inx = fx >= 0 && fx < bw, iny = fy >= 0 && fy < bh;
        if (valid && !((inx || selfx) && (iny || selfy))) {
            const int k = atomicAdd(&halo_count, 1);
            halo_node[k] = y * nx + x;
            halo_cell[k] = c;
        }
    }
    uint32_t step0 = 0;
    if (sizeof(ST) == 2 && p.rounding) step0 = p.step_ctr[p.parity];

    // nodes of this tile: own nodes first, then (with the correction term) the nodes around
    // the tile whose u (1 - theta) the derivatives read, on axes that have other tiles
    const int own = bw * bh;
    const int hx = CORR && !selfx ? 2 * bh : 0, hy = CORR && !selfy ? 2 * bw : 0;
    const int tasks = own + hx + hy;
    auto node_of = [&](int t, ResNode& d) {  // false: outside the lattice
        if (t < own) {
            d.ly = t / bw;
            d.lx = t - d.ly * bw;
        } else if (t < own + hx) {
            t -= own;
            d.lx = t < bh ? -1 : bw;
            d.ly = t < bh ? t : t - bh;
        } else {
            t -= own + hx;
            d.ly = t < bw ? -1 : bh;
            d.lx = t < bw ? t : t - bw;
        }
        int x = x0 + d.lx, y = y0 + d.ly;
        if (p.xper) x = x < 0 ? x + nx : (x >= nx ? x - nx : x); else if (x < 0 || x >= nx) return false;
        if (p.yper) y = y < 0 ? y + ny : (y >= ny ? y - ny : y); else if (y < 0 || y >= ny) return false;
        d.x = x;
        d.y = y;
        d.i = (d.ly + R) * FX + d.lx + R;
        d.side = wall_side_of(p, x, y);
        d.in = (d.side == SIDE_XM ? 1 : (d.side == SIDE_XP ? -1 : 0)) + FX * (d.side == SIDE_YM ? 1 : (d.side == SIDE_YP ? -1 : 0));
        d.one_x = d.side == SIDE_XM ? 1 : (d.side == SIDE_XP ? -1 : 0);
        d.one_y = d.side == SIDE_YM ? 1 : (d.side == SIDE_YP ? -1 : 0);
        return true;
    };
    // the other frame positions, within r cells around the tile, of the tile's cell (lx, ly)
    // on an axis that wraps onto this tile
    auto images = [&](const ResNode& d, int r, auto&& put) {
        for (int fy = selfy ? d.ly - ((d.ly + r) / bh) * bh : d.ly; fy < bh + r; fy += selfy ? bh : bh + 2 * r)
            for (int fx = selfx ? d.lx - ((d.lx + r) / bw) * bw : d.lx; fx < bw + r; fx += selfx ? bw : bw + 2 * r)
                if (fx != d.lx || fy != d.ly) put((fy + R) * FX + fx + R);
    };
    auto moments = [&](const float* fr, const ResNode& d, float* f, float* h) {
        res_pull<KIND, CELLS>(fr, d.i, FX, f, h);
        if (d.side >= 0) {
            float ff[9], hf[9];
            res_pull<KIND, CELLS>(fr, d.i + d.in, FX, ff, hf);
            wall_rebuild<THERMAL>(p, d.side, d.x, d.y, f, h, ff, hf);
        }
        return macro_of<THERMAL, FAST>(p, f, h, d.x, d.y);
    };
    auto publish_phi = [&](const ResNode& d, bool own_node, const Macro& m) {
        const float a = phi_x(m), b = phi_y(m);
        phx[d.i] = a;
        phy[d.i] = b;
        if (self && own_node)
            images(d, 1, [&](int c) {
                phx[c] = a;
                phy[c] = b;
            });
    };
    const bool boards = gx > 1 || gy > 1;
    auto update = [&](int s, float* fw, const ResNode& d, const float* f, const float* h, const Macro& m) {
        float dxv = 0.0f, dyv = 0.0f;
        if (CORR) {
            const float *px = phx + d.i, *py = phy + d.i;
            dxv = 0.5f * (px[1] - px[-1]);
            dyv = 0.5f * (py[FX] - py[-FX]);
            if (d.side >= 0) {
                if (d.one_x > 0) dxv = 0.5f * (-3.0f * px[0] + 4.0f * px[1] - px[2]);
                if (d.one_x < 0) dxv = 0.5f * (3.0f * px[0] - 4.0f * px[-1] + px[-2]);
                if (d.one_y > 0) dyv = 0.5f * (-3.0f * py[0] + 4.0f * py[FX] - py[2 * FX]);
                if (d.one_y < 0) dyv = 0.5f * (3.0f * py[0] - 4.0f * py[-FX] + py[-2 * FX]);
            }
        }
        float v[18];
        collide<THERMAL, FAST>(p, f, h, m, dxv, dyv, v, v + 9);
        round_node<ST, NP>(p, d.x, d.y, step0 + (uint32_t)s, v);
        if (s + 1 < n) {
            const unsigned tag = tag0 + (unsigned)s + 1u;
            const bool edge = (gx > 1 && (d.lx < R || d.lx >= bw - R)) || (gy > 1 && (d.ly < R || d.ly >= bh - R));
            if (boards && edge && d.y != p.skip_row) {  // (test hook: a row that is never published)
                uint4* b = board + ((long long)(tag & 1u) * N + (d.y * nx + d.x)) * W;
#pragma unroll
                for (int w = 0; w < W; ++w) board_st(b + w, v[3 * w], v[3 * w + 1], v[3 * w + 2], tag);
            }
#pragma unroll
            for (int q = 0; q < NP; ++q) fw[q * CELLS + d.i] = v[q];
            if (self)
                images(d, R, [&](int c) {
#pragma unroll
                    for (int q = 0; q < NP; ++q) fw[q * CELLS + c] = v[q];
                });
        } else {
            ST* o = dst + ((long long)d.y * p.pitch + d.x);
#pragma unroll
            for (int q = 0; q < NP; ++q) Store<ST>::st(o + q * p.plane, v[q]);
        }
    };
    ResNode nd = {};
    bool active = false;
    if (!MULTI && tid < tasks) active = node_of(tid, nd);
    const bool mine = tid < own;
    __syncthreads();
    // the board words this thread reads every step: the first ITEMS of them from registers
    const int items = halo_count * W;
    int it_src[ITEMS], it_dst[ITEMS], nit = 0;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const int i = tid + j * T;
        it_src[j] = it_dst[j] = 0;
        if (i < items) {
            const int k = i / W, w = i - k * W;
            it_src[j] = halo_node[k] * W + w;
            it_dst[j] = 3 * w * CELLS + halo_cell[k];
            nit = j + 1;
        }
    }

    const bool quiet = (long long)gridDim.x * items > kResQuietWords;

    for (int s = 0; s < n; ++s) {
        float* const fr = frame + (s & 1) * NP * CELLS;
        float* const fw = frame + ((s & 1) ^ 1) * NP * CELLS;
        if (s > 0) {
            const unsigned tag = tag0 + (unsigned)s;  // number of the state this step starts from
            const uint4* b = board + (long long)(tag & 1u) * N * W;
            float v[ITEMS][3];
            unsigned got[ITEMS];
            int fail = 0;
            // Every word in flight at once, and those that were not there yet read again.  With
            // many words on the board (quiet) one lane of a warp first waits for its own, so
            // that the polling does not flood the L2 that the neighbours' stores go through.
            long long deadline = 0;
            int tries = 0;
            auto give_up = [&]() {  // the error word and the clock only now and then: each is a round trip
                if ((++tries & 63) != 0) return false;
                const long long now = res_timer_ns();
                if (deadline == 0) deadline = now + 1000000000LL;
                const bool late = now > deadline;
                if (late) atomicExch(err, 3);
                return late || *(volatile int*)err != 0;
            };
            if (quiet && (tid & 31) == 0 && nit > 0)
                while (board_ld(b + it_src[0], v[0][0], v[0][1], v[0][2]) != tag)
                    if (give_up()) {
                        fail = 1;
                        break;
                    }
            __syncwarp();
            bool all;
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) {
                got[j] = tag;
                if (j < nit) got[j] = board_ld(b + it_src[j], v[j][0], v[j][1], v[j][2]);
            }
            do {
                all = true;
#pragma unroll
                for (int j = 0; j < ITEMS; ++j) all = all && got[j] == tag;
                if (!all) {
                    if (fail || give_up()) {
                        fail = 1;
                        break;
                    }
#pragma unroll
                    for (int j = 0; j < ITEMS; ++j)
                        if (got[j] != tag) got[j] = board_ld(b + it_src[j], v[j][0], v[j][1], v[j][2]);
                }
            } while (!all);
#pragma unroll
            for (int j = 0; j < ITEMS; ++j)
                if (j < nit) {
                    float* d = fr + it_dst[j];
                    d[0] = v[j][0];
                    d[CELLS] = v[j][1];
                    d[2 * CELLS] = v[j][2];
                }
            if (items > ITEMS * T) {  // long thin tiles: the rest, one word after another
                for (int i = tid + ITEMS * T; i < items && !fail; i += T) {
                    const int k = i / W, w = i - k * W;
                    float a0, a1, a2;
                    while (board_ld(b + ((long long)halo_node[k] * W + w), a0, a1, a2) != tag && !fail)
                        if (give_up()) fail = 1;
                    float* d = fr + 3 * w * CELLS + halo_cell[k];
                    d[0] = a0;
                    d[CELLS] = a1;
                    d[2 * CELLS] = a2;
                }
            }
            if (__syncthreads_or(fail)) return;
        }
        float f[9], h[9];
        Macro m;
        if (!MULTI) {
            if (active) {
                m = moments(fr, nd, f, h);
                if (CORR) publish_phi(nd, mine, m);
            }
            if (CORR) __syncthreads();
            if (mine) update(s, fw, nd, f, h, m);
        } else {
            ResNode d;
            for (int t = tid; t < own; t += T) {
                node_of(t, d);
                m = moments(fr, d, f, h);
                update(s, fw, d, f, h, m);
            }
        }
    }
}

// Advances the stochastic-rounding counters of a lattice by n >= 1 steps (after a resident run
// or a chain of launches that left them alone): `to` is the copy the state ended in.  Both get
// what one launch per step would leave in them -- all steps in the copy of the state, one
// fewer in the other -- so that new fields, which always start from copy 0, and launches that a
// caller captured earlier go on with the same draws whatever ran before.
static __global__ void tclbm_count_steps(const DevParams p, int to, unsigned n) {
    const unsigned total = p.step_ctr[p.parity] + n;
    p.step_ctr[to] = total;
    p.step_ctr[to ^ 1] = total - 1u;
}

}  // namespace tclbm
