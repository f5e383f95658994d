// tclbm_api.cu -- host side of the C ABI declared in include/tclbm.h: parameter
// validation and derived constants, device memory, the step loop (CUDA graphs for
// short launches), field initialisation, moments, FP64 diagnostics and population
// transfer kernels.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <unistd.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdarg>
#include <cstring>
#include <mutex>
#include <type_traits>
#include <new>

#include "tclbm.h"
#include "tclbm_device.cuh"
#include "tclbm_fields.cuh"
#include "tclbm_internal.h"
#include "tclbm_launch.h"

using namespace tclbm;

namespace {
thread_local char g_err[512] = "";
thread_local int64_t g_refuse_in = -1;  // test hook: step launches left before one is refused
}  // namespace

bool tclbm::refuse_launch() { return g_refuse_in >= 0 && g_refuse_in-- == 0; }

tclbm_status tclbm::fail(tclbm_status st, const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof g_err, fmt, ap);
    va_end(ap);
    return st;
}

tclbm_status tclbm::cuda_fail(cudaError_t e, const char* what) {
    return fail(TCLBM_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

namespace {
constexpr int kDiagBlock = 256;
constexpr int kDiagMaxBlocks = 1024;
}  // namespace

void tclbm::set_last_error(const char* msg) { snprintf(g_err, sizeof g_err, "%s", msg); }

struct tclbm::StreamUse {
    int dev;
    cudaStream_t stream;
    int handles;
    StreamUse* next;
};

namespace {
std::mutex g_use_mutex;
StreamUse* g_uses = nullptr;
}  // namespace

StreamUse* tclbm::use_stream(cudaStream_t s) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    std::lock_guard<std::mutex> lock(g_use_mutex);
    // (the per-thread stream is another one in each thread: an entry for each handle)
    if (s != cudaStreamPerThread)
        for (StreamUse* u = g_uses; u; u = u->next)
            if (u->dev == dev && u->stream == s) {
                ++u->handles;
                return u;
            }
    StreamUse* u = new (std::nothrow) StreamUse{dev, s, 1, g_uses};
    if (u) g_uses = u;
    return u;
}

void tclbm::unuse_stream(StreamUse* u) {
    if (!u) return;
    std::lock_guard<std::mutex> lock(g_use_mutex);
    if (--u->handles > 0) return;
    StreamUse** at = &g_uses;
    while (*at != u) at = &(*at)->next;
    *at = u->next;
    delete u;
}

bool tclbm::only_stream(const StreamUse* u) {
    if (!u) return false;
    std::lock_guard<std::mutex> lock(g_use_mutex);
    for (const StreamUse* v = g_uses; v; v = v->next)
        if (v != u && v->dev == u->dev) return false;
    return true;
}

void* tclbm::dev_alloc(tclbm_lattice* L, size_t bytes) {
    if (bytes == 0) return nullptr;
    if (L->alloc) return L->alloc(bytes, (void*)L->stream, L->ctx);
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return p;
}

void tclbm::dev_free(tclbm_lattice* L, void* p, size_t bytes) {
    if (!p) return;
    if (L->free_fn)
        L->free_fn(p, bytes, (void*)L->stream, L->ctx);
    else
        cudaFree(p);
}

namespace {

bool walls_ok(const tclbm_params* p) {
    for (int s = 0; s < 4; ++s) {
        const int k = p->wall[s].kind;
        if (k < TCLBM_WALL_PERIODIC || k > TCLBM_WALL_EQUILIBRIUM) return false;
        if (p->wall[s].therm != TCLBM_THERM_FIXED_T && p->wall[s].therm != TCLBM_THERM_ADIABATIC) return false;
    }
    return true;
}

tclbm_status validate(const tclbm_params* p) {
    if (!p) return fail(TCLBM_EINVAL, "params is NULL");
    if (p->nx < 1 || p->ny < 1) return fail(TCLBM_EINVAL, "nx, ny must be >= 1 (got %d, %d)", p->nx, p->ny);
    if ((long long)p->nx * p->ny > (1LL << 34)) return fail(TCLBM_EINVAL, "lattice too large");
    if (!walls_ok(p)) return fail(TCLBM_EINVAL, "unknown wall kind or thermal treatment");
    const bool xper = p->wall[TCLBM_SIDE_XM].kind == TCLBM_WALL_PERIODIC;
    const bool yper = p->wall[TCLBM_SIDE_YM].kind == TCLBM_WALL_PERIODIC;
    if (xper != (p->wall[TCLBM_SIDE_XP].kind == TCLBM_WALL_PERIODIC) ||
        yper != (p->wall[TCLBM_SIDE_YP].kind == TCLBM_WALL_PERIODIC))
        return fail(TCLBM_EINVAL, "opposite sides must both be periodic or both walls");
    if (!xper && !yper) return fail(TCLBM_EUNSUPPORTED, "walls on both axes are not supported");
    if (!xper && p->nx < 3) return fail(TCLBM_EINVAL, "a walled x axis needs nx >= 3");
    if (!yper && p->ny < 3) return fail(TCLBM_EINVAL, "a walled y axis needs ny >= 3");
    if (!(p->gamma > 1.0) || !(p->Pr > 0.0) || !(p->R > 0.0) || !(p->T0 > 0.0))
        return fail(TCLBM_EINVAL, "gamma > 1, Pr > 0, R > 0, T0 > 0 required");
    if (p->visc_law < TCLBM_VISC_NU || p->visc_law > TCLBM_VISC_W1) return fail(TCLBM_EINVAL, "bad visc_law");
    if (p->visc_law == TCLBM_VISC_W1 ? !(p->visc > 0.0 && p->visc < 2.0) : !(p->visc > 0.0))
        return fail(TCLBM_EINVAL, "viscosity (or w1) out of range");
    if (!p->bgk)
        for (double w : {p->w2, p->w3, p->w4})
            if (!(w > 0.0 && w < 2.0)) return fail(TCLBM_EINVAL, "w2, w3, w4 must lie in (0, 2)");
    if (p->force_kind < TCLBM_FORCE_NONE || p->force_kind > TCLBM_FORCE_TAYLOR_GREEN)
        return fail(TCLBM_EINVAL, "bad force_kind");
    if (p->correction && !p->thermal) return fail(TCLBM_EINVAL, "the correction term needs thermal = 1");
    if (p->work && !p->thermal) return fail(TCLBM_EINVAL, "the work term needs thermal = 1");
    if (p->storage < TCLBM_STORE_FP32 || p->storage > TCLBM_STORE_FP16) return fail(TCLBM_EINVAL, "bad storage");
    if (p->rounding != TCLBM_ROUND_NEAREST && p->rounding != TCLBM_ROUND_STOCHASTIC)
        return fail(TCLBM_EINVAL, "bad rounding");
    return TCLBM_OK;
}

int pitch_of(int nx) { return (nx + 31) / 32 * 32; }

size_t elem_of(int storage) { return storage == TCLBM_STORE_FP32 ? 4 : 2; }

void derive(tclbm_lattice* L) {
    const tclbm_params& p = L->prm;
    FieldParams& d = L->dp;
    memset(&d, 0, sizeof d);
    d.skip_row = -1;  // the timeout test hook is off
    d.nx = p.nx;
    d.ny = p.ny;
    d.pitch = pitch_of(p.nx);
    d.plane = (long long)p.ny * d.pitch;
    d.xper = p.wall[TCLBM_SIDE_XM].kind == TCLBM_WALL_PERIODIC;
    d.yper = p.wall[TCLBM_SIDE_YM].kind == TCLBM_WALL_PERIODIC;
    d.visc_law = p.visc_law;
    d.visc = (float)p.visc;
    d.w2 = (float)p.w2;
    d.w3 = (float)p.w3;
    d.w4 = (float)p.w4;
    d.bgk = p.bgk;
    const double b = 2.0 / (p.gamma - 1.0);
    d.R = (float)p.R;
    d.T0 = (float)p.T0;
    d.b = (float)b;
    d.two_over_b = (float)(2.0 / b);
    d.inv_R = (float)(1.0 / p.R);
    // Rest state of the deviations: RT0 and Et0 on a 2^-10 grid near R T0 and b R T0 / 2,
    // so that f^eq(1, 0, RT0), h^eq(1, 0, RT0) and their moment identities are exact in
    // float (each value needs at most 21 significant bits).
    const double RTb = std::max(1.0, std::round(p.R * p.T0 * 1024.0)) / 1024.0;
    const double Etb = std::max(1.0, std::round(0.5 * b * RTb * 1024.0)) / 1024.0;
    d.RT0 = (float)RTb;
    d.Et0 = (float)Etb;
    d.cRT = (float)(2.0 / b * Etb - RTb);
    d.RTp = (float)(p.R * p.T0);
    d.inv_RTp = (float)(1.0 / (p.R * p.T0));
    d.inv_w1_fixed = p.visc_law == TCLBM_VISC_W1 ? (float)(1.0 / p.visc) : 0.0f;
    d.inv_Pr = (float)(1.0 / p.Pr);
    d.Pr_m1 = (float)(p.Pr - 1.0);
    d.force_kind = p.force_kind;
    // zero without a uniform acceleration, so that instances which know no other force read none
    d.ax = p.force_kind == TCLBM_FORCE_ACCEL ? (float)p.ax : 0.0f;
    d.ay = p.force_kind == TCLBM_FORCE_ACCEL ? (float)p.ay : 0.0f;
    d.famp = (float)p.famp;
    d.rounding = p.storage != TCLBM_STORE_FP32 && p.rounding == TCLBM_ROUND_STOCHASTIC;
    for (int s = 0; s < 4; ++s) {
        d.wall_kind[s] = p.wall[s].kind;
        d.wall_therm[s] = p.wall[s].therm;
        d.wall_rho[s] = (float)p.wall[s].rho;
        d.wall_ux[s] = (float)p.wall[s].ux;
        d.wall_uy[s] = (float)p.wall[s].uy;
        d.wall_T[s] = (float)p.wall[s].T;
        d.wall_RT[s] = (float)(p.R * p.wall[s].T);
        d.wall_dRT[s] = (float)(p.R * p.wall[s].T - RTb);
    }
    d.dRTp = (float)(p.R * p.T0 - RTb);
    d.inv_bR2 = 2.0 / (b * p.R);  // the same FP64 expression tclbm_diagnostics_noalloc() takes
    d.work = p.thermal && p.work;
    d.T0d = p.T0;
    // rest-state populations f^eq(1, 0, RT0), h^eq(1, 0, RT0) with Et = Et0
    const double x0 = 1.0 - RTb, x1 = 0.5 * RTb;
    const double fr[9] = {x0 * x0, x1 * x0, x0 * x1, x1 * x0, x0 * x1, x1 * x1, x1 * x1, x1 * x1, x1 * x1};
    const double C0 = RTb * (Etb + RTb);
    const double hr[9] = {Etb - 2.0 * C0, 0.5 * C0, 0.5 * C0, 0.5 * C0, 0.5 * C0, 0, 0, 0, 0};
    for (int q = 0; q < 9; ++q) {
        d.fbase[q] = (float)fr[q];
        d.hbase[q] = p.thermal ? (float)hr[q] : 0.0f;
        d.fbase_d[q] = d.fbase[q];  // (exact)
        d.hbase_d[q] = d.hbase[q];
        d.hrest += d.hbase_d[q];
    }
}

// Lattices that fit in L2 are latency-bound: 2-D tiles of one node per thread (or the
// direct-load kernel with short strips where tiles do not apply) expose the most
// parallelism (runs of 8 or more steps of lattices that fit in shared memory stay there:
// resident_steps).  Larger lattices stream rows through the TMA ring in 128-wide strips
// (rows per CTA: default_shape).
constexpr long long kSmallNodes = 1LL << 21, kChainNodes = 1LL << 20;

// Launch shape a kernel variant gets by default: (tx, rows per CTA) for the marching
// kernels, the tile (BX, BY) for KERNEL_TILE.
void default_shape(const tclbm_params& p, int kernel, int& tx, int& ty) {
    if (kernel == KERNEL_TILE) {
        tx = kTileBX;
        ty = kTileBY;
    } else if (kernel == KERNEL_DIRECT) {
        tx = p.nx >= 96 ? 64 : 32;
        const long long strips = (p.nx + tx - 1) / tx;
        long long t = (long long)p.ny * strips / (8LL * 152);
        ty = (int)(t < 2 ? 2 : (t > 16 ? 16 : t));
    } else {
        // Without the correction term: 16 rows per CTA, or 32 (fewer halo rows per node) where
        // the last wave's tail weighs little: where the 32-row grid spans more than two waves
        // of the kernel's resident CTAs, so its tail of half-height segments applies (ny a
        // multiple of 8), else where it spans at least 8 waves (16 rows win by 12-20 % on
        // athermal 2048 x 2048, which has no short tail at 32).
        tx = p.nx >= 512 ? 128 : (p.nx >= 96 ? 64 : 32);
        const long long strips = (p.nx + tx - 1) / tx;
        const long long resident = tma_resident(p.storage, tx, p.thermal && p.correction, p.thermal);
        if (p.thermal && p.correction) {
            // Chained launches overlap consecutive steps, so the tail no longer sets the
            // segment height: the tallest segments whose grid spans 1.65 waves of resident
            // CTAs.  Measured (us per step at 16 / 32 / 48 / 64 rows): 4096 x 2048 FP32 245 /
            // 227 / 220 / 217 with 9.0 / 4.9 / 3.5 / 2.7 waves, FP16 234 / 218 / 214 / 210 with
            // 6.8 / 3.8 / 2.7 / 1.7; 2048 x 2048 bf16 120 / 109 / 151 / 130 with 3.4 / 1.7 /
            // 1.1 / 0.8; 2051 x 1537 FP32 104 / 98 / 101 / 124 with 3.6 / 1.8 / 1.2 / 0.9.
            DevParams d = {};
            d.nx = p.nx;
            d.ny = p.ny;
            for (int rows : {96, 64, 48, 32, 16}) {
                const SegPlan plan = tma_seg_plan(d, tx, rows, resident);
                if (20 * strips * (plan.full + plan.half) >= 33 * resident) {
                    ty = rows;
                    return;
                }
            }
            ty = 8;
            return;
        }
        if (p.ny % 8 == 0)
            ty = strips * (p.ny / 32) > 2 * resident ? 32 : 16;
        else
            ty = strips * ((p.ny + 31) / 32) >= 8 * resident ? 32 : 16;
    }
}

bool tile_fits(const tclbm_params& p, int bx, int by) {
    const bool xper = p.wall[TCLBM_SIDE_XM].kind == TCLBM_WALL_PERIODIC;
    const bool yper = p.wall[TCLBM_SIDE_YM].kind == TCLBM_WALL_PERIODIC;
    return tile_kernel_fits(p.nx, p.ny, xper, yper, p.thermal, p.correction, bx, by);
}

void default_launch(const tclbm_params& p, int& tx, int& ty, int& kernel) {
    const long long n = (long long)p.nx * p.ny;
    // With the correction term chained TMA launches take over from the tiles at 2^20 nodes
    // (us per step, tiles / chained: 2048 x 1024 FP32 81 / 68, FP16 87 / 66; 1024 x 1024 42.5 /
    // 39; 1024 x 512 19.5 / 26).  The work term, which the tiles round their own way, and
    // lattices whose last strip is too narrow to chain stay with them up to 2^21.
    const int tail = p.nx % 128;
    const bool chains = p.thermal && p.correction && !p.work && (tail == 0 || tail >= 3);
    if (n <= kSmallNodes && !(chains && n >= kChainNodes && p.nx >= 512))
        kernel = tile_fits(p, kTileBX, kTileBY) ? KERNEL_TILE : KERNEL_DIRECT;
    else
        kernel = KERNEL_TMA;
    default_shape(p, kernel, tx, ty);
}

void default_tile(const tclbm_params& p, int kernel, int& tx, int& ty) { default_shape(p, kernel, tx, ty); }

// ------------------------------------------------------------------ small kernels

__device__ __forceinline__ int wrapi(int i, int n) {
    i %= n;
    return i < 0 ? i + n : i;
}

// f_bar = f^eq - S/2, h_bar = h^eq at each node (FP64), written where the pull of the
// next step reads it: buffer_q(x - e_q) = value_q(x).  Bound by the FP64 pipe: the values
// are formed with as few of its instructions as give the same rounding.
template <class ST>
__global__ void init_kernel(const FieldParams p, const double* __restrict__ rho, const double* __restrict__ ux,
                            const double* __restrict__ uy, const double* __restrict__ T, ST* __restrict__ dst,
                            int thermal, double R, double T0, double b, int force_kind, double ax, double ay,
                            double famp) {
    const long long n = (long long)p.nx * p.ny;
    const bool wide = wide_nodes(n);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        int x, y;
        node_xy(i, p.nx, wide, x, y);
        const double r = rho[i], vx = ux[i], vy = uy[i], t = thermal ? T[i] : T0;
        const double RT = __dmul_rn(R, t), ux2 = __dmul_rn(vx, vx), uy2 = __dmul_rn(vy, vy);
        const double qx = __dadd_rn(RT, ux2), qy = __dadd_rn(RT, uy2);
        // r X(e_x) and Y(e_y), e = 0, +1, -1
        const double rx[3] = {__dmul_rn(r, __dsub_rn(__dsub_rn(1.0, RT), ux2)), __dmul_rn(r, __dmul_rn(0.5, __dadd_rn(qx, vx))),
                              __dmul_rn(r, __dmul_rn(0.5, __dsub_rn(qx, vx)))};
        const double py[3] = {__dsub_rn(__dsub_rn(1.0, RT), uy2), __dmul_rn(0.5, __dadd_rn(qy, vy)),
                              __dmul_rn(0.5, __dsub_rn(qy, vy))};
        constexpr int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, ey[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
        double hS[9];  // S/2 by Eq. 3 of its raw moments
        double Fx = 0, Fy = 0;
        if (force_kind != FORCE_NONE) {
            double Ax = ax, Ay = ay;
            if (force_kind == FORCE_ACCEL) {
                Fx = r * ax;
                Fy = r * ay;
            } else {
                const double kx = 6.283185307179586 / p.nx, ky = 6.283185307179586 / p.ny;
                Fx = famp * sin(kx * x) * sin(ky * y);
                Fy = famp * cos(kx * x) * cos(ky * y);
                Ax = Fx / r;
                Ay = Fy / r;
            }
            const double axx = Ax * vx, ayy = Ay * vy, uxy2 = 2.0 * (vx * vy);
            const double ep = 2.0 * axx, em = 2.0 * ayy, E = ep + em;  // (E + N) / 2, (E - N) / 2, E
            const double P = fma(Ax, vy, Ay * vx);
            const double s21 = fma(Ay, ux2, Ax * uxy2), s12 = fma(Ax, uy2, Ay * uxy2), s22 = uxy2 * P;
            const double hr = 0.25 * r, qr = 0.125 * r;  // half of r/2, r/4
            const double c1 = ep - s22, c2 = em - s22, m1 = Ax - s12, m2 = Ay - s21;
            const double sp = s21 + s12, sm = s21 - s12, pp = s22 + P, pm = s22 - P;
            hS[0] = (0.5 * r) * (s22 - E);
            hS[1] = hr * (c1 + m1);
            hS[2] = hr * (c2 + m2);
            hS[3] = hr * (c1 - m1);
            hS[4] = hr * (c2 - m2);
            hS[5] = qr * (pp + sp);
            hS[6] = qr * (pm + sm);
            hS[7] = qr * (pp - sp);
            hS[8] = qr * (pm - sm);
        } else {
#pragma unroll
            for (int q = 0; q < 9; ++q) hS[q] = 0.0;
        }
        // source rows and columns of the pull, or none past a wall
        auto wrap = [](int s, int m, int per) { return s < 0 ? (per ? s + m : -1) : (s >= m ? (per ? s - m : -1) : s); };
        const int xs[3] = {x, wrap(x - 1, p.nx, p.xper), wrap(x + 1, p.nx, p.xper)};
        const int ys[3] = {y, wrap(y - 1, p.ny, p.yper), wrap(y + 1, p.ny, p.yper)};
        auto put = [&](int q, int plane, double v) {
            const int sx = xs[ex[q] == 0 ? 0 : (ex[q] > 0 ? 1 : 2)], sy = ys[ey[q] == 0 ? 0 : (ey[q] > 0 ? 1 : 2)];
            if (sx >= 0 && sy >= 0) Store<ST>::st(dst + plane * p.plane + ((long long)sy * p.pitch + sx), d2f(v));
        };
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const double a = rx[ex[q] == 0 ? 0 : (ex[q] > 0 ? 1 : 2)], c = py[ey[q] == 0 ? 0 : (ey[q] > 0 ? 1 : 2)];
            put(q, q, __dsub_rn(__fma_rn(a, c, -hS[q]), p.fbase_d[q]));
        }
        if (thermal) {
            const double uu = __dadd_rn(ux2, uy2), Et = __dmul_rn(0.5, __fma_rn(b, RT, uu)), A = __dadd_rn(Et, RT),
                         B = __fma_rn(2.0, RT, Et), C = __dmul_rn(RT, A);
            const double hr = __dmul_rn(0.5, r), bx = __dmul_rn(B, ux2), by = __dmul_rn(B, uy2);
            const double qb = __dmul_rn(__dmul_rn(__dmul_rn(__dmul_rn(0.25, r), B), vx), vy);
            double hv[9];
            hv[0] = __dmul_rn(r, __fma_rn(-2.0, C, __fma_rn(-B, uu, Et)));
            hv[1] = __dmul_rn(hr, __dadd_rn(__fma_rn(A, vx, bx), C));
            hv[2] = __dmul_rn(hr, __dadd_rn(__fma_rn(A, vy, by), C));
            hv[3] = __dmul_rn(hr, __dadd_rn(__fma_rn(-A, vx, bx), C));
            hv[4] = __dmul_rn(hr, __dadd_rn(__fma_rn(-A, vy, by), C));
            hv[5] = hv[7] = qb;
            hv[6] = hv[8] = -qb;
            if (p.work) {  // h_bar = h^eq - q / 2, q_a = W_a F.u
                const double fu = __fma_rn(Fx, vx, __dmul_rn(Fy, vy));
#pragma unroll
                for (int q = 0; q < 9; ++q)
                    hv[q] = __fma_rn(-0.5 * (q == 0 ? 4.0 / 9.0 : (q <= 4 ? 1.0 / 9.0 : 1.0 / 36.0)), fu, hv[q]);
            }
#pragma unroll
            for (int q = 0; q < 9; ++q) put(q, 9 + q, __dsub_rn(hv[q], p.hbase_d[q]));
        }
    }
}

// Arbitrary populations (double [9][ny][nx] each) written in the pull layout.
template <class ST>
__global__ void set_pops_kernel(const FieldParams p, const double* __restrict__ f, const double* __restrict__ h,
                                ST* __restrict__ dst, int thermal) {
    const long long n = (long long)p.nx * p.ny;
    const int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, ey[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
    NodeWalk w(blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, p.nx);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x, w.next(p.nx)) {
        const int x = w.x, y = w.y;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            int xs = x - ex[q], ys = y - ey[q];
            if (p.xper) xs = wrapi(xs, p.nx); else if (xs < 0 || xs >= p.nx) continue;
            if (p.yper) ys = wrapi(ys, p.ny); else if (ys < 0 || ys >= p.ny) continue;
            const long long o = (long long)ys * p.pitch + xs;
            Store<ST>::st(dst + q * p.plane + o, d2f(f[q * n + i] - p.fbase_d[q]));
            if (thermal) Store<ST>::st(dst + (9 + q) * p.plane + o, d2f(h[q * n + i] - p.hbase_d[q]));
        }
    }
}

// Observable state: streamed populations with wall schemes applied (double [9][ny][nx]).
template <bool THERMAL, class ST>
__global__ void get_pops_kernel(const FieldParams p, const ST* __restrict__ src, double* __restrict__ f,
                                double* __restrict__ h) {
    const long long n = (long long)p.nx * p.ny;
    NodeWalk w(blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, p.nx);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x, w.next(p.nx)) {
        const int x = w.x, y = w.y;
        float fv[9], hv[9];
        load_node<THERMAL, ST>(p, src, x, y, fv, hv);
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            f[q * n + i] = p.fbase_d[q] + f2d(fv[q]);
            if (THERMAL && h) h[q * n + i] = p.hbase_d[q] + f2d(hv[q]);
        }
    }
}

// Eq. 20 and the temperature of Section IV in FP64 from the observable state.
template <bool THERMAL, class ST>
__global__ void moments_kernel(const FieldParams p, const ST* __restrict__ src, double* __restrict__ rho,
                               double* __restrict__ ux, double* __restrict__ uy, double* __restrict__ T) {
    const long long n = (long long)p.nx * p.ny;
    NodeWalk w(blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, p.nx);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x, w.next(p.nx)) {
        const int x = w.x, y = w.y;
        float fv[9], hv[9];
        load_node<THERMAL, ST>(p, src, x, y, fv, hv);
        const NodeTotals s = node_totals<THERMAL>(p, node_sums<THERMAL>(fv, hv), fv, hv);
        const NodeFields v = node_velocity(p, s, x, y);
        rho[i] = v.rho;
        ux[i] = v.ux;
        uy[i] = v.uy;
        T[i] = node_temperature<THERMAL>(p, v, s.sh, THERMAL ? __fma_rn(v.ux, v.ux, v.uy * v.uy) : 0.0, x, y);
    }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// FP64 sums (see tclbm_diagnostics) -> one partial per block, summed by diag_finish.
template <bool THERMAL, class ST>
__global__ void __launch_bounds__(kDiagBlock) diag_kernel(const FieldParams p, const ST* __restrict__ src,
                                                          const float* __restrict__ usnap, double T_ref,
                                                          double* __restrict__ partial) {
    __shared__ double red[kDiagBlock / 32][TCLBM_NDIAG];
    double acc[TCLBM_NDIAG] = {0, 0, 0, 0, 0, 0, 0, 0};
    const long long n = (long long)p.nx * p.ny;
    // the linear sums stay FP32 error-free sums of deviations until the thread's last node
    // (where a node's are narrow; the others enter acc at once)
    Running drho, jx, jy, sdh;
    double nodes = 0, Fxs = 0, Fys = 0;  // narrow nodes seen; the Taylor-Green forces of all
    NodeWalk w(blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, p.nx);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x, w.next(p.nx)) {
        const int x = w.x, y = w.y;
        float fv[9], hv[9];
        load_node<THERMAL, ST>(p, src, x, y, fv, hv);
        const NodeSums s = node_sums<THERMAL>(fv, hv);
        const NodeTotals total = node_totals<THERMAL>(p, s, fv, hv);
        const NodeFields v = node_velocity(p, total, x, y);
        const double uu = __fma_rn(v.ux, v.ux, v.uy * v.uy);
        if (s.narrow()) {
            drho.add(s.drho);
            jx.add(s.jx);
            jy.add(s.jy);
            if (THERMAL) sdh.add(s.sdh);
            nodes += 1.0;
        } else {
            acc[0] += total.rho;
            acc[1] += total.jx;
            acc[2] += total.jy;
            acc[3] += total.sh;
        }
        if (p.force_kind == FORCE_TAYLOR_GREEN) {
            Fxs = __fma_rn(f2d(p.sx[x]), f2d(p.sy[y]), Fxs);
            Fys = __fma_rn(f2d(p.cx[x]), f2d(p.cy[y]), Fys);
        }
        const double t = node_temperature<THERMAL>(p, v, total.sh, uu, x, y);
        acc[4] = __fma_rn(v.rho, uu, acc[4]);
        acc[5] = __fma_rn(v.uy, t - T_ref, acc[5]);
        if (usnap) {
            const double dx = v.ux - f2d(usnap[2 * i]), dy = v.uy - f2d(usnap[2 * i + 1]);
            acc[6] = __fma_rn(dx, dx, __fma_rn(dy, dy, acc[6]));
        }
        acc[7] += uu;
    }
    // sum rho, sum (j + F/2), sum h_bar and the kinetic energy of this thread's nodes
    acc[0] += nodes + drho.value();
    acc[1] += jx.value();
    acc[2] += jy.value();
    if (p.force_kind == FORCE_TAYLOR_GREEN) {
        acc[1] = __fma_rn(0.5 * (double)p.famp, Fxs, acc[1]);
        acc[2] = __fma_rn(0.5 * (double)p.famp, Fys, acc[2]);
    } else if (p.force_kind == FORCE_ACCEL) {
        acc[1] = __fma_rn(0.5 * (double)p.ax, acc[0], acc[1]);
        acc[2] = __fma_rn(0.5 * (double)p.ay, acc[0], acc[2]);
    }
    if (THERMAL) acc[3] += __fma_rn(nodes, p.hrest, sdh.value());
    acc[4] *= 0.5;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < TCLBM_NDIAG; ++k) {
        const double v = warp_sum(acc[k]);
        if (lane == 0) red[wid][k] = v;
    }
    __syncthreads();
    if (threadIdx.x < TCLBM_NDIAG) {
        double s = 0;
        for (int w = 0; w < kDiagBlock / 32; ++w) s += red[w][threadIdx.x];
        partial[blockIdx.x * TCLBM_NDIAG + threadIdx.x] = s;
    }
}

// Warp k sums quantity k over the block partials (a single thread's chain of 1024 additions
// took 45 us); the error word of the step kernels rides along in out[TCLBM_NDIAG].
__global__ void diag_finish(const double* __restrict__ partial, int nblocks, const int* __restrict__ err,
                            double* __restrict__ out) {
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s = 0;
    for (int b = lane; b < nblocks; b += 32) s += partial[b * TCLBM_NDIAG + k];
    s = warp_sum(s);
    if (lane == 0) out[k] = s;
    if (threadIdx.x == 0) out[TCLBM_NDIAG] = (double)*err;
}

template <bool THERMAL, class ST>
__global__ void snapshot_kernel(const FieldParams p, const ST* __restrict__ src, float* __restrict__ usnap) {
    const long long n = (long long)p.nx * p.ny;
    NodeWalk w(blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, p.nx);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x, w.next(p.nx)) {
        const int x = w.x, y = w.y;
        float fv[9], hv[9];
        load_node<THERMAL, ST>(p, src, x, y, fv, hv);
        const NodeFields v = node_velocity(p, node_totals<false>(p, node_sums<false>(fv, hv), fv, hv), x, y);
        usnap[2 * i] = d2f(v.ux);
        usnap[2 * i + 1] = d2f(v.uy);
    }
}

// Pageable host arrays a call is about to fill.  Their pages are made present by the host while
// the call's own kernel runs: a device-to-host copy into pages nobody has touched yet (a fresh
// array of a hundred kilobytes or more) faults them in one by one from the copy's side (moments
// of 256 x 128 into fresh arrays 270 to 500 us against 90 to 190, of 1024 x 512 1130 / 720).  Work
// queued on the handle earlier may still read the arrays, so it is waited for first.  Plain
// stores: populating the range by madvise, or reading a byte and storing it back, took 16 served
// requests from 39 to 45-100 ms a pass where the heap is growing.
struct HostOutputs {
    volatile char* array[4];
    int count = 0;
    size_t bytes = 0;

    // the arrays of `n` given that are pageable and large enough; waits for queued work if any
    tclbm_status begin(const tclbm_lattice* L, double* const* given, int n, size_t size) {
        bytes = size;
        for (int k = 0; k < n && bytes >= 65536; ++k) {
            // what CUDA knows is present, or not for the host to write
            cudaPointerAttributes at;
            if (!given[k]) continue;
            if (cudaPointerGetAttributes(&at, given[k]) == cudaSuccess && at.type == cudaMemoryTypeUnregistered)
                array[count++] = reinterpret_cast<volatile char*>(given[k]);
            else
                cudaGetLastError();
        }
        if (count > 0) CK(cudaStreamSynchronize(L->stream));
        return TCLBM_OK;
    }
    void touch() const {
        static const size_t page = (size_t)sysconf(_SC_PAGESIZE);
        for (int k = 0; k < count; ++k) {
            array[k][0] = 0;
            for (size_t i = page - (uintptr_t)array[k] % page; i < bytes; i += page) array[k][i] = 0;
        }
    }
};

int grid_for(long long n, int block) {
    long long g = (n + block - 1) / block;
    if (g > 152 * 16) g = 152 * 16;
    if (g < 1) g = 1;
    return (int)g;
}

// ---------------------------------------------------------------- storage dispatch

template <class F>
tclbm_status with_storage(int storage, F&& fn) {
    switch (storage) {
        case TCLBM_STORE_FP32: return fn((float*)nullptr);
        case TCLBM_STORE_BF16: return fn((__nv_bfloat16*)nullptr);
        default: return fn((__half*)nullptr);
    }
}

tclbm_status ensure_maps(tclbm_lattice* L);

StepLaunch step_launch(tclbm_lattice* L, int src) {
    StepLaunch k;
    k.thermal = L->prm.thermal;
    k.correction = L->prm.correction;
    k.tx = L->tx;
    k.ty = L->ty;
    k.kernel = L->kernel;
    k.src_map = &L->maps[src];
    k.err = L->err;
    k.parity = src;
    return k;
}

// Whether consecutive TMA launches of L can be chained: the correction-term kernel, row
// segments of at least 4 rows (half-height tails of 8-row plans), and a last strip at least
// as wide as the three columns its neighbours read of it.  (The row copies bring more
// columns than that; what they bring of a strip further away is never used.)
bool chainable(const tclbm_lattice* L) {
    const int tail = L->prm.nx % L->tx;
    return L->kernel == KERNEL_TMA && L->prm.thermal && L->prm.correction && L->ty >= 8 && (tail == 0 || tail >= 3);
}

// Whether a caller is capturing `s` (a replayed launch would reuse tickets and step numbers).
bool capturing(cudaStream_t s) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) {
        cudaGetLastError();
        return true;
    }
    return cap != cudaStreamCaptureStatusNone;
}

// Launches that do not chain (a call of fewer than kChainSteps steps, a stream being captured)
// of a lattice the library gave to the TMA kernel for its chains: 2-D tiles where these are
// the faster single steps, i.e. below 1.5 M nodes and where the last strip leaves more than a
// tenth of the strips empty.  Measured (us per step in calls of one step, TMA / tiles):
// 1024 x 1024 FP32 51.7 / 43.0, FP16 46.9 / 46.3; 1200 x 1000 FP32 56.8 / 49.6; 515 x 4000
// 94.0 / 84.9; but 1448 x 1448 80.1 / 82.8, 2048 x 1024 77.5 / 81.5.  In calls of two steps
// 1411 x 801 takes 52.5 / 47.3, of four 46 / 47.  The states are the same bit for bit.
constexpr int64_t kChainSteps = 4;
bool tiles_unchained(const tclbm_lattice* L) {
    const tclbm_params& p = L->prm;
    const long long nodes = (long long)p.nx * p.ny, strips = (p.nx + L->tx - 1) / L->tx;
    if (!L->auto_kernel || L->kernel != KERNEL_TMA || nodes > kSmallNodes || p.work || !tile_fits(p, kTileBX, kTileBY))
        return false;
    return nodes < 3 * (kSmallNodes / 4) || 10LL * p.nx < 9LL * strips * L->tx;
}

tclbm_status launch_steps(tclbm_lattice* L, int64_t n) {
    const bool chains = n > 1 && chainable(L) && !capturing(L->stream);
    const bool tiles = (n < kChainSteps || !chains) && tiles_unchained(L);
    if (n > 0 && L->kernel == KERNEL_TMA && !tiles) {
        tclbm_status st = ensure_maps(L);
        if (st != TCLBM_OK) return st;
    }
    // TMA launches with the correction term publish per-item completion tickets; after the
    // first launch of this run the next one waits for each item's neighbours only
    const bool tickets = L->kernel == KERNEL_TMA && L->prm.thermal && L->prm.correction && !tiles;
    const bool chain = chains && !tiles;
    const int first = L->cur;
    tclbm_status st = TCLBM_OK;
    int64_t s = 0;
    for (; s < n; ++s) {
        StepLaunch k = step_launch(L, L->cur);
        if (tiles) {
            k.kernel = KERNEL_TILE;
            k.tx = kTileBX;
            k.ty = kTileBY;
        }
        if (tickets) {
            k.seg_done = L->seg_done;
            k.seg_cap = (long long)(L->seg_bytes / sizeof(unsigned));
            k.ticket = ++L->ticket;
            k.chain = chain && s > 0;
        }
        if (chain && L->dp.rounding) {  // no launch of the chain may write the counter others read
            k.ctr_copy = first;
            k.ctr_add = (unsigned)s;
        }
        const cudaError_t e = refuse_launch() ? cudaErrorLaunchOutOfResources
                                              : launch_step_kernel(L->prm.storage, k, L->dp, L->buf[L->cur],
                                                                   L->buf[L->cur ^ 1], L->stream);
        if (e != cudaSuccess) {
            st = cuda_fail(e, "step kernel launch");
            break;
        }
        L->cur ^= 1;
        ++L->steps;
    }
    if (chain && L->dp.rounding && s > 0) {  // also after a failure: the steps that were launched count
        DevParams p = L->dp;
        p.parity = first;
        tclbm_count_steps<<<1, 1, 0, L->stream>>>(p, L->cur, (unsigned)s);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess && st == TCLBM_OK) st = cuda_fail(e, "step counter");
    }
    return st;
}

// Steps of one resident launch at most (1.5 to 6 ms, which work of other streams may have to
// wait for), and the fewest steps worth one: filling and emptying the shared memory costs
// about as much as two steps, and 2-D tiles take little longer than a resident step (320 x 170
// FP16 4.5 us; calls of 8 steps 4.9 resident, of 12 4.5, long runs 4.2).
constexpr int64_t kResMaxSteps = 1024, kResMinSteps = 8, kResMinStepsTiles = 12;
int64_t res_min_steps(const tclbm_lattice* L) { return L->kernel == KERNEL_TILE ? kResMinStepsTiles : kResMinSteps; }

// Resident launches of one lattice that the device has to hold at once for lattices on several
// streams to run so.  A resident launch keeps its multiprocessors to itself for hundreds of
// steps, where one-step launches of several lattices share them.  Measured (us per step of all,
// K lattices on streams of their own, resident / one launch per step): 64 x 32 thermal with the
// correction term (15 fit) K = 4 2.6 / 3.1, K = 16 3.7 / 6.5; 64 x 64 (7.6 fit) K = 8 4.0 / 3.5;
// 256 x 128 (1 fits) K = 2 5.9 / 4.0, K = 16 47.7 / 18.7; athermal 80 x 80 (9.5 fit) K = 16
// 3.6 / 8.8, 192 x 192 (2.0 fit) K = 8 8.5 / 5.4.
constexpr long long kResShared = 8;

int res_kind(const tclbm_params& p) { return !p.thermal ? RES_ATHERMAL : (p.correction ? RES_CORR : RES_THERMAL); }

// Whether L runs resident where enough steps are asked for (planned on first use): the library
// chose its kernel and shape, it fits, and it has the device to itself or takes little of it.
bool resident_planned(tclbm_lattice* L) {
    if (!L->auto_kernel || L->dp.work) return false;
    if (L->res_state == 0) {
        int dev = 0, coop = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess) {
            cudaGetLastError();
            coop = 0;
        }
        L->res_state = coop && res_plan(L->dp, res_kind(L->prm), sm_count(), L->res_plan) ? 1 : -1;
    }
    if (L->res_state < 0 || only_stream(L->use)) return L->res_state > 0;
    if (L->res_small < 0)
        L->res_small = (long long)resident_per_sm(L->storage, res_kind(L->prm), L->res_plan, L->dp) * sm_count() >=
                       kResShared * L->res_plan.gx * L->res_plan.gy;
    return L->res_small > 0;
}

// Advances L by as many of n steps as resident launches take (`done`); 0 where they do not
// apply: a kernel or shape chosen by the caller, a lattice too large, the work term (whose
// rounding differs between the one-step kernels), a capturing stream (a replayed launch
// would reuse its step numbers), no memory for the board.
tclbm_status resident_steps(tclbm_lattice* L, int64_t n, int64_t& done) {
    done = 0;
    const int64_t fewest = res_min_steps(L);
    if (n < fewest || !resident_planned(L)) return TCLBM_OK;
    if (capturing(L->stream)) return TCLBM_OK;
    if (!L->board) {
        L->board_bytes = 2 * (size_t)L->prm.nx * L->prm.ny * (size_t)(L->nplanes / 3) * 16;
        {
            // cudaMalloc would break a global-mode capture of another stream that is open just
            // now; this allocation is no part of one (this stream is not capturing)
            cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
            CK(cudaThreadExchangeStreamCaptureMode(&mode));
            L->board = dev_alloc(L, L->board_bytes);
            CK(cudaThreadExchangeStreamCaptureMode(&mode));
        }
        if (!L->board) {
            L->res_state = -1;
            return TCLBM_OK;
        }
        L->res_tag = 0xffffffffu;  // cleared below
    }
    while (n - done >= fewest) {
        const int64_t k = n - done < kResMaxSteps ? n - done : kResMaxSteps;
        if (L->res_tag > 0xffffffffu - (unsigned)k) {  // step numbers start over on a cleared board
            CK(cudaMemsetAsync(L->board, 0, L->board_bytes, L->stream));
            L->res_tag = 0;
        }
        ResLaunch r;
        r.plan = L->res_plan;
        r.kind = res_kind(L->prm);
        r.parity = L->cur;
        r.n = (int)k;
        r.tag0 = L->res_tag;
        r.board = L->board;
        r.err = L->err;
        const int to = L->cur ^ (int)(k & 1);  // the copy that k launches would end in
        const cudaError_t e = refuse_launch()
                                  ? cudaErrorLaunchOutOfResources
                                  : launch_resident(L->prm.storage, r, L->dp, L->buf[L->cur], L->buf[to], L->stream);
        if (e == cudaErrorCooperativeLaunchTooLarge) {  // fewer multiprocessors than the device has are ours
            cudaGetLastError();
            L->res_state = -1;
            return TCLBM_OK;
        }
        if (e != cudaSuccess) return cuda_fail(e, "resident kernel launch");
        L->res_tag += (unsigned)k;
        L->cur = to;
        L->steps += k;
        done += k;
    }
    return TCLBM_OK;
}

tclbm_status build_graph(tclbm_lattice* L) {
    if (L->graph && L->graph_tx == L->tx && L->graph_ty == L->ty && L->graph_kernel == L->kernel) return TCLBM_OK;
    if (L->kernel == KERNEL_TMA) {
        tclbm_status st = ensure_maps(L);
        if (st != TCLBM_OK) return st;
    }
    if (L->graph) {
        cudaGraphExecDestroy(L->graph);
        L->graph = nullptr;
    }
    cudaStream_t cs;
    CK(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        for (int s = 0; s < 2 * kGraphPairs && e == cudaSuccess; ++s)
            e = launch_step_kernel(L->prm.storage, step_launch(L, s & 1), L->dp, L->buf[s & 1], L->buf[(s & 1) ^ 1],
                                   cs);
        cudaError_t e2 = cudaStreamEndCapture(cs, &g);
        if (e == cudaSuccess) e = e2;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&L->graph, g, 0);
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cs);
    if (e != cudaSuccess) {
        L->graph = nullptr;
        return cuda_fail(e, "step graph capture");
    }
    L->graph_tx = L->tx;
    L->graph_ty = L->ty;
    L->graph_kernel = L->kernel;
    return TCLBM_OK;
}

}  // namespace

// TMA descriptors of both copies of L for strips of tx columns: 3-D (x, y, plane), box
// (tx + 2M, 1, planes).
tclbm_status tclbm::encode_row_maps(const tclbm_lattice* L, int tx, CUtensorMap out[2]) {
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        cudaDriverEntryPointQueryResult q;
        void* fn = nullptr;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn)
            return fail(TCLBM_ECUDA, "cuTensorMapEncodeTiled is not available");
        encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    const CUtensorMapDataType dt = L->prm.storage == TCLBM_STORE_FP32   ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                   : L->prm.storage == TCLBM_STORE_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                                        : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
    const cuuint64_t dims[3] = {(cuuint64_t)L->dp.pitch, (cuuint64_t)L->prm.ny, (cuuint64_t)L->nplanes};
    const cuuint64_t strides[2] = {(cuuint64_t)L->dp.pitch * L->elem, (cuuint64_t)L->dp.plane * L->elem};
    const cuuint32_t box[3] = {(cuuint32_t)tma_box_width(L->prm.storage, tx), 1u, (cuuint32_t)L->nplanes};
    const cuuint32_t estr[3] = {1u, 1u, 1u};
    for (int b = 0; b < 2; ++b) {
        const CUresult r = encode(&out[b], dt, 3, L->buf[b], dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                  CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return fail(TCLBM_ECUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
    }
    return TCLBM_OK;
}

namespace {

tclbm_status ensure_maps(tclbm_lattice* L) {
    if (L->maps_tx == L->tx) return TCLBM_OK;
    tclbm_status st = encode_row_maps(L, L->tx, L->maps);
    if (st != TCLBM_OK) return st;
    L->maps_tx = L->tx;
    return TCLBM_OK;
}

// Error word of the step kernels (a bounded wait expired): ETIMEOUT once, then cleared.
tclbm_status check_kernel_error(tclbm_lattice* L) {
    int v = 0;
    CK(cudaMemcpyAsync(&v, L->err, sizeof v, cudaMemcpyDeviceToHost, L->stream));
    CK(cudaStreamSynchronize(L->stream));
    if (v) {
        CK(cudaMemsetAsync(L->err, 0, sizeof(int), L->stream));
        return fail(TCLBM_ETIMEOUT, "a step kernel's pipeline wait expired (%d)", v);
    }
    return TCLBM_OK;
}

}  // namespace

// Entries of the completion-ticket array of the TMA kernel's work items: strips of at
// least 32 columns times segments of at least 4 rows (half-height segments of 8-row plans).
static size_t seg_entries(int nx, int ny) { return (size_t)((nx + 31) / 32) * (size_t)(ny / 4 + 2); }

// ==================================================================== C ABI

extern "C" {

const char* tclbm_last_error(void) { return g_err; }

size_t tclbm_state_bytes(const tclbm_params* p) {
    if (!p || p->nx < 1 || p->ny < 1) return 0;
    const size_t n = (size_t)p->nx * p->ny;
    const size_t planes = p->thermal ? 18 : 9;
    const size_t pops = 2 * planes * (size_t)p->ny * pitch_of(p->nx) * elem_of(p->storage);
    const size_t tables = sizeof(float) * 2 * ((size_t)p->nx + p->ny);
    const size_t diag = sizeof(double) * ((kDiagMaxBlocks + 1) * TCLBM_NDIAG + 1);
    return pops + tables + diag + n * 4 * sizeof(double) + seg_entries(p->nx, p->ny) * sizeof(unsigned);
}

tclbm_status tclbm_create(const tclbm_params* params, tclbm_alloc_fn alloc, tclbm_free_fn free_fn, void* ctx,
                          void* stream, tclbm_lattice** out) {
    if (!out) return fail(TCLBM_EINVAL, "out is NULL");
    *out = nullptr;
    tclbm_status st = validate(params);
    if (st != TCLBM_OK) return st;
    if ((alloc == nullptr) != (free_fn == nullptr)) return fail(TCLBM_EINVAL, "alloc and free must be given together");
    tclbm_lattice* L = new (std::nothrow) tclbm_lattice;
    if (!L) return fail(TCLBM_ENOMEM, "host allocation failed");
    L->prm = *params;
    L->alloc = alloc;
    L->free_fn = free_fn;
    L->ctx = ctx;
    L->stream = (cudaStream_t)stream;
    L->storage = params->storage;
    L->elem = elem_of(params->storage);
    L->nplanes = params->thermal ? 18 : 9;
    derive(L);
    default_launch(L->prm, L->tx, L->ty, L->kernel);
    const size_t n = (size_t)params->nx * params->ny;
    L->buf_bytes = (size_t)L->nplanes * L->dp.plane * L->elem;
    L->tables_bytes = sizeof(float) * 2 * ((size_t)params->nx + params->ny);
    L->diag_bytes = sizeof(double) * ((kDiagMaxBlocks + 1) * TCLBM_NDIAG + 1);
    L->stage_bytes = n * 4 * sizeof(double);
    L->buf[0] = dev_alloc(L, L->buf_bytes);
    L->buf[1] = dev_alloc(L, L->buf_bytes);
    L->tables = (float*)dev_alloc(L, L->tables_bytes);
    L->diag = (double*)dev_alloc(L, L->diag_bytes);
    L->stage = (double*)dev_alloc(L, L->stage_bytes);
    L->err = (int*)dev_alloc(L, 256);
    L->seg_bytes = seg_entries(params->nx, params->ny) * sizeof(unsigned);
    L->seg_done = (unsigned*)dev_alloc(L, L->seg_bytes);
    if (!L->buf[0] || !L->buf[1] || !L->tables || !L->diag || !L->stage || !L->err || !L->seg_done) {
        tclbm_destroy(L);
        return fail(TCLBM_ENOMEM, "device allocation of %zu bytes failed", tclbm_state_bytes(params));
    }
    // Taylor-Green force tables: sin/cos of 2 pi x / nx and 2 pi y / ny
    {
        const int nx = params->nx, ny = params->ny;
        float* h = new (std::nothrow) float[2 * ((size_t)nx + ny)];
        if (!h) {
            tclbm_destroy(L);
            return fail(TCLBM_ENOMEM, "host allocation failed");
        }
        for (int i = 0; i < nx; ++i) {
            h[i] = (float)std::sin(2.0 * M_PI * i / nx);
            h[nx + i] = (float)std::cos(2.0 * M_PI * i / nx);
        }
        for (int j = 0; j < ny; ++j) {
            h[2 * nx + j] = (float)std::sin(2.0 * M_PI * j / ny);
            h[2 * nx + ny + j] = (float)std::cos(2.0 * M_PI * j / ny);
        }
        cudaError_t e = cudaMemcpyAsync(L->tables, h, L->tables_bytes, cudaMemcpyHostToDevice, L->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(L->stream);
        delete[] h;
        if (e != cudaSuccess) {
            tclbm_destroy(L);
            return cuda_fail(e, "table upload");
        }
        L->dp.sx = L->tables;
        L->dp.cx = L->tables + nx;
        L->dp.sy = L->tables + 2 * nx;
        L->dp.cy = L->tables + 2 * nx + ny;
    }
    cudaError_t e = cudaMemsetAsync(L->buf[0], 0, L->buf_bytes, L->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(L->err, 0, 256, L->stream);
    L->dp.step_ctr = reinterpret_cast<unsigned*>(L->err) + 4;  // two counters after the error word
    if (e == cudaSuccess) e = cudaMemsetAsync(L->buf[1], 0, L->buf_bytes, L->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(L->seg_done, 0, L->seg_bytes, L->stream);  // tickets start at 1
    if (e != cudaSuccess) {
        tclbm_destroy(L);
        return cuda_fail(e, "state clear");
    }
    {
        // dynamic shared-memory limits of the TMA kernels, set before any launch or capture
        const cudaError_t pe = params->storage == TCLBM_STORE_FP32   ? prepare_step_fp32()
                               : params->storage == TCLBM_STORE_BF16 ? prepare_step_bf16()
                                                                     : prepare_step_fp16();
        if (pe != cudaSuccess) {
            tclbm_destroy(L);
            return cuda_fail(pe, "step kernel attributes");
        }
    }
    snprintf(L->desc, sizeof L->desc, "unset");
    L->use = use_stream(L->stream);
    *out = L;
    return TCLBM_OK;
}

tclbm_status tclbm_destroy(tclbm_lattice* L) {
    if (!L) return TCLBM_OK;
    if (L->graph) cudaGraphExecDestroy(L->graph);
    cudaStreamSynchronize(L->stream);  // work queued on the handle may still use its memory
    dev_free(L, L->buf[0], L->buf_bytes);
    dev_free(L, L->buf[1], L->buf_bytes);
    dev_free(L, L->tables, L->tables_bytes);
    dev_free(L, L->diag, L->diag_bytes);
    dev_free(L, L->usnap, L->usnap_bytes);
    dev_free(L, L->stage, L->stage_bytes);
    dev_free(L, L->err, 256);
    dev_free(L, L->seg_done, L->seg_bytes);
    dev_free(L, L->board, L->board_bytes);
    if (L->copy_event) cudaEventDestroy(L->copy_event);
    unuse_stream(L->use);
    delete L;
    return TCLBM_OK;
}

tclbm_status tclbm_set_stream(tclbm_lattice* L, void* stream) {
    if (!L) return fail(TCLBM_EINVAL, "lattice is NULL");
    if (L->stream == (cudaStream_t)stream) return TCLBM_OK;
    unuse_stream(L->use);
    L->stream = (cudaStream_t)stream;
    L->use = use_stream(L->stream);
    return TCLBM_OK;
}

int64_t tclbm_steps_done(const tclbm_lattice* L) { return L ? L->steps : -1; }

tclbm_status tclbm_set_tile(tclbm_lattice* L, int32_t tx, int32_t ty) {
    if (!L) return fail(TCLBM_EINVAL, "lattice is NULL");
    int dtx, dty;
    default_tile(L->prm, L->kernel, dtx, dty);
    const int ntx = tx ? tx : dtx, nty = ty ? ty : dty;
    if (L->kernel == KERNEL_TILE) {
        if (!tile_fits(L->prm, ntx, nty))
            return fail(TCLBM_EINVAL, "tile shape %dx%d is not available for this lattice", ntx, nty);
    } else {
        if (tx != 0 && tx != 32 && tx != 64 && tx != 128) return fail(TCLBM_EINVAL, "tx must be 0, 32, 64 or 128");
        if (ty < 0) return fail(TCLBM_EINVAL, "ty must be 0 or >= 1");
    }
    L->tx = ntx;
    L->ty = nty;
    if (tx || ty) L->auto_kernel = false;
    return TCLBM_OK;
}

tclbm_status tclbm_test_skip_row(tclbm_lattice* L, int32_t row) {
    if (!L) return fail(TCLBM_EINVAL, "lattice is NULL");
    if (row < -1 || row >= L->prm.ny) return fail(TCLBM_EINVAL, "row must be -1 or in [0, ny)");
    L->dp.skip_row = row;
    if (L->graph) {  // a captured graph holds the old parameters
        cudaGraphExecDestroy(L->graph);
        L->graph = nullptr;
    }
    return TCLBM_OK;
}

tclbm_status tclbm_test_run_number(tclbm_lattice* L, uint32_t number) {
    if (!L) return fail(TCLBM_EINVAL, "lattice is NULL");
    if (!L->board || number < L->res_tag) return fail(TCLBM_EINVAL, "no resident run yet, or numbers would come again");
    L->res_tag = number;
    return TCLBM_OK;
}

tclbm_status tclbm_test_fail_launch(int64_t after) {
    if (after < -1) return fail(TCLBM_EINVAL, "after must be >= -1");
    g_refuse_in = after;
    return TCLBM_OK;
}

namespace {
// The reciprocal the collision takes of R T, mu/p + 1/2 and the thermal rate's argument.
__global__ void rcp_kernel(const float* __restrict__ x, float* __restrict__ y, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = tclbm::rcp(x[i]);
}

// The quotient the field conversions take.
__global__ void div_kernel(const double* __restrict__ a, const double* __restrict__ x, double* __restrict__ y,
                           long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = div_d(a[i], x[i], rcp_d(x[i]));
}
}  // namespace

tclbm_status tclbm_test_rcp(const float* x, float* y, int64_t n, void* stream) {
    if (n < 0 || (n > 0 && (!x || !y))) return fail(TCLBM_EINVAL, "x, y must be device arrays of n >= 0 floats");
    if (n == 0) return TCLBM_OK;
    cudaStream_t s = (cudaStream_t)stream;
    rcp_kernel<<<grid_for(n, 256), 256, 0, s>>>(x, y, n);
    CK(cudaGetLastError());
    CK(cudaStreamSynchronize(s));
    return TCLBM_OK;
}

tclbm_status tclbm_test_div(const double* a, const double* x, double* y, int64_t n, void* stream) {
    if (n < 0 || (n > 0 && (!a || !x || !y))) return fail(TCLBM_EINVAL, "a, x, y must be device arrays of n >= 0 doubles");
    if (n == 0) return TCLBM_OK;
    cudaStream_t s = (cudaStream_t)stream;
    div_kernel<<<grid_for(n, 256), 256, 0, s>>>(a, x, y, n);
    CK(cudaGetLastError());
    CK(cudaStreamSynchronize(s));
    return TCLBM_OK;
}

tclbm_status tclbm_test_node_walk(uint32_t first, uint32_t stride, int32_t nx, int64_t count, int32_t divide, int32_t* x,
                                  int32_t* y) {
    if (nx < 1 || count < 0 || (count > 0 && (!x || !y))) return fail(TCLBM_EINVAL, "bad node walk");
    NodeWalk w(first, stride, nx);
    for (int64_t k = 0; k < count; ++k, w.next(nx)) {
        x[k] = w.x;
        y[k] = w.y;
    }
    const bool wide = wide_nodes(first + (count > 0 ? count - 1 : 0) * (long long)stride + 1);
    for (int64_t k = 0; divide && k < count; ++k) node_xy(first + k * (long long)stride, nx, wide, x[k], y[k]);
    return TCLBM_OK;
}

tclbm_status tclbm_set_kernel(tclbm_lattice* L, int32_t kind) {
    if (!L) return fail(TCLBM_EINVAL, "lattice is NULL");
    if (kind != KERNEL_TMA && kind != KERNEL_DIRECT && kind != KERNEL_TILE)
        return fail(TCLBM_EINVAL, "kernel kind must be 0, 1 or 2");
    if (kind == KERNEL_TILE && !tile_fits(L->prm, kTileBX, kTileBY))
        return fail(TCLBM_EUNSUPPORTED,
                    "2-D tiles need the correction term, nx %% %d != 1 on a walled x axis and ny %% %d != 1 on a "
                    "walled y axis",
                    kTileBX, kTileBY);
    if (kind != L->kernel) default_shape(L->prm, kind, L->tx, L->ty);
    L->kernel = kind;
    L->auto_kernel = false;
    return TCLBM_OK;
}

const char* tclbm_describe(const tclbm_lattice* L) {
    if (!L) return "";
    tclbm_lattice* M = const_cast<tclbm_lattice*>(L);
    describe_step_kernel(L->prm.storage, step_launch(M, 0), L->dp, M->desc, sizeof M->desc);
    if (resident_planned(M)) {
        const size_t n = strlen(M->desc);
        snprintf(M->desc + n, sizeof M->desc - n, "; %d steps or more: tclbm_resident grid (%d, %d) block (%d)",
                 (int)res_min_steps(L), L->res_plan.gx, L->res_plan.gy, L->res_plan.threads);
    }
    if (tiles_unchained(M)) {
        const size_t n = strlen(M->desc);
        snprintf(M->desc + n, sizeof M->desc - n, "; fewer than %d steps: tclbm_step_tile<%d,%d>", (int)kChainSteps, kTileBX,
                 kTileBY);
    }
    return L->desc;
}

tclbm_status tclbm_init_fields(tclbm_lattice* L, const double* rho, const double* ux, const double* uy,
                               const double* T, int32_t on_device) {
    if (!L || !rho || !ux || !uy || (!T && L->prm.thermal)) return fail(TCLBM_EINVAL, "NULL argument");
    const size_t n = (size_t)L->prm.nx * L->prm.ny;
    const double* d[4] = {rho, ux, uy, T ? T : rho};
    if (!on_device) {
        for (int k = 0; k < 4; ++k) {
            if (k == 3 && !T) break;
            CK(cudaMemcpyAsync(L->stage + k * n, d[k], n * sizeof(double), cudaMemcpyHostToDevice, L->stream));
        }
        d[0] = L->stage;
        d[1] = L->stage + n;
        d[2] = L->stage + 2 * n;
        d[3] = T ? L->stage + 3 * n : L->stage;
    }
    const tclbm_params& p = L->prm;
    const double b = 2.0 / (p.gamma - 1.0);
    tclbm_status st = with_storage(p.storage, [&](auto* tag) -> tclbm_status {
        using ST = std::remove_pointer_t<decltype(tag)>;
        init_kernel<ST><<<grid_for((long long)n, 256), 256, 0, L->stream>>>(
            L->dp, d[0], d[1], d[2], d[3], (ST*)L->buf[0], p.thermal, p.R, p.T0, b, p.force_kind, p.ax, p.ay, p.famp);
        return TCLBM_OK;
    });
    if (st != TCLBM_OK) return st;
    CK(cudaGetLastError());
    // (the draws go on from copy 0 of the step counter: tclbm_count_steps)
    L->cur = 0;
    L->steps = 0;
    if (!on_device) CK(cudaStreamSynchronize(L->stream));  // host arrays may be freed on return
    return TCLBM_OK;
}

tclbm_status tclbm_step(tclbm_lattice* L, int64_t nsteps) {
    if (!L) return fail(TCLBM_EINVAL, "lattice is NULL");
    if (nsteps < 0) return fail(TCLBM_EINVAL, "nsteps must be >= 0");
    int64_t left = nsteps;
    {
        int64_t done = 0;
        const tclbm_status st = resident_steps(L, left, done);
        if (st != TCLBM_OK) return st;
        left -= done;
    }
    // long runs of short launches go through a captured graph of 2*kGraphPairs steps
    const long long nodes = (long long)L->prm.nx * L->prm.ny;
    // (chained TMA launches overlap on the device, which a graph's whole-grid waits do not)
    if (left >= 2 * kGraphPairs && nodes <= (1LL << 22) && !chainable(L)) {
        if (L->cur != 0) {
            tclbm_status st = launch_steps(L, 1);
            if (st != TCLBM_OK) return st;
            --left;
        }
        tclbm_status st = build_graph(L);
        if (st != TCLBM_OK) return st;
        while (left >= 2 * kGraphPairs) {
            CK(cudaGraphLaunch(L->graph, L->stream));
            left -= 2 * kGraphPairs;
            L->steps += 2 * kGraphPairs;
        }
    }
    return launch_steps(L, left);
}

tclbm_status tclbm_moments(tclbm_lattice* L, double* rho, double* ux, double* uy, double* T, int32_t on_device) {
    if (!L) return fail(TCLBM_EINVAL, "lattice is NULL");
    const size_t n = (size_t)L->prm.nx * L->prm.ny;
    double* out[4] = {rho, ux, uy, T};
    double* dst[4];
    for (int k = 0; k < 4; ++k) dst[k] = (on_device && out[k]) ? out[k] : L->stage + k * n;
    HostOutputs host;
    tclbm_status st = on_device ? TCLBM_OK : host.begin(L, out, 4, n * sizeof(double));
    if (st != TCLBM_OK) return st;
    st = with_storage(L->prm.storage, [&](auto* tag) -> tclbm_status {
        using ST = std::remove_pointer_t<decltype(tag)>;
        const ST* src = (const ST*)L->buf[L->cur];
        if (L->prm.thermal)
            moments_kernel<true, ST><<<grid_for((long long)n, 256), 256, 0, L->stream>>>(L->dp, src, dst[0], dst[1],
                                                                                         dst[2], dst[3]);
        else
            moments_kernel<false, ST><<<grid_for((long long)n, 256), 256, 0, L->stream>>>(L->dp, src, dst[0], dst[1],
                                                                                          dst[2], dst[3]);
        return TCLBM_OK;
    });
    if (st != TCLBM_OK) return st;
    CK(cudaGetLastError());
    if (!on_device) {
        host.touch();
        for (int k = 0; k < 4; ++k)
            if (out[k])
                CK(cudaMemcpyAsync(out[k], dst[k], n * sizeof(double), cudaMemcpyDeviceToHost, L->stream));
    }
    return check_kernel_error(L);  // synchronises
}

tclbm_status tclbm_snapshot_velocity(tclbm_lattice* L) {
    if (!L) return fail(TCLBM_EINVAL, "lattice is NULL");
    const size_t n = (size_t)L->prm.nx * L->prm.ny;
    if (!L->usnap) {
        L->usnap_bytes = 2 * n * sizeof(float);
        L->usnap = (float*)dev_alloc(L, L->usnap_bytes);
        if (!L->usnap) return fail(TCLBM_ENOMEM, "velocity snapshot allocation failed");
    }
    return with_storage(L->prm.storage, [&](auto* tag) -> tclbm_status {
        using ST = std::remove_pointer_t<decltype(tag)>;
        const ST* src = (const ST*)L->buf[L->cur];
        if (L->prm.thermal)
            snapshot_kernel<true, ST><<<grid_for((long long)n, 256), 256, 0, L->stream>>>(L->dp, src, L->usnap);
        else
            snapshot_kernel<false, ST><<<grid_for((long long)n, 256), 256, 0, L->stream>>>(L->dp, src, L->usnap);
        CK(cudaGetLastError());
        return TCLBM_OK;
    });
}

tclbm_status tclbm_diagnostics(tclbm_lattice* L, double out[TCLBM_NDIAG]) {
    if (!L || !out) return fail(TCLBM_EINVAL, "NULL argument");
    const long long n = (long long)L->prm.nx * L->prm.ny;
    long long nb = (n + kDiagBlock - 1) / kDiagBlock;
    if (nb > kDiagMaxBlocks) nb = kDiagMaxBlocks;
    double* res = L->diag + kDiagMaxBlocks * TCLBM_NDIAG;
    tclbm_status st = with_storage(L->prm.storage, [&](auto* tag) -> tclbm_status {
        using ST = std::remove_pointer_t<decltype(tag)>;
        const ST* src = (const ST*)L->buf[L->cur];
        if (L->prm.thermal)
            diag_kernel<true, ST><<<(int)nb, kDiagBlock, 0, L->stream>>>(L->dp, src, L->usnap, L->prm.T_ref, L->diag);
        else
            diag_kernel<false, ST><<<(int)nb, kDiagBlock, 0, L->stream>>>(L->dp, src, L->usnap, L->prm.T_ref, L->diag);
        diag_finish<<<1, 32 * TCLBM_NDIAG, 0, L->stream>>>(L->diag, (int)nb, L->err, res);
        return TCLBM_OK;
    });
    if (st != TCLBM_OK) return st;
    CK(cudaGetLastError());
    double got[TCLBM_NDIAG + 1];
    CK(cudaMemcpyAsync(got, res, sizeof got, cudaMemcpyDeviceToHost, L->stream));
    CK(cudaStreamSynchronize(L->stream));
    memcpy(out, got, TCLBM_NDIAG * sizeof(double));
    if (got[TCLBM_NDIAG] != 0.0) return check_kernel_error(L);  // reports and clears it
    for (int k = 0; k < TCLBM_NDIAG; ++k)
        if (!std::isfinite(out[k])) return fail(TCLBM_ENONFINITE, "non-finite diagnostic %d", k);
    return TCLBM_OK;
}

tclbm_status tclbm_get_populations(tclbm_lattice* L, double* f, double* h, int32_t on_device) {
    if (!L || !f) return fail(TCLBM_EINVAL, "NULL argument");
    const size_t n = (size_t)L->prm.nx * L->prm.ny;
    const size_t bytes = 9 * n * sizeof(double);
    double *df = f, *dh = h;
    double* tmp = nullptr;
    HostOutputs host;
    if (!on_device) {
        double* const out[2] = {f, L->prm.thermal ? h : nullptr};
        const tclbm_status hs = host.begin(L, out, 2, bytes);
        if (hs != TCLBM_OK) return hs;
        tmp = (double*)dev_alloc(L, 2 * bytes);
        if (!tmp) return fail(TCLBM_ENOMEM, "staging allocation failed");
        df = tmp;
        dh = tmp + 9 * n;
    }
    tclbm_status st = with_storage(L->prm.storage, [&](auto* tag) -> tclbm_status {
        using ST = std::remove_pointer_t<decltype(tag)>;
        const ST* src = (const ST*)L->buf[L->cur];
        if (L->prm.thermal)
            get_pops_kernel<true, ST><<<grid_for((long long)n, 256), 256, 0, L->stream>>>(L->dp, src, df, dh);
        else
            get_pops_kernel<false, ST><<<grid_for((long long)n, 256), 256, 0, L->stream>>>(L->dp, src, df, nullptr);
        return TCLBM_OK;
    });
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && !on_device) {
        host.touch();
        e = cudaMemcpyAsync(f, df, bytes, cudaMemcpyDeviceToHost, L->stream);
        if (e == cudaSuccess && h && L->prm.thermal) e = cudaMemcpyAsync(h, dh, bytes, cudaMemcpyDeviceToHost, L->stream);
    }
    if (e == cudaSuccess && tmp) e = cudaStreamSynchronize(L->stream);
    if (tmp) dev_free(L, tmp, 2 * bytes);
    if (st != TCLBM_OK) return st;
    if (e != cudaSuccess) return cuda_fail(e, "get_populations");
    return check_kernel_error(L);
}

tclbm_status tclbm_set_populations(tclbm_lattice* L, const double* f, const double* h, int32_t on_device) {
    if (!L || !f || (L->prm.thermal && !h)) return fail(TCLBM_EINVAL, "NULL argument");
    const size_t n = (size_t)L->prm.nx * L->prm.ny;
    const size_t bytes = 9 * n * sizeof(double);
    const double *df = f, *dh = h;
    double* tmp = nullptr;
    cudaError_t e = cudaSuccess;
    if (!on_device) {
        tmp = (double*)dev_alloc(L, 2 * bytes);
        if (!tmp) return fail(TCLBM_ENOMEM, "staging allocation failed");
        e = cudaMemcpyAsync(tmp, f, bytes, cudaMemcpyHostToDevice, L->stream);
        if (e == cudaSuccess && L->prm.thermal) e = cudaMemcpyAsync(tmp + 9 * n, h, bytes, cudaMemcpyHostToDevice, L->stream);
        df = tmp;
        dh = tmp + 9 * n;
    }
    if (e == cudaSuccess) {
        with_storage(L->prm.storage, [&](auto* tag) -> tclbm_status {
            using ST = std::remove_pointer_t<decltype(tag)>;
            set_pops_kernel<ST><<<grid_for((long long)n, 256), 256, 0, L->stream>>>(L->dp, df, dh, (ST*)L->buf[L->cur],
                                                                                    L->prm.thermal);
            return TCLBM_OK;
        });
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(L->stream);
    if (tmp) dev_free(L, tmp, 2 * bytes);
    if (e != cudaSuccess) return cuda_fail(e, "set_populations");
    return TCLBM_OK;
}

// Slab decomposition along y: whole rows of every population plane, in the storage
// format as stored (post-collision values at their own node, ready for the next pull).
tclbm_status tclbm_copy_rows(tclbm_lattice* dst, int32_t dst_row, tclbm_lattice* src, int32_t src_row,
                             int32_t rows) {
    if (!dst || !src) return fail(TCLBM_EINVAL, "lattice is NULL");
    if (dst->prm.nx != src->prm.nx || dst->storage != src->storage || dst->nplanes != src->nplanes)
        return fail(TCLBM_EINVAL, "lattices differ in nx, storage format or thermal flag");
    if (rows < 0 || src_row < 0 || dst_row < 0 || (int64_t)src_row + rows > src->prm.ny ||
        (int64_t)dst_row + rows > dst->prm.ny)
        return fail(TCLBM_EINVAL, "rows [%d, %d) of %d and [%d, %d) of %d are not all inside the lattices", src_row,
                    src_row + rows, src->prm.ny, dst_row, dst_row + rows, dst->prm.ny);
    if (dst == src && dst_row < src_row + rows && src_row < dst_row + rows)
        return fail(TCLBM_EINVAL, "source and destination rows overlap");
    if (rows == 0) return TCLBM_OK;
    const size_t row_bytes = (size_t)dst->dp.pitch * dst->elem;
    const size_t width = (size_t)rows * row_bytes;
    const size_t dplane = (size_t)dst->dp.plane * dst->elem, splane = (size_t)src->dp.plane * src->elem;
    char* d = (char*)dst->buf[dst->cur] + (size_t)dst_row * row_bytes;
    const char* s = (const char*)src->buf[src->cur] + (size_t)src_row * row_bytes;
    const bool cross = dst->stream != src->stream;
    if (cross) {  // the copy follows work queued on the source's stream
        if (!src->copy_event) CK(cudaEventCreateWithFlags(&src->copy_event, cudaEventDisableTiming));
        if (!dst->copy_event) CK(cudaEventCreateWithFlags(&dst->copy_event, cudaEventDisableTiming));
        CK(cudaEventRecord(src->copy_event, src->stream));
        CK(cudaStreamWaitEvent(dst->stream, src->copy_event, 0));
    }
    if (dplane <= (size_t)INT32_MAX && splane <= (size_t)INT32_MAX) {
        CK(cudaMemcpy2DAsync(d, dplane, s, splane, width, (size_t)dst->nplanes, cudaMemcpyDeviceToDevice,
                             dst->stream));
    } else {
        for (int q = 0; q < dst->nplanes; ++q)
            CK(cudaMemcpyAsync(d + q * dplane, s + q * splane, width, cudaMemcpyDeviceToDevice, dst->stream));
    }
    if (cross) {  // and the source's later steps, which overwrite these rows, follow the copy
        CK(cudaEventRecord(dst->copy_event, dst->stream));
        CK(cudaStreamWaitEvent(src->stream, dst->copy_event, 0));
    }
    return TCLBM_OK;
}

}  // extern "C"
