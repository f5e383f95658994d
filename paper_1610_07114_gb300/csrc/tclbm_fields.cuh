// tclbm_fields.cuh -- FP64 arithmetic of the field conversions (initial fields, moments,
// diagnostics, population transfer), arranged for sm_103a's FP64 rate.
//
// The FP64 pipe takes 64 cycles a warp instruction on this part (1/64 of FP32), so these
// kernels were bound by it, not by memory: 1.96 ms for the moments of a 4096 x 2048
// lattice whose bytes take 0.13 ms.  What the pipe does not have to do is moved off it:
//   - conversions between FP32 and FP64 are exact bit moves (or one rounding) in integer
//     instructions;
//   - sums over a node's populations are taken on the stored FP32 deviations by
//     error-free transformations (Knuth's two-sum: s = a + b and its exact error), carried as
//     an unevaluated sum of three floats, and enter FP64 once; the base values' sums are
//     exact;
//   - one reciprocal of rho serves the three divisions, each corrected by its remainder.
// The results are as near the exact ones as those of the plain FP64 expressions (compared
// with quad precision over the flows of the performance cases).
// Measured before / after (us): 4096 x 2048 FP32, moments 1962 / 596, diagnostics 2447 / 838,
// velocity snapshot 1155 / 413, initial fields 3337 / 1983 (their bytes take 129, 89, 99 and
// 129); 2048 x 1024 populations in 258 / 186, out 236 / 113.  An FP64 instruction per node
// costs 23 us at 4096 x 2048; about 26, 36, 18 and 86 are left.
#pragma once

#include "tclbm_device.cuh"

namespace tclbm {

// Column and row of the nodes first, first + stride, ... that one thread of a conversion
// visits: two divisions, and an addition with carry from node to node.  `first` and `stride` are
// numbers of threads (below 2^32); the nodes may go beyond that, where a 32-bit division of the
// node number would give wrong rows (a lattice has up to 2^34 nodes).
struct NodeWalk {
    int x, y, dx, dy;
    __host__ __device__ __forceinline__ NodeWalk(unsigned first, unsigned stride, int nx) {
        const unsigned m = (unsigned)nx, fy = first / m, sy = stride / m;
        y = (int)fy;
        x = (int)(first - fy * m);
        dy = (int)sy;
        dx = (int)(stride - sy * m);
    }
    __host__ __device__ __forceinline__ void next(int nx) {
        const unsigned t = (unsigned)x + (unsigned)dx;  // (below 2 nx < 2^32)
        const bool over = t >= (unsigned)nx;
        x = (int)(over ? t - (unsigned)nx : t);
        y += dy + (over ? 1 : 0);
    }
};

// The same of node i by division, for the initial fields: bound by the FP64 pipe, they lose 2.4 %
// to the counted walk (4096 x 2048 1983 / 2030 us), where storing populations gains from it
// (2048 x 1024 234 / 186).  `wide`: more than 2^32 nodes.
__host__ __device__ __forceinline__ void node_xy(long long i, int nx, bool wide, int& x, int& y) {
    if (wide) {
        const long long r = i / nx;
        y = (int)r;
        x = (int)(i - r * nx);
    } else {
        const unsigned r = (unsigned)i / (unsigned)nx;
        y = (int)r;
        x = (int)((unsigned)i - r * (unsigned)nx);
    }
}
__host__ __device__ __forceinline__ bool wide_nodes(long long n) { return n > (1LL << 32); }

// A lattice's constants with those of the field conversions in FP64: T = inv_bR2 (E - u^2/2)
// with inv_bR2 = 2 / (b R), and T0, as the FP64 initialisation uses them; the rest-state
// populations and sum hbase.
struct FieldParams : DevParams {
    double inv_bR2, T0d;
    double fbase_d[9], hbase_d[9], hrest;
};

// (double)v without the FP64 pipe for zeros and normal numbers.
__device__ __forceinline__ double f2d(float v) {
    const unsigned u = __float_as_uint(v), m = u & 0x7fffffffu;
    if (m - 0x00800000u < 0x7f000000u)  // normal
        return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
    if (m == 0) return __hiloint2double((int)u, 0);
    return (double)v;
}

// (float)v, rounded to nearest even, without the FP64 pipe where the result is zero or normal.
__device__ __forceinline__ float d2f(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v), m = hi & 0x7fffffffu;
    if (m - 0x38100000u < 0x0fd00000u) {  // exponents -126 .. 126
        const unsigned t = ((m - 0x38000000u) << 3) | (lo >> 29), rem = lo << 3;
        const unsigned up = rem > 0x80000000u || (rem == 0x80000000u && (t & 1u)) ? 1u : 0u;
        return __uint_as_float((hi & 0x80000000u) | (t + up));
    }
    if ((m | lo) == 0) return __uint_as_float(hi);
    return __double2float_rn(v);
}

// An unevaluated sum hi + mid + lo.
struct Sum3 {
    float hi, mid, lo;
};
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}
__device__ __forceinline__ void sum_add(Sum3& p, float v) {
    float e;
    two_sum(p.hi, v, p.hi, e);
    two_sum(p.mid, e, p.mid, e);
    p.lo = __fadd_rn(p.lo, e);
}
// base + sum, for sums that are narrow()
__device__ __forceinline__ double sum_value(double base, const Sum3& p) {
    return base + f2d(p.hi) + (f2d(p.mid) + f2d(p.lo));
}
__device__ __forceinline__ double sum_value(const Sum3& p) { return f2d(p.hi) + (f2d(p.mid) + f2d(p.lo)); }
template <int N>
__device__ __forceinline__ Sum3 sum_of(const float (&v)[N]) {
    Sum3 p;
    two_sum(v[0], v[1], p.hi, p.mid);
    p.lo = 0.0f;
#pragma unroll
    for (int q = 2; q < N; ++q) sum_add(p, v[q]);
    return p;
}

// Whether |x| is in 2^-63 .. 2^63, where the reciprocal below starts from FP32.
__device__ __forceinline__ bool rcp_range(double x) {
    return ((unsigned)__double2hiint(x) & 0x7fffffffu) - 0x3c000000u < 0x07f00000u;
}

// 1/x: the FP32 approximation (2^-23) and one third-order iteration of Newton's kind,
// y (1 + e + e^2) with e = 1 - x y, whose own error is e^3; plain division outside rcp_range().
__device__ __forceinline__ double rcp_d(double x) {
    if (!rcp_range(x)) return 1.0 / x;
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d2f(x)));
    const double y = f2d(r), e = __fma_rn(-x, y, 1.0);
    return __fma_rn(y, __fma_rn(e, e, e), y);
}

// a / x, r = rcp_d(x): the quotient corrected by its remainder (P. Markstein's method; within
// one unit in the last place), where x, the quotient and the remainder are ordinary numbers;
// zeros, infinities, NaN and the ends of the exponent range divide plainly.
__device__ __forceinline__ double div_d(double a, double x, double r) {
    const double q = a * r;
    if (rcp_range(x)) {
        if (((unsigned)__double2hiint(q) & 0x7fffffffu) - 0x0ad00000u < 0x6d800000u)  // 2^-850 .. 2^902
            return __fma_rn(__fma_rn(-q, x, a), r, q);
        if ((((unsigned)__double2hiint(a) & 0x7fffffffu) | (unsigned)__double2loint(a)) == 0) return q;
    }
    return a / x;
}

// Sums of a node's deviations: rho - 1, the momentum without the force, sum h_bar less its
// rest value.
struct NodeSums {
    Sum3 drho, jx, jy, sdh;
    // Whether they can be carried in FP32 (and summed over the 2^15 nodes a thread sees of the
    // largest lattice): not where a sum comes near FP32's range, is infinite or undefined.
    __device__ __forceinline__ bool narrow() const {
        return fabsf(drho.hi) + fabsf(jx.hi) + fabsf(jy.hi) + fabsf(sdh.hi) < 7.9e28f;  // 2^96
    }
};
template <bool THERMAL>
__device__ __forceinline__ NodeSums node_sums(const float (&f)[9], const float (&h)[9]) {
    NodeSums s;
    s.drho = sum_of(f);
    s.jx = sum_of({f[1], -f[3], f[5], -f[6], f[8], -f[7]});
    s.jy = sum_of({f[2], -f[4], f[5], -f[7], f[6], -f[8]});
    if (THERMAL)
        s.sdh = sum_of(h);
    else
        s.sdh = Sum3{0.0f, 0.0f, 0.0f};
    return s;
}

// The sums themselves: rho, the momentum without the force, sum h_bar; in plain FP64 arithmetic
// where the FP32 parts do not hold them.
struct NodeTotals {
    double rho, jx, jy, sh;
};
template <bool THERMAL>
__device__ __forceinline__ NodeTotals node_totals(const FieldParams& p, const NodeSums& s, const float (&f)[9],
                                                  const float (&h)[9]) {
    if (s.narrow())
        return NodeTotals{sum_value(1.0, s.drho), sum_value(s.jx), sum_value(s.jy),
                          THERMAL ? sum_value(p.hrest, s.sdh) : 0.0};
    const int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, ey[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
    NodeTotals t = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const double fq = p.fbase_d[q] + (double)f[q];
        t.rho += fq;
        if (ex[q] != 0) t.jx += fq * ex[q];
        if (ey[q] != 0) t.jy += fq * ey[q];
        if (THERMAL) t.sh += p.hbase_d[q] + (double)h[q];
    }
    return t;
}

// rho and u of Eq. 20 from the sums (Fx, Fy: the Taylor-Green force, else unused).
struct NodeFields {
    double rho, irho, ux, uy;
};
__device__ __forceinline__ NodeFields node_velocity(const DevParams& p, const NodeTotals& s, int x, int y) {
    NodeFields n;
    n.rho = s.rho;
    n.irho = rcp_d(n.rho);
    double jx = s.jx, jy = s.jy;
    if (p.force_kind == FORCE_TAYLOR_GREEN) {
        const double a = 0.5 * f2d(p.famp);
        jx = __fma_rn(a * f2d(p.sx[x]), f2d(p.sy[y]), jx);
        jy = __fma_rn(a * f2d(p.cx[x]), f2d(p.cy[y]), jy);
    } else if (p.force_kind == FORCE_ACCEL) {
        jx = __fma_rn(0.5 * f2d(p.ax), n.rho, jx);
        jy = __fma_rn(0.5 * f2d(p.ay), n.rho, jy);
    }
    n.ux = div_d(jx, n.rho, n.irho);
    n.uy = div_d(jy, n.rho, n.irho);
    return n;
}

// Temperature of Section IV; hrest: the rest value of sum h_bar, uu = |u|^2.
template <bool THERMAL>
__device__ __forceinline__ double node_temperature(const FieldParams& p, const NodeFields& n, double sh, double uu, int x,
                                                   int y) {
    if (!THERMAL) return p.T0d;
    if (p.work) {  // rho E = sum h_bar + F.u / 2
        double Fx = 0.0, Fy = 0.0;
        if (p.force_kind == FORCE_TAYLOR_GREEN) {
            Fx = f2d(p.famp) * f2d(p.sx[x]) * f2d(p.sy[y]);
            Fy = f2d(p.famp) * f2d(p.cx[x]) * f2d(p.cy[y]);
        } else if (p.force_kind == FORCE_ACCEL) {
            Fx = n.rho * f2d(p.ax);
            Fy = n.rho * f2d(p.ay);
        }
        sh = __fma_rn(0.5, __fma_rn(Fx, n.ux, Fy * n.uy), sh);
    }
    return p.inv_bR2 * __fma_rn(-0.5, uu, div_d(sh, n.rho, n.irho));
}

// A running sum of narrow() FP32 values in three parts (error-free to far below FP64's rounding).
struct Running {
    float a = 0.0f, b = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float v) {
        float e;
        two_sum(a, v, a, e);
        two_sum(b, e, b, e);
        c = __fadd_rn(c, e);
    }
    __device__ __forceinline__ void add(const Sum3& p) {
        add(p.hi);
        add(p.mid);  // (lo is below 2^-48 of this node's sum)
    }
    __device__ __forceinline__ double value() const { return (f2d(c) + f2d(b)) + f2d(a); }
};

}  // namespace tclbm
