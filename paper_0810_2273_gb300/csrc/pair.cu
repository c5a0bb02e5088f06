// Pair kernels of the vdW-DF double sum (paper section 2, eq. (2)) and of its
// adjoint, with periodic images under a spherical cutoff (section 3).
//
// For active points i, j and image vectors L (periodic axes),
//   r = |r_i - r_j + L|,  D = r (q_i + q_j)/2,  delta = |q_i - q_j|/(q_i + q_j),
//   phi = bicubic B-spline of the node table at (D, delta)         if D <= Dmax,
//   phi = g phi17,  phi17 = -C / (d1^2 d2^2 (d1^2 + d2^2))            otherwise,
// d1 = q_i r, d2 = q_j r (section 2: the kernel "can be redefined to depend on two
// quantities D and delta"; Dion eq. 17 for large D).  The factor
//   g = rho(delta*) + (1 - rho(0)) (1 - (Dmax/D)^2),  delta* = max(0, 1 - min(d1, d2)/Dmax),
// with rho the cubic spline of phi(Dmax, delta) / phi17(Dmax, delta), carries the
// table's departure from eq. 17 at Dmax to larger D along the smaller argument
// (on which that departure depends once the larger one is big), so phi is
// continuous at Dmax and tends to eq. 17 as both arguments grow.
// Energy mode sums each unordered pair once with weight 2 (phi is symmetric in
// i, j); potential mode gives, per point,
//   A_i = sum_{j,L} n_j phi,   U_i = n_i sum_{j,L} n_j r dphi/dd1,
//   r dphi/dd1 = r/2 phi_D + (1 - ds)/(q_i + q_j) phi_ds,  ds = (q_i - q_j)/(q_i + q_j),
// and beyond the table g r dphi17/dd1 + phi17 r dg/dd1 with
// r dphi17/dd1 = -2 phi17 (1/q_i + q_i/(q_i^2 + q_j^2)) and
// r dg/dd1 = (1 - rho(0)) (Dmax/D)^2 r/D - [d1 < d2] rho'(delta*) r/Dmax.
//
// Work decomposition: persistent CTAs keep a band of B-spline rows resident in
// shared memory (FP32 path, staged once; which rows is chosen on the device from
// a sampled histogram of the call's D cells); the rest comes from the table's
// texture copy.  Each warp then works on its own:
// it pulls work items (instance, tile of kTile i points, range of j tiles) from
// one queue in global memory, culls every (j tile, image) against its i tile
// by bounding boxes and then every (j point, image) against the i box, stages
// surviving j tiles in a private shared-memory buffer (warp-synchronous, no
// block barrier), and runs the pair loop with each lane owning one i (two in
// FP32), the j points read as broadcasts and the images of a pair innermost.
// FP32 partial sums over one j tile are folded into FP64 accumulators.  The work
// loop is bounded (max_iters); nothing waits on another warp or CTA.
#include <cuda_runtime.h>

#include <type_traits>

#include "common.cuh"

namespace vdwdf {

namespace {

// floor of a non-negative float below 2^22 without a conversion instruction:
// adding 1.5 * 2^23 rounded toward minus infinity leaves floor(x) in the low
// mantissa bits.
__device__ __forceinline__ int floor_split(float x, float &frac) {
    const float b = __fadd_rd(x, 12582912.0f);
    frac = x - (b - 12582912.0f);
    return __float_as_int(b) - 0x4B400000;
}
__device__ __forceinline__ int floor_split(double x, double &frac) {
    const double f = floor(x);
    frac = x - f;
    return static_cast<int>(f);
}

// Cubic B-spline weights times 6 and their t-derivatives times 6.
template <typename R>
__device__ __forceinline__ void bw(R t, R w[4]) {
    const R t2 = t * t, t3 = t2 * t, s = R(1) - t;
    w[0] = s * s * s;
    w[1] = R(3) * t3 - R(6) * t2 + R(4);
    w[2] = R(-3) * t3 + R(3) * t2 + R(3) * t + R(1);
    w[3] = t3;
}
template <typename R>
__device__ __forceinline__ void bdw(R t, R d[4]) {
    const R t2 = t * t, s = R(1) - t;
    d[0] = R(-3) * s * s;
    d[1] = R(9) * t2 - R(12) * t;
    d[2] = R(-9) * t2 + R(6) * t + R(3);
    d[3] = R(3) * t2;
}

__device__ __forceinline__ float recip(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }
__device__ __forceinline__ float rlen(float r2) { return r2 * rsqrtf(fmaxf(r2, 1e-30f)); }
__device__ __forceinline__ double rlen(double r2) { return sqrt(r2); }

// One-instruction reciprocal and reciprocal root of normal values (the same bits as
// the functions that also take denormals, without their scaling steps).
__device__ __forceinline__ float rcp_ftz(float x) {
    float v;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(v) : "f"(x));
    return v;
}
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float v;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(v) : "f"(x));
    return v;
}

__device__ __forceinline__ float lds32(uint32_t a) {
    float v;
    asm("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}

// Two FP32 values side by side, one operation each.  Not the packed FP32x2
// instructions: a packed multiply-add holds the scheduler's dispatch for 2.3 clocks,
// two single ones for 2.2 (16 warps on an SM, independent chains; beside an integer
// operation 3.8 against 3.3), and single ones take immediate operands where packed
// ones need a register pair filled with each constant.  Both ways E + v of the
// 36 x 63 x 90 monolayer takes 102.7 ms; single operations are 4 % faster on the open
// molecule and 3 % on the slab.
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    return make_float2(__fmaf_rn(a.x, b.x, c.x), __fmaf_rn(a.y, b.y, c.y));
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    return make_float2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y));
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    return make_float2(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y));
}

// floor_split of two values at once (both non-negative and below 2^22): the floors as
// floats, and as the low mantissa bits of the shifted values.
__device__ __forceinline__ float2 floor2(float2 x, unsigned &b0, unsigned &b1) {
    const float s0 = __fadd_rd(x.x, 12582912.0f), s1 = __fadd_rd(x.y, 12582912.0f);
    b0 = __float_as_uint(s0);
    b1 = __float_as_uint(s1);
    return make_float2(s0 - 12582912.0f, s1 - 12582912.0f);
}

// bw and bdw (without dw[0], which the differences leave out) of two offsets at once.
__device__ __forceinline__ void bw2(float2 t, float2 w[4]) {
    const float2 s = sub2(f2(1.0f), t), t2 = mul2(t, t), s2 = mul2(s, s);
    w[0] = mul2(s2, s);
    w[1] = fma2(t2, fma2(t, f2(3.0f), f2(-6.0f)), f2(4.0f));
    w[2] = fma2(s2, fma2(s, f2(3.0f), f2(-6.0f)), f2(4.0f));
    w[3] = mul2(t2, t);
}
__device__ __forceinline__ void bdw2(float2 t, float2 d[4]) {
    const float2 s = sub2(f2(1.0f), t);
    d[1] = mul2(t, fma2(t, f2(9.0f), f2(-12.0f)));
    d[2] = mul2(s, fma2(s, f2(-9.0f), f2(12.0f)));
    d[3] = mul2(mul2(t, t), f2(3.0f));
}
// The last three weights and derivative weights (not times 6), for sums over the
// differences from the first coefficient.
__device__ __forceinline__ void bw_diff2(float2 t, float2 w[4], float2 d[4]) {
    const float2 t2 = mul2(t, t), h = f2(0.5f);
    w[1] = fma2(t2, fma2(h, t, f2(-1.0f)), f2(2.0f / 3.0f));
    w[2] = fma2(t, fma2(t, fma2(t, f2(-0.5f), h), h), f2(1.0f / 6.0f));
    w[3] = mul2(mul2(t, f2(1.0f / 6.0f)), t2);
    d[1] = mul2(t, fma2(t, f2(1.5f), f2(-2.0f)));
    d[2] = fma2(t, fma2(t, f2(-1.5f), f2(1.0f)), h);
    d[3] = mul2(t2, h);
}

// The delta-derivative weights sum to zero, so sum_n dwd[n] c[n] is taken as
// sum_{n>=1} dwd[n] (c[n] - c[0]): neighbouring coefficients differ little and
// their differences are exact, which keeps the small derivative of an O(phi)
// row free of the cancellation that would otherwise scale its error by the
// number of delta cells.
template <bool POT, typename R>
__device__ __forceinline__ void combine(const R c[4][4], const R wD[4], const R dwD[4],
                                        const R wd[4], const R dwd[4], R &phi, R &pt, R &pu) {
    R p = 0, a = 0, b = 0;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const R row = wd[0] * c[m][0] + wd[1] * c[m][1] + wd[2] * c[m][2] + wd[3] * c[m][3];
        p += wD[m] * row;
        if (POT) {
            const R drow = dwd[1] * (c[m][1] - c[m][0]) + dwd[2] * (c[m][2] - c[m][0]) +
                           dwd[3] * (c[m][3] - c[m][0]);
            // along D the same in FP32, from the differences to the first row
            a += dwD[m] * (sizeof(R) == 8 ? row
                                          : wd[0] * (c[m][0] - c[0][0]) + wd[1] * (c[m][1] - c[0][1]) +
                                                wd[2] * (c[m][2] - c[0][2]) + wd[3] * (c[m][3] - c[0][3]));
            b += wD[m] * drow;
        }
    }
    phi = p;
    pt = a;
    pu = b;
}

template <typename R>
using Consts = LoopConsts<R>;

template <typename R>
struct Table {
    const R *g;      // bicubic coefficients / 36 in global memory, row stride S
    const R *rho;    // rho(delta) coefficients / 6 (after the bicubic block)
    uint32_t s;      // shared-memory address of the resident band (FP32), row stride SB
    int k0, kn;      // band rows [k0, k0 + kn)
    int S, SB;
};

template <bool POT, typename R>
__device__ __forceinline__ void interp(const Table<R> &tb, int k, int l, const R wD[4],
                                       const R dwD[4], const R wd[4], const R dwd[4], R &p, R &pt,
                                       R &pu) {
    R c[4][4];
    const R *g = tb.g + static_cast<size_t>(k) * tb.S + l;
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
        for (int n = 0; n < 4; ++n) c[m][n] = __ldg(g + m * tb.S + n);
    combine<POT, R>(c, wD, dwD, wd, dwd, p, pt, pu);
}

// The delta-dependent part of a pair, shared by all its periodic images: the
// delta cell and weights, the scale from r to the table's D coordinate, and the
// factors that turn the delta-derivative into r dphi/dd1 and r dphi/dd2.
// With ds = (q_i - q_j)/(q_i + q_j): dds/dd1 = (1 - ds)/(2D), dds/dd2 = -(1 + ds)/(2D),
// so b1 = cd sign(ds) (1 - ds)/(q_i + q_j) and b2 = -cd sign(ds) (1 + ds)/(q_i + q_j).
template <typename R>
struct Delta {
    R sqcD, b1, b2;  // (q_i + q_j) cD; the delta-derivative factors
    R wd[4], dwd[4];
    int l;
    bool cl;  // delta beyond the last node (weights continued linearly)
};

template <bool POT, typename R>
__device__ __forceinline__ void delta_part(R qi, R qj, const Consts<R> &K, Delta<R> &d) {
    const R sq = qi + qj;
    const R dq = qi - qj;
    const R isq = recip(sq);
    // beyond the last node the spline continues linearly with its end slope (it has
    // zero curvature there): the weights become w(u) + e w'(u), e the distance past
    // the node in cells.  No index leaves the table.
    const R dl = fabs(dq) * isq;
    const R td0 = dl * K.cd;
    d.cl = td0 > K.tdmax;
    const R td = fmin(fmax(td0, R(0)), K.tdclamp);
    R u;
    int l = floor_split(td, u);
    if (sizeof(R) == 8 && l > K.lmax) {  // FP64 keeps the exact end node: last cell at u = 1
        l = K.lmax;
        u = td - R(l);
    }
    d.l = l;
    bw<R>(u, d.wd);
    if (POT || d.cl) bdw<R>(u, d.dwd);
    if (d.cl) {
        const R e = td0 - td;
#pragma unroll
        for (int n = 0; n < 4; ++n) d.wd[n] += e * d.dwd[n];
    }
    const R bq = isq * K.cd;
    d.sqcD = sq * K.cD;
    d.b1 = bq * (dq > R(0) ? (R(1) - dl) : -(R(1) + dl));   // sign(ds) (1 - ds)
    d.b2 = -bq * (dq > R(0) ? (R(1) + dl) : -(R(1) - dl));  // sign(ds) (1 + ds)
}

// The delta parts of two pairs (i0, j) and (i1, j) in the two halves of packed
// FP32 values: the quantities of delta_part, two pairs per instruction.
struct Delta2 {
    float2 sqcD;          // (q_i + q_j) cD
    float2 b1, sb;        // r dphi/dd1 = a + b1 pu, r dphi/dd2 = a + (b1 - 2 sb) pu
    float2 wd[4], dwd[4]; // E + v: bw_diff2's (no [0]), else bw2's
    float2 fl;            // the delta cells' third columns, l + 2, as texture coordinates
    uint32_t l0, l1;
};

template <bool POT>
__device__ __forceinline__ void delta_part2(float2 qi, float qj, const Consts<float> &K, Delta2 &d, bool &cl0,
                                            bool &cl1) {
    const float2 sq = add2(qi, f2(qj)), ndq = sub2(f2(qj), qi);
    const float2 isq = make_float2(rcp_ftz(sq.x), rcp_ftz(sq.y));
    const float2 nds = mul2(ndq, isq);  // -ds = (q_j - q_i)/(q_i + q_j)
    const float2 td0 = mul2(nds, f2(K.cd));
    cl0 = fabsf(td0.x) > K.tdmax;
    cl1 = fabsf(td0.y) > K.tdmax;
    const float2 td = make_float2(fminf(fabsf(td0.x), K.tdclamp), fminf(fabsf(td0.y), K.tdclamp));
    unsigned b0, b1;
    const float2 f = floor2(td, b0, b1), u = sub2(td, f);
    d.l0 = b0 - 0x4B400000u;
    d.l1 = b1 - 0x4B400000u;
    d.fl = make_float2(f.x + 3.0f, f.y + 3.0f);
    if (POT)
        bw_diff2(u, d.wd, d.dwd);
    else
        bw2(u, d.wd);
    if (cl0 || cl1) {
        // past the last node the weights continue linearly: + e w'(u), and the derivative
        // weights sum to zero
        float2 dw[4];
        if (POT)
            dw[1] = d.dwd[1], dw[2] = d.dwd[2], dw[3] = d.dwd[3];
        else
            bdw2(u, dw);
        const float2 e = make_float2(cl0 ? fabsf(td0.x) - td.x : 0.0f, cl1 ? fabsf(td0.y) - td.y : 0.0f);
        if (!POT) d.wd[0] = sub2(d.wd[0], mul2(e, add2(dw[1], add2(dw[2], dw[3]))));
#pragma unroll
        for (int n = 1; n < 4; ++n) d.wd[n] = fma2(e, dw[n], d.wd[n]);
    }
    d.sqcD = mul2(sq, f2(K.cD));
    // sign(ds) cd/(q_i + q_j), and times (1 - ds)
    const float2 bq = mul2(isq, f2(K.cd));
    d.sb = make_float2(copysignf(bq.x, -ndq.x), copysignf(bq.y, -ndq.y));
    d.b1 = fma2(d.sb, nds, d.sb);
}

// phi and (POT) r dphi/dd1, r dphi/dd2 past the table (D > Dmax, tD = r (q_i + q_j) cD):
// g(delta*) times eq. (17).
template <bool POT, typename R>
__device__ __forceinline__ void past_part(R r, R r2, R tD, R qi, R qj, R inv_qi, R qi2, const Consts<R> &K,
                                          const R *rho_c, R &phi, R &rd, R &rd2) {
    const R r4 = r2 * r2;
    const R qj2 = qj * qj;
    const R s2 = qi2 + qj2;
    const R p17 = -K.C * recip(r4 * r2 * qi2 * qj2 * s2);
    // rho at delta* = 1 - min(d1, d2)/Dmax, in delta cells; at or below 0 the
    // spline's value at delta = 0 with zero slope (its end condition), past the
    // last node its linear continuation.  No index leaves the rho block.
    const bool i_small = qi < qj;
    const R ts0 = (R(1) - r * fmin(qi, qj) * K.iDmax) * K.cd;
    const bool up = ts0 > R(0);
    const bool past = ts0 > K.tdmax;
    const R ts = fmin(fmax(ts0, R(0)), K.tdclamp);
    R u;
    int l = floor_split(ts, u);
    if (sizeof(R) == 8 && l > K.lmax) {
        l = K.lmax;
        u = ts - R(l);
    }
    R w[4], dw[4];
    bw<R>(u, w);
    const R *rc = rho_c + l;
    const R c0 = __ldg(rc), c1 = __ldg(rc + 1), c2 = __ldg(rc + 2), c3 = __ldg(rc + 3);
    R rho = w[0] * c0 + w[1] * c1 + w[2] * c2 + w[3] * c3;
    R drho = R(0);  // d rho / d delta*, in cells
    if (POT || past) {
        bdw<R>(u, dw);
        drho = up ? dw[1] * (c1 - c0) + dw[2] * (c2 - c0) + dw[3] * (c3 - c0) : R(0);
        if (past) rho += (ts0 - ts) * drho;
    }
    const R Dr = K.tDmax * recip(tD);  // Dmax / D
    const R Dr2 = Dr * Dr;
    const R g = rho + K.om_rho0 * (R(1) - Dr2);
    phi = g * p17;
    if (POT) {
        const R is2 = recip(s2);
        // (1 - rho(0)) (Dmax/D)^2 r/D with r/D = 2 cD r / tD, and rho'(delta*) r/Dmax
        const R ramp = K.om_rho0 * Dr2 * R(2) * K.cD * r * recip(tD);
        const R sl = drho * K.cd * r * K.iDmax;
        rd = g * (R(-2) * p17 * (inv_qi + qi * is2)) + p17 * (i_small ? ramp - sl : ramp);
        rd2 = g * (R(-2) * p17 * (recip(qj) + qj * is2)) + p17 * (i_small ? ramp : ramp - sl);
    }
}

// The distance-dependent part: phi and (POT) r dphi/dd1, r dphi/dd2 at r^2.
template <bool POT, typename R>
__device__ __forceinline__ void dist_part(R r, R r2, R qi, R qj, R inv_qi, R qi2, const Delta<R> &d,
                                          const Consts<R> &K, const Table<R> &tb, R &phi, R &rd,
                                          R &rd2) {
    R tD = r * d.sqcD;
    // the table is read only for 0 <= tD <= nD - 1 (false for NaN as well)
    if (tD >= R(0) && tD <= K.tDmax) {
        tD = fmin(tD, K.tDclamp);
        R t;
        int k = floor_split(tD, t);
        if (sizeof(R) == 8 && k > K.kmax) {
            k = K.kmax;
            t = tD - R(k);
        }
        R wD[4], dwD[4];
        bw<R>(t, wD);
        if (POT) bdw<R>(t, dwD);
        R pt = 0, pu = 0;
        interp<POT, R>(tb, k, d.l, wD, dwD, d.wd, d.dwd, phi, pt, pu);
        if (POT) {
            const R a = r * K.cD * pt;
            rd = a + pu * d.b1;
            rd2 = a + pu * d.b2;
        }
    } else {
        past_part<POT, R>(r, r2, tD, qi, qj, inv_qi, qi2, K, tb.rho, phi, rd, rd2);
    }
}

// One pair: phi and (POT) r dphi/dd1, r dphi/dd2; counts a delta past the last node.
template <bool POT, typename R>
__device__ __forceinline__ void pair_phi(R r2, R qi, R qj, R inv_qi, R qi2, const Consts<R> &K,
                                         const Table<R> &tb, R &phi, R &rd, R &rd2, unsigned &ncl) {
    Delta<R> d;
    delta_part<POT, R>(qi, qj, K, d);
    ncl += d.cl ? 1u : 0u;
    dist_part<POT, R>(rlen(r2), r2, qi, qj, inv_qi, qi2, d, K, tb, phi, rd, rd2);
}

template <typename R>
__device__ __forceinline__ void make_consts(const PairShared &sh, Consts<R> &K) {
    if constexpr (sizeof(R) == 4)
        K = sh.k32;
    else
        K = sh.k64;
}

template <typename R>
__device__ void make_table(const PairShared &sh, Table<R> &tb) {
    tb.S = sh.S;
    tb.SB = band_stride(sh.S);
    tb.g = sizeof(R) == 4 ? reinterpret_cast<const R *>(sh.tab32) : reinterpret_cast<const R *>(sh.tab64);
    tb.rho = tb.g + static_cast<size_t>(sh.nD + 2) * sh.S;
    tb.s = 0;
    tb.k0 = 0;
    tb.kn = 0;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// r of an index displacement in FP64, -1 outside the cutoff.
template <bool SKEW>
__device__ __forceinline__ double index_r(const PairParams &p, int dx, int dy, int dz) {
    const double X = dx, Y = dy, Z = dz;
    double e = p.h2[0] * (X * X) + p.h2[1] * (Y * Y) + p.h2[2] * (Z * Z);
    if (SKEW) e += p.g2x[0] * (X * Y) + p.g2x[1] * (X * Z) + p.g2x[2] * (Y * Z);
    return p.use_cut && e > p.rc2 ? -1.0 : sqrt(e);
}

// Spherical cutoff, inclusive: a pair is inside iff r^2 <= rc2 (the host folds a
// 1e-12 relative allowance into rc2 so that distances equal to the cutoff up to
// rounding count as inside in every path).  FP32 decides pairs clearly away from
// the boundary and re-checks the rest in FP64 from the exact index offsets.
struct Cut {
    const PairParams *pp;  // FP64 metric and cutoff (kernel parameters), read only
                           // by the recheck near the boundary
};
template <bool SKEW>
__device__ __forceinline__ bool beyond(float r2, float dx, float dy, float dz, const Cut &c) {
    const PairParams &p = *c.pp;
    if (r2 > p.cut_hi) return true;
    if (r2 <= p.cut_lo) return false;
    const double X = dx, Y = dy, Z = dz;
    double e = p.h2[0] * (X * X) + p.h2[1] * (Y * Y) + p.h2[2] * (Z * Z);
    if (SKEW) e += p.g2x[0] * (X * Y) + p.g2x[1] * (X * Z) + p.g2x[2] * (Y * Z);
    return e > p.rc2;
}
// Squared distance between the i box shifted by image m and the j box.
__device__ __forceinline__ float box_gap2(const float ilo[3], const float ihi[3], const float jl[3],
                                          const float jh[3], const int m[3], const int dims[3],
                                          const float h2[3]) {
    float d2 = 0.0f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float s = static_cast<float>(m[a] * dims[a]);
        const float g = fmaxf(0.0f, fmaxf(ilo[a] - jh[a] + s, jl[a] - ihi[a] - s));
        d2 += h2[a] * g * g;
    }
    return d2;
}

// Skewed cells: squared distance between the Cartesian box of the i tile shifted
// by image m (L = sum_a m_a N_a v_a) and the Cartesian box of the j tile.
__device__ __forceinline__ float box_gap2_cart(const float4 &il, const float4 &ih, const float4 &jl,
                                               const float4 &jh, const int m[3], const int dims[3],
                                               const CellRows &vr) {
    const float s0 = static_cast<float>(m[0] * dims[0]), s1 = static_cast<float>(m[1] * dims[1]),
                s2 = static_cast<float>(m[2] * dims[2]);
    const float L0 = s0 * vr.v[0] + s1 * vr.v[3] + s2 * vr.v[6];
    const float L1 = s0 * vr.v[1] + s1 * vr.v[4] + s2 * vr.v[7];
    const float L2 = s0 * vr.v[2] + s1 * vr.v[5] + s2 * vr.v[8];
    const float g0 = fmaxf(0.0f, fmaxf(il.x + L0 - jh.x, jl.x - ih.x - L0));
    const float g1 = fmaxf(0.0f, fmaxf(il.y + L1 - jh.y, jl.y - ih.y - L1));
    const float g2 = fmaxf(0.0f, fmaxf(il.z + L2 - jh.z, jl.z - ih.z - L2));
    return g0 * g0 + g1 * g1 + g2 * g2;
}

// The counters of a finished work item, summed over the warp and added by lane 0
// to the instance's totals (integer atomics: the totals do not depend on order).
__device__ __forceinline__ void count_item(Stats *s, unsigned long long cnt, unsigned nclamp,
                                           unsigned long long evals, unsigned long long cnt_warp = 0ull) {
    const unsigned long long pairs = warp_sum(cnt) + cnt_warp;
    const unsigned clamped = warp_sum(nclamp);
    if ((threadIdx.x & 31) == 0) {
        if (pairs) atomicAdd(&s->pairs, pairs);
        if (evals) atomicAdd(&s->evals, evals);
        if (clamped) atomicAdd(&s->clamped, static_cast<unsigned long long>(clamped));
    }
}

// One FP32 evaluation: the two i points of a lane (halves) against one image of a
// j point.  Table cells come from two memories at once: twelve of the sixteen
// coefficients from the resident band by shared loads, the 2 x 2 block of the
// third and fourth rows' third and fourth columns by a texture gather, whose
// pipe otherwise idles.  Random stencils cost 3.1 SM clocks per shared load (bank
// conflicts) and 22 per gather, side by side: 49.7 clocks for sixteen loads, 42.0
// for twelve and one gather (448 threads on an SM, measured on random cells).
// Energy mode has less arithmetic to hide the loads behind: there the shared pipe is
// 89 % busy, and one of the two halves takes a second block from the texture, the same
// rows' first and second columns, which levels the two pipes (20 loads and 3 gathers
// for both halves).  Energies: Kr dimer 24 x 18 x 18 0.193 -> 0.183 ms, 36 x 63 x 90
// monolayer 78.0 -> 75.6 ms, 36 x 36 x 90 hexagonal cell 49.1 -> 47.2 ms.  With the
// potential nothing is won: issue bounds it.
__device__ __forceinline__ float4 tex_block(unsigned long long tex, float x, float y) {
    return tex2Dgather<float4>(static_cast<cudaTextureObject_t>(tex), x, y, 0);
}

// One row of the stencil: row = sum_n wd[n] c[n], with POT (weights that sum to one,
// 1/6 of the others) from the differences c[n] - c[0], which the delta derivative needs
// for its accuracy in any case (see combine).
template <bool POT>
__device__ __forceinline__ void row2(const float2 c[4], const float2 wd[4], const float2 dwd[4], float2 &row,
                                     float2 &drow) {
    if (POT) {
        const float2 d1 = sub2(c[1], c[0]), d2 = sub2(c[2], c[0]), d3 = sub2(c[3], c[0]);
        row = fma2(wd[3], d3, fma2(wd[2], d2, fma2(wd[1], d1, c[0])));
        drow = fma2(dwd[3], d3, fma2(dwd[2], d2, mul2(dwd[1], d1)));
    } else {
        row = fma2(wd[3], c[3], fma2(wd[2], c[2], fma2(wd[1], c[1], mul2(wd[0], c[0]))));
    }
}

// Six times the cubic B-spline of the rows r at offset t of their middle cell, and
// (POT) a third of six times its t-derivative and six times the spline of dr.  With
// three results the weights pay (25 operations a half against 28 from powers of t and
// the differences of neighbours), with one the differences do (14 against 16).
// E + v with these weights and with row2's differences, against neither: 36 x 63 x 90
// monolayer 102.2 -> 100.2 ms.
template <bool POT>
__device__ __forceinline__ void rows2(const float2 r[4], const float2 dr[4], float2 t, float2 &p, float2 &pt,
                                      float2 &pu) {
    if (POT) {
        const float2 s = sub2(f2(1.0f), t), t2 = mul2(t, t), s2 = mul2(s, s), w0 = mul2(s2, s), w3 = mul2(t2, t);
        const float2 w1 = fma2(t2, fma2(t, f2(3.0f), f2(-6.0f)), f2(4.0f)),
                     w2 = fma2(s2, fma2(s, f2(3.0f), f2(-6.0f)), f2(4.0f));
        p = fma2(w3, r[3], fma2(w2, r[2], fma2(w1, r[1], mul2(w0, r[0]))));
        pu = fma2(w3, dr[3], fma2(w2, dr[2], fma2(w1, dr[1], mul2(w0, dr[0]))));
        const float2 c1 = fma2(add2(t, t), s, f2(1.0f));
        pt = fma2(t2, sub2(r[3], r[2]), fma2(c1, sub2(r[2], r[1]), mul2(s2, sub2(r[1], r[0]))));
    } else {
        // 6 r1 + v + 3 t y + 3 t^2 v + t^3 x
        const float2 u0 = sub2(r[1], r[0]), u1 = sub2(r[2], r[1]), u2 = sub2(r[3], r[2]);
        const float2 v = sub2(u1, u0), x = sub2(sub2(u2, u1), v), y = add2(u0, u1), z = fma2(t, v, y);
        p = fma2(f2(3.0f), fma2(t, z, add2(r[1], r[1])), fma2(mul2(mul2(t, t), t), x, v));
    }
}

// Both halves in the resident band: t the offsets in their D cells (fk: the cells'
// first rows), a0 and a1 the shared addresses of their first coefficients.
template <bool POT>
__device__ __forceinline__ void band_pair2(unsigned long long tex, uint32_t rs, float2 t, float2 fk, uint32_t a0,
                                           uint32_t a1, float2 fl, const float2 wd[4], const float2 dwd[4],
                                           float2 &p, float2 &pt, float2 &pu) {
    const float4 g0 = tex_block(tex, fl.x, fk.x + 3.0f), g1 = tex_block(tex, fl.y, fk.y + 3.0f);
    float4 h0;  // (energy mode) the first half's first and second columns
    if (!POT) h0 = tex_block(tex, fl.x - 2.0f, fk.x + 3.0f);
    float2 r[4], dr[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        float2 c[4];
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            if (!POT && m >= 2 && n < 2)
                c[n] = make_float2(m == 2 ? (n == 0 ? h0.w : h0.z) : (n == 0 ? h0.x : h0.y),
                                   lds32(a1 + m * rs + 4u * n));
            else if (m < 2 || n < 2)
                c[n] = make_float2(lds32(a0 + m * rs + 4u * n), lds32(a1 + m * rs + 4u * n));
            else if (m == 2)
                c[n] = n == 2 ? make_float2(g0.w, g1.w) : make_float2(g0.z, g1.z);
            else
                c[n] = n == 2 ? make_float2(g0.x, g1.x) : make_float2(g0.y, g1.y);
        }
        row2<POT>(c, wd, dwd, r[m], dr[m]);
    }
    rows2<POT>(r, dr, t, p, pt, pu);
}

// Rows k, k + 1 (y0 = k + 1) of one half's stencil: from the band where the half is in
// it (a0 its shared address), else from the texture.
__device__ __forceinline__ void row_pair(bool inb, uint32_t a0, uint32_t rs, unsigned long long tex, float x, float y,
                                         float lo[4], float hi[4]) {
    if (inb) {
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            lo[n] = lds32(a0 + 4u * n);
            hi[n] = lds32(a0 + rs + 4u * n);
        }
    } else {
        const float4 l = tex_block(tex, x - 2.0f, y), r = tex_block(tex, x, y);
        lo[0] = l.w, lo[1] = l.z, lo[2] = r.w, lo[3] = r.z;
        hi[0] = l.x, hi[1] = l.y, hi[2] = r.x, hi[3] = r.y;
    }
}

// The same two evaluations where some lane is off the resident band: each half reads
// the band or, off it, the texture (four gathers for a whole stencil: 89 SM clocks
// against 310 for sixteen global loads, measured on random cells).
template <bool POT>
__device__ __forceinline__ void table_pair2(unsigned long long tex, uint32_t rs, bool inb0, bool inb1, uint32_t a0,
                                            uint32_t a1, float2 tD, float2 fl, const float2 wd[4],
                                            const float2 dwd[4], float2 &p, float2 &pt, float2 &pu) {
    unsigned b0, b1;
    const float2 fk = floor2(tD, b0, b1), t = sub2(tD, fk);
    float2 r[4], dr[4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float lo0[4], hi0[4], lo1[4], hi1[4];
        row_pair(inb0, a0 + 2u * h * rs, rs, tex, fl.x, fk.x + (1.0f + 2.0f * h), lo0, hi0);
        row_pair(inb1, a1 + 2u * h * rs, rs, tex, fl.y, fk.y + (1.0f + 2.0f * h), lo1, hi1);
        const float2 ca[4] = {make_float2(lo0[0], lo1[0]), make_float2(lo0[1], lo1[1]), make_float2(lo0[2], lo1[2]),
                              make_float2(lo0[3], lo1[3])};
        const float2 cb[4] = {make_float2(hi0[0], hi1[0]), make_float2(hi0[1], hi1[1]), make_float2(hi0[2], hi1[2]),
                              make_float2(hi0[3], hi1[3])};
        row2<POT>(ca, wd, dwd, r[2 * h], dr[2 * h]);
        row2<POT>(cb, wd, dwd, r[2 * h + 1], dr[2 * h + 1]);
    }
    rows2<POT>(r, dr, t, p, pt, pu);
}

// Warp sums of two values: the total of v0 ends in lanes 0-15, that of v1 in lanes
// 16-31 (hi: the lane is one of these).  One halving exchange and four butterflies.
__device__ __forceinline__ float warp_sum2(float v0, float v1, bool hi) {
    float x = (hi ? v1 : v0) + __shfl_xor_sync(0xffffffffu, hi ? v0 : v1, 16);
    x += __shfl_xor_sync(0xffffffffu, x, 8);
    x += __shfl_xor_sync(0xffffffffu, x, 4);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    return x;
}

// Shared memory of a warp in the FP32 kernel: the staged j tile, the image shifts
// and the j tile's sums.
struct Warp32 {
    float4 p[kTile];
    float4 img[kTile];
    float n[kTile];
    float js[2][kTile];
};

// A pair on a table that is too large for a texture, scalar, from the band and the
// global copy (out of line: no ordinary table comes here).
template <bool POT>
__device__ __noinline__ float3 table_generic(float r2, float qi, float qj, const PairShared *sh) {
    Table<float> tb;
    make_table<float>(*sh, tb);
    unsigned ncl = 0u;
    float3 v = make_float3(0.0f, 0.0f, 0.0f);
    pair_phi<POT, float>(r2, qi, qj, 1.0f / qi, qi * qi, sh->k32, tb, v.x, v.y, v.z, ncl);
    return v;
}

// r^2 of an index displacement in FP32: the packed loop's operations, one value.
template <bool SKEW>
__device__ __forceinline__ float dist2(float dx, float dy, float dz, const PairParams &pp) {
    float r2 = pp.h2f[2] * (dz * dz);
    r2 = fmaf(pp.h2f[1], dy * dy, r2);
    r2 = fmaf(pp.h2f[0], dx * dx, r2);
    if (SKEW) {
        r2 = fmaf(pp.g2f[0], dx * dy, r2);
        r2 = fmaf(pp.g2f[1], dx * dz, r2);
        r2 = fmaf(pp.g2f[2], dy * dz, r2);
    }
    return r2;
}

// The FP32 work items of one warp.  An item is 64 i points (two tiles, a lane owns
// one point of each) against a range of j points from the i points on.  All 64
// share the image masks of a j point, its loop and its part of the j side; an image
// that keeps the whole i box inside the cutoff (most of them) needs no test, weight
// or count per lane.
//
// Bound by instruction issue: 334 instructions a step (a j point's image against 64
// i points), 199 of them FP32 arithmetic, with the schedulers 81 % busy and the
// shared-memory pipe 73 % (24 x 42 x 60 monolayer, E + v; energy 238 instructions, 73 %
// and 79 %).  The kernel before this one (a lane's halves held two j points, 14 warps of
// 128 registers, packed arithmetic) against this one, ms per pass, E + v / E:
//   monolayer 36 x 63 x 90  123.0 / 99.7 -> 98.1 / 75.2    slab 48 x 42 x 75  63.2 / - -> 49.7 / -
//   hexagonal 36 x 36 x 90      - / 62.6 ->    - / 46.9    molecule 48^3      58.0 / - -> 39.7 / 30.2
// What lies off the band costs code as well as loads: with one more copy of the step
// (for tiles whose images all stay inside) the instruction cache no longer held
// the loop, and the slab took 119 ms.
//
// OPEN: cells without images or a cutoff.  One image, no masks, tests or counts but in
// ragged and diagonal tiles.  The general instance against it when it came, ms per pass: molecule
// 48^3 E + v 48.5 -> 42.2, E 36.0 -> 30.6, binding curve 69.8 -> 58.0, Kr dimer
// 24 x 18 x 18 E 0.221 -> 0.191.
template <int MODE, int NT, bool SKEW, bool OPEN>
__device__ __forceinline__ void pair_items_f32(const PairLaunch &pl, unsigned char *smem_raw,
                                               const unsigned int *s_prefix, const int *s_C,
                                               unsigned int n_items, unsigned int stride, const Table<float> &tb) {
    constexpr bool POT = (MODE == 1);
    constexpr float kUnit = POT ? 6.0f : 1.0f;  // bw_diff2's weights lack this factor
    const int warp = threadIdx.x >> 5;
    int lane = threadIdx.x & 31;
    asm volatile("" : "+r"(lane));  // kept, not read from the special register again
    const bool hi = (lane & 16) != 0;
    // the warp's shared memory by an address that stays in a register: otherwise it is
    // formed again from the thread index at each use (E + v: molecule 48^3 42.2 -> 40.5 ms,
    // slab 48 x 42 x 75 51.4 -> 49.9, monolayer 36 x 63 x 90 102.2 -> 100.2)
    uint32_t sw_addr = static_cast<uint32_t>(__cvta_generic_to_shared(reinterpret_cast<Warp32 *>(smem_raw) + warp));
    asm volatile("" : "+r"(sw_addr));
    Warp32 &sw = *reinterpret_cast<Warp32 *>(__cvta_shared_to_generic(sw_addr));
    const PairShared &sh = pl.sh;
    const Consts<float> &K = sh.k32;
    const unsigned long long tex = sh.tex32;
    const uint32_t rs = 4u * static_cast<uint32_t>(tb.SB);
    // cells [k0, k0 + span) have all four rows in the band (none without a texture)
    const unsigned span =
        tex ? static_cast<unsigned>(max(0, min(tb.k0 + tb.kn - 3, sh.nD - 1) - tb.k0)) : 0u;
    const float band_lo = static_cast<float>(tb.k0);
    const unsigned kbits = 0x4B400000u + static_cast<unsigned>(tb.k0);

    for (unsigned int iter = 0;; ++iter) {
        if (iter >= sh.max_iters) {
            if (lane == 0) atomicAdd(&pl.inst[0].stats->guard_trips, 1u);
            break;
        }
        unsigned int item = 0;
        if (lane == 0) item = atomicAdd(sh.queue, 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= n_items) break;
        item *= stride;
        int k = 0;
        while (k + 1 < pl.ninst && item >= s_prefix[k + 1]) ++k;
        const PairParams &pp = pl.inst[k];
        const unsigned int local = item - s_prefix[k];
        const int C = s_C[k];
        const int I = static_cast<int>(local / C), c = static_cast<int>(local % C);
        const int n_act = pp.stats->n_active;
        const int j_first = I * 64 + c * sh.jpts, j_end = min(n_act, j_first + sh.jpts);
        if (j_first >= j_end) {
            if (!POT && lane == 0 && sh.item_E && item < sh.item_cap) sh.item_E[item] = 0.0;
            continue;
        }
        const int i0 = I * 64 + lane, i1 = i0 + 32;
        const bool act0 = i0 < n_act, act1 = i1 < n_act;
        const int ni_act = min(64, n_act - I * 64);
        float2 xi = f2(0.0f), yi = f2(0.0f), zi = f2(0.0f), qi = f2(1.0f), ni = f2(0.0f);
        if (act0) {
            const float4 p = __ldg(pp.p32 + i0);
            xi.x = p.x, yi.x = p.y, zi.x = p.z, qi.x = p.w;
            ni.x = __ldg(pp.n32 + i0);
        }
        if (act1) {
            const float4 p = __ldg(pp.p32 + i1);
            xi.y = p.x, yi.y = p.y, zi.y = p.z, qi.y = p.w;
            ni.y = __ldg(pp.n32 + i1);
        }
        const bool use_cut = pp.use_cut != 0;
        Cut cut;
        cut.pp = &pp;
        const float2 H0 = f2(pp.h2f[0]), H1 = f2(pp.h2f[1]), H2 = f2(pp.h2f[2]);
        double E64 = 0.0;  // energy mode: this lane's part of the item's sum
        unsigned int cnt = 0, nclamp = 0;  // per lane: images that are only partly inside
        unsigned int cnt_full = 0;         // (j point, image) steps with all 64 i points inside
        unsigned int evals = 0;            // (j point, image) steps
        const int T0 = 2 * I, T1 = min(2 * I + 1, (n_act - 1) / kTile);  // the i tiles
        for (int J = j_first / kTile; J * kTile < j_end; ++J) {
            const int jb = J * kTile;
            const int jl0 = max(0, j_first - jb), jl1 = min(kTile, j_end - jb);
            const bool mine = lane >= jl0 && lane < jl1;
            const bool diag = (J >> 1) == I;
            const bool special = diag || ni_act < 64;
            bool staged = false;
            int n_cand = 1;
            float ilo[3], ihi[3], jl[3], jh[3];
            {
                const float4 a0 = __ldg(pp.blo + T0), a1 = __ldg(pp.blo + T1), b0 = __ldg(pp.bhi + T0),
                             b1 = __ldg(pp.bhi + T1), jlo = __ldg(pp.blo + J), jhi = __ldg(pp.bhi + J);
                ilo[0] = fminf(a0.x, a1.x), ilo[1] = fminf(a0.y, a1.y), ilo[2] = fminf(a0.z, a1.z);
                ihi[0] = fmaxf(b0.x, b1.x), ihi[1] = fmaxf(b0.y, b1.y), ihi[2] = fmaxf(b0.z, b1.z);
                jl[0] = jlo.x, jl[1] = jlo.y, jl[2] = jlo.z;
                jh[0] = jhi.x, jh[1] = jhi.y, jh[2] = jhi.z;
            }
            float4 cil = make_float4(0.f, 0.f, 0.f, 0.f), cih = cil, cjl = cil, cjh = cil;
            if (SKEW) {  // Cartesian boxes
                const float4 a0 = __ldg(pp.clo + T0), a1 = __ldg(pp.clo + T1), b0 = __ldg(pp.chi + T0),
                             b1 = __ldg(pp.chi + T1);
                cil = make_float4(fminf(a0.x, a1.x), fminf(a0.y, a1.y), fminf(a0.z, a1.z), 0.f);
                cih = make_float4(fmaxf(b0.x, b1.x), fmaxf(b0.y, b1.y), fmaxf(b0.z, b1.z), 0.f);
                cjl = __ldg(pp.clo + J);
                cjh = __ldg(pp.chi + J);
            }
            const float rc2_box = pp.box_out, rc2_in = pp.box_in;
            // culling metric: h2 on orthogonal cells, a lower bound of r^2/|d|^2 on skewed ones
            const float cull[3] = {pp.cull_h2[0], pp.cull_h2[1], pp.cull_h2[2]};
            int mlo[3], nm[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (pp.M[a] == 0) {
                    mlo[a] = 0;
                    nm[a] = 1;
                } else {
                    const float N = static_cast<float>(pp.dims[a]), rcm = pp.rcm[a];
                    mlo[a] = max(-pp.M[a], static_cast<int>(ceilf((-rcm - (ihi[a] - jl[a])) / N)));
                    const int mhi = min(pp.M[a], static_cast<int>(floorf((rcm - (ilo[a] - jh[a])) / N)));
                    nm[a] = max(0, mhi - mlo[a] + 1);
                }
            }
            if (!OPEN) n_cand = nm[0] * nm[1] * nm[2];
            // candidate images in chunks of 32, one per lane (an open cell has the one at 0)
            for (int c0 = 0; c0 < n_cand; c0 += 32) {
                unsigned bal = 1u, jm = mine ? 1u : 0u, jf = 0u;
                if constexpr (OPEN) {
                    __syncwarp();  // earlier reads of p, n, js are done
                    if (mine) {
                        sw.p[lane] = __ldg(pp.p32 + jb + lane);
                        sw.n[lane] = __ldg(pp.n32 + jb + lane);
                    }
                    __syncwarp();
                } else {
                const int t = c0 + lane;
                bool ok = false;
                int mm[3] = {0, 0, 0};
                if (t < n_cand) {
                    mm[2] = mlo[2] + t % nm[2];
                    const int t1 = t / nm[2];
                    mm[1] = mlo[1] + t1 % nm[1];
                    mm[0] = mlo[0] + t1 / nm[1];
                    if (SKEW)
                        ok = !use_cut || box_gap2_cart(cil, cih, cjl, cjh, mm, pp.dims, pp.vrow) <= rc2_box;
                    else
                        ok = !use_cut || box_gap2(ilo, ihi, jl, jh, mm, pp.dims, cull) <= rc2_box;
                }
                bal = __ballot_sync(0xffffffffu, ok);
                if (bal == 0u) continue;
                __syncwarp();  // earlier reads of img, p, n, js are done
                if (ok)
                    sw.img[__popc(bal & ((1u << lane) - 1u))] =
                        make_float4(static_cast<float>(mm[0] * pp.dims[0]), static_cast<float>(mm[1] * pp.dims[1]),
                                    static_cast<float>(mm[2] * pp.dims[2]), 0.0f);
                if (!staged) {
                    if (mine) {
                        sw.p[lane] = __ldg(pp.p32 + jb + lane);
                        sw.n[lane] = __ldg(pp.n32 + jb + lane);
                    }
                    staged = true;
                }
                __syncwarp();
                const int nimg = __popc(bal);
                // this lane's j point: images that bring the i box within the cutoff (jm), and
                // those that keep all of it inside (jf; none in ragged or diagonal tiles)
                jm = 0u;
                if (mine) {
                    const float4 pj = sw.p[lane];
                    for (int b = 0; b < nimg; ++b) {
                        const float4 sft = sw.img[b];
                        float d2, f2max;
                        if (SKEW) {
                            // the point less the shift, in Cartesian coordinates, against the i box
                            const float ux = pj.x - sft.x, uy = pj.y - sft.y, uz = pj.z - sft.z;
                            const CellRows &vr = pp.vrow;
                            const float q0c = ux * vr.v[0] + uy * vr.v[3] + uz * vr.v[6];
                            const float q1c = ux * vr.v[1] + uy * vr.v[4] + uz * vr.v[7];
                            const float q2c = ux * vr.v[2] + uy * vr.v[5] + uz * vr.v[8];
                            const float lx = cil.x - q0c, hx = q0c - cih.x, ly = cil.y - q1c, hy = q1c - cih.y,
                                        lz = cil.z - q2c, hz = q2c - cih.z;
                            const float gx = fmaxf(0.0f, fmaxf(lx, hx)), gy = fmaxf(0.0f, fmaxf(ly, hy)),
                                        gz = fmaxf(0.0f, fmaxf(lz, hz));
                            d2 = gx * gx + gy * gy + gz * gz;
                            const float ex = fminf(lx, hx), ey = fminf(ly, hy), ez = fminf(lz, hz);
                            f2max = ex * ex + ey * ey + ez * ez;
                        } else {
                            const float lx = ilo[0] + sft.x - pj.x, hx = pj.x - ihi[0] - sft.x,
                                        ly = ilo[1] + sft.y - pj.y, hy = pj.y - ihi[1] - sft.y,
                                        lz = ilo[2] + sft.z - pj.z, hz = pj.z - ihi[2] - sft.z;
                            const float gx = fmaxf(0.0f, fmaxf(lx, hx)), gy = fmaxf(0.0f, fmaxf(ly, hy)),
                                        gz = fmaxf(0.0f, fmaxf(lz, hz));
                            d2 = cull[0] * gx * gx + cull[1] * gy * gy + cull[2] * gz * gz;
                            // the farther face along each axis: the lower of the two (signed) gaps
                            const float ex = fminf(lx, hx), ey = fminf(ly, hy), ez = fminf(lz, hz);
                            f2max = cull[0] * ex * ex + cull[1] * ey * ey + cull[2] * ez * ez;
                        }
                        if (!use_cut || d2 <= rc2_box) jm |= 1u << b;
                        if (!use_cut || f2max <= rc2_in) jf |= 1u << b;
                    }
                    if (special) jf = 0u;
                }
                }
                float2 a_acc = f2(0.0f), u_acc = f2(0.0f);
                float2 cwt = f2(0.0f);
                if (OPEN) {
                    evals += static_cast<unsigned>(jl1 - jl0);
                    if (!special) cnt_full += static_cast<unsigned>(jl1 - jl0);
                }
                unsigned jset = OPEN ? 0u : __ballot_sync(0xffffffffu, jm != 0u);
                for (int jo = jl0; OPEN ? jo < jl1 : jset != 0u; ++jo) {
                    const int jj = OPEN ? jo : __ffs(jset) - 1;
                    unsigned m = 1u, mf = special ? 0u : 1u;
                    if (!OPEN) {
                        jset &= jset - 1u;
                        m = __shfl_sync(0xffffffffu, jm, jj);
                        mf = __shfl_sync(0xffffffffu, jf, jj);
                        evals += static_cast<unsigned>(__popc(m));
                        cnt_full += static_cast<unsigned>(__popc(mf));
                    }
                    const float4 pj = sw.p[jj];
                    const float nj = sw.n[jj];
                    Delta2 dp;
                    bool cl0, cl1;
                    delta_part2<POT>(qi, pj.w, K, dp, cl0, cl1);
                    const uint32_t c0a = tb.s + 4u * dp.l0, c1a = tb.s + 4u * dp.l1;
                    float2 A2 = f2(0.0f), V2 = f2(0.0f);
                    // r dphi/dd1 = cD r pt + b1 pu with b1, b2 fixed for the j point: the
                    // sums of r pt and of pu over the images are scaled once at the end
                    float2 Srpt = f2(0.0f), Spu = f2(0.0f);
                    unsigned mfar = 0u;  // images with some pair past the table
                    float2 cw = f2(0.0f);  // partly inside images: those that count, per half
                    unsigned mr = m;
                    do {
                        const unsigned bit = OPEN ? 1u : mr & (0u - mr);
                        // integers: every sum is exact
                        float2 dx = sub2(xi, f2(pj.x)), dy = sub2(yi, f2(pj.y)), dz = sub2(zi, f2(pj.z));
                        if (!OPEN) {
                            const float4 sft = sw.img[__ffs(mr) - 1];
                            mr ^= bit;
                            dx = add2(xi, f2(sft.x - pj.x)), dy = add2(yi, f2(sft.y - pj.y)),
                            dz = add2(zi, f2(sft.z - pj.z));
                        }
                        float2 r2 = mul2(H2, mul2(dz, dz));
                        r2 = fma2(H1, mul2(dy, dy), r2);
                        r2 = fma2(H0, mul2(dx, dx), r2);
                        if (SKEW) {
                            r2 = fma2(f2(pp.g2f[0]), mul2(dx, dy), r2);
                            r2 = fma2(f2(pp.g2f[1]), mul2(dx, dz), r2);
                            r2 = fma2(f2(pp.g2f[2]), mul2(dy, dz), r2);
                        }
                        float2 rr = mul2(r2, make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y)));
                        float2 tD = mul2(rr, dp.sqcD);
                        float2 w = f2(kUnit);  // 0 in a half that does not count
                        uint32_t l0a = c0a, l1a = c1a;
                        if (OPEN ? special : (mf & bit) == 0u) {
                            bool in0 = true, in1 = true;
                            if (!OPEN && use_cut) {
                                in0 = !beyond<SKEW>(r2.x, dx.x, dy.x, dz.x, cut);
                                in1 = !beyond<SKEW>(r2.y, dx.y, dy.y, dz.y, cut);
                            }
                            if (special) {
                                // ragged i tile, or a diagonal one, where only j >= i counts, self-images (j =
                                // i, r > 0) for i only, and the self term is added in FP64 at the end
                                if (!(r2.x > 0.0f)) in0 = false, rr.x = 0.0f;
                                if (!(r2.y > 0.0f)) in1 = false, rr.y = 0.0f;
                                in0 = in0 && act0 && (!diag || jb + jj >= i0);
                                in1 = in1 && act1 && (!diag || jb + jj >= i1);
                                cnt -= (in0 && diag && jb + jj == i0 ? 1u : 0u) + (in1 && diag && jb + jj == i1 ? 1u : 0u);
                            }
                            w = make_float2(in0 ? kUnit : 0.0f, in1 ? kUnit : 0.0f);
                            cw = add2(cw, make_float2(in0 ? 1.0f : 0.0f, in1 ? 1.0f : 0.0f));
                            // an idle half reads the band's first cell (one address for all)
                            if (!in0) tD.x = band_lo, l0a = tb.s;
                            if (!in1) tD.y = band_lo, l1a = tb.s;
                        }
                        unsigned kb0, kb1;
                        const float2 fk = floor2(tD, kb0, kb1);
                        kb0 -= kbits;
                        kb1 -= kbits;
                        if (__all_sync(0xffffffffu, kb0 < span && kb1 < span)) {
                            float2 p, pt, pu;
                            band_pair2<POT>(tex, rs, sub2(tD, fk), fk, l0a + kb0 * rs, l1a + kb1 * rs, dp.fl, dp.wd,
                                            dp.dwd, p, pt, pu);
                            A2 = fma2(w, p, A2);
                            if (POT) {
                                Srpt = fma2(mul2(w, rr), pt, Srpt);
                                Spu = fma2(w, pu, Spu);
                            }
                        } else {
                            // some lane off the band: what lies on the table from its texture copy, what
                            // lies past it (false for NaN as well) in the loop below
                            const bool on0 = tD.x >= 0.0f && tD.x <= K.tDmax, on1 = tD.y >= 0.0f && tD.y <= K.tDmax;
                            if (tex) {
                                const float2 tq = make_float2(on0 ? fminf(tD.x, K.tDclamp) : 0.0f,
                                                              on1 ? fminf(tD.y, K.tDclamp) : 0.0f);
                                const float2 wt = make_float2(on0 ? w.x : 0.0f, on1 ? w.y : 0.0f);
                                float2 p, pt, pu;
                                table_pair2<POT>(tex, rs, kb0 < span, kb1 < span, l0a + kb0 * rs, l1a + kb1 * rs, tq,
                                                 dp.fl, dp.wd, dp.dwd, p, pt, pu);
                                A2 = fma2(wt, p, A2);
                                if (POT) {
                                    Srpt = fma2(make_float2(wt.x == 0.0f ? 0.0f : kUnit * rr.x,
                                                            wt.y == 0.0f ? 0.0f : kUnit * rr.y), pt, Srpt);
                                    Spu = fma2(wt, pu, Spu);
                                }
                            }
                            if (__any_sync(0xffffffffu, (w.x != 0.0f && !(tex && on0)) || (w.y != 0.0f && !(tex && on1))))
                                mfar |= bit;
                        }
                    } while (!OPEN && mr != 0u);
                    // ordered pairs: two for every inside evaluation (once for i, once for j), less
                    // the one of a self-image taken off above
                    cwt = add2(cwt, cw);
                    if (cl0 || cl1) {
                        const float nf = OPEN ? (special ? 0.0f : 1.0f) : static_cast<float>(__popc(mf));
                        nclamp += 2u * static_cast<unsigned>((cl0 ? nf + cw.x : 0.0f) + (cl1 ? nf + cw.y : 0.0f));
                    }
                    if (POT) {
                        const float2 a = mul2(Srpt, f2(3.0f * K.cD));  // rows2 gives a third of the derivative
                        const float2 u = fma2(Spu, dp.b1, a), v = mul2(Spu, dp.sb);
                        u_acc = fma2(f2(nj), u, u_acc);
                        V2 = sub2(sub2(u, v), v);
                    }
                    // the halves past the table (once more from the geometry, so that the loop above
                    // keeps nothing for them in registers)
                    while (mfar != 0u) {
                        const float4 sft = OPEN ? make_float4(0.f, 0.f, 0.f, 0.f) : sw.img[__ffs(mfar) - 1];
                        const bool part = OPEN ? special : (mf & mfar & (0u - mfar)) == 0u;
                        mfar &= mfar - 1u;
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const float q = h ? qi.y : qi.x;
                            const float dx = (h ? xi.y : xi.x) + (sft.x - pj.x), dy = (h ? yi.y : yi.x) + (sft.y - pj.y),
                                        dz = (h ? zi.y : zi.x) + (sft.z - pj.z);
                            const float r2 = dist2<SKEW>(dx, dy, dz, pp);
                            const float r = r2 * rsqrt_ftz(fmaxf(r2, 1e-30f)), tD = r * ((q + pj.w) * K.cD);
                            const bool on = tD >= 0.0f && tD <= K.tDmax;
                            if ((tex && on) || !(r2 > 0.0f)) continue;
                            if (part && (!(h ? act1 : act0) || (diag && jb + jj < (h ? i1 : i0)) ||
                                         (!OPEN && use_cut && beyond<SKEW>(r2, dx, dy, dz, cut))))
                                continue;
                            float phi, rd = 0.0f, rd2 = 0.0f;
                            if (on) {  // (only with a table too large for a texture)
                                const float3 g = table_generic<POT>(r2, q, pj.w, &sh);
                                phi = g.x, rd = g.y, rd2 = g.z;
                            } else
                                past_part<POT, float>(r, r2, tD, q, pj.w, 1.0f / q, q * q, K, tb.rho, phi, rd, rd2);
                            const float p0 = h ? 0.0f : phi, p1 = h ? phi : 0.0f, u0 = h ? 0.0f : rd, u1 = h ? rd : 0.0f;
                            A2 = add2(A2, make_float2(p0, p1));
                            if (POT) {
                                u_acc = fma2(f2(nj), make_float2(u0, u1), u_acc);
                                V2 = add2(V2, make_float2(h ? 0.0f : rd2, h ? rd2 : 0.0f));
                            }
                        }
                    }
                    if (POT) {
                        a_acc = fma2(f2(nj), A2, a_acc);
                        // (j = i counts for i only)
                        const float2 nb = make_float2(diag && jb + jj == i0 ? 0.0f : ni.x,
                                                      diag && jb + jj == i1 ? 0.0f : ni.y);
                        const float tot = warp_sum2(nb.x * A2.x + nb.y * A2.y, nb.x * V2.x + nb.y * V2.y, hi);
                        if ((lane & 15) == 0) sw.js[lane >> 4][jj] = tot;
                    } else {
                        // every pair counts for i and for j, j = i for i only
                        const float n2 = nj + nj;
                        a_acc = fma2(make_float2(diag && jb + jj == i0 ? nj : n2, diag && jb + jj == i1 ? nj : n2), A2,
                                     a_acc);
                    }
                }
                cnt += 2u * static_cast<unsigned>(cwt.x + cwt.y);
                // the j tile's FP32 sums, folded into FP64
                if (POT) {
                    if (act0) {
                        atomicAdd(pp.A + i0, static_cast<double>(a_acc.x));
                        atomicAdd(pp.U + i0, static_cast<double>(ni.x) * static_cast<double>(u_acc.x));
                    }
                    if (act1) {
                        atomicAdd(pp.A + i1, static_cast<double>(a_acc.y));
                        atomicAdd(pp.U + i1, static_cast<double>(ni.y) * static_cast<double>(u_acc.y));
                    }
                    __syncwarp();
                    if (jm != 0u) {
                        const float ja = sw.js[0][lane], ju = sw.js[1][lane];
                        if (ja != 0.0f) atomicAdd(pp.A + jb + lane, static_cast<double>(ja));
                        if (ju != 0.0f)
                            atomicAdd(pp.U + jb + lane, static_cast<double>(sw.n[lane]) * static_cast<double>(ju));
                    }
                } else {
                    E64 += static_cast<double>(ni.x) * static_cast<double>(a_acc.x) +
                           static_cast<double>(ni.y) * static_cast<double>(a_acc.y);
                }
            }
        }
        // the self terms n_i phi(0, 0) of the i points whose own j lies in this item, from
        // the table's node: near a nucleus they outweigh the rest of A_i, and FP32 sums that
        // hold them round at their size (r dphi/dd1 is 0 there)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = h ? i1 : i0;
            if (i < n_act && i >= j_first && i < j_end) {
                const double n = __ldg(pp.n64 + i);
                if (POT)
                    atomicAdd(pp.A + i, n * sh.phi00);
                else
                    E64 += n * n * sh.phi00;
            }
        }
        count_item(pp.stats, cnt, nclamp, static_cast<unsigned long long>(evals) * static_cast<unsigned long long>(ni_act),
                   128ull * cnt_full);
        if (!POT) {
            // the item's energy partial, summed over lanes in a fixed order (items
            // beyond the partials' capacity are added atomically)
            const double e = warp_sum(E64);
            if (lane == 0) {
                if (sh.item_E && item < sh.item_cap)
                    sh.item_E[item] = e;
                else if (e != 0.0)
                    atomicAdd(&pp.stats->E_pair, e);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// FP64
// ---------------------------------------------------------------------------

// The cell of a coordinate x in [0, n): floor(x) in k and x - k, from the low word of x
// shifted by 1.5 2^52 (rounded down).  False for x outside and for NaN.
__device__ __forceinline__ bool cell_of(double x, int n, int &k, double &t) {
    const double b = __dadd_rd(x, 6755399441055744.0);
    k = __double2loint(b);
    t = x - (b - 6755399441055744.0);
    return __double2hiint(b) == 0x43380000 && static_cast<unsigned>(k) < static_cast<unsigned>(n);
}

// The delta part of a pair in FP64, for all lanes of a warp (the quantities of delta_part): (q_i + q_j) cD, the
// derivative factors b1 and sb (see Delta2), the delta cell and weights.
struct Delta64 {
    double sqcD, b1, sb;
    double wd[4], dwd[4];
    int l;
    bool cl;
};
template <bool POT>
__device__ __forceinline__ void delta_part64(double qi, double qj, const Consts<double> &K, Delta64 &d) {
    const double sq = qi + qj, dq = qi - qj, isq = rcp_newton(sq), ds = dq * isq;
    const double td0 = fabs(ds) * K.cd;
    double u;
    d.cl = false;
    double e = 0.0;
    const bool ok = cell_of(td0, K.lmax + 1, d.l, u);
    // (a vote, so that the operations of the rare case are not run for all)
    if (__any_sync(0xffffffffu, !ok)) {
        // the last node itself (its cell at u = 1), or past it: the weights continue
        // linearly (see delta_part)
        const double td = fmin(fmax(td0, 0.0), K.tdmax);
        const int l = min(static_cast<int>(td), K.lmax);
        d.cl = td0 > K.tdmax;
        e = td0 - td;
        u = ok ? u : td - l;
        d.l = ok ? d.l : l;
    }
    const double s = 1.0 - u, u2 = u * u, s2 = s * s;
    d.wd[0] = s2 * s;
    d.wd[1] = fma(u2, fma(u, 3.0, -6.0), 4.0);
    d.wd[2] = fma(s2, fma(s, 3.0, -6.0), 4.0);
    d.wd[3] = u2 * u;
    if (POT || __any_sync(0xffffffffu, d.cl)) {
        d.dwd[0] = -3.0 * s2;
        d.dwd[1] = u * fma(u, 9.0, -12.0);
        d.dwd[2] = s * fma(s, -9.0, 12.0);
        d.dwd[3] = 3.0 * u2;
    }
    if (__any_sync(0xffffffffu, d.cl)) {
#pragma unroll
        for (int n = 0; n < 4; ++n) d.wd[n] = fma(d.cl ? e : 0.0, d.dwd[n], d.wd[n]);
    }
    d.sqcD = sq * K.cD;
    d.sb = copysign(isq * K.cd, dq);
    d.b1 = fma(-ds, d.sb, d.sb);
}

// The spline at cell (k, l), offset t along D: phi and, with POT, the cell-coordinate
// derivatives.  poly holds, per D cell and delta column, the column's cubic in t.
template <bool POT>
__device__ __forceinline__ void spline64(const double *poly, int S, int k, double t, const Delta64 &d, double &p,
                                         double &pt, double &pu) {
    const double2 *c = reinterpret_cast<const double2 *>(poly) + 2 * (static_cast<size_t>(k) * S + d.l);
    double s[4], P1 = 0.0, P2 = 0.0, P3 = 0.0;
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        const double2 a = __ldg(c + 2 * n), b = __ldg(c + 2 * n + 1);
        s[n] = fma(t, fma(t, fma(t, b.y, b.x), a.y), a.x);
        if (POT) {
            P1 = n ? fma(d.wd[n], a.y, P1) : d.wd[0] * a.y;
            P2 = n ? fma(d.wd[n], b.x, P2) : d.wd[0] * b.x;
            P3 = n ? fma(d.wd[n], b.y, P3) : d.wd[0] * b.y;
        }
    }
    p = fma(d.wd[3], s[3], fma(d.wd[2], s[2], fma(d.wd[1], s[1], d.wd[0] * s[0])));
    if (POT) {
        pt = fma(t, fma(t, 3.0 * P3, P2 + P2), P1);
        // the derivative weights sum to zero: differences to the first column
        pu = fma(d.dwd[3], s[3] - s[0], fma(d.dwd[2], s[2] - s[0], d.dwd[1] * (s[1] - s[0])));
    }
}

// past_part in FP64 with one reciprocal (of eq. (17)'s denominator times tD) in place
// of five divisions.  y = q_i q_j and s2 = q_i^2 + q_j^2.  False, and nothing written,
// where that product (27 (q r)^7 at equal q) is not within 2^-500 .. 2^501: past_part
// takes such pairs, whose divisions by an infinity give the 0 that they contribute.
template <bool POT>
__device__ __forceinline__ bool past_part64(double r, double tD, double qi, double qj, const Consts<double> &K,
                                            const double *rho_c, double &phi, double &rd, double &rd2) {
    const double r2 = r * r, r6 = r2 * r2 * r2, y = qi * qj, s2 = fma(qi, qi, qj * qj);
    const double z = r6 * (y * y), X = z * s2, XtD = X * tD;
    // (by the exponent, off the FP64 pipe)
    if (static_cast<unsigned>(__double2hiint(XtD) - ((1023 - 500) << 20)) >= (1001u << 20)) return false;
    const double w = rcp_newton(XtD);
    const double inv = w * tD, itD = w * X;  // 1/X, 1/tD
    const double p17 = -K.C * inv;
    const bool i_small = qi < qj;
    // rho at delta* (see past_part)
    const double a = r * K.iDmax * K.cd, ts0 = fma(-(i_small ? qi : qj), a, K.cd);
    double u, e = 0.0;
    int l;
    bool up = true;
    if (!cell_of(ts0, K.lmax + 1, l, u)) {
        const double ts = fmin(fmax(ts0, 0.0), K.tdmax);
        up = ts0 > 0.0;
        l = min(static_cast<int>(ts), K.lmax);
        u = ts - l;
        e = ts0 > K.tdmax ? ts0 - ts : 0.0;
    }
    const double s = 1.0 - u, u2 = u * u, s2u = s * s;
    const double c0 = __ldg(rho_c + l), c1 = __ldg(rho_c + l + 1), c2 = __ldg(rho_c + l + 2), c3 = __ldg(rho_c + l + 3);
    double rho = fma(u2 * u, c3, fma(fma(s2u, fma(s, 3.0, -6.0), 4.0), c2,
                                     fma(fma(u2, fma(u, 3.0, -6.0), 4.0), c1, s2u * s * c0)));
    double drho = 0.0;
    if (POT || e != 0.0) {
        drho = up ? fma(3.0 * u2, c3 - c0, fma(s * fma(s, -9.0, 12.0), c2 - c0, u * fma(u, 9.0, -12.0) * (c1 - c0)))
                  : 0.0;
        rho = fma(e, drho, rho);
    }
    const double Dr = K.tDmax * itD, m = K.om_rho0 * (Dr * Dr);
    const double g = rho + (K.om_rho0 - m);
    phi = g * p17;
    if (POT) {
        const double is2 = inv * z, iy = inv * (r6 * s2 * y);  // 1/s2, 1/(q_i q_j)
        const double ramp = m * (2.0 * K.cD) * r * itD, sl = drho * a, t = -2.0 * phi;
        rd = fma(t, fma(qi, is2, qj * iy), p17 * (i_small ? ramp - sl : ramp));
        rd2 = fma(t, fma(qj, is2, qi * iy), p17 * (i_small ? ramp : ramp - sl));
    }
    return true;
}

// FP64 warp sums of two values (as warp_sum2).
__device__ __forceinline__ double warp_sum2(double v0, double v1, bool hi) {
    double x = (hi ? v1 : v0) + __shfl_xor_sync(0xffffffffu, hi ? v0 : v1, 16);
    x += __shfl_xor_sync(0xffffffffu, x, 8);
    x += __shfl_xor_sync(0xffffffffu, x, 4);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    return x;
}

// r of an index displacement, negative outside the cutoff: from the table of
// k_r_table, or computed where there is none.
template <bool SKEW>
__device__ __forceinline__ double pair_r(const PairParams &pp, int dx, int dy, int dz) {
    if (pp.rt) {
        if (SKEW) {
            if (dz < 0) dx = -dx, dy = -dy, dz = -dz;
            const unsigned ux = static_cast<unsigned>(dx + pp.rtm[0]), uy = static_cast<unsigned>(dy + pp.rtm[1]);
            const unsigned wx = 2u * pp.rtm[0] + 1u, wy = 2u * pp.rtm[1] + 1u;
            if (ux >= wx || uy >= wy || dz > pp.rtm[2]) return -1.0;
            return __ldg(pp.rt + (static_cast<size_t>(ux) * wy + uy) * (pp.rtm[2] + 1) + dz);
        }
        dx = abs(dx), dy = abs(dy), dz = abs(dz);
        if (dx > pp.rtm[0] || dy > pp.rtm[1] || dz > pp.rtm[2]) return -1.0;
        return __ldg(pp.rt + (static_cast<size_t>(dx) * (pp.rtm[1] + 1) + dy) * (pp.rtm[2] + 1) + dz);
    }
    return index_r<SKEW>(pp, dx, dy, dz);
}

// The table of pair_r: entry (x, y, z) of extents rtm + 1, or 2 rtm + 1 along the
// first two axes of a skewed cell (signed differences; z >= 0 by inversion).
template <bool SKEW>
__global__ void k_r_table(const __grid_constant__ PairParams pp, double *__restrict__ rt) {
    const int wx = SKEW ? 2 * pp.rtm[0] + 1 : pp.rtm[0] + 1, wy = SKEW ? 2 * pp.rtm[1] + 1 : pp.rtm[1] + 1,
              wz = pp.rtm[2] + 1;
    const long long total = static_cast<long long>(wx) * wy * wz;
    for (long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; e < total;
         e += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int z = static_cast<int>(e % wz), y = static_cast<int>(e / wz % wy),
                  x = static_cast<int>(e / (static_cast<long long>(wz) * wy));
        rt[e] = index_r<SKEW>(pp, SKEW ? x - pp.rtm[0] : x, SKEW ? y - pp.rtm[1] : y, z);
    }
}

// Shared memory of a warp in the FP64 kernel: the j tile, image shifts, j sums.
struct Warp64 {
    int4 p[kTile];    // index coordinates
    int4 img[kTile];
    double2 qn[kTile];
    double js[2][kTile];
};

// What every CTA does first: the table, with the resident band staged (FP32), the first
// item of each instance and its chunks.  The band starts behind the warps' parts (NW).
template <typename R, int NW>
__device__ __forceinline__ void pair_begin(const PairLaunch &pl, unsigned char *smem_raw, unsigned int *s_prefix,
                                           int *s_C, Table<R> &tb) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const PairShared &sh = pl.sh;
    make_table<R>(sh, tb);
    if constexpr (sizeof(R) == 4) {
        float *band = reinterpret_cast<float *>(smem_raw + sizeof(Warp32) * NW);
        tb.s = static_cast<uint32_t>(__cvta_generic_to_shared(band));
        tb.k0 = sh.ks0 >= 0 ? sh.ks0 : pl.inst[0].stats->band_row0;
        tb.kn = sh.ksn;
        const int S = sh.S, SB = tb.SB;
        const float *src = sh.tab32 + static_cast<size_t>(tb.k0) * S;
        for (int row = warp; row < sh.ksn; row += NW)
            for (int col = lane; col < S; col += 32) band[row * SB + col] = __ldg(src + row * S + col);
    }
    // work items per instance: (i tiles) x (chunks of jtiles_per_item j tiles)
    if (threadIdx.x == 0) {
        unsigned int acc = 0;
        for (int k = 0; k < pl.ninst; ++k) {
            const int na = pl.inst[k].stats->n_active;
            s_prefix[k] = acc;
            s_C[k] = max(1, (na + sh.jpts - 1) / sh.jpts);
            acc += static_cast<unsigned int>(pair_items(na, sh.itile, sh.jpts));
        }
        s_prefix[pl.ninst] = acc;
    }
    __syncthreads();  // the only block barrier: table band and item counts ready
}

// MODE 0: energy (unordered pairs), MODE 1: potential (A, U per point).
//
// Per work item the warp holds an i tile (lane = i point; two of them in FP32,
// pair_items_f32).  For each j tile it lists the images whose shifted i box comes
// within the cutoff of the j box, then each lane marks, for its own j point, which
// of those images bring the i box within the cutoff of that point.  The pair loop
// runs over j points (broadcast) and, inside, over the marked images: the delta part
// of a pair is computed once for all its images.
//
// The FP64 instances are bound by the FP64 pipe (1.7 lanes an SM and clock, 1/73 of
// FP32), so what need not run on it does not: r comes from a table over index
// displacements (k_r_table; it also holds the cutoff test), the D cell's cubic from
// a table of polynomials instead of weights and rows (spline64), cells and signs from
// integer operations on the bits.  Rare cases (past the table, the last delta node)
// stand behind votes: behind a lane's branch the compiler ran them for all, predicated.
// FP64 operations per evaluation 136 -> 89 (16 x 28 x 40 monolayer, E + v, a third of
// whose warps hold a lane past the table), the pipe 88 % busy as before.  ms per pass,
// 24 x 42 x 60 monolayer E + v 453 -> 274 and E 242 -> 143, hexagonal 20 x 20 x 50
// 93 -> 47, slab 32 x 28 x 50 185 -> 138, open dimer 31 x 23 x 19 E 16.7 -> 14.0.
template <typename R, int MODE, int NT, bool SKEW>
__global__ void __launch_bounds__(NT, 1) k_pair(const __grid_constant__ PairLaunch pl) {
    constexpr bool POT = (MODE == 1);
    constexpr int NW = NT / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned int s_prefix[kMaxInst + 1];
    __shared__ int s_C[kMaxInst];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const PairShared &sh = pl.sh;
    Table<R> tb;
    pair_begin<R, NW>(pl, smem_raw, s_prefix, s_C, tb);
    // autotuning samples every item_stride-th item (item * stride < the total)
    const unsigned int stride = max(1u, sh.item_stride);
    const unsigned int n_items = min((s_prefix[pl.ninst] + stride - 1u) / stride, sh.item_limit);
    if constexpr (sizeof(R) == 4) {
        pair_items_f32<MODE, NT, SKEW, false>(pl, smem_raw, s_prefix, s_C, n_items, stride, tb);
        return;
    } else {
    const Consts<double> &K = sh.k64;
    const double *poly = sh.poly64;
    const bool hi = (lane & 16) != 0;
    Warp64 &sw = reinterpret_cast<Warp64 *>(smem_raw)[warp];

    for (unsigned int iter = 0;; ++iter) {
        if (iter >= sh.max_iters) {
            if (lane == 0) atomicAdd(&pl.inst[0].stats->guard_trips, 1u);
            break;
        }
        unsigned int item = 0;
        if (lane == 0) item = atomicAdd(sh.queue, 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= n_items) break;
        item *= stride;
        int k = 0;
        while (k + 1 < pl.ninst && item >= s_prefix[k + 1]) ++k;
        const PairParams &pp = pl.inst[k];
        const unsigned int local = item - s_prefix[k];
        const int C = s_C[k];
        const int I = static_cast<int>(local / C), c = static_cast<int>(local % C);
        const int n_act = pp.stats->n_active;
        const int nT = (n_act + kTile - 1) / kTile;
        const int Js = I;  // i <-> j folded: j tiles from the i tile on
        const int J0 = Js + c * (sh.jpts / kTile);
        const int J1 = min(nT, J0 + sh.jpts / kTile);
        if (J0 >= J1) {
            if (!POT && lane == 0 && sh.item_E && item < sh.item_cap) sh.item_E[item] = 0.0;
            continue;
        }

        float rcm[3];
        int dims[3], M[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            dims[a] = pp.dims[a];
            M[a] = pp.M[a];
            // cutoff in index units along a, widened so that rounding never drops an image
            rcm[a] = pp.rcm[a];
        }
        // culling metric: h2 on orthogonal cells, a lower bound of r^2/|d|^2 on skewed ones
        const float cull[3] = {pp.cull_h2[0], pp.cull_h2[1], pp.cull_h2[2]};
        const float rc2_box = pp.box_out;
        const bool use_cut = pp.use_cut != 0;

        const int ig = I * kTile + lane;
        const bool act = ig < n_act;
        const int ni_act = min(kTile, n_act - I * kTile);
        int xi = 0, yi = 0, zi = 0;
        double qi = 1.0, ni = 0.0;
        if (act) {
            const float4 pi = __ldg(pp.p32 + ig);
            xi = static_cast<int>(pi.x);
            yi = static_cast<int>(pi.y);
            zi = static_cast<int>(pi.z);
            qi = __ldg(pp.q64 + ig);
            ni = __ldg(pp.n64 + ig);
        }
        const float4 ib0 = __ldg(pp.blo + I), ib1 = __ldg(pp.bhi + I);
        const float ilo[3] = {ib0.x, ib0.y, ib0.z}, ihi[3] = {ib1.x, ib1.y, ib1.z};
        float4 cil = make_float4(0.f, 0.f, 0.f, 0.f), cih = cil;  // skewed: Cartesian i box
        if (SKEW) {
            cil = __ldg(pp.clo + I);
            cih = __ldg(pp.chi + I);
        }
        double A64 = 0.0, U64 = 0.0;
        unsigned int cnt = 0, nclamp = 0;
        unsigned int item_evals = 0;  // (j point, image) steps of this item (times ni_act at the end)
        for (int J = J0; J < J1; ++J) {
            const int jb = J * kTile;
            const int jn = min(kTile, n_act - jb);
            const float4 jlo = __ldg(pp.blo + J), jhi = __ldg(pp.bhi + J);
            const float jl[3] = {jlo.x, jlo.y, jlo.z}, jh[3] = {jhi.x, jhi.y, jhi.z};
            int mlo[3], nm[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (M[a] == 0) {
                    mlo[a] = 0;
                    nm[a] = 1;
                } else {
                    const float N = static_cast<float>(dims[a]);
                    mlo[a] = max(-M[a], static_cast<int>(ceilf((-rcm[a] - (ihi[a] - jl[a])) / N)));
                    const int mhi = min(M[a], static_cast<int>(floorf((rcm[a] - (ilo[a] - jh[a])) / N)));
                    nm[a] = max(0, mhi - mlo[a] + 1);
                }
            }
            const int n_cand = nm[0] * nm[1] * nm[2];
            float4 cjl = make_float4(0.f, 0.f, 0.f, 0.f), cjh = cjl;  // skewed: Cartesian j box
            if (SKEW) {
                cjl = __ldg(pp.clo + J);
                cjh = __ldg(pp.chi + J);
            }
            const bool diag = (J == I);
            bool staged = false;
            // candidate images in chunks of 32, one per lane
            for (int c0 = 0; c0 < n_cand; c0 += 32) {
                const int t = c0 + lane;
                bool ok = false;
                int mm[3] = {0, 0, 0};
                if (t < n_cand) {
                    mm[2] = mlo[2] + t % nm[2];
                    const int t1 = t / nm[2];
                    mm[1] = mlo[1] + t1 % nm[1];
                    mm[0] = mlo[0] + t1 / nm[1];
                    if (SKEW)
                        ok = !use_cut || box_gap2_cart(cil, cih, cjl, cjh, mm, dims, pp.vrow) <= rc2_box;
                    else
                        ok = !use_cut || box_gap2(ilo, ihi, jl, jh, mm, dims, cull) <= rc2_box;
                }
                const unsigned bal = __ballot_sync(0xffffffffu, ok);
                if (bal == 0u) continue;
                __syncwarp();  // earlier reads of simg, sp, sn are done
                if (ok)
                    sw.img[__popc(bal & ((1u << lane) - 1u))] =
                        make_int4(mm[0] * dims[0], mm[1] * dims[1], mm[2] * dims[2], 0);
                if (!staged) {
                    if (lane < jn) {
                        const float4 pj = __ldg(pp.p32 + jb + lane);
                        sw.p[lane] = make_int4(static_cast<int>(pj.x), static_cast<int>(pj.y), static_cast<int>(pj.z), 0);
                        sw.qn[lane] = make_double2(__ldg(pp.q64 + jb + lane), __ldg(pp.n64 + jb + lane));
                    }
                    staged = true;
                }
                __syncwarp();
                const int nimg = __popc(bal);
                // this lane's j point: images that bring the i box within the cutoff
                unsigned jm = 0u;
                if (lane < jn) {
                    const int4 pjl = sw.p[lane];
                    const float px = static_cast<float>(pjl.x), py = static_cast<float>(pjl.y),
                                pz = static_cast<float>(pjl.z);
                    for (int b = 0; b < nimg; ++b) {
                        const int4 sft = sw.img[b];
                        const float sx = static_cast<float>(sft.x), sy = static_cast<float>(sft.y),
                                    sz = static_cast<float>(sft.z);
                        float d2;
                        if (SKEW) {
                            // the point less the shift, in Cartesian coordinates, against the i box
                            const float ux = px - sx, uy = py - sy, uz = pz - sz;
                            const CellRows &vr = pp.vrow;
                            const float q0c = ux * vr.v[0] + uy * vr.v[3] + uz * vr.v[6];
                            const float q1c = ux * vr.v[1] + uy * vr.v[4] + uz * vr.v[7];
                            const float q2c = ux * vr.v[2] + uy * vr.v[5] + uz * vr.v[8];
                            const float gx = fmaxf(0.0f, fmaxf(cil.x - q0c, q0c - cih.x));
                            const float gy = fmaxf(0.0f, fmaxf(cil.y - q1c, q1c - cih.y));
                            const float gz = fmaxf(0.0f, fmaxf(cil.z - q2c, q2c - cih.z));
                            d2 = gx * gx + gy * gy + gz * gz;
                        } else {
                            const float gx = fmaxf(0.0f, fmaxf(ilo[0] + sx - px, px - ihi[0] - sx));
                            const float gy = fmaxf(0.0f, fmaxf(ilo[1] + sy - py, py - ihi[1] - sy));
                            const float gz = fmaxf(0.0f, fmaxf(ilo[2] + sz - pz, pz - ihi[2] - sz));
                            d2 = cull[0] * gx * gx + cull[1] * gy * gy + cull[2] * gz * gz;
                        }
                        if (!use_cut || d2 <= rc2_box) jm |= 1u << b;
                    }
                }
                for (unsigned jset = __ballot_sync(0xffffffffu, jm != 0u); jset != 0u; jset &= jset - 1u) {
                    const int jj = __ffs(jset) - 1;
                    unsigned m = __shfl_sync(0xffffffffu, jm, jj);
                    item_evals += static_cast<unsigned>(__popc(m));
                    const int4 pj = sw.p[jj];
                    const double2 qnj = sw.qn[jj];
                    const double qj = qnj.x, nj = qnj.y;
                    // off the diagonal every pair counts for i and for j; in the diagonal tile j > i
                    // for both, j = i (self-images; the self term is added at the end) for i only
                    const bool both = !diag || jj > lane;
                    const bool lane_ok = act && (both || jj == lane);
                    Delta64 dp;
                    delta_part64<POT>(qi, qj, K, dp);
                    double A = 0.0, Srpt = 0.0, Spu = 0.0, Uf = 0.0, Vf = 0.0;
                    unsigned ins = 0;
                    do {
                        const int4 sft = sw.img[__ffs(m) - 1];
                        m &= m - 1u;
                        double r = pair_r<SKEW>(pp, xi + (sft.x - pj.x), yi + (sft.y - pj.y), zi + (sft.z - pj.z));
                        const bool in = lane_ok && __double2hiint(r) > 0;  // r <= 0: outside, or the self term
                        ins += in ? 1u : 0u;
                        r = in ? r : 0.0;
                        const double tD = r * dp.sqcD;
                        int kc;
                        double t;
                        bool on = cell_of(tD, K.kmax + 1, kc, t);
                        if (__any_sync(0xffffffffu, !on || !poly)) {
                            const bool end = !on && tD == K.tDmax;  // the last node: its cell at t = 1
                            on = on || end;
                            kc = end ? K.kmax : (on ? kc : 0);
                            t = end ? 1.0 : (on ? t : 0.0);
                            if (in && !(on && poly)) {
                                double phi, rd = 0.0, rd2 = 0.0;
                                if (on || !past_part64<POT>(r, tD, qi, qj, K, tb.rho, phi, rd, rd2)) {
                                    // a table too large for polynomials, from its coefficients, or a
                                    // pair past it that past_part64 leaves
                                    Delta<double> dd;
                                    delta_part<POT, double>(qi, qj, K, dd);
                                    dist_part<POT, double>(r, r * r, qi, qj, 1.0 / qi, qi * qi, dd, K, tb, phi, rd, rd2);
                                }
                                A += phi;
                                if (POT) {
                                    Uf += rd;
                                    Vf += rd2;
                                }
                            }
                            if (!poly) continue;
                        }
                        double p, pt, pu;
                        spline64<POT>(poly, sh.S, kc, t, dp, p, pt, pu);
                        A += in && on ? p : 0.0;
                        if (POT) {
                            Srpt = fma(on ? r : 0.0, pt, Srpt);
                            Spu += in && on ? pu : 0.0;
                        }
                    } while (m != 0u);
                    const unsigned wt = both ? 2u : 1u;  // ordered pairs represented
                    cnt += ins * wt;
                    nclamp += dp.cl ? ins * wt : 0u;
                    if (POT) {
                        const double u = fma(Spu, dp.b1, Srpt * K.cD), v = Spu * dp.sb;
                        A64 = fma(nj, A, A64);
                        U64 = fma(nj, u + Uf, U64);
                        const double nb = both ? ni : 0.0;
                        const double tot = warp_sum2(nb * A, nb * ((u - v) - v + Vf), hi);
                        if ((lane & 15) == 0) sw.js[lane >> 4][jj] = tot;
                    } else {
                        A64 = fma(both ? nj + nj : nj, A, A64);
                    }
                }
                if (POT) {
                    __syncwarp();
                    if (jm != 0u) {
                        const double ja = sw.js[0][lane], ju = sw.js[1][lane];
                        if (ja != 0.0) atomicAdd(pp.A + jb + lane, ja);
                        if (ju != 0.0) atomicAdd(pp.U + jb + lane, sw.qn[lane].y * ju);
                    }
                }
            }
        }
        // the self term n_i phi(0, 0) of the i points whose diagonal tile this item holds
        if (act && c == 0) A64 = fma(ni, sh.phi00, A64);
        if (act && POT) {
            if (A64 != 0.0) atomicAdd(pp.A + ig, A64);
            if (U64 != 0.0) atomicAdd(pp.U + ig, ni * U64);
        }
        count_item(pp.stats, act ? cnt : 0u, act ? nclamp : 0u,
                   static_cast<unsigned long long>(item_evals) * static_cast<unsigned long long>(ni_act));
        if (!POT) {
            // the item's energy partial, summed over lanes in a fixed order (items
            // beyond the partials' capacity are added atomically)
            const double e = warp_sum(act ? ni * A64 : 0.0);
            if (lane == 0) {
                if (sh.item_E && item < sh.item_cap)
                    sh.item_E[item] = e;
                else if (e != 0.0)
                    atomicAdd(&pp.stats->E_pair, e);
            }
        }
    }
    }
}

// Cells without images or a cutoff (FP32; see pair_items_f32).
template <int MODE, int NT, bool SKEW>
__global__ void __launch_bounds__(NT, 1) k_pair_open(const __grid_constant__ PairLaunch pl) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned int s_prefix[kMaxInst + 1];
    __shared__ int s_C[kMaxInst];
    Table<float> tb;
    pair_begin<float, NT / 32>(pl, smem_raw, s_prefix, s_C, tb);
    const unsigned int stride = max(1u, pl.sh.item_stride);
    const unsigned int n_items = min((s_prefix[pl.ninst] + stride - 1u) / stride, pl.sh.item_limit);
    pair_items_f32<MODE, NT, SKEW, true>(pl, smem_raw, s_prefix, s_C, n_items, stride, tb);
}

// Per D cell k and delta column l the cubic in t (times 1, as the coefficients / 36 give
// it) through rows k .. k + 3 of the bicubic coefficients: poly[(k S + l) 4 ...].
__global__ void k_table_poly(const double *__restrict__ c, long long n, int S, double *__restrict__ poly) {
    const long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    if (e >= n) return;
    const double c0 = c[e], c1 = c[e + S], c2 = c[e + 2LL * S], c3 = c[e + 3LL * S];
    poly[4 * e] = c0 + 4.0 * c1 + c2;
    poly[4 * e + 1] = 3.0 * (c2 - c0);
    poly[4 * e + 2] = 3.0 * ((c0 - c1) + (c2 - c1));
    poly[4 * e + 3] = (c3 - c0) + 3.0 * (c1 - c2);
}

// The splitmix64 output function (Steele, Lea and Flood, "Fast splittable
// pseudorandom number generators", 2014): a counter-based stream for sampling.
__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

constexpr int kBandSamples = 8;  // samples per thread of k_band_hist

// Sampled histogram of the table's D cell over the evaluations of one problem:
// uniform (i, j, image) triples (image index uniform in [-M_a, M_a] per periodic
// axis), kept where r <= r_cut, binned by the stencil's first row floor(tD);
// evaluations past the table (tD > nD - 1) read no row and are not counted.
// The counts depend only on the sample indices: the result is reproducible.
__global__ void k_band_hist(const __grid_constant__ PairShared sh, const __grid_constant__ PairParams pp,
                            unsigned int *__restrict__ hist, unsigned int salt) {
    __shared__ unsigned int h[kBandBins];
    for (int b = threadIdx.x; b < kBandBins; b += blockDim.x) h[b] = 0u;
    __syncthreads();
    const int na = pp.stats->n_active;
    const int kmax = sh.nD - 2;
    if (na > 0 && kmax < kBandBins) {
        const float h0 = static_cast<float>(pp.h2[0]), h1 = static_cast<float>(pp.h2[1]),
                    h2 = static_cast<float>(pp.h2[2]);
        const float g0 = static_cast<float>(pp.g2x[0]), g1 = static_cast<float>(pp.g2x[1]),
                    g2 = static_cast<float>(pp.g2x[2]);
        const float rc2 = static_cast<float>(pp.rc2), cD = static_cast<float>(sh.cD),
                    tmax = static_cast<float>(sh.nD - 1);
        const unsigned long long t0 =
            (static_cast<unsigned long long>(blockIdx.x) * blockDim.x + threadIdx.x) * kBandSamples;
        for (int s = 0; s < kBandSamples; ++s) {
            const unsigned long long x = mix64((static_cast<unsigned long long>(salt) << 40) + t0 + s);
            const unsigned long long y = mix64(x ^ 0x9e3779b97f4a7c15ull);
            const int i = static_cast<int>((x & 0xffffffffull) % static_cast<unsigned>(na));
            const int j = static_cast<int>((x >> 32) % static_cast<unsigned>(na));
            int m[3];
#pragma unroll
            for (int a = 0; a < 3; ++a)
                m[a] = pp.M[a] > 0 ? static_cast<int>((y >> (21 * a)) % (2u * pp.M[a] + 1u)) - pp.M[a] : 0;
            const float4 pi = __ldg(pp.p32 + i), pj = __ldg(pp.p32 + j);
            const float dx = (pi.x - pj.x) + static_cast<float>(m[0] * pp.dims[0]);
            const float dy = (pi.y - pj.y) + static_cast<float>(m[1] * pp.dims[1]);
            const float dz = (pi.z - pj.z) + static_cast<float>(m[2] * pp.dims[2]);
            const float r2 = h0 * dx * dx + h1 * dy * dy + h2 * dz * dz + g0 * dx * dy + g1 * dx * dz + g2 * dy * dz;
            if (pp.use_cut && r2 > rc2) continue;
            const float t = sqrtf(fmaxf(r2, 0.0f)) * (pi.w + pj.w) * cD;
            if (!(t <= tmax)) continue;
            atomicAdd(&h[min(static_cast<int>(t), kmax)], 1u);
        }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < kBandBins; b += blockDim.x)
        if (h[b]) atomicAdd(hist + b, h[b]);
}

// The band start r0 in [0, nD + 2 - ksn] whose stencils [r0, r0 + ksn - 4] hold the
// most sampled evaluations; among starts within 0.2 % of the total of the best,
// the last (evaluations that miss the band then have small D, where a warp's lanes
// tend to miss together).  The block stages the histogram in shared memory; one
// thread then slides the window over at most kBandBins rows.
__global__ void k_band_choose(const __grid_constant__ PairShared sh, const unsigned int *__restrict__ hist,
                              Stats *out) {
    __shared__ unsigned int h[kBandBins];
    for (int b = threadIdx.x; b < kBandBins; b += blockDim.x) h[b] = hist[b];
    __syncthreads();
    if (threadIdx.x != 0) return;
    const int nk = sh.nD - 1;              // stencil starts 0 .. nD - 2
    const int span = sh.ksn - 3;           // stencil starts a band of ksn rows holds
    const int r0max = sh.nD + 2 - sh.ksn;  // last start that keeps the band in the table
    int choice = 0;
    if (nk <= kBandBins && span > 0 && r0max > 0) {
        unsigned long long total = 0, cov = 0;
        for (int k = 0; k < nk; ++k) total += h[k];
        for (int k = 0; k < min(span, nk); ++k) cov += h[k];
        unsigned long long best = cov, c = cov;
        for (int r0 = 1; r0 <= r0max; ++r0) {
            c -= h[r0 - 1];
            if (r0 + span - 1 < nk) c += h[r0 + span - 1];
            best = c > best ? c : best;
        }
        const unsigned long long tol = total / 500;
        c = cov;
        for (int r0 = 0; r0 <= r0max; ++r0) {
            if (r0 > 0) {
                c -= h[r0 - 1];
                if (r0 + span - 1 < nk) c += h[r0 + span - 1];
            }
            if (c + tol >= best) choice = r0;
        }
    }
    out->band_row0 = choice;
}

// Fixed-order sum of an instance's energy-mode item partials (block k: instance k).
__global__ void k_reduce_items(const __grid_constant__ PairLaunch pl) {
    const int k = blockIdx.x;
    if (k >= pl.ninst) return;
    unsigned int lo = 0;
    for (int t = 0; t < k; ++t)
        lo += static_cast<unsigned int>(pair_items(pl.inst[t].stats->n_active, pl.sh.itile, pl.sh.jpts));
    const unsigned int n = static_cast<unsigned int>(pair_items(pl.inst[k].stats->n_active, pl.sh.itile, pl.sh.jpts));
    const unsigned int hi = min(lo + n, pl.sh.item_cap);
    double s = 0.0;
    for (unsigned int i = lo + threadIdx.x; i < hi; i += blockDim.x) s += pl.sh.item_E[i];
    __shared__ double part[256];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (static_cast<int>(threadIdx.x) < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(&pl.inst[k].stats->E_pair, part[0]);
}

// Voxel-averaged kernel at delta = 0 (the diagonal "phi0" step):
//   phi0(q) = int_{[-1,1]^3} prod_a (1 - |t_a|) phi_0(q |sum_a t_a v_a|) d^3t,
// phi_0(D) the kernel at delta = 0 for D >= D_1 and -(2/pi) ln D + psi0 + c2 D^2
// below (the divergence of eq. 14 at D -> 0 that the table's row 0 softens).
// Block (q, octant): one of the eight sign octants of t times a tensor rule of
// nn nodes (x, w on [0, 1]) per axis.  The integrand is evaluated in FP32 (the
// FP32 table path, errors ~1e-7 relative per term, far below the rule's
// ~1e-5) and summed in FP64; the octant sums are added in a fixed order.
__global__ void k_phi0(const PairShared sh, Phi0Rule rule, const double *__restrict__ q,
                       const double *__restrict__ xw, double *__restrict__ part) {
    Table<float> tb;
    make_table<float>(sh, tb);
    Consts<float> K;
    make_consts<float>(sh, K);
    const int nn = rule.nn;
    const float qq = static_cast<float>(q[blockIdx.x]);
    const int sg = blockIdx.y;
    const float s0 = (sg & 1) ? -1.0f : 1.0f, s1 = (sg & 2) ? -1.0f : 1.0f, s2 = (sg & 4) ? -1.0f : 1.0f;
    float v[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) v[k] = static_cast<float>(rule.v[k]);
    const float D1 = static_cast<float>(rule.D1), psi0 = static_cast<float>(rule.psi0),
                c2 = static_cast<float>(rule.c2);
    const int total = nn * nn * nn;
    double acc = 0.0;
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
        const int i = e / (nn * nn), j = (e / nn) % nn, k = e % nn;
        const float t0 = s0 * static_cast<float>(xw[i]), t1 = s1 * static_cast<float>(xw[j]),
                    t2 = s2 * static_cast<float>(xw[k]);
        const float r0 = t0 * v[0] + t1 * v[3] + t2 * v[6];
        const float r1 = t0 * v[1] + t1 * v[4] + t2 * v[7];
        const float r2 = t0 * v[2] + t1 * v[5] + t2 * v[8];
        const float D = qq * sqrtf(r0 * r0 + r1 * r1 + r2 * r2);
        float phi;
        if (D < D1) {
            phi = -0.63661977236758134f * logf(D) + psi0 + c2 * D * D;
        } else {
            float rd = 0.0f, rd2 = 0.0f;
            unsigned ncl = 0;
            pair_phi<false, float>(D * D, 1.0f, 1.0f, 1.0f, 1.0f, K, tb, phi, rd, rd2, ncl);
        }
        const double wt = xw[nn + i] * xw[nn + j] * xw[nn + k] * (1.0 - xw[i]) * (1.0 - xw[j]) * (1.0 - xw[k]);
        acc += wt * static_cast<double>(phi);
    }
    __shared__ double red[256];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (static_cast<int>(threadIdx.x) < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x * 8 + blockIdx.y] = red[0];
}

__global__ void k_phi0_sum(const double *__restrict__ part, int nq, double *__restrict__ out) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nq; t += gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int o = 0; o < 8; ++o) s += part[t * 8 + o];
        out[t] = s;
    }
}

// The kernel at given (r, q_i, q_j), for isolated checks of the interpolation.
template <typename R>
__global__ void k_kernel_eval(const PairShared sh, int64_t npts, const double *r,
                              const double *qi, const double *qj, double *phi, double *rd) {
    Table<R> tb;
    make_table<R>(sh, tb);
    Consts<R> K;
    make_consts<R>(sh, K);
    for (int64_t p = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; p < npts;
         p += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const R rr = static_cast<R>(r[p]);
        const R a = static_cast<R>(qi[p]), b = static_cast<R>(qj[p]);
        R ph, rdv = 0, rd2 = 0;
        unsigned ncl = 0;
        pair_phi<true, R>(rr * rr, a, b, R(1) / a, a * a, K, tb, ph, rdv, rd2, ncl);
        phi[p] = static_cast<double>(ph);
        rd[p] = static_cast<double>(rdv);
    }
}

template <typename R, int MODE, int NT, bool SKEW, bool OPEN = false>
int launch_one(const PairLaunch &pl, int nctas, size_t smem, cudaStream_t st) {
    void (*kern)(PairLaunch) = nullptr;
    if constexpr (OPEN)
        kern = k_pair_open<MODE, NT, SKEW>;
    else
        kern = k_pair<R, MODE, NT, SKEW>;
    VDWDF_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        static_cast<int>(smem)));
    kern<<<nctas, NT, smem, st>>>(pl);
    count_launches(1);
    VDWDF_CUDA_TRY(cudaGetLastError());
    return VDWDF_OK;
}

template <typename R, int MODE>
int launch_nt(int threads, bool skew, const PairLaunch &pl, int nctas, size_t smem, cudaStream_t st) {
    if constexpr (sizeof(R) == 4) {
        // cells with neither images nor a cutoff: the instance without either (13-17 %
        // faster, see pair_items_f32), at the default's threads and, so that a tuned shape
        // can have it as well, at 512 on orthogonal cells (binding curve with the shape tuned
        // on the batch 72.6 -> 57.7 ms, default 54.8)
        bool open = threads == 640 || (threads == 512 && !skew);
        for (int k = 0; k < pl.ninst; ++k) {
            const PairParams &p = pl.inst[k];
            open = open && !p.use_cut && p.M[0] == 0 && p.M[1] == 0 && p.M[2] == 0;
        }
        if (open && threads == 512) return launch_one<R, MODE, 512, false, true>(pl, nctas, smem, st);
        if (open)
            return skew ? launch_one<R, MODE, 640, true, true>(pl, nctas, smem, st)
                        : launch_one<R, MODE, 640, false, true>(pl, nctas, smem, st);
        if (threads == 640)
            return skew ? launch_one<R, MODE, 640, true>(pl, nctas, smem, st)
                        : launch_one<R, MODE, 640, false>(pl, nctas, smem, st);
    }
    if (skew) {
        if (threads == 448) return launch_one<R, MODE, 448, true>(pl, nctas, smem, st);
        return threads == 384 ? launch_one<R, MODE, 384, true>(pl, nctas, smem, st)
                              : launch_one<R, MODE, 512, true>(pl, nctas, smem, st);
    }
    switch (threads) {
        case 256: return launch_one<R, MODE, 256, false>(pl, nctas, smem, st);
        case 384: return launch_one<R, MODE, 384, false>(pl, nctas, smem, st);
        case 448: return launch_one<R, MODE, 448, false>(pl, nctas, smem, st);
        case 1024: return launch_one<R, MODE, 1024, false>(pl, nctas, smem, st);
        default: return launch_one<R, MODE, 512, false>(pl, nctas, smem, st);
    }
}

}  // namespace

int pair_smem_bytes(int precision, int threads, int ksn, int S) {
    // per warp: j tile (points, densities) and image shifts; FP32: the table band
    const size_t warp = precision == VDWDF_FP64 ? sizeof(Warp64) : sizeof(Warp32);
    size_t b = warp * static_cast<size_t>(threads / 32);
    if (precision != VDWDF_FP64) b += static_cast<size_t>(ksn) * band_stride(S) * sizeof(float);
    return static_cast<int>(b);
}

// The displacement table of an instance into rt.
static int launch_r_table(const PairParams &pp, bool skew, double *rt, cudaStream_t st) {
    const long long n = r_table_entries(pp.rtm, skew);
    const int nb = static_cast<int>(n < (1LL << 18) ? (n + 255) / 256 : 1024);
    if (skew)
        k_r_table<true><<<nb, 256, 0, st>>>(pp, rt);
    else
        k_r_table<false><<<nb, 256, 0, st>>>(pp, rt);
    count_launches(1);
    VDWDF_CUDA_TRY(cudaGetLastError());
    return VDWDF_OK;
}

int launch_pair(int precision, bool potential, bool skew, int threads, const PairLaunch &pl, int nctas,
                cudaStream_t st) {
    if (skew && threads != 640 && threads != 512 && threads != 448 && threads != 384) return VDWDF_EINVAL;  // skewed: 384, 448, 512
    const size_t smem = static_cast<size_t>(pair_smem_bytes(precision, threads, pl.sh.ksn, pl.sh.S));
    if (precision == VDWDF_FP64)
        for (int k = 0; k < pl.ninst; ++k)
            if (pl.inst[k].rt) {
                const int rc = launch_r_table(pl.inst[k], skew, const_cast<double *>(pl.inst[k].rt), st);
                if (rc) return rc;
            }
    if (precision == VDWDF_FP64)
        return potential ? launch_nt<double, 1>(threads, skew, pl, nctas, smem, st)
                         : launch_nt<double, 0>(threads, skew, pl, nctas, smem, st);
    return potential ? launch_nt<float, 1>(threads, skew, pl, nctas, smem, st)
                     : launch_nt<float, 0>(threads, skew, pl, nctas, smem, st);
}

int launch_table_poly(const double *coef, int nD, int S, double *poly) {
    const long long n = static_cast<long long>(nD - 1) * S;
    k_table_poly<<<static_cast<int>((n + 255) / 256), 256>>>(coef, n, S, poly);
    VDWDF_CUDA_TRY(cudaGetLastError());
    return VDWDF_OK;
}

int launch_band_choose(const PairLaunch &pl, unsigned int *hist, cudaStream_t st) {
    VDWDF_CUDA_TRY(cudaMemsetAsync(hist, 0, sizeof(unsigned int) * kBandBins, st));
    int dev = 0, sms = 0;
    VDWDF_CUDA_TRY(cudaGetDevice(&dev));
    VDWDF_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    for (int k = 0; k < pl.ninst; ++k)
        k_band_hist<<<2 * (sms > 0 ? sms : 1), 256, 0, st>>>(pl.sh, pl.inst[k], hist, static_cast<unsigned>(k));
    k_band_choose<<<1, 256, 0, st>>>(pl.sh, hist, pl.inst[0].stats);
    count_launches(pl.ninst + 1);
    VDWDF_CUDA_TRY(cudaGetLastError());
    return VDWDF_OK;
}

int launch_reduce_items(const PairLaunch &pl, cudaStream_t st) {
    if (!pl.sh.item_E) return VDWDF_OK;
    k_reduce_items<<<pl.ninst, 256, 0, st>>>(pl);
    count_launches(1);
    VDWDF_CUDA_TRY(cudaGetLastError());
    return VDWDF_OK;
}

int launch_phi0(const PairShared &sh, const Phi0Rule &rule, int nq, const double *q, const double *xw,
                double *part, double *out, cudaStream_t st) {
    if (nq <= 0) return VDWDF_OK;
    k_phi0<<<dim3(nq, 8), 256, 0, st>>>(sh, rule, q, xw, part);
    k_phi0_sum<<<(nq + 255) / 256, 256, 0, st>>>(part, nq, out);
    count_launches(2);
    VDWDF_CUDA_TRY(cudaGetLastError());
    return VDWDF_OK;
}

int launch_kernel_eval(int precision, const PairShared &sh, int64_t npts, const double *r,
                       const double *qi, const double *qj, double *phi, double *rdphi,
                       cudaStream_t st) {
    const int bs = 256;
    int64_t nb = (npts + bs - 1) / bs;
    if (nb > 65535) nb = 65535;
    if (nb < 1) nb = 1;
    if (precision == VDWDF_FP64)
        k_kernel_eval<double><<<static_cast<int>(nb), bs, 0, st>>>(sh, npts, r, qi, qj, phi, rdphi);
    else
        k_kernel_eval<float><<<static_cast<int>(nb), bs, 0, st>>>(sh, npts, r, qi, qj, phi, rdphi);
    count_launches(1);
    VDWDF_CUDA_TRY(cudaGetLastError());
    return VDWDF_OK;
}

}  // namespace vdwdf
