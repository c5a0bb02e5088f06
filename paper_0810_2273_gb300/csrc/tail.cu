// Far field past the pair cutoff from the kernel's asymptote alone (the paper's
// section 7 names image sums sped up by the asymptotic form as future work;
// sections 3 and 6.2 repeat the cell until the energy converges).
//
// Every pair beyond r_cut takes eq. (17), phi17 = -C / (u_i u_j (u_i + u_j) r^6)
// with u = q0^2, and the lattice images beyond r_cut are replaced by the
// lattice's continuum.  Per pair of points that gives
//   K_ij = (2 pi / A) / (4 max(r_cut, |z_ij|)^4)   (two periodic axes, area A,
//          z_ij the separation normal to the periodic plane),
//   K    = (4 pi / V) / (3 r_cut^3)                 (three periodic axes),
// and the tail T = 1/2 dV^2 sum_ij n_i n_j (-C / (u_i u_j (u_i + u_j))) K_ij.
//
// On the grid, z depends only on the plane of the non-periodic axis, and
// 1/(u_i + u_j) = int_0^inf exp(-(u_i + u_j) s) ds separates i from j.  With
// s = e^x and the trapezoidal rule in x (step hx = ln 2 / 3; the integrand is analytic
// in the strip |Im x| < pi/2, so the error falls like exp(-pi^2 / hx)),
//   T = -1/2 dV^2 C sum_k hx s_k sum_{p, p'} K(p, p') F_k(p) F_k(p'),
//   F_k(p) = sum over active points of plane p of (n / u) exp(-u s_k).
// That is O(N_grid) work for the planes and O(planes^2) for the pairs of planes,
// instead of O(N_active^2).  Its potential (the derivative of T with the active mask
// frozen) comes from the same sums, point by point (k_tail_AU), in the pair sum's
// adjoint form.
//
// Few exponentials: FP64 ones were all of the time (165 per point and pass).
// - Nodes with u_max s_k <= 1/16 (three quarters of them) need none: there
//   exp(-u s) is its Taylor polynomial of degree 8 (3e-17), so F_k is a combination of
//   the nine moments M_j = sum (n / u) (u / u_max)^j, and K acts on the moments.
// - The others come in three runs of doubling s (s_{k+3} = 2 s_k): one exponential
//   starts a run, the rest are squares, carried as 1 - exp(-x) while that is small.
// Bound by the FP64 pipe still.  ms per call before -> after (with the potential):
// monolayer 48 x 84 x 120 2.27 (5.28) -> 0.61 (1.28), the same with three periodic
// axes, whose one plane now has many blocks, 36.0 -> 0.79, chain 24 x 72 x 72 with its
// product of lines over 76 rows instead of 176 nodes 7.84 (8.88) -> 3.93 (4.20).
//
// One periodic axis a (length |a|): the images of a pair lie on a line, and
// their continuum beyond r_cut gives
//   K_ij = (2 / |a|) I(rho_ij, x0),  I(rho, x0) = int_{x0}^inf dx / (rho^2 + x^2)^3,
// rho_ij the distance of r_i - r_j from the axis direction and
// x0 = sqrt(max(0, r_cut^2 - rho^2)).  rho depends only on the grid lines along
// a that hold i and j, so the lines take the place of the planes: F_k per
// line with an active point, K as a table over the lines' index differences
// (k_tail_line_Ktab), G_k = K F_k as a tiled FP64 product (k_tail_line_G).
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"

namespace vdwdf {

namespace {

constexpr int kRun = 20;           // nodes of a run per block column of the sums
constexpr int kTailThreads = 256;
constexpr int kMom = kTailMoments;

constexpr double kTailPi = 3.14159265358979323846;

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Grid index of the t-th point of plane p (the points whose index along axis
// `ax` is p); one plane holding every point when np == 1.
__device__ __forceinline__ long long plane_point(int d0, int d1, int d2, int ax, int np, int p, long long t) {
    if (np == 1) return t;
    if (ax == 0) return static_cast<long long>(p) * d1 * d2 + t;
    if (ax == 1) return (t / d2 * d1 + p) * static_cast<long long>(d2) + t % d2;
    return t * d2 + p;
}

// exp(-x) along a run of doublings: e = exp(-x), f = 1 - e to full relative accuracy
// while f < 1/2 (squaring e there would lose it), then frozen.
__device__ __forceinline__ void run_start(double x, double &f, double &e) {
    if (x < 0.7) {
        f = -expm1(-x);
        e = 1.0 - f;
    } else {
        f = 1.0;
        e = exp(-x);
    }
}
__device__ __forceinline__ void run_double(double &f, double &e) {
    const bool small = __double2hiint(f) < 0x3FE00000;  // f < 1/2
    const double f2 = fma(-f, f, f + f), ea = 1.0 - f2, eb = e * e;
    e = small ? ea : eb;
    f = small ? f2 : f;
}

// Columns of the sums: column 0 the moments, then run r = (col - 1) % 3, doublings
// from kRun ((col - 1) / 3) on.  Adds one point's terms (u = q0^2, a = n / u).
__device__ __forceinline__ void tail_add(int col, const TailNodes &q, double s0, double u, double a, double acc[kRun]) {
    if (col == 0) {
        const double x = u * q.iumax;
#pragma unroll
        for (int j = 0; j < kMom; ++j) {
            acc[j] += a;
            a *= x;
        }
        return;
    }
    double f, e;
    run_start(u * s0, f, e);
#pragma unroll
    for (int j = 0; j < kRun; ++j) {
        acc[j] = fma(a, e, acc[j]);
        run_double(f, e);
    }
}
// s of a column's first node, and the row of F of its entry j (below 0: none).
__device__ __forceinline__ double tail_s0(int col, const TailNodes &q) {
    return col == 0 ? 0.0 : ldexp(q.s[(col - 1) % 3], kRun * ((col - 1) / 3));
}
__device__ __forceinline__ int tail_row(int col, int j, const TailNodes &q) {
    if (col == 0) return j < kMom ? j : -1;
    const int k = (col - 1) % 3 + 3 * (kRun * ((col - 1) / 3) + j);
    return k < q.nb ? kMom + k : -1;
}

// F[row * np + p] of column blockIdx.y, for the blockIdx.z-th part of the points of
// plane p = blockIdx.x (parts are then added in order): threads stride the points,
// then warp and block trees, all in a fixed order.
__global__ void __launch_bounds__(kTailThreads) k_tail_planes(int d0, int d1, int d2, int ax, int np,
                                                              const double *__restrict__ n,
                                                              const double *__restrict__ q0, double n_cut,
                                                              const __grid_constant__ TailNodes q,
                                                              double *__restrict__ F) {
    __shared__ double red[kTailThreads / 32][kRun];
    const int p = blockIdx.x, col = blockIdx.y;
    const double s0 = tail_s0(col, q);
    const long long per_plane = (np == 1) ? static_cast<long long>(d0) * d1 * d2
                                          : static_cast<long long>(d0) * d1 * d2 / np;
    double acc[kRun];
#pragma unroll
    for (int c = 0; c < kRun; ++c) acc[c] = 0.0;
    for (long long t = blockIdx.z * static_cast<long long>(blockDim.x) + threadIdx.x; t < per_plane;
         t += static_cast<long long>(gridDim.z) * blockDim.x) {
        const long long m = plane_point(d0, d1, d2, ax, np, p, t);
        const double nm = n[m];
        if (!(nm >= n_cut)) continue;  // inactive (NaN as well)
        const double u = q0[m] * q0[m];
        tail_add(col, q, s0, u, nm / u, acc);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < kRun; ++c) {
        const double v = warp_sum_d(acc[c]);
        if (lane == 0) red[warp][c] = v;
    }
    __syncthreads();
    const int row = threadIdx.x < kRun ? tail_row(col, static_cast<int>(threadIdx.x), q) : -1;
    if (row >= 0) {
        double s = 0.0;
        for (int w = 0; w < kTailThreads / 32; ++w) s += red[w][threadIdx.x];
        F[(static_cast<long long>(blockIdx.z) * (kMom + q.nb) + row) * np + p] = s;
    }
}

// F[e] += the parts' sums, in order (parts of n values one after the other).
__global__ void k_tail_fold(long long n, int parts, double *__restrict__ F) {
    for (long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; e < n;
         e += static_cast<long long>(gridDim.x) * blockDim.x) {
        double s = F[e];
        for (int z = 1; z < parts; ++z) s += F[z * n + e];
        F[e] = s;
    }
}

// G[r * np + p] = sum_{p'} K(p, p') F[r * np + p'] for row r = blockIdx.x, with
// K(p, p') = c2 / max(rc, |p - p'| dz)^4 (two periodic axes) or c3 (three).  K by |p - p'|
// and the row of F stand in shared memory (sh) when they fit.
__global__ void __launch_bounds__(kTailThreads) k_tail_pairs(int np, const double *__restrict__ F, double dz,
                                                             double rc, double c2, double c3, int sh,
                                                             double *__restrict__ G) {
    extern __shared__ double sm[];
    const double *f = F + static_cast<long long>(blockIdx.x) * np;
    auto kern = [&](int d) {
        if (np == 1) return c3;
        const double z = d * dz, R = z > rc ? z : rc, R2 = R * R;
        return c2 / (R2 * R2);
    };
    if (sh) {
        for (int p = threadIdx.x; p < np; p += blockDim.x) {
            sm[p] = kern(p);
            sm[np + p] = f[p];
        }
        __syncthreads();
    }
    for (int p = threadIdx.x; p < np; p += blockDim.x) {
        double row = 0.0;
        for (int pp = 0; pp < np; ++pp) {
            const int d = p > pp ? p - pp : pp - p;
            row += sh ? sm[d] * sm[np + pp] : kern(d) * f[pp];
        }
        G[static_cast<long long>(blockIdx.x) * np + p] = row;
    }
}

// Dot products over the groups: block b < nb that of node b's rows of F and G, then
// the kMom x kMom products of the moments' rows.  One block each, fixed order.
__global__ void __launch_bounds__(kTailThreads) k_tail_dots(int ng, int nb, const double *__restrict__ F,
                                                            const double *__restrict__ G, double *__restrict__ dots) {
    __shared__ double red[kTailThreads / 32];
    const int b = blockIdx.x;
    const long long rf = b < nb ? kMom + b : (b - nb) / kMom, rg = b < nb ? kMom + b : (b - nb) % kMom;
    double acc = 0.0;
    for (int a = threadIdx.x; a < ng; a += blockDim.x) acc += F[rf * ng + a] * G[rg * ng + a];
    acc = warp_sum_d(acc);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kTailThreads / 32; ++w) s += red[w];
        dots[b] = s;
    }
}

__device__ __forceinline__ double sign_over_factorial(int j) {
    double v = 1.0;
    for (int i = 2; i <= j; ++i) v *= i;
    return ((j & 1) ? -1.0 : 1.0) / v;
}

// out = scale sum_k hx s_k F_k . G_k: the nodes' products in order, and for the nodes
// of the Taylor polynomial sum_{j, j'} (-1)^{j + j'} / (j! j'!) W_{j + j'} M_j . K M_j'.
__global__ void k_tail_final(const __grid_constant__ TailNodes q, const double *__restrict__ dots, double scale,
                             double *__restrict__ out) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double s = 0.0;
    for (int j = 0; j < kMom; ++j)
        for (int i = 0; i < kMom; ++i)
            s += sign_over_factorial(j) * sign_over_factorial(i) * q.W[j + i] * dots[q.nb + j * kMom + i];
    for (int k = 0; k < q.nb; ++k) s += q.hx * ldexp(q.s[k % 3], k / 3) * dots[k];
    *out = scale * s;
}

// Per group p the Taylor nodes' part of S0 and S1 (k_tail_AU) as polynomials in
// x = u / u_max: coef[j * ng + p] and coef[(kMom + j) * ng + p].
__global__ void k_tail_coef(int ng, const __grid_constant__ TailNodes q, const double *__restrict__ G,
                            double *__restrict__ coef) {
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < ng; p += gridDim.x * blockDim.x)
        for (int j = 0; j < kMom; ++j) {
            double c0 = 0.0, c1 = 0.0;
            for (int i = 0; i < kMom; ++i) {
                const double g = sign_over_factorial(i) * G[static_cast<long long>(i) * ng + p];
                c0 += q.W[j + i] * g;
                c1 += q.W[j + i + 1] * g;
            }
            coef[static_cast<long long>(j) * ng + p] = sign_over_factorial(j) * c0;
            coef[static_cast<long long>(kMom + j) * ng + p] = sign_over_factorial(j) * c1 * q.iumax;
        }
}

// The far field's potential in the pair sum's adjoint form, per grid point m:
// with S0 = sum_k hx s_k e^{-u s_k} G_k(p) and S1 = sum_k hx s_k^2 e^{-u s_k} G_k(p)
// (u = q0_m^2, p the plane of m),
//   sum_j n_j f(u, u_j) K_mj = S0 / u,   sum_j n_j df/du K_mj = -S0 / u^2 - S1 / u,
// f(a, b) = 1 / (a b (a + b)), since 1/(a + b) and 1/(a + b)^2 are the integrals of
// e^{-(a + b) s} and s e^{-(a + b) s}.  A = -C S0 / u and U = -2 C n q (-S0/u^2 - S1/u)
// at active points (slot[m] = m), slot[m] = -1 elsewhere.
__global__ void __launch_bounds__(kTailThreads) k_tail_AU(int d0, int d1, int d2, int ax, int np,
                                                          const int *__restrict__ line_slot,
                                                          const double *__restrict__ n,
                                                          const double *__restrict__ q0, double n_cut,
                                                          const __grid_constant__ TailNodes q,
                                                          const double *__restrict__ G,
                                                          const double *__restrict__ coef, double C,
                                                          int *__restrict__ slot, double *__restrict__ A,
                                                          double *__restrict__ U) {
    const long long N = static_cast<long long>(d0) * d1 * d2;
    for (long long m = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; m < N;
         m += static_cast<long long>(gridDim.x) * blockDim.x) {
        const double nm = n[m];
        if (!(nm >= n_cut)) {
            slot[m] = -1;
            continue;
        }
        int p = 0;
        const long long c2i = m % d2, c1i = (m / d2) % d1, c0i = m / (static_cast<long long>(d1) * d2);
        if (line_slot) {
            // one periodic axis: the active line of m
            const long long ib = ax == 0 ? c1i : c0i, ic = ax == 2 ? c1i : c2i;
            p = line_slot[ib * (ax == 2 ? d1 : d2) + ic];
        } else if (np > 1) {
            p = static_cast<int>(ax == 0 ? c0i : (ax == 1 ? c1i : c2i));
        }
        const double qm = q0[m], u = qm * qm, x = u * q.iumax;
        double S0 = 0.0, S1 = 0.0;
#pragma unroll
        for (int j = kMom - 1; j >= 0; --j) {
            S0 = fma(S0, x, coef[static_cast<long long>(j) * np + p]);
            S1 = fma(S1, x, coef[static_cast<long long>(kMom + j) * np + p]);
        }
        for (int r = 0; r < 3; ++r) {
            double s = q.s[r], f, e;
            run_start(u * s, f, e);
            for (int k = r; k < q.nb; k += 3) {
                const double t = (q.hx * s) * (e * G[static_cast<long long>(kMom + k) * np + p]);
                S0 += t;
                S1 = fma(s, t, S1);
                s += s;
                run_double(f, e);
            }
        }
        slot[m] = static_cast<int>(m);
        const double iu = 1.0 / u;
        A[m] = -C * S0 * iu;
        U[m] = 2.0 * C * nm * qm * (S0 * iu + S1) * iu;
    }
}

// ---------------------------------------------------------------------------
// one periodic axis: lines along it
// ---------------------------------------------------------------------------

// The grid index of the t-th point of line (ib, ic) along ax.
__device__ __forceinline__ long long line_point(int d1, int d2, int ax, int ib, int ic, long long t) {
    if (ax == 0) return (t * d1 + ib) * static_cast<long long>(d2) + ic;
    if (ax == 1) return (static_cast<long long>(ib) * d1 + t) * d2 + ic;
    return (static_cast<long long>(ib) * d1 + ic) * d2 + t;
}

// The line (ib * N_c + ic) of grid point m.
__device__ __forceinline__ long long line_of(int d1, int d2, int ax, long long m) {
    const long long i2 = m % d2, i1 = (m / d2) % d1, i0 = m / (static_cast<long long>(d1) * d2);
    const long long ib = ax == 0 ? i1 : i0, ic = ax == 2 ? i1 : i2;
    return ib * (ax == 2 ? d1 : d2) + ic;
}

// flags[line] = 1 where the line holds an active point (the line of grid point m
// is ib * Nc + ic).
__global__ void k_tail_line_flags(int d0, int d1, int d2, int ax, const double *__restrict__ n, double n_cut,
                                  int *__restrict__ flags) {
    const long long N = static_cast<long long>(d0) * d1 * d2;
    for (long long m = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; m < N;
         m += static_cast<long long>(gridDim.x) * blockDim.x) {
        if (!(n[m] >= n_cut)) continue;
        flags[line_of(d1, d2, ax, m)] = 1;
    }
}

// F[row * La + a] over the active points of line lines[a]: one warp per line and
// column blockIdx.y (see tail_add), sums in a fixed order.
__global__ void __launch_bounds__(kTailThreads) k_tail_line_F(int d0, int d1, int d2, int ax, int La,
                                                              const int *__restrict__ lines,
                                                              const double *__restrict__ n,
                                                              const double *__restrict__ q0, double n_cut,
                                                              const __grid_constant__ TailNodes q,
                                                              double *__restrict__ F) {
    const int lane = threadIdx.x & 31, col = blockIdx.y;
    const int a = blockIdx.x * (kTailThreads / 32) + (threadIdx.x >> 5);
    if (a >= La) return;
    const double s0 = tail_s0(col, q);
    const int Nc = ax == 2 ? d1 : d2, len = ax == 0 ? d0 : (ax == 1 ? d1 : d2);
    const int l = lines[a], ib = l / Nc, ic = l % Nc;
    double acc[kRun];
#pragma unroll
    for (int c = 0; c < kRun; ++c) acc[c] = 0.0;
    for (int t = lane; t < len; t += 32) {
        const long long m = line_point(d1, d2, ax, ib, ic, t);
        const double nm = n[m];
        if (!(nm >= n_cut)) continue;
        const double u = q0[m] * q0[m];
        tail_add(col, q, s0, u, nm / u, acc);
    }
#pragma unroll
    for (int c = 0; c < kRun; ++c) {
        const double v = warp_sum_d(acc[c]);
        const int row = tail_row(col, c, q);
        if (lane == 0 && row >= 0) F[static_cast<long long>(row) * La + a] = v;
    }
}

// I(rho, x0) = int_{x0}^inf dx / (rho^2 + x^2)^3.  x0 = 0: 3 pi / (16 rho^5).  For
// e = rho / x0 < 1/2, x0^-5 sum_k (-1)^k (k+1)(k+2)/2 e^2k / (2k + 5) (the binomial
// series of (1 + e^2/t^2)^-3 integrated over t >= 1); otherwise the closed form
// 3 atan(rho / x0) / (8 rho^5) - x0 / (4 rho^2 s^2) - 3 x0 / (8 rho^4 s), s = rho^2 + x0^2.
__device__ double line_tail_I(double rho, double x0) {
    if (!(x0 > 0.0)) {
        const double r2 = rho * rho;
        return 3.0 * kTailPi / (16.0 * r2 * r2 * rho);
    }
    const double e = rho / x0;
    if (e < 0.5) {
        const double e2 = e * e;
        double sum = 0.0, p = 1.0;
        for (int k = 0; k < 80; ++k) {
            const double term = 0.5 * (k + 1.0) * (k + 2.0) * p / (2.0 * k + 5.0);
            sum += (k & 1) ? -term : term;
            if (term < 1e-19) break;
            p *= e2;
        }
        const double x2 = x0 * x0;
        return sum / (x2 * x2 * x0);
    }
    const double r2 = rho * rho, s = r2 + x0 * x0;
    return 3.0 * atan(e) / (8.0 * r2 * r2 * rho) - x0 / (4.0 * r2 * s * s) - 3.0 * x0 / (8.0 * r2 * r2 * s);
}

// Kt[db * (2 N_c - 1) + dc + N_c - 1] = K between two lines whose index differences
// are (db, dc), 0 <= db < N_b, |dc| < N_c: the squared distance through the metric
// (gbb, gbc, gcc) of the axis steps with their components along the periodic axis
// removed.  K depends on the lines only through (db, dc), and K(-db, -dc) = K(db, dc).
__global__ void k_tail_line_Ktab(int Nb, int Nc, double gbb, double gbc, double gcc, double rc, double pref,
                                 double *__restrict__ Kt) {
    const int W = 2 * Nc - 1;
    const long long total = static_cast<long long>(Nb) * W;
    for (long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; e < total;
         e += static_cast<long long>(gridDim.x) * blockDim.x) {
        const double db = static_cast<double>(e / W), dc = static_cast<double>(e % W - (Nc - 1));
        double p2 = gbb * db * db + 2.0 * gbc * db * dc + gcc * dc * dc;
        p2 = p2 > 0.0 ? p2 : 0.0;
        // x0 = sqrt(rc^2 - rho^2) is singular at rho = rc, where lattice-aligned line
        // pairs sit exactly: a difference within 1e-12 rc^2 of zero counts as zero
        // (as the pair sum's inclusive cutoff), so rounding does not decide them
        const double x2 = rc * rc - p2;
        Kt[e] = pref * line_tail_I(sqrt(p2), x2 > 1e-12 * rc * rc ? sqrt(x2) : 0.0);
    }
}

// G[k * La + i] = sum_a K(lines[i], lines[a]) F[k * La + a] for every active line i
// and row k (moment or node): a 32 x 32 output tile per block of 16 x 16 threads (2 x 2 each), the a
// range in shared-memory tiles of 32, K from the table Kt, summed in a fixed order.
constexpr int kGT = 32;
__global__ void __launch_bounds__(256) k_tail_line_G(int La, int nodes, const int *__restrict__ lines, int Nc,
                                                     const double *__restrict__ Kt, const double *__restrict__ F,
                                                     double *__restrict__ G) {
    __shared__ double sK[kGT][kGT + 1], sF[kGT][kGT + 1];
    __shared__ int rb[kGT], rcl[kGT];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int i0 = blockIdx.x * kGT, k0 = blockIdx.y * kGT;
    const int W = 2 * Nc - 1;
    if (threadIdx.x < kGT) {
        const int l = (i0 + threadIdx.x < La) ? lines[i0 + threadIdx.x] : 0;
        rb[threadIdx.x] = l / Nc;
        rcl[threadIdx.x] = l % Nc;
    }
    double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
    for (int a0 = 0; a0 < La; a0 += kGT) {
        __syncthreads();  // rb, rcl written; the previous tiles read
        for (int e = threadIdx.x; e < kGT * kGT; e += 256) {
            const int r = e / kGT, cc = e % kGT;
            const int i = i0 + r, k = k0 + r, a = a0 + cc;
            double kv = 0.0;
            if (i < La && a < La) {
                const int l2 = lines[a];
                int db = rb[r] - l2 / Nc, dc = rcl[r] - l2 % Nc;
                if (db < 0) {
                    db = -db;
                    dc = -dc;
                }
                kv = Kt[static_cast<long long>(db) * W + dc + Nc - 1];
            }
            sK[r][cc] = kv;
            sF[r][cc] = (k < nodes && a < La) ? F[static_cast<long long>(k) * La + a] : 0.0;
        }
        __syncthreads();
#pragma unroll 8
        for (int j = 0; j < kGT; ++j) {
            const double k_0 = sK[ty][j], k_1 = sK[ty + 16][j];
            const double f_0 = sF[tx][j], f_1 = sF[tx + 16][j];
            acc[0][0] += k_0 * f_0;
            acc[0][1] += k_0 * f_1;
            acc[1][0] += k_1 * f_0;
            acc[1][1] += k_1 * f_1;
        }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const int i = i0 + ty + 16 * u, k = k0 + tx + 16 * v;
            if (i < La && k < nodes) G[static_cast<long long>(k) * La + i] = acc[u][v];
        }
}

}  // namespace

int launch_far_tail_line_flags(const int dims[3], int ax, const double *n, double n_cut, int *flags,
                               cudaStream_t st) {
    const long long N = static_cast<long long>(dims[0]) * dims[1] * dims[2];
    long long nb = (N + kTailThreads - 1) / kTailThreads;
    if (nb > 152 * 16) nb = 152 * 16;
    k_tail_line_flags<<<static_cast<int>(nb), kTailThreads, 0, st>>>(dims[0], dims[1], dims[2], ax, n, n_cut, flags);
    count_launches(1);
    VDWDF_CUDA_TRY(cudaGetLastError());
    return VDWDF_OK;
}

// Columns of the sums that hold the moments and every node.
static int tail_columns(const TailNodes &q) { return 1 + 3 * ((q.nb + 3 * kRun - 1) / (3 * kRun)); }

static int tail_finish(int ng, const TailNodes &q, const double *F, const double *G, double scale, double *dots,
                       double *out, cudaStream_t st) {
    k_tail_dots<<<q.nb + kMom * kMom, kTailThreads, 0, st>>>(ng, q.nb, F, G, dots);
    k_tail_final<<<1, 32, 0, st>>>(q, dots, scale, out);
    count_launches(2);
    VDWDF_CUDA_TRY(cudaGetLastError());
    return VDWDF_OK;
}

int launch_far_tail_lines(const int dims[3], int ax, int La, const int *lines, const double *n, const double *q0,
                          double n_cut, const TailNodes &q, double gbb, double gbc, double gcc, double rc, double pref,
                          double scale, double *F, double *Kt, double *G, double *dots, double *out,
                          cudaStream_t st) {
    // lines are ib * N_c + ic, b < c the other two axes
    const int Nb = ax == 0 ? dims[1] : dims[0], Nc = ax == 2 ? dims[1] : dims[2];
    const int wpb = kTailThreads / 32, rows = kMom + q.nb;
    k_tail_line_F<<<dim3((La + wpb - 1) / wpb, tail_columns(q)), kTailThreads, 0, st>>>(dims[0], dims[1], dims[2], ax,
                                                                                     La, lines, n, q0, n_cut, q, F);
    const long long kt = static_cast<long long>(Nb) * (2 * Nc - 1);
    k_tail_line_Ktab<<<static_cast<int>(std::min<long long>((kt + kTailThreads - 1) / kTailThreads, 152 * 8)),
                       kTailThreads, 0, st>>>(Nb, Nc, gbb, gbc, gcc, rc, pref, Kt);
    k_tail_line_G<<<dim3((La + kGT - 1) / kGT, (rows + kGT - 1) / kGT), 256, 0, st>>>(La, rows, lines, Nc, Kt, F, G);
    count_launches(3);
    VDWDF_CUDA_TRY(cudaGetLastError());
    return tail_finish(La, q, F, G, scale, dots, out, st);
}

int launch_far_tail_AU(const int dims[3], int ax, int np, const int *line_slot, const double *n, const double *q0,
                       double n_cut, const TailNodes &q, const double *G, double *coef, double C, int *slot, double *A,
                       double *U, cudaStream_t st) {
    k_tail_coef<<<(np + 127) / 128, 128, 0, st>>>(np, q, G, coef);
    const long long N = static_cast<long long>(dims[0]) * dims[1] * dims[2];
    long long nb = (N + kTailThreads - 1) / kTailThreads;
    if (nb > 152 * 16) nb = 152 * 16;
    k_tail_AU<<<static_cast<int>(nb), kTailThreads, 0, st>>>(dims[0], dims[1], dims[2], ax, np, line_slot, n, q0,
                                                             n_cut, q, G, coef, C, slot, A, U);
    count_launches(2);
    VDWDF_CUDA_TRY(cudaGetLastError());
    return VDWDF_OK;
}

// Parts of a plane's points: enough blocks for two rounds of the chip.
int far_tail_parts(const TailNodes &q, int np, long long points) {
    const long long blocks = static_cast<long long>(np) * tail_columns(q);
    const long long want = (152 * 8 + blocks - 1) / blocks, most = (points / np + 4 * kTailThreads - 1) / (4 * kTailThreads);
    return static_cast<int>(std::max<long long>(1, std::min<long long>(std::min(want, most), 64)));
}

int launch_far_tail(const int dims[3], int ax, int np, const double *n, const double *q0, double n_cut,
                    const TailNodes &q, int parts, double dz, double rc, double c2, double c3, double scale, double *F,
                    double *G, double *dots, double *out, cudaStream_t st) {
    const int rows = kMom + q.nb;
    k_tail_planes<<<dim3(np, tail_columns(q), parts), kTailThreads, 0, st>>>(dims[0], dims[1], dims[2], ax, np, n, q0,
                                                                             n_cut, q, F);
    count_launches(1);
    if (parts > 1) {
        const long long e = static_cast<long long>(rows) * np;
        k_tail_fold<<<static_cast<int>(std::min<long long>((e + 255) / 256, 152 * 8)), 256, 0, st>>>(e, parts, F);
        count_launches(1);
    }
    const size_t smem = 2 * sizeof(double) * static_cast<size_t>(np);
    const int sh = smem <= 48 * 1024 ? 1 : 0;
    k_tail_pairs<<<rows, kTailThreads, sh ? smem : 0, st>>>(np, F, dz, rc, c2, c3, sh, G);
    count_launches(1);
    VDWDF_CUDA_TRY(cudaGetLastError());
    return tail_finish(np, q, F, G, scale, dots, out, st);
}

}  // namespace vdwdf
