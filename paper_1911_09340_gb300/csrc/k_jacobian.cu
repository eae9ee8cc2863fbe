// Residual Jacobians for Gauss-Newton refinement of the best seeds (FP64, uniform axial field).
//
// The seed is parameterised by theta = (z0, phi, pz, pT) with the vertex (vx, vy) fixed, as in the
// lattice.  With P = px + i py and X = x + i y, one RK4 step of length h in B = (0, 0, Bz) is the
// linear map P' = m P, X' = X + n P, z' = z + dz, whose coefficients depend on P0 = |p| and h only
// (device.cuh), and so do those of any product of steps: after a path of length L, X = X_0 + N P_0 and
// z = z_0 + L pz / |p|.  The derivatives of the recorded states in theta therefore need the maps'
// derivatives in one variable, |p|: the path is carried as X and P, each with its derivative in ln(1/|p|)
// (forward mode), and the chain rule in (z0, phi, pz, pT) is applied once, at its end.  This part's FP64
// unit holds its scheduler for 64 cycles per warp instruction, whatever the active lanes, so the
// kernel's time is its longest lane's count of FP64 instructions.  A whole call with four derivatives
// carried through every step and through the maps' powers, and so: 16 seeds x 134 wires x 138 states
// 438 and 95 us, 64 x 134 x 2229 584 and 232, 1000 x 134 x 138 1856 and 663.
//
// The DCA of a wire is the distance at the point of closest approach (PCA) found as in the scan: the
// closest recorded state (searched in FP32, settled in FP64 among its neighbours), then the local
// virtual-plane Newton refinement of Algorithm 2, each refinement step being one RK4 step of the
// axial map.  At the PCA the distance is stationary along the track, so dD/dtheta = nhat . dx/dtheta at
// the fixed arc length of the PCA (envelope theorem): the refinement steps enter the product of maps with
// their lengths held fixed.  nhat is the unit vector from the wire to the PCA.
//
// Smoothed residual (Eq. 1 with a differentiable cap): e = min_j |D - r_j| over the wire's unmasked
// hits, w = sigmoid((lambda - e) / tau), term = w e^2 + (1 - w) lambda^2.  Gauss-Newton treats w as
// fixed within an iteration: residual rho = D - r_j* with weight w.
#include <math.h>

#include "device.cuh"
#include "internal.h"

namespace comet {

namespace {

// A complex number and its derivative D = -P0 d/dP0.
struct Cd {
    double re, im, dre, dim;
};

// a + m b
__device__ __forceinline__ Cd mul_add(const Cd &a, const Cd &m, const Cd &b)
{
    return Cd{a.re + (m.re * b.re - m.im * b.im), a.im + (m.re * b.im + m.im * b.re),
              a.dre + ((m.dre * b.re - m.dim * b.im) + (m.re * b.dre - m.im * b.dim)),
              a.dim + ((m.dre * b.im + m.dim * b.re) + (m.re * b.dim + m.im * b.dre))};
}

// The map of a path: P' = (1 + A) P, X' = X + N P.
struct PathMap {
    Cd A, N;
};

// One RK4 step of length h: A = m - 1 = -t^2 (1/2 - t^2/24) - i t (1 - t^2/6), N = hp (1 - t^2/6) -
// i hp t (1/2 - t^2/24), with t = h w and hp = h / P0 (w and 1 / P0 both have D = themselves).
__device__ __forceinline__ PathMap step_map(double ip, double w, double h)
{
    const double t = h * w, t2 = t * t, hp = h * ip;
    const double u = 1.0 - t2 * (1.0 / 6.0), v = 0.5 - t2 * (1.0 / 24.0), q = 1.0 - 0.5 * t2;
    const double tu = t * u;
    return PathMap{Cd{-(t2 * v), -tu, -(t2 * u), -(t * q)}, Cd{hp * u, -(hp * (t * v)), hp * q, -(hp * tu)}};
}

__device__ __forceinline__ void cmul(double ar, double ai, double br, double bi, double &r, double &i)
{
    r = ar * br - ai * bi;
    i = ar * bi + ai * br;
}
__device__ __forceinline__ void crecip(double re, double im, double &r, double &i)
{
    const double inv = 1.0 / (re * re + im * im);
    r = re * inv;
    i = -im * inv;
}

// Passes of one map s: A_k = (1 + A)^k - 1 by binary powering on values ((1 + a)(1 + b) - 1 = a + b + a b:
// nothing cancels), N_k = N S with S = A_k / A, and from them D A_k = k (1 + A_k) q with q = DA / (1 + A)
// and D S = (D A_k - S DA) / A: the derivatives cost the same whatever k.
struct Powers {
    PathMap s;
    double ir, ii, qr, qi;   // 1 / A and q
    bool turns;
    __device__ __forceinline__ explicit Powers(const PathMap &m) : s(m)
    {
        turns = s.A.re != 0.0 || s.A.im != 0.0;
        crecip(s.A.re, s.A.im, ir, ii);
        double r, i;
        crecip(1.0 + s.A.re, s.A.im, r, i);
        cmul(s.A.dre, s.A.dim, r, i, qr, qi);
    }
    __device__ __forceinline__ PathMap operator()(int k) const   // k >= 0
    {
        double Rr = 0.0, Ri = 0.0, Br = s.A.re, Bi = s.A.im;
        for (int e = k; e > 0; e >>= 1) {
            double r, i;
            if (e & 1) {
                cmul(Rr, Ri, Br, Bi, r, i);
                Rr = (Rr + Br) + r;
                Ri = (Ri + Bi) + i;
            }
            if (e > 1) {
                cmul(Br, Bi, Br, Bi, r, i);
                Br = 2.0 * Br + r;
                Bi = 2.0 * Bi + i;
            }
        }
        PathMap m;
        Cd S{(double)k, 0.0, 0.0, 0.0};
        m.A = Cd{Rr, Ri, 0.0, 0.0};
        if (turns) {
            cmul(1.0 + Rr, Ri, (double)k * qr, (double)k * qi, m.A.dre, m.A.dim);
            cmul(Rr, Ri, ir, ii, S.re, S.im);
            double r, i;
            cmul(S.re, S.im, s.A.dre, s.A.dim, r, i);
            cmul(m.A.dre - r, m.A.dim - i, ir, ii, S.dre, S.dim);
        }
        m.N = mul_add(Cd{0.0, 0.0, 0.0, 0.0}, s.N, S);
        return m;
    }
};

// A path from the seed per unit of transverse momentum: X = X_0 + pT x, P = pT p, both functions of P0 at
// a fixed phi.
struct Path {
    Cd x, p;
};
__device__ __forceinline__ void apply(const PathMap &s, Path &y)
{
    y.x = mul_add(y.x, s.N, y.p);
    y.p = mul_add(y.p, s.A, y.p);
}
// values only
__device__ __forceinline__ void apply_values(const PathMap &s, Path &y)
{
    const double pr = y.p.re, pi = y.p.im;
    y.x.re += s.N.re * pr - s.N.im * pi;
    y.x.im += s.N.re * pi + s.N.im * pr;
    y.p.re += s.A.re * pr - s.A.im * pi;
    y.p.im += s.A.re * pi + s.A.im * pr;
}

constexpr int kMaxSteps = 64;    // refinement steps at most (max_iter is capped)
constexpr int kWalkTile = 256;   // recorded states staged at a time

// One warp: one seed and 32 of its wires, or with few wires 32 / G seeds and G >= W lanes for each (G a
// power of two), so that no more than half the lanes idle.  Lanes past the last wire or seed repeat it
// without writing.
__global__ void __launch_bounds__(32) jacobian_kernel(JacArgs a, int G)
{
    __shared__ float4 walk_s[kWalkTile];
    const int chunks = (a.W + G - 1) / G;
    const int g = threadIdx.x / G, lane = threadIdx.x & (G - 1);   // lane of the group
    const int64_t sg = (int64_t)(blockIdx.x / chunks) * (32 / G) + g;
    const int i = (int)(blockIdx.x % chunks) * G + lane;
    const bool has = i < a.W && sg < a.S;
    const int64_t s = sg < a.S ? sg : a.S - 1;
    const int iw = i < a.W ? i : a.W - 1;
    const int tile = kWalkTile / 32 * G;
    float4 *walk = walk_s + g * tile;

    // seed: theta = (z0, phi, pz, pT)
    const double *th = a.theta + s * 4;
    const double z0 = th[0], pz = th[2], pt = th[3];
    double sphi, cphi;
    sincos(th[1], &sphi, &cphi);
    const double P0 = sqrt(pt * pt + pz * pz), ip = 1.0 / P0;
    const double w = kKappa * a.charge * a.bz * ip;
    const PathMap one = step_map(ip, w, a.h);
    const Powers itv(a.stride == 1 ? one : Powers(one)(a.stride));
    const double tz = pz * ip, tt = pt * ip;
    const double dz = (double)a.stride * (a.h * tz);

    // wire
    const double *wr = (const double *)a.wires + iw;
    const double ax = wr[0 * a.ldw], ay = wr[1 * a.ldw], az = wr[2 * a.ldw];
    const double ux = wr[3 * a.ldw], uy = wr[4 * a.ldw], uz = wr[5 * a.ldw];

    // closest recorded state, recording as the scan does: state 0, then each interval, stopping
    // after the first state outside the target region.  The walk runs in FP32 (FP64 instructions
    // are scarce on this part), the seed's states once into shared memory and then each lane's wire
    // against them; the argmin is settled in FP64 among the FP32 choice and its two neighbours.
    const float am1f = (float)itv.s.A.re, bbf = (float)-itv.s.A.im, ccf = (float)itv.s.N.re,
                ddf = (float)-itv.s.N.im, dzf = (float)dz;
    float f[5] = {(float)a.vx, (float)a.vy, (float)z0, (float)(pt * cphi), (float)(pt * sphi)};
    const float axf = (float)ax, ayf = (float)ay, azf = (float)az, uxf = (float)ux, uyf = (float)uy,
                uzf = (float)uz;
    const float zminf = (float)a.zmin, zmaxf = (float)a.zmax, rmax2f = (float)a.rmax2;
    float bestf = INFINITY;
    int kbest = 0, nvalid = a.n_rec;
    auto step = [&]() {
        const float px = f[3], py = f[4];
        f[0] += ccf * px + ddf * py;
        f[1] += ccf * py - ddf * px;
        f[2] += dzf;
        f[3] += am1f * px + bbf * py;
        f[4] += am1f * py - bbf * px;
    };
    // a track that provably stays inside the region needs no test per state (0.1 um of rounding per
    // plain float state)
    const bool inside = stays_inside(f[0], f[1], f[2], f[3], f[4], AxialStep<float>{am1f, bbf, ccf, ddf, dzf},
                                     a.n_rec, zminf, zmaxf, rmax2f, 1e-7f);
    for (int kt = 0; __any_sync(0xffffffffu, kt < nvalid); kt += tile) {
        const int ke = min(kt + tile, nvalid);
        int k = kt;
        if (inside) {
#pragma unroll 4
            for (; k < ke; ++k) {
                if (k > 0) step();
                if (lane == (k & (G - 1))) walk[k - kt] = make_float4(f[0], f[1], f[2], 0.f);
            }
        } else {
            for (; k < ke; ++k) {
                if (k > 0) step();
                if (lane == (k & (G - 1))) walk[k - kt] = make_float4(f[0], f[1], f[2], 0.f);
                if (f[2] < zminf || f[2] > zmaxf || f[0] * f[0] + f[1] * f[1] > rmax2f) {
                    nvalid = ++k;
                    break;
                }
            }
        }
        __syncwarp();
#pragma unroll 4
        for (int j = 0; j < k - kt; ++j) {
            const float4 p = walk[j];
            const float d2 = line_dist2<float>(p.x, p.y, p.z, axf, ayf, azf, uxf, uyf, uzf);
            if (d2 < bestf) {
                bestf = d2;
                kbest = kt + j;
            }
        }
        __syncwarp();
    }
    // FP64: states kbest - 1 .. kbest + 1, the lowest distance, ties to the lower index
    const int k0 = kbest > 0 ? kbest - 1 : 0;
    Path y{Cd{0.0, 0.0, 0.0, 0.0}, Cd{cphi, sphi, 0.0, 0.0}};
    apply(itv(k0), y);
    {
        double best = INFINITY;
        int kb = kbest;
        Path c = y;
        for (int k = k0; k <= kbest + 1 && k < nvalid; ++k) {
            if (k > k0) apply_values(itv.s, c);
            const double d2 = line_dist2<double>(a.vx + pt * c.x.re, a.vy + pt * c.x.im, z0 + (double)k * dz, ax, ay,
                                                 az, ux, uy, uz);
            if (d2 < best) {
                best = d2;
                kb = k;
            }
        }
        kbest = kb;
    }
    for (int k = k0; k < kbest; ++k) apply(itv.s, y);

    // local virtual-plane refinement from there, on the position relative to the wire's point
    const double vx = a.vx - ax, vy = a.vy - ay, vz = (z0 - az) + (double)kbest * dz;
    int conv = 0;
    double sigma = 0.0;
    const int max_iter = a.max_iter < kMaxSteps ? a.max_iter : kMaxSteps;
    for (int it = 0;; ++it) {
        // t = p / P0: |p| stays P0 in a magnetic field (refine_dca)
        const double tx = tt * y.p.re, ty = tt * y.p.im;
        const double tu = tx * ux + ty * uy + tz * uz;
        const double nx = tx - tu * ux, ny = ty - tu * uy, nz = tz - tu * uz;
        const double nn2 = nx * nx + ny * ny + nz * nz;
        if (nn2 < 1e-18) break;
        const double rn = rsqrt(nn2);
        const double dist = ((vx + pt * y.x.re) * nx + (vy + pt * y.x.im) * ny + (vz + sigma * tz) * nz) * rn;
        if (fabs(dist) < a.tol) {
            conv = 1;
            break;
        }
        if (it >= max_iter) break;
        double target = sigma - dist * rn;
        target = target > a.h_rec ? a.h_rec : target;
        target = target < -a.h_rec ? -a.h_rec : target;
        const double ds = target - sigma;
        if (ds == 0.0) break;
        apply(step_map(ip, w, ds), y);
        sigma = target;
    }

    // D and dD/dtheta = nhat . dx/dtheta at the path's fixed length
    const double rx = vx + pt * y.x.re, ry = vy + pt * y.x.im, rz = vz + sigma * tz;
    const double al = rx * ux + ry * uy + rz * uz;
    const double ex = rx - al * ux, ey = ry - al * uy, ez = rz - al * uz;
    const double D = sqrt(ex * ex + ey * ey + ez * ez);
    const double inv = D > 0.0 ? 1.0 / D : 0.0;
    const double hx = ex * inv, hy = ey * inv, hz = ez * inv;
    // X = X_0 + pT x: dX/dphi = i pT x, dX/dpT = x + pT dx/dP0 dP0/dpT, dX/dpz = pT dx/dP0 dP0/dpz;
    // z = z_0 + L pz / P0, so dz/dpz = (L / P0) (1 - tz^2), dz/dpT = -(L / P0) tz tt
    const double hq = -tt * (hx * y.x.dre + hy * y.x.dim);   // nhat . pT dx/dP0
    const double lz = (((double)kbest * a.stride) * a.h + sigma) * ip * hz;
    double J[4];
    J[0] = hz;
    J[1] = pt * (hy * y.x.re - hx * y.x.im);
    J[2] = hq * tz + lz * (1.0 - tz * tz);
    J[3] = hq * tt + (hx * y.x.re + hy * y.x.im) - lz * tz * tt;

    // smoothed residual of the wire
    if (!has) return;
    const int hb = a.offs[i], he = a.offs[i + 1];
    bool any = false;
    double e = INFINITY, r_best = 0.0;
    for (int j = hb; j < he; ++j) {
        if (a.mask[j]) continue;
        any = true;
        const double ej = fabs(D - a.drift[j]);
        if (ej < e) {
            e = ej;
            r_best = a.drift[j];
        }
    }
    double term = 0.0, dterm = 0.0, wgt = 0.0, rho = 0.0;
    if (any) {
        const double lam = a.lambda;
        wgt = 1.0 / (1.0 + exp(-(lam - e) / a.tau));
        term = wgt * e * e + (1.0 - wgt) * lam * lam;
        const double dw = -wgt * (1.0 - wgt) / a.tau;
        const double sgn = D >= r_best ? 1.0 : -1.0;
        dterm = sgn * (2.0 * wgt * e + dw * (e * e - lam * lam));
        rho = D - r_best;
    }
    const int64_t tid = s * a.W + i;
    double *out = a.work + tid * 11;   // flag, term, dterm, w, rho, J[0..3], nhat_x, nhat_y
    out[0] = any ? 1.0 : 0.0;
    out[1] = term;
    out[2] = dterm;
    out[3] = wgt;
    out[4] = rho;
    if (a.dca_out) a.dca_out[tid] = D;
    if (a.jac_out) {
#pragma unroll
        for (int j = 0; j < 4; ++j) a.jac_out[tid * 4 + j] = J[j];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) out[5 + j] = J[j];
    out[9] = hx;    // dD/dx0 and dD/dy0: the recorded X_k depend on (x0, y0) additively
    out[10] = hy;
    if (!conv && any && a.n_unconv) atomicAdd(a.n_unconv, 1);
}

// Per seed, ascending wire order: smoothed RSS, its gradient, J^T W J and J^T W rho.  One warp per seed: the
// terms of 32 wires at a time go to shared memory, then lane q adds product q of the 27 sums wire by
// wire (the order, and the one rounding per product, of a single thread doing them all, which waited
// on memory for every wire: 210 us for 16 seeds x 100 wires).
__global__ void __launch_bounds__(32) jacobian_reduce_kernel(JacArgs a)
{
    // factors of a wire's products: f[0] = 1, [1] = dterm, [2] = w rho, [3..6] = w J, g[0] = term,
    // [1..4] = J, [5..6] = nhat
    __shared__ double sf[32][7], sg[32][7];
    __shared__ int any[32];
    const int64_t s = blockIdx.x;
    const int q = threadIdx.x;
    // sum q: 0 smoothed RSS, 1-4 gradient, 5-8 J^T W rho, 9-24 J^T W J, 25-26 gradient in (x0, y0)
    const int fi = q == 0 ? 0 : q < 5 ? 1 : q < 9 ? 2 : q < 25 ? 3 + (q - 9) / 4 : 1;
    const int gi = q == 0 ? 0 : q < 5 ? q : q < 9 ? q - 4 : q < 25 ? 1 + (q - 9) % 4 : q < 27 ? q - 20 : 0;
    double acc = 0.0;
    for (int i0 = 0; i0 < a.W; i0 += 32) {
        const int n = min(32, a.W - i0);
        if (q < n) {
            const double *o = a.work + (s * a.W + i0 + q) * 11;
            any[q] = o[0] != 0.0;
            sf[q][0] = 1.0;
            sf[q][1] = o[2];
            sf[q][2] = o[3] * o[4];
            sg[q][0] = o[1];
            sg[q][5] = o[9];
            sg[q][6] = o[10];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                sf[q][3 + j] = o[3] * o[5 + j];
                sg[q][1 + j] = o[5 + j];
            }
        }
        __syncwarp();
        for (int t = 0; t < n; ++t)
            if (any[t]) acc = fma(sf[t][fi], sg[t][gi], acc);
        __syncwarp();
    }
    if (q == 0) a.srss_out[s] = acc;
    else if (q < 5) a.grad_out[s * 4 + q - 1] = acc;
    else if (q < 9) a.jtr_out[s * 4 + q - 5] = acc;
    else if (q < 25) a.jtj_out[s * 16 + q - 9] = acc;
    if (a.grad6_out) {
        // (x0, y0, z0, px, py, pz): phi = atan2(py, px) and pT = hypot(px, py), by the chain rule
        double g[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) g[j] = __shfl_sync(0xffffffffu, acc, 1 + j);
        const double phi = a.theta[s * 4 + 1], pt = a.theta[s * 4 + 3];
        const double cp = cos(phi), sp = sin(phi);
        double *o = a.grad6_out + s * 6;
        if (q == 25 || q == 26) o[q - 25] = acc;
        if (q == 0) {
            o[2] = g[0];
            o[3] = -g[1] * sp / pt + g[3] * cp;
            o[4] = g[1] * cp / pt + g[3] * sp;
            o[5] = g[2];
        }
    }
}

// Solves (J^T W J + mu diag(J^T W J)) x = -J^T W rho for one seed by Cholesky; returns false (x
// untouched) when the damped matrix is not positive definite.
__device__ bool damped_normal_solve(const double *jtj, const double *jtr, double mu, double x[4])
{
    double A[4][4], L[4][4] = {}, r[4];
    for (int j = 0; j < 4; ++j) {
        for (int k = 0; k < 4; ++k) A[j][k] = jtj[j * 4 + k];
        A[j][j] *= 1.0 + mu;
        r[j] = -jtr[j];
    }
    for (int j = 0; j < 4; ++j) {
        double d = A[j][j];
        for (int k = 0; k < j; ++k) d -= L[j][k] * L[j][k];
        if (!(d > 0.0)) return false;
        L[j][j] = sqrt(d);
        for (int i = j + 1; i < 4; ++i) {
            double v = A[i][j];
            for (int k = 0; k < j; ++k) v -= L[i][k] * L[j][k];
            L[i][j] = v / L[j][j];
        }
    }
    double z[4];
    for (int j = 0; j < 4; ++j) {
        double v = r[j];
        for (int k = 0; k < j; ++k) v -= L[j][k] * z[k];
        z[j] = v / L[j][j];
    }
    for (int j = 3; j >= 0; --j) {
        double v = z[j];
        for (int k = j + 1; k < 4; ++k) v -= L[k][j] * x[k];
        x[j] = v / L[j][j];
    }
    return true;
}

// theta += delta, (J^T W J + mu diag(J^T W J)) delta = -J^T W rho, by Cholesky; a seed whose
// matrix is not positive definite keeps its theta
__global__ void gn_step_kernel(double *theta, int64_t S, const double *jtj, const double *jtr, double mu)
{
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    double x[4];
    if (!damped_normal_solve(jtj + s * 16, jtr + s * 4, mu, x)) return;
    for (int j = 0; j < 4; ++j) theta[s * 4 + j] += x[j];
}

// Levenberg-Marquardt bookkeeping of one seed: judge the trial (accept it when its smoothed RSS is
// lower: it becomes the current seed with its normal equations, and the damping shrinks; else the
// damping grows), then form the next trial from the current seed.
__global__ void lm_step_kernel(LmArgs a)
{
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= a.S) return;
    double mu = a.mu[s];
    if (!a.first) {
        const double ft = a.srss_try[s];
        if (ft < a.srss[s]) {
            a.srss[s] = ft;
            for (int j = 0; j < 4; ++j) a.theta[s * 4 + j] = a.theta_try[s * 4 + j];
            for (int j = 0; j < 4; ++j) a.jtr[s * 4 + j] = a.jtr_try[s * 4 + j];
            for (int j = 0; j < 16; ++j) a.jtj[s * 16 + j] = a.jtj_try[s * 16 + j];
            mu = fmax(mu * a.down, a.mu_min);
        } else {
            mu = fmin(mu * a.up, a.mu_max);
        }
        a.mu[s] = mu;
    }
    double x[4] = {0.0, 0.0, 0.0, 0.0};
    damped_normal_solve(a.jtj + s * 16, a.jtr + s * 4, mu, x);
    for (int j = 0; j < 4; ++j) a.theta_try[s * 4 + j] = a.theta[s * 4 + j] + x[j];
}

} // namespace

cudaError_t launch_jacobian(const JacArgs &a, cudaStream_t st)
{
    if (a.W > 0) {
        // one warp per block: a few dozen warps of long FP64 chains, spread over as many SMs as possible
        int G = 32;
        while (G > 1 && G / 2 >= a.W) G /= 2;
        const int64_t blocks = (a.S + 32 / G - 1) / (32 / G) * ((a.W + G - 1) / G);
        jacobian_kernel<<<(unsigned)blocks, 32, 0, st>>>(a, G);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    jacobian_reduce_kernel<<<(unsigned)a.S, 32, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_gn_step(double *theta, int64_t S, const double *jtj, const double *jtr, double mu,
                           cudaStream_t st)
{
    gn_step_kernel<<<(unsigned)((S + 63) / 64), 64, 0, st>>>(theta, S, jtj, jtr, mu);
    return cudaGetLastError();
}

cudaError_t launch_lm_step(const LmArgs &a, cudaStream_t st)
{
    lm_step_kernel<<<(unsigned)((a.S + 63) / 64), 64, 0, st>>>(a);
    return cudaGetLastError();
}

} // namespace comet
