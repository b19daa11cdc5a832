// ocmc_tables.cu -- physics tables of the transport kernel, built on the GPU in
// double precision from closed-form models, then stored as FP32.
//
// The paper stores per-material photon attenuation per channel, restricted
// stopping powers and macroscopic cross sections as 2D images indexed by
// energy and material (Sec. 2.1, Sec. 2.2.2). Here the same quantities come
// from published closed forms (one table row per material, uniform in ln E):
//   photons  : Klein-Nishina (free electrons), K-shell Born photoelectric,
//              Maximon's pair expansions with Z(Z+1);
//   electrons: ICRU-37 restricted collision stopping power with the
//              Sternheimer-Peierls density effect, complete-screening
//              Bethe-Heitler bremsstrahlung with Z(Z+1), Moller cross section,
//              screened-Rutherford transport cross section (Moliere screening).
// The CSDA range R(E) is the integral of 1/L (8-point Gauss-Legendre per
// table interval), inverted on a uniform ln R grid.
//
// What bounds the build: GB300's narrow FP64 pipe (about two multiply-adds per clock and SM) and the
// length of FP64 chains, so the work is spread over all SMs in short pieces: per-composition constants
// once per material (k_mconst), eight lanes per node for the majorant's scan and the quadratures'
// abscissas (k_nodes), secant steps instead of 60 bisections for the inverse range (k_range_inverse),
// bracketed Newton steps instead of 100 for the screening table (extra blocks of k_nodes). The sums keep
// the order of the plain loops. The three built-in materials: 6.1 ms
// with a thread per node and bisections, 0.2 ms so.
#include "ocmc_internal.h"

#include <cmath>

namespace ocmc {

namespace {


constexpr double RE = 2.8179403262e-13;
constexpr double ALPHA = 1.0 / 137.035999084;
constexpr double NAV = 6.02214076e23;
constexpr double PI = 3.14159265358979323846;

using MC = MatConst;

// Per-gram constants of one composition: a warp per material, a lane per element for the logarithms
// and cube roots, then the sums in element order.
__global__ void k_mconst(Tables t)
{
    const MatDef& d = t.mats[blockIdx.x];
    const int lane = threadIdx.x;
    double ws = 0.0;
    for (int i = 0; i < d.n; ++i) ws += d.w[i];
    double n_l = 0.0, l_l = 0.0;
    if (lane < d.n) {
        const double z3 = cbrt((double)d.Z[lane]);
        n_l = NAV * d.w[lane] / ws / d.A[lane];
        l_l = log(183.0 / z3);
        t.elem[(size_t)blockIdx.x * MAX_ELEM + lane] = make_double2(n_l, z3);
    }
    MC c;
    c.ne = c.photo = c.pairZ = c.S1 = c.S2 = 0.0;
    for (int i = 0; i < d.n; ++i) {
        const double Z = d.Z[i], n = __shfl_sync(0xFFFFFFFFu, n_l, i), l = __shfl_sync(0xFFFFFFFFu, l_l, i);
        c.ne += n * Z;
        c.photo += n * Z * Z * Z * Z * Z;
        c.pairZ += n * Z * (Z + 1.0);
        c.S1 += n * Z * (Z + 1.0) * l;
        c.S2 += n * Z * (Z + 1.0) / 9.0;
    }
    c.I = d.I_eV;
    double hw = 28.816 * sqrt(d.rho0 * c.ne / NAV);
    double C = 2.0 * log(d.I_eV / hw) + 1.0;
    double x0, x1;
    if (d.I_eV < 100.0) { x1 = 2.0; x0 = C < 3.681 ? 0.2 : 0.326 * C - 1.0; }
    else                { x1 = 3.0; x0 = C < 5.215 ? 0.2 : 0.326 * C - 1.5; }
    c.dC = C; c.dX0 = x0; c.dX1 = x1;
    double span = x1 - x0;
    c.dA = (C - 2.0 * log(10.0) * x0) / (span * span * span);
    if (lane == 0) {
        t.mc[blockIdx.x] = c;
        t.msc[2 * blockIdx.x] = (float)c.S1;
        t.msc[2 * blockIdx.x + 1] = (float)c.S2;
    }
}

__device__ double kn_total(double E)
{
    double k = E / MC2, a = 1.0 + 2.0 * k, l = log(a);
    return 2.0 * PI * RE * RE *
           ((1.0 + k) / (k * k) * (2.0 * (1.0 + k) / a - l / k) + l / (2.0 * k) - (1.0 + 3.0 * k) / (a * a));
}

__device__ double pair_phi(double E)
{
    double k = E / MC2;
    if (k <= 2.0) return 0.0;
    double v;
    if (k <= 4.0) {
        double e = (2.0 * k - 4.0) / (2.0 + k + 2.0 * sqrt(2.0 * k));
        double r = 1.0 - 2.0 / k;
        v = (2.0 * PI / 3.0) * r * r * r *
            (1.0 + e * (0.5 + e * (23.0 / 40.0 + e * (11.0 / 60.0 + e * 29.0 / 960.0))));
    } else {
        double L = log(2.0 * k), q2 = 4.0 / (k * k);
        const double zeta3 = 1.2020569031595942;
        v = 28.0 / 9.0 * L - 218.0 / 27.0 +
            q2 * (6.0 * L - 3.5 + (2.0 / 3.0) * L * L * L - L * L - (PI * PI / 3.0) * L + 2.0 * zeta3 +
                  PI * PI / 6.0) -
            q2 * q2 * (3.0 / 16.0 * L + 0.125) -
            q2 * q2 * q2 * (29.0 / 2304.0 * L - 77.0 / 13824.0);
    }
    return v > 0.0 ? v : 0.0;
}

// 0 total, 1 Compton, 2 photoelectric, 3 pair  (cm^2/g)
__device__ void mu_channels(const MC& c, double E, double mu[4])
{
    double sC = c.ne * kn_total(E);
    double sigT = 8.0 * PI / 3.0 * RE * RE;
    double sP = c.photo * 4.0 * sqrt(2.0) * ALPHA * ALPHA * ALPHA * ALPHA * sigT * pow(MC2 / E, 3.5);
    double sQ = c.pairZ * ALPHA * RE * RE * pair_phi(E);
    mu[0] = sC + sP + sQ;
    mu[1] = sC;
    mu[2] = sP;
    mu[3] = sQ;
}

__device__ double density_delta(const MC& c, double T)
{
    double tau = T / MC2;
    double x = 0.5 * log10(tau * (tau + 2.0));
    if (x < c.dX0) return 0.0;
    double r = 2.0 * log(10.0) * x - c.dC;
    if (x < c.dX1) {
        double y = c.dX1 - x;
        r += c.dA * y * y * y;
    }
    return r;
}

__device__ double L_col(const MC& c, double T, double wcc)
{
    double tau = T / MC2, g = tau + 1.0, b2 = 1.0 - 1.0 / (g * g);
    double d = fmin(wcc, 0.5 * T) / MC2;
    double I = c.I * 1e-6 / MC2;
    double F = -1.0 - b2 + log((tau - d) * d) + tau / (tau - d) +
               (0.5 * d * d + (2.0 * tau + 1.0) * log(1.0 - d / tau)) / (g * g);
    return 2.0 * PI * RE * RE * MC2 * c.ne / b2 * (log(2.0 * (tau + 2.0) / (I * I)) + F - density_delta(c, T));
}

__device__ double L_rad(const MC& c, double T, double wcb)
{
    double E = T + MC2, k = fmin(wcb, T);
    double a = c.S1 * (4.0 / 3.0 * k - 2.0 / 3.0 * k * k / E + k * k * k / (3.0 * E * E));
    double b = c.S2 * (k - 0.5 * k * k / E);
    return 4.0 * ALPHA * RE * RE * (a + b);
}

__device__ double L_tot(const MC& c, double T, const PhysParams& pp)
{
    T = fmax(T, 1e-3);
    return L_col(c, T, pp.w_cc) + L_rad(c, T, pp.w_cb);
}

__device__ double sig_moller(const MC& c, double T, double wcc)
{
    if (T <= 2.0 * wcc) return 0.0;
    double tau = T / MC2, g = tau + 1.0, b2 = 1.0 - 1.0 / (g * g);
    double cc = (tau / g) * (tau / g), dd = (2.0 * tau + 1.0) / (g * g), e0 = wcc / T;
    // integral over eps in [e0, 1/2] of 1/e^2 + 1/(1-e)^2 + cc - dd/(e(1-e))
    double I = (1.0 / e0 - 2.0) + (2.0 - 1.0 / (1.0 - e0)) + cc * (0.5 - e0) - dd * log((1.0 - e0) / e0);
    return 2.0 * PI * RE * RE * MC2 * c.ne / (b2 * T) * I;
}

__device__ double sig_brems(const MC& c, double T, double wcb)
{
    if (T <= wcb) return 0.0;
    double E = T + MC2, l = log(T / wcb), dk = T - wcb;
    double a = c.S1 * (4.0 / 3.0 * l - 4.0 / 3.0 * dk / E + (T * T - wcb * wcb) / (2.0 * E * E));
    double b = c.S2 * (l - dk / E);
    return 4.0 * ALPHA * RE * RE * (a + b);
}

// One element's factors of 1/lambda_1 at energy T: the sum over elements is of f.x * f.y.
__device__ double2 lambda1_factors(double2 elem, double Z, double T)
{
    double pc = sqrt(T * (T + 2.0 * MC2)), beta = pc / (T + MC2), q = MC2 / (pc * beta);
    double a = ALPHA * elem.y * MC2 / (0.885 * pc);
    double az = ALPHA * Z / beta;
    double eta = 0.25 * a * a * (1.13 + 3.76 * az * az);
    return make_double2(elem.x * 2.0 * PI * Z * (Z + 1.0) * RE * RE * q * q, log1p(1.0 / eta) - 1.0 / (1.0 + eta));
}

__device__ double wentzel_mean(double A)
{
    if (A > 1e3) {
        double x = 1.0 / A;
        return 1.0 - x * (1.0 / 3.0 - x * (1.0 / 6.0 - x / 10.0));
    }
    return 2.0 * A * ((1.0 + A) * log1p(1.0 / A) - 1.0);
}

// ln A with wentzel_mean(A) = 1 - exp(-G1): Newton steps in ln A inside a shrinking bracket, a
// bisection where a step would leave it.
__device__ double wentzel_solve(double G1)
{
    const double target = -expm1(-G1);
    double lo = log(1e-40), hi = log(1e15);
    // 2 A (ln(1/A) - 1) for small A, 1 - 1/(3A) for large
    double x = G1 < 1.0 ? log(target / (2.0 * (log(2.0 / target) + 3.0))) : G1 - 1.0986122886681098;
    double last = 1e300;
    for (int it = 0; it < 60; ++it) {
        const double A = exp(x), m = wentzel_mean(A);
        const double L = log1p(1.0 / A), dm = A > 1e3 ? (1.0 / 3.0 - 1.0 / (3.0 * A)) / A : 2.0 * A * ((1.0 + 2.0 * A) * L - 2.0);
        const double step = (target - m) / dm;
        // done, or the steps no longer shrink: the rounding of the mean (near A = 1e3) is reached
        if (fabs(step) <= 4e-16 * fabs(x) || (it > 4 && fabs(step) < 1e-6 && fabs(step) > 0.25 * last)) break;
        if (m < target) lo = x; else hi = x;
        last = fabs(step);
        x = x + step > lo && x + step < hi ? x + step : 0.5 * (lo + hi);
    }
    return x;
}

// integral of dT / L(T) over [a, b], 8-point Gauss-Legendre: each of the eight lanes of a group takes one
// abscissa, every lane gets the sum (in the order of the plain loop over the four pairs)
__device__ double inv_L_integral(const MC& c, double a, double b, const PhysParams& pp)
{
    const double x[4] = {0.1834346424956498, 0.5255324099163290, 0.7966664774136267, 0.9602898564975363};
    const double w[4] = {0.3626837833783620, 0.3137066458778873, 0.2223810344533745, 0.1012285362903763};
    const int sub = threadIdx.x & 7;
    const double xs = (sub >> 1) == 0 ? x[0] : (sub >> 1) == 1 ? x[1] : (sub >> 1) == 2 ? x[2] : x[3];
    double mid = 0.5 * (a + b), h = 0.5 * (b - a), s = 0.0;
    const double v = 1.0 / L_tot(c, sub & 1 ? mid - h * xs : mid + h * xs, pp);
#pragma unroll
    for (int k = 0; k < 4; ++k)
        s += w[k] * (__shfl_sync(0xFFFFFFFFu, v, 2 * k, 8) + __shfl_sync(0xFFFFFFFFu, v, 2 * k + 1, 8));
    return s * h;
}

__device__ __forceinline__ double node_E(int i)
{
    double d = log(E_HI / E_LO) / (NE - 1);
    return exp(log(E_LO) + d * i);
}

// Blocks [0, node_blocks): electron rows, eight lanes per node. Then photon rows, a thread per node
// (short: one warp a block), and the screening table, a thread per entry.
constexpr int NODE_THREADS = 64, ROW_THREADS = 32;

__global__ void __launch_bounds__(NODE_THREADS) k_nodes(Tables t, PhysParams pp, int node_blocks, int photon_blocks)
{
    if ((int)blockIdx.x >= node_blocks) {
        if (threadIdx.x >= ROW_THREADS) return;
        const int r = (int)blockIdx.x - node_blocks;
        if (r >= photon_blocks) {
            const int j = (r - photon_blocks) * ROW_THREADS + threadIdx.x;
            if (j >= NG) return;
            double lg = log(G1_LO) + (log(G1_ISO) - log(G1_LO)) * j / (NG - 1);
            t.msA[j] = (float)wentzel_solve(exp(lg));
            return;
        }
        const int idx = r * ROW_THREADS + threadIdx.x;
        if (idx >= t.n_mat * NE) return;
        const MC& c = t.mc[idx / NE];
        const double E = node_E(idx % NE);
        double mu[4];
        mu_channels(c, E, mu);
        t.ph[idx] = make_float4((float)log(mu[0]), (float)(mu[1] / mu[0]), (float)(mu[2] / mu[0]), (float)mu[0]);
        return;
    }
    const int sub = threadIdx.x & 7;
    const int idx0 = (int)(blockIdx.x * NODE_THREADS + threadIdx.x) >> 3;
    const int idx = min(idx0, t.n_mat * NE - 1);              // whole groups stay together for the shuffles
    const int m = idx / NE, i = idx % NE;
    const MC c = t.mc[m];
    const double E = node_E(i);
    // step limit d_maxe (mass thickness) and the hard-event majorant on [E_i, E_i+1),
    // covering the energies a step starting there can reach (down to E (1 - f_maxe)).
    const double dRf = inv_L_integral(c, E * (1.0 - pp.f_maxe), E, pp);
    double Ehi = E * exp(log(E_HI / E_LO) / (NE - 1));
    double Elo = E * (1.0 - pp.f_maxe) * 0.99, mx = 0.0;
    for (int k = sub; k <= 32; k += 8) {
        double e = Elo + (Ehi - Elo) * k / 32.0;
        mx = fmax(mx, sig_moller(c, e, pp.w_cc) + sig_brems(c, e, pp.w_cb));
    }
    for (int o = 4; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o, 8));
    const double part = inv_L_integral(c, i ? node_E(i - 1) : E * (1.0 - pp.f_maxe), E, pp);
    // 1/lambda_1: two rounds of eight elements, summed in element order
    const MatDef& d = t.mats[m];
    double l1 = 0.0;
    for (int e0 = 0; e0 < MAX_ELEM; e0 += 8) {
        double2 f = make_double2(0.0, 0.0);
        if (e0 + sub < d.n) f = lambda1_factors(t.elem[m * MAX_ELEM + e0 + sub], d.Z[e0 + sub], E);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const double fx = __shfl_sync(0xFFFFFFFFu, f.x, k, 8), fy = __shfl_sync(0xFFFFFFFFu, f.y, k, 8);
            if (e0 + k < d.n) l1 += fx * fy;
        }
    }
    if (sub == 0 && idx0 == idx) {
        t.el[idx] = make_float4(0.f, (float)l1, (float)sig_moller(c, E, pp.w_cc), (float)sig_brems(c, E, pp.w_cb));
        t.el2[idx] = make_float2((float)dRf, (float)(1.02 * mx));
        t.scratch[idx] = i == 0 ? E / L_tot(c, E, pp) : part;
    }
}

// cumulative ranges at the nodes, one block per material: the additions one after the other
__global__ void __launch_bounds__(NE) k_range_scan(Tables t)
{
    __shared__ double s[NE];
    double* R = t.scratch + (size_t)blockIdx.x * NE;
    s[threadIdx.x] = R[threadIdx.x];
    __syncthreads();
    if (threadIdx.x == 0) {
        double r = 0.0;
#pragma unroll 16
        for (int i = 0; i < NE; ++i) {
            r += s[i];
            s[i] = r;
        }
    }
    __syncthreads();
    R[threadIdx.x] = s[threadIdx.x];
}

// Eight lanes per entry j of ln E at ln R_j, and ln R at node j. The energy solves
// R[a] + integral(E_a .. E) = R_j between the nodes a and a + 1: secant steps from the linear guess
// (three or four evaluations; the root is the bisection's to the last bits of a double, far below FP32's).
__global__ void __launch_bounds__(NODE_THREADS) k_range_inverse(Tables t, PhysParams pp)
{
    static_assert(NE == NR, "one group of lanes per node and per entry");
    const int sub = threadIdx.x & 7;
    const int idx0 = (int)(blockIdx.x * NODE_THREADS + threadIdx.x) >> 3;
    const int idx = min(idx0, t.n_mat * NR - 1);
    const int m = idx / NR, j = idx % NR;
    const MC c = t.mc[m];
    const double* R = t.scratch + m * NE;
    // one logarithm a lane: of the first, the last and the j-th range
    const double lr = log(R[sub == 0 ? 0 : sub == 1 ? NE - 1 : j]);
    const double lo = __shfl_sync(0xFFFFFFFFu, lr, 0, 8), hi = __shfl_sync(0xFFFFFFFFu, lr, 1, 8),
                 lrj = __shfl_sync(0xFFFFFFFFu, lr, 2, 8);
    const double Rt = exp(lo + (hi - lo) * j / (NR - 1));
    int a = 0, b = NE - 1;                          // R[a] <= Rt <= R[b]
    while (b - a > 1) {
        int mid = (a + b) / 2;
        if (R[mid] <= Rt) a = mid; else b = mid;
    }
    const double en = node_E(sub & 1 ? b : a);
    const double e0 = __shfl_sync(0xFFFFFFFFu, en, 0, 8), e1 = __shfl_sync(0xFFFFFFFFu, en, 1, 8), Ra = R[a];
    double x0 = e0, f0 = Ra - Rt;                   // f = range - R_j: <= 0 at e0, >= 0 at e1
    double x = e0 + (e1 - e0) * (Rt - Ra) / (R[b] - Ra);
    bool go = j > 0 && j < NR - 1;
    for (int it = 0; it < 12 && __any_sync(0xFFFFFFFFu, go); ++it) {
        const double f = Ra + inv_L_integral(c, e0, x, pp) - Rt;
        if (go) {
            const double df = f - f0;
            double xn = df != 0.0 ? x - f * (x - x0) / df : x;
            xn = fmin(fmax(xn, e0), e1);
            go = fabs(xn - x) > 2e-16 * x;
            x0 = x;
            f0 = f;
            x = xn;
        }
    }
    if (sub == 0 && idx0 == idx) {
        t.rinv[idx] = (float)log(j == 0 ? node_E(0) : j == NR - 1 ? node_E(NE - 1) : x);
        t.el[idx].x = (float)lrj;
        if (j == 0) {
            t.rmeta[2 * m] = (float)lo;
            t.rmeta[2 * m + 1] = (float)((NR - 1) / (hi - lo));
        }
    }
}

// Per-material maximum density and the validity check. Maxima are gathered in shared memory
// first (one global atomic per material and block): with every voxel's atomic going to the same
// few global words the scan took 1.3 ms on a 128^3 phantom.
__global__ void k_phantom_scan(const float* density, const uint8_t* material, long long nvox, int n_mat,
                               unsigned int* rho_max, int* err)
{
    __shared__ unsigned int s_max[MAX_STAGED];
    __shared__ int s_bad;
    for (int m = threadIdx.x; m < MAX_STAGED; m += blockDim.x) s_max[m] = 0u;
    if (threadIdx.x == 0) s_bad = 0;
    __syncthreads();
    bool bad = false;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < nvox; v += (long long)gridDim.x * blockDim.x) {
        float r = density[v];
        int m = material[v];
        const bool ok = m < n_mat && r >= 0.f && r <= 30.f;
        bad |= !ok;
        // lanes of one material take their maximum together; one shared atomic per material
        const unsigned key = ok ? (unsigned)m : 0xFFu;
        const unsigned grp = __match_any_sync(__activemask(), key);
        const unsigned mx = __reduce_max_sync(grp, ok && r > 0.f ? __float_as_uint(r) : 0u);   // non-negative floats order as their bits
        if (ok && mx && (threadIdx.x & 31) == __ffs(grp) - 1) atomicMax(s_max + m, mx);
    }
    if (bad) s_bad = 1;
    __syncthreads();
    for (int m = threadIdx.x; m < n_mat; m += blockDim.x)
        if (s_max[m]) atomicMax(rho_max + m, s_max[m]);
    if (threadIdx.x == 0 && s_bad) atomicOr(err, ERR_PHANTOM);
}

__global__ void k_photon_majorant(Tables t)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NE) return;
    float best = -1e30f;
    for (int m = 0; m < t.n_mat; ++m) {
        float r = __uint_as_float(t.rho_max[m]);
        if (r > 0.f) best = fmaxf(best, (float)log((double)r) + t.ph[m * NE + i].x);
    }
    t.phmaj[i] = best > -1e29f ? best + 1e-6f : best;   // small margin over FP32 rounding
    // voxel-crossing electron steps: max over materials of rho_max * (hard-event majorant of a
    // step starting in [E_i, E_i+1)), so a step's candidate events may fall in any voxel
    float hm = 0.f;
    for (int m = 0; m < t.n_mat; ++m) hm = fmaxf(hm, __uint_as_float(t.rho_max[m]) * t.el2[m * NE + i].y);
    t.elmaj[i] = hm * 1.00001f;
}

}  // namespace

void material_defs(MatDef out[NMAT_DEFAULT])
{
    // mass fractions: water H2O; cortical bone (ICRP); lung (ICRP)
    MatDef water = {2, {1, 8}, {1.008, 15.999}, {0.111894, 0.888106}, 75.0, 1.0};
    MatDef bone = {9, {1, 6, 7, 8, 12, 15, 16, 20, 30},
                   {1.008, 12.011, 14.007, 15.999, 24.305, 30.974, 32.06, 40.078, 65.38},
                   {0.047234, 0.144330, 0.041990, 0.446096, 0.002200, 0.104970, 0.003150, 0.209930, 0.000100},
                   106.4, 1.85};
    MatDef lung = {13, {1, 6, 7, 8, 11, 12, 15, 16, 17, 19, 20, 26, 30},
                   {1.008, 12.011, 14.007, 15.999, 22.990, 24.305, 30.974, 32.06, 35.45, 39.098, 40.078, 55.845, 65.38},
                   {0.101278, 0.102310, 0.028650, 0.757072, 0.001840, 0.000730, 0.000800, 0.002250, 0.002660,
                    0.001940, 0.000090, 0.000370, 0.000010},
                   75.3, 0.26};
    out[0] = water;
    out[1] = bone;
    out[2] = lung;
}

// Material tables for the t.n_mat staged materials defs[0 .. n_mat) (table row m = defs[m]):
// they depend on the compositions and the physics parameters only, not on the phantom.
cudaError_t build_material_tables(const Tables& t, const PhysParams& pp, const MatDef* defs, cudaStream_t s)
{
    if (t.n_mat < 1 || t.n_mat > MAX_STAGED) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemcpyAsync(t.mats, defs, sizeof(MatDef) * t.n_mat, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    const int rows = t.n_mat * NE, node_blocks = (rows * 8 + NODE_THREADS - 1) / NODE_THREADS,
              photon_blocks = (rows + ROW_THREADS - 1) / ROW_THREADS, ms_blocks = (NG + ROW_THREADS - 1) / ROW_THREADS;
    k_mconst<<<t.n_mat, 32, 0, s>>>(t);
    k_nodes<<<node_blocks + photon_blocks + ms_blocks, NODE_THREADS, 0, s>>>(t, pp, node_blocks, photon_blocks);
    k_range_scan<<<t.n_mat, NE, 0, s>>>(t);
    k_range_inverse<<<node_blocks, NODE_THREADS, 0, s>>>(t, pp);
    return cudaGetLastError();
}

// Phantom-dependent part: per-material maximum density (with the phantom's validity check) and
// the photon majorant built from it.
cudaError_t build_phantom_tables(const Tables& t, const float* density, const uint8_t* material, long long nvox,
                                 int* d_err, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(t.rho_max, 0, t.n_mat * sizeof(unsigned int), s);
    if (e != cudaSuccess) return e;
    k_phantom_scan<<<1024, 256, 0, s>>>(density, material, nvox, t.n_mat, t.rho_max, d_err);
    k_photon_majorant<<<(NE + 127) / 128, 128, 0, s>>>(t);
    return cudaGetLastError();
}

cudaError_t build_tables(const Tables& t, const PhysParams& pp, const float* density, const uint8_t* material,
                         long long nvox, int* d_err, const MatDef* defs, cudaStream_t s)
{
    cudaError_t e = build_material_tables(t, pp, defs, s);
    return e != cudaSuccess ? e : build_phantom_tables(t, density, material, nvox, d_err, s);
}

}  // namespace ocmc
