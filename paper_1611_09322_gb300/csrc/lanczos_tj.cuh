// T_j^{1/2} e_1 of the Lanczos loop and its stop test (Sec. II B 1), device
// code of one warp, sm_103a.
#pragma once
#include "pse_internal.cuh"

namespace pse {

// One warp.  The matrix square root as an integral, discretised after Hale,
// Higham & Trefethen, SIAM J. Numer. Anal. 46, 2505 (2008), method 3:
//   T^{1/2} e_1 = sum_l w_l T (T + s_l I)^{-1} e_1,
// nodes s_l and weights w_l from Jacobi elliptic functions for a spectrum in
// [2^-18, 1], scaled by the power of four c >= ||T|| (exactly: shifts c s_l,
// weights c^{1/2} w_l).  31 nodes leave a relative error of 1.5e-17 on that
// interval (evaluated with 40 digits), so the result is T^{1/2} e_1 to
// rounding: 1-2e-16 of its norm from a 40-digit value for j = 1..64 and
// condition numbers up to 1e3, where an eigendecomposition in doubles is off
// by up to 6e-15.  Lane l
// solves the system of node l through the trailing determinants
//   phi_i = (alpha_i + s) phi_{i+1} - beta_i^2 phi_{i+2},
//   x_i = (-1)^{i+1} beta_1 .. beta_{i-1} phi_{i+1} / phi_1,
// j dependent multiply-adds and one division, where QL sweeps chain dozens of
// divisions and square roots (FP64 latency is what this costs).  (T x)_i =
// -s x_i for i >= 2, so no component cancels.  Lane 31 runs the recurrence at
// the shift -2^-18 c: all phi_i > 0 there means that the spectrum lies above
// it (Sylvester); otherwise (a zero mode of coincident spheres, or no
// convergence) the QL route below is taken.
// It was one launch of 12-19 us after each update (Newton-Schulz, QL).
__device__ const double c_hht_s[32] = {
    5.7983172601720927e-8, 5.4321516364628967e-7, 1.6334814437543627e-6, 3.5979661192943067e-6,
    6.9216981084029469e-6, 1.2425309911265321e-5, 2.1467667841819654e-5, 3.6281423144883104e-5,
    6.0524386131848248e-5, 0.00010018300523163798, 0.00016505141758121806, 0.00027115231705414841,
    0.00044470021775750382, 0.00072859332384748145, 0.0011930574307098304, 0.001953125,
    0.0031974129387513047, 0.0052357016469499542, 0.0085781322187369926, 0.014068466414259757,
    0.023112175112024554, 0.038077289224902505, 0.063027442481034705, 0.10514188625930458,
    0.17769500132631345, 0.30701023096143713, 0.55112158980091238, 1.0602371281842982,
    2.3353171719278134, 7.0224425253874365, 65.789729924363965, -3.814697265625e-6};
__device__ const double c_hht_w[32] = {
    0.00030813623989951382, 0.00032687093299644554, 0.00036547944964625105, 0.00042630934808390455,
    0.00051305944420673084, 0.00063100491451650686, 0.00078731848148126131, 0.0009915074693214191,
    0.0012559938481394102, 0.0015968736736132673, 0.0020349044825956523, 0.002596785671713454,
    0.0033168201568205391, 0.0042390802236798112, 0.0054202550989604143, 0.0069334495341588189,
    0.0088733664177913662, 0.011363614366040764, 0.014567486387701018, 0.018704789507856225,
    0.024079907193853152, 0.031131965811612131, 0.040530984970311739, 0.053375470369097509,
    0.071630110008854434, 0.099187181846279507, 0.14477216591543603, 0.23141836745246686,
    0.43699734258975575, 1.1752613581759009, 10.379366401483795, 0.0};

// y[0..k-1] = T_k^{1/2} e_1 by the QL eigendecomposition (Golub & Van Loan,
// Sec. 8.3): every lane runs the scalar recurrences redundantly and applies
// each plane rotation to its own rows of the eigenvector matrix, then
// y = Q diag(sqrt(max(lambda, 0))) Q^T e_1.  ws: PSE_QL_WORK doubles.
__device__ __noinline__ void tri_sqrt_e1_ql(int k, const double *alpha, const double *beta, double *y, double *ws) {
    double *Q = ws, *d = ws + PSE_MAXIT * (PSE_MAXIT + 1), *e = d + PSE_MAXIT + 1;
    constexpr int LD = PSE_MAXIT + 1;
    const int lane = threadIdx.x & 31;
    for (int i = lane; i < k; i += 32) {
        d[i] = alpha[i + 1];
        e[i] = (i + 1 < k) ? beta[i + 1] : 0.0;
        for (int c = 0; c < k; ++c) Q[i * LD + c] = (i == c) ? 1.0 : 0.0;
    }
    __syncwarp();
    const double eps = 2.220446049250313e-16;
    for (int l = 0; l < k; ++l) {
        for (int sweep = 0; sweep < 60; ++sweep) {
            int m = l;
            for (; m < k - 1; ++m) {
                const double dd = fabs(d[m]) + fabs(d[m + 1]);
                if (fabs(e[m]) <= eps * dd) break;
            }
            if (m == l) break;
            // shift from the leading 2x2 block (entries are O(mobility), far
            // from overflow, so plain square roots replace hypot)
            double g = (d[l + 1] - d[l]) / (2.0 * e[l]);
            double r = sqrt(fma(g, g, 1.0));
            g = d[m] - d[l] + e[l] / (g + (g >= 0 ? r : -r));
            double s = 1.0, c = 1.0, p = 0.0;
            int i = m - 1;
            bool deflated = false;
            for (; i >= l; --i) {
                const double f = s * e[i], b = c * e[i];
                r = sqrt(fma(f, f, g * g));
                __syncwarp();
                if (lane == 0) e[i + 1] = r;
                __syncwarp();
                if (r == 0.0) {
                    if (lane == 0) { d[i + 1] -= p; e[m] = 0.0; }
                    __syncwarp();
                    deflated = true;
                    break;
                }
                const double rinv = 1.0 / r;  // one division per rotation
                s = f * rinv;
                c = g * rinv;
                g = d[i + 1] - p;
                r = (d[i] - g) * s + 2.0 * c * b;
                p = s * r;
                __syncwarp();
                if (lane == 0) d[i + 1] = g + p;
                __syncwarp();
                g = c * r - b;
                for (int row = lane; row < k; row += 32) {
                    const double qa = Q[row * LD + i], qb = Q[row * LD + i + 1];
                    Q[row * LD + i + 1] = s * qa + c * qb;
                    Q[row * LD + i] = c * qa - s * qb;
                }
                __syncwarp();
            }
            if (deflated && i >= l) continue;
            __syncwarp();
            if (lane == 0) { d[l] -= p; e[l] = g; e[m] = 0.0; }
            __syncwarp();
        }
    }
    __syncwarp();
    for (int c = lane; c < k; c += 32) e[c] = sqrt(fmax(d[c], 0.0)) * Q[c];
    __syncwarp();
    for (int row = lane; row < k; row += 32) {
        double acc = 0.0;
        for (int c = 0; c < k; ++c) acc += Q[row * LD + c] * e[c];
        y[row] = acc;
    }
    __syncwarp();
}

// phi_{i+1} (then its share of the sums) of each lane's node lie in shared
// memory for j <= 8 and in the global workspace above: the 17 KB that j = 64
// needs would change the SMs' split between L1 and shared memory, which costs
// the kernels of the wave branch beside this one (64-system batch 0.5% slower).
#define PSE_EIG_ROWS 8
struct EigSmem {
    double ph[PSE_EIG_ROWS][33];
    double a[PSE_MAXIT + 2], b[PSE_MAXIT + 2], p[PSE_MAXIT + 2], y[PSE_MAXIT + 2];
};
static_assert(PSE_QL_WORK >= PSE_MAXIT * 33, "the rational sum's terms fit the QL workspace");

// What the T_j warp reads, fetched at once and before j is known (one round
// of loads instead of three): alpha_{l+1}, beta_{l+1}, y_l of lane l and its
// node.
struct EigIn {
    double a, b, y, s, w, tmax;
    __device__ __forceinline__ void fetch(const LzState *lz, int lane) {
        a = lz->alpha[lane + 1];
        b = lz->beta[lane + 1];
        y = lz->y[lane];
        s = __ldg(c_hht_s + lane);
        w = __ldg(c_hht_w + lane);
        tmax = lz->tmax;
    }
};

// The T_j block of one update launch (its first warp): y_j = T_k^{1/2} e_1
// (k = j) by the rational sum, QL where the spectrum is too wide for it, the
// stop test without beta_j (||y_j - y_{j-1}||^2 < tol^2 ||y_j||^2), the state.
// Every step of the chain is one dependent FP64 operation of ~70 cycles: the
// recurrence takes one per row (its other term a step ahead), the reciprocal
// of phi_1 three instead of a division's ~3500 cycles, the beta products run
// beside it and scale the row sums at the end: 13000 -> 4500 cycles at k = 4.
__device__ __forceinline__ void lz_eig_body(LzState *lz, int k, const LzStop &st, EigSmem *sm, double *qlws,
                                            const EigIn &in) {
    const int lane = threadIdx.x & 31;
    sm->a[lane + 1] = in.a;
    sm->b[lane + 1] = in.b;
    for (int i = lane + 33; i <= k; i += 32) {
        sm->a[i] = lz->alpha[i];
        sm->b[i] = lz->beta[i];
    }
    if (lane == 0) sm->b[0] = 0.0;
    __syncwarp();
    // largest row sum of |T|: rows < k with their beta, row k without beta_k
    double tmax = in.tmax;
    {
        const double b1 = sm->b[k - 1], b2 = k > 1 ? sm->b[k - 2] : 0.0;
        if (k > 1) tmax = fmax(tmax, sm->a[k - 1] + b1 + b2);
        tmax = fmax(tmax, sm->a[k] + b1);
    }
    // c = 4^p >= tmax
    const int thi = __double2hiint(tmax), p = ((thi >> 20) - 1023 + 2) >> 1;
    bool pos = thi > 0 && normal_f64(thi) && p > -400 && p < 400;
    const double s = in.s * __hiloint2double((1023 + 2 * p) << 20, 0);
    double(*ph)[33] = k <= PSE_EIG_ROWS ? sm->ph : reinterpret_cast<double(*)[33]>(qlws);
    {
        double p1 = 1.0, u = 0.0, as = sm->a[k] + s;  // phi_{i+1}, beta_i^2 phi_{i+2}, alpha_i + s
        double bp = 1.0;                              // (-1)^{i+1} beta_1 .. beta_{i-1}
        for (int i = k, r = 1; i >= 1; --i, ++r) {
            ph[i - 1][lane] = p1;
            const double b = sm->b[i - 1];
            const double t = fma(as, p1, -u);
            u = b * b * p1;
            as = sm->a[i > 1 ? i - 1 : 1] + s;
            p1 = t;
            const int hi = __double2hiint(t);
            pos = pos && hi > 0 && normal_f64(hi);
            if (lane == 0) sm->p[r] = bp;
            bp *= -sm->b[r];
        }
        if (__all_sync(0xffffffffu, pos)) {
            const double f = in.w * __hiloint2double((1023 + p) << 20, 0) * rcp_f64(p1);  // w_l / phi_1
            double v = sm->a[1] * ph[0][lane];
            if (k > 1) v = fma(-sm->b[1] * sm->b[1], ph[1][lane], v);
            ph[0][lane] = v * f;
            const double g = -s * f;
            for (int i = 1; i < k; ++i) ph[i][lane] *= g;
            __syncwarp();
        } else {
            tri_sqrt_e1_ql(k, lz->alpha, lz->beta, sm->y, qlws);
            pos = false;
        }
        pos = __all_sync(0xffffffffu, pos);
    }
    double num = 0.0, den = 0.0;
    if (pos && k <= PSE_EIG_ROWS) {  // four lanes per row
        const int row = lane >> 2, l0 = (lane & 3) * 8;
        double y = 0.0;
        if (row < k) {
            const double *q = ph[row] + l0;
            y = ((q[0] + q[1]) + (q[2] + q[3])) + ((q[4] + q[5]) + (q[6] + q[7]));
        }
        y += __shfl_xor_sync(0xffffffffu, y, 1);
        y += __shfl_xor_sync(0xffffffffu, y, 2);
        const double prev = __shfl_sync(0xffffffffu, in.y, row);
        if (row < k) {
            y *= sm->p[row + 1];
            const double d = row < k - 1 ? y - prev : y;
            num = d * d;
            den = y * y;
            if ((lane & 3) == 0) lz->y[row] = y;
        }
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            num += __shfl_xor_sync(0xffffffffu, num, o);
            den += __shfl_xor_sync(0xffffffffu, den, o);
        }
    } else {
        for (int row = lane; row < k; row += 32) {
            double y = sm->y[row];
            if (pos) {
                y = 0.0;
                for (int l = 0; l < 32; ++l) y += ph[row][l];
                y *= sm->p[row + 1];
            }
            const double d = row < k - 1 ? y - lz->y[row] : y;
            num += d * d;
            den += y * y;
            lz->y[row] = y;
        }
        num = warp_sum(num);
        den = warp_sum(den);
    }
    if (lane == 0) {
        int conv, stop;
        if (st.fixed_iter > 0) {
            stop = conv = k >= st.fixed_iter;
        } else {
            conv = k >= 2 && den > 0.0 && num < st.tol * st.tol * den;
            stop = conv || k >= st.max_iter;
        }
        lz->tmax = tmax;
        lz->num = num;
        lz->den = k >= 2 ? den : 0.0;
        lz->stop_y = stop;
        lz->converged = conv;
    }
}

}  // namespace pse
