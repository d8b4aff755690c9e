// moss_finalize.cu -- estimators and variances in FP64 on the device.
//
//   MOSS-4 (Sec. 4.1.2, Theorems 2-3): p_i = 2 phi^(1)_i / Gamma,
//     n_i = m_i / (K p_i), i in {1,3,4,5,6}; n_2 = Lambda_3 - n_4 - 2 n_5 - 4 n_6
//     (eq. 2); Var(n_i) = n_i/K (1/p_i - n_i); Var(n_2) of Theorem 3.  The
//     collisions r = w are triangles, each reached by 6 ordered draws of
//     probability 1/Gamma, so they also estimate the triangle count.
//   MOSS-5 (Theorems 6-10, Sec. 5.1.3): eta^(l)_i = m^(l)_i / (K_l p^(l)_i),
//     p^(l)_i = 2 phi^(l)_i / Gamma^(l); classes of Omega_1 and Omega_2 are
//     mixed with lambda^(1) = V2/(V1+V2), lambda^(2) = V1/(V1+V2); eta_2 =
//     Lambda_4 - sum_{Omega_3*} phi^(3)_i eta_i with the variance of Theorem 10
//     and the covariances Cov(eta_i, eta_j) = -eta_i eta_j sum_l a_i a_j / K_l.
//   The unknown eta in a variance is replaced by the estimate (one source) or
//   by the pooled value (m1 + m2) / (K1 p1 + K2 p2) (two sources).
//   MOSS-4 with MOSS-4Min (Sec. 4.2, Theorems 1 and 5): a MOSS-4Min hit of
//     class i in {3, 5, 6} whose CIS has c centred 3-paths was drawn with
//     probability 2 c / Gamma-check, so n-check_i = Gamma-check / (2 K-check)
//     sum_c m_{i,c} / c; Var(n-check_i) = (S_i - n_i^2) / K-check with
//     S_i = n_i Gamma-check h_i / 2, h_i the mean of 1/c over the class
//     (sum_c m_{i,c}/c^2 over sum_c m_{i,c}/c; 1, 1, 1/3 without hits, the
//     values of Theorem 4).  Both variances take the plug-in
//     n_i = (K n-hat_i + K-check n-check_i) / (K + K-check), the weights are
//     V_other / (V_1 + V_2) (Theorem 1), n_2 follows eq. (2).
#include "../../include/moss.h"
#include "moss_internal.cuh"

namespace moss {

namespace {

// Sec. 4.1.2: copies of M_1^(4) in M_1..M_6 (phi^(1)) and of M_2^(4) (phi^(2))
__device__ const double kPhi4[6][2] = {{1, 0}, {0, 1}, {4, 0}, {2, 1}, {6, 2}, {12, 4}};
// Table 2: forks, 5-paths, 4-stars in M_1^(5)..M_21^(5)
__device__ const double kPhi5[21][3] = {
    {0, 1, 0},  {0, 0, 1},  {1, 0, 0},   {1, 2, 0},   {2, 2, 0},   {0, 5, 0},   {2, 1, 0},
    {2, 0, 1},  {4, 4, 0},  {4, 7, 0},   {5, 2, 1},   {4, 4, 1},   {6, 6, 0},   {10, 10, 1},
    {9, 6, 1},  {12, 6, 2}, {10, 14, 0}, {20, 24, 1}, {20, 18, 2}, {36, 36, 3}, {60, 60, 5}};

__device__ __forceinline__ double u128_to_double(u128 x) {
    return (double)(uint64_t)(x >> 64) * 18446744073709551616.0 + (double)(uint64_t)x;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

// Row `row` of the covariance matrix, lane i its column i: c between sampled
// classes, c2 in column 2 and its mirror in row 2, zeros elsewhere; row 2
// itself holds its variance (when have2) and the zeros of what is no class.
__device__ __forceinline__ void cov_row(double *cov, int row, int i, bool sampled, bool row_sampled, double c,
                                        double c2, bool have2, double var2) {
    if (i >= kSlots) return;
    if (row == 2) {
        if (i == 2) cov[2 * kSlots + 2] = have2 ? var2 : 0.0;
        else if (!sampled) cov[2 * kSlots + i] = 0.0;
    } else if (row_sampled) {
        cov[row * kSlots + i] = i == 2 ? c2 : c;
        if (i == 2) cov[2 * kSlots + row] = c2;
    } else {
        cov[row * kSlots + i] = 0.0;
    }
}

// MOSS-5 with one warp: lane i is class i (1..21); the sums over classes
// (the eta_2 identity, its variance, the concentrations) are warp sums.
// hits0/hits1: counts of the two sub-methods (either may be null); cov
// (nullable, 22 x 22 row-major) receives row `row` of the covariance matrix,
// and its mirror in row 2 (cov_row).
__device__ void finalize5_warp(const FinalizeIn &in, const uint64_t *hits0, const uint64_t *hits1,
                               const DevTotals *tot, moss_result *out, double *cov, int row) {
    const int i = threadIdx.x & 31;
    const bool cls = i >= 1 && i <= 21;
    const double G0 = u128_to_double(tot->gamma[1]), G1 = u128_to_double(tot->gamma[2]);
    const double K0 = (double)in.K[0], K1 = (double)in.K[1];
    const bool av0 = in.K[0] > 0 && G0 > 0, av1 = in.K[1] > 0 && G1 > 0;
    const uint64_t h0 = (i < kSlots && hits0) ? hits0[i] : 0, h1 = (i < kSlots && hits1) ? hits1[i] : 0;
    const double f0 = cls ? kPhi5[i - 1][0] : 0.0, f1 = cls ? kPhi5[i - 1][1] : 0.0, f3 = cls ? kPhi5[i - 1][2] : 0.0;
    const bool s0 = av0 && f0 > 0, s1 = av1 && f1 > 0;
    double p0 = 0.0, p1 = 0.0, e0 = 0.0, e1 = 0.0;
    if (s0) {
        p0 = 2.0 * f0 / G0;                               // Theorem 6
        e0 = (double)h0 / (K0 * p0);
    }
    if (s1) {
        p1 = 2.0 * f1 / G1;                               // Theorem 8
        e1 = (double)h1 / (K1 * p1);
    }
    double est = 0.0, var = 0.0, plug = 0.0, a0 = 0.0, a1 = 0.0;
    if (cls && i != 2 && (s0 || s1)) {
        if (s0 != s1) {
            const double e = s0 ? e0 : e1, K = s0 ? K0 : K1, p = s0 ? p0 : p1;
            plug = e;
            est = e;
            var = e / K * (1.0 / p - e);                  // Theorems 7, 9
            if (s0) a0 = 1.0; else a1 = 1.0;
        } else {
            const double e = ((double)h0 + (double)h1) / (K0 * p0 + K1 * p1);
            plug = e;
            const double V1 = fmax(e / K0 * (1.0 / p0 - e), 0.0);
            const double V2 = fmax(e / K1 * (1.0 / p1 - e), 0.0);
            if (V1 + V2 > 0.0) {
                a0 = V2 / (V1 + V2);
                a1 = V1 / (V1 + V2);
                var = V1 * V2 / (V1 + V2);                // Theorem 10
            } else {
                a0 = a1 = 0.5;
                var = 0.0;
            }
            est = a0 * e0 + a1 * e1;
        }
    }
    // eta_2 = Lambda_4 - sum_{Omega_3*} phi^(3)_i eta_i and its variance
    const bool om3 = cls && i != 2 && f3 > 0;
    const double s = warp_sum_d(om3 ? f3 * est : 0.0);
    double v2 = warp_sum_d(om3 ? f3 * f3 * var : 0.0);
    // sum_{i != j} phi_i phi_j Cov(i, j), Cov = -sum_l b_i b_j / K_l with
    // b_i = phi_i a^(l)_i plug_i: per l, (sum b)^2 - sum b^2
    const double b0 = om3 ? f3 * (a0 * plug) : 0.0, b1 = om3 ? f3 * (a1 * plug) : 0.0;
    const double sb0 = warp_sum_d(b0), sbb0 = warp_sum_d(b0 * b0);
    const double sb1 = warp_sum_d(b1), sbb1 = warp_sum_d(b1 * b1);
    if (av0) v2 -= (sb0 * sb0 - sbb0) / K0;
    if (av1) v2 -= (sb1 * sb1 - sbb1) / K1;
    if (i == 2) {
        est = u128_to_double(tot->lambda4) - s;
        var = v2;
    }
    const double t = warp_sum_d(cls ? est : 0.0);         // concentrations (Sec. 6.3)
    if (out && i < kSlots) {
        out->hits[0][i] = h0;
        out->hits[1][i] = h1;
        out->est[i] = est;
        out->var[i] = var;
        out->lambda[0][i] = a0;
        out->lambda[1][i] = a1;
        out->conc[i] = (cls && t != 0.0) ? est / t : 0.0;
    }
    if (out && i == 0) {
        out->k = 5;
        out->n_classes = 21;
        out->K[0] = in.K[0];
        out->K[1] = in.K[1];
        out->triangles = 0.0;
        out->triangles_var = 0.0;
    }
    if (cov) {
        // Cov(eta_r, eta_i) = -plug_r plug_i sum_l a_r a_i / K_l off the diagonal
        const bool sampled = cls && i != 2, rowr = row >= 1 && row <= 21 && row != 2;
        const double c0 = a0 * plug, c1 = a1 * plug;
        const double c0r = __shfl_sync(0xffffffffu, c0, row), c1r = __shfl_sync(0xffffffffu, c1, row);
        double c = 0.0;
        if (rowr && sampled) {
            if (i == row) {
                c = var;
            } else {
                if (av0) c -= c0r * c0 / K0;
                if (av1) c -= c1r * c1 / K1;
            }
        }
        // eta_2's linear identity: Cov(eta_2, eta_r) = -sum phi^(3)_j Cov(eta_j, eta_r)
        double c2 = 0.0;
        for (int j = 1; j <= 21; ++j) {
            const double cj = __shfl_sync(0xffffffffu, c, j);
            if (j != 2 && kPhi5[j - 1][2] > 0) c2 -= kPhi5[j - 1][2] * cj;
        }
        cov_row(cov, row, i, sampled, rowr, c, c2, true, var);
    }
}

// k = 4, alone (MOSS-4) or mixed with MOSS-4Min, with one warp: lane i is
// class i (1..6); the eta_2 identity, its variance and the covariances are
// formed on every lane from the values of classes 4, 5, 6 gathered by
// shuffles, in the order the formulas are written; the concentrations' sum
// is a warp sum.  The divisions, the slow part (FP64 runs at 1/64 of the FP32
// rate: about 1 us each in a dependent chain), are spread over the lanes: a
// lane per (class, c) slot of MOSS-4Min and per term of n_2's variance (one
// lane did 24 divisions in turn before, 52 us for the mix from a cold start).
__device__ void finalize4_warp(const FinalizeIn &in, const uint64_t *hits0, const uint64_t *hits1,
                               const DevTotals *tot, moss_result *out, double *cov, int row) {
    const int i = threadIdx.x & 31;
    const bool cls = i >= 1 && i <= 6, mix = in.mix != 0;
    const double G = u128_to_double(tot->gamma[0]), Gm = mix ? u128_to_double(tot->gamma[3]) : 0.0;
    const double K = (double)in.K[0], Km = (double)in.K[1];
    const bool av0 = in.K[0] > 0 && G > 0, av1 = mix && in.K[1] > 0 && Gm > 0;
    const uint64_t h0 = (i < kSlots && hits0) ? hits0[i] : 0, h1 = (i < kSlots && hits1) ? hits1[i] : 0;
    const bool s0 = av0 && cls && i != 2;
    double p = 0.0, e4 = 0.0;
    if (s0) {
        p = 2.0 * kPhi4[i - 1][0] / G;                    // Theorem 2
        e4 = (double)h0 / (K * p);
    }
    // MOSS-4Min: classes 3, 5, 6 from their (class, c) slots (Theorems 4, 5)
    const int first = i == 3 ? 0 : (i == 5 ? 4 : 10), nslot = i == 3 ? 4 : (i == 5 ? 6 : (i == 6 ? 12 : 0));
    const bool s1 = av1 && nslot > 0;
    double em = 0.0, h = 0.0;
    if (av1) {   // warp-uniform: lane l holds slot l's hits over its c and c^2
        const int c = i < 4 ? i + 1 : (i < 10 ? i - 3 : i - 9);
        const double ma = (double)h1 / c, mb = (double)h1 / (c * c);
        double sa = 0.0, sb = 0.0;
        for (int k = 0; k < 12; ++k) {
            const double x = __shfl_sync(0xffffffffu, ma, first + k), y = __shfl_sync(0xffffffffu, mb, first + k);
            if (k < nslot) {
                sa += x;
                sb += y;
            }
        }
        if (s1) em = Gm / (2.0 * Km) * sa;
        if (s1) h = sa > 0 ? sb / sa : (i == 6 ? 1.0 / 3.0 : 1.0);
    }
    double est = 0.0, var = 0.0, plug = 0.0, a0 = 0.0, a1 = 0.0;
    if (s0 != s1) {
        if (s0) {
            plug = est = e4;
            var = e4 / K * (1.0 / p - e4);                 // Theorem 3
            a0 = 1.0;
        } else {
            plug = est = em;
            var = (em * Gm * h / 2.0 - em * em) / Km;      // Theorem 5, per-CIS probabilities
            a1 = 1.0;
        }
    } else if (s0) {
        const double e = (K * e4 + Km * em) / (K + Km);
        plug = e;
        const double V1 = fmax(e / K * (1.0 / p - e), 0.0);
        const double V2 = fmax((e * Gm * h / 2.0 - e * e) / Km, 0.0);
        if (V1 + V2 > 0.0) {
            a0 = V2 / (V1 + V2);
            a1 = V1 / (V1 + V2);
            var = V1 * V2 / (V1 + V2);                     // Theorem 1
        } else {
            a0 = a1 = 0.5;
            var = 0.0;
        }
        est = a0 * e4 + a1 * em;
    }
    // classes 4, 5, 6 on every lane: n_2 = Lambda_3 - n_4 - 2 n_5 - 4 n_6 (eq. 2)
    double E[7], Vv[7], P[7], B0[7], B1[7];
    for (int c = 4; c <= 6; ++c) {
        E[c] = __shfl_sync(0xffffffffu, est, c);
        Vv[c] = __shfl_sync(0xffffffffu, var, c);
        P[c] = __shfl_sync(0xffffffffu, p, c);
        B0[c] = __shfl_sync(0xffffffffu, a0 * plug, c);
        B1[c] = __shfl_sync(0xffffffffu, a1 * plug, c);
    }
    const double est2 = u128_to_double(tot->lambda3) - E[4] - 2.0 * E[5] - 4.0 * E[6];
    const double coef[7] = {0, 0, 0, 0, 1.0, 2.0, 4.0};
    double v2 = 0.0;
    if (!mix) {
        if (av0) {
            const double s = E[4] + 2.0 * E[5] + 4.0 * E[6];
            v2 = (E[4] / P[4] + 4.0 * E[5] / P[5] + 16.0 * E[6] / P[6] - s * s) / K;
        }
    } else if (av0 || av1) {   // lane 3 (r - 4) + c - 4 forms the term of classes r, c
        const int l = i < 9 ? i : 0, r = 4 + l / 3, c = 4 + l % 3;
        auto of = [](const double (&x)[7], int k) { return k == 4 ? x[4] : (k == 5 ? x[5] : x[6]); };
        double cv = of(Vv, r);
        if (r != c) {
            cv = 0.0;
            if (av0) cv -= of(B0, r) * of(B0, c) / K;
            if (av1) cv -= of(B1, r) * of(B1, c) / Km;
        }
        for (int k = 0; k < 9; ++k) v2 += coef[4 + k / 3] * coef[4 + k % 3] * __shfl_sync(0xffffffffu, cv, k);
    }
    if (i == 2) {
        est = est2;
        var = v2;
    }
    const double t = warp_sum_d(cls ? est : 0.0);          // concentrations (Sec. 6.3)
    if (out && i < kSlots) {
        out->hits[0][i] = h0;
        out->hits[1][i] = h1;
        out->est[i] = est;
        out->var[i] = var;
        out->lambda[0][i] = mix ? a0 : 0.0;
        out->lambda[1][i] = mix ? a1 : 0.0;
        out->conc[i] = (cls && t != 0.0) ? est / t : 0.0;
    }
    if (out && i == 0) {
        out->k = 4;
        out->n_classes = 6;
        out->K[0] = mix ? (av0 ? in.K[0] : 0) : in.K[0];
        out->K[1] = mix ? (av1 ? in.K[1] : 0) : in.K[1];
        const double tri = av0 ? (double)h0 * G / (6.0 * K) : 0.0;
        out->triangles = tri;
        out->triangles_var = av0 ? tri / K * (G / 6.0 - tri) : 0.0;
    }
    if (cov) {
        // Cov(n_r, n_i) = -sum_l b_r b_i / K_l off the diagonal (b = a^(l) plug;
        // -n_r n_i / K for MOSS-4 alone)
        const bool have = mix || av0;
        const bool sampled = cls && i != 2, rowr = row >= 1 && row <= 6 && row != 2;
        const double b0 = mix ? a0 * plug : est, b1 = a1 * plug;
        const double b0r = __shfl_sync(0xffffffffu, b0, row), b1r = __shfl_sync(0xffffffffu, b1, row);
        double c = 0.0;
        if (have && rowr && sampled) {
            if (i == row) {
                c = var;
            } else if (mix) {
                if (av0) c -= b0r * b0 / K;
                if (av1) c -= b1r * b1 / Km;
            } else {
                c = -b0r * b0 / K;
            }
        }
        double c2 = 0.0;   // n_2's linear identity (eq. 2)
        for (int j = 4; j <= 6; ++j) c2 -= coef[j] * __shfl_sync(0xffffffffu, c, j);
        cov_row(cov, row, i, sampled, rowr, c, c2, have, v2);
    }
}

// called by a whole warp: a lane per class; out and cov are nullable
__device__ void finalize_any(const FinalizeIn &in, const uint64_t *hits0, const uint64_t *hits1,
                             const DevTotals *tot, moss_result *out, double *cov = nullptr, int row = 0) {
    if (in.k == 5 && !in.mix) finalize5_warp(in, hits0, hits1, tot, out, cov, row);
    else finalize4_warp(in, hits0, hits1, tot, out, cov, row);
}

// A block of one warp; with cov a block per row: every block finalizes (so
// nothing passes between them) and writes its row, block 0 also the result.
// One warp walking the 22 rows took 51 us, all of it FP64 division latency.
__global__ void k_finalize(FinalizeIn in, const __grid_constant__ HitsArg hits, const DevTotals *tot, moss_result *out,
                           double *cov) {
    const int row = blockIdx.x;
    await_previous();
    const uint64_t *h = hits.dev ? hits.dev : hits.h;
    finalize_any(in, h, h + kSlots, tot, row == 0 ? out : nullptr, cov, row);
}

// one warp per request of a batch
constexpr int kFinalizeWarps = 4;
__global__ void k_finalize_batch(const BatchRequest *reqs, int nreq, const uint64_t *task_counts,
                                 moss_result *out) {
    const int r = blockIdx.x * kFinalizeWarps + (threadIdx.x >> 5);
    if (r >= nreq) return;   // warp-uniform
    const BatchRequest q = reqs[r];
    const uint64_t *h0 = q.task[0] >= 0 ? task_counts + (uint64_t)q.task[0] * kSlots : nullptr;
    const uint64_t *h1 = q.task[1] >= 0 ? task_counts + (uint64_t)q.task[1] * kSlots : nullptr;
    finalize_any(q.in, h0, h1, q.tot, out + r);
}

}  // namespace

cudaError_t launch_finalize(const FinalizeIn &in, const HitsArg &hits, const DevTotals *tot, void *result, double *cov,
                            cudaStream_t s, bool early) {
    return launch_early(early, k_finalize, cov ? kSlots : 1, 32, s, in, hits, tot, static_cast<moss_result *>(result), cov);
}

cudaError_t launch_finalize_batch(const BatchRequest *reqs, int nreq, const uint64_t *task_counts, void *results,
                                  cudaStream_t s) {
    if (nreq <= 0) return cudaSuccess;
    k_finalize_batch<<<(nreq + kFinalizeWarps - 1) / kFinalizeWarps, 32 * kFinalizeWarps, 0, s>>>(
        reqs, nreq, task_counts, static_cast<moss_result *>(results));
    return cudaGetLastError();
}

}  // namespace moss
