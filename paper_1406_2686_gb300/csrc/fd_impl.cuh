#pragma once
// Device code of the FENE-P update that its kernels share: one node's update
// from a gathered stencil, and its feedback stress (scheme and stored variables:
// fd_kernels.cu).
#include "vefd_internal.cuh"

namespace vefd {

namespace {

template <int NC>
__device__ __forceinline__ constexpr int tidx(int i, int j) {
    // stored component of (i, j), -1 when identically zero (D2Q9 xz, yz)
    if (NC == 6) {
        return (i == 0) ? j : (i == 1 ? (j == 0 ? 1 : (j == 1 ? 3 : 4)) : (j == 0 ? 2 : (j == 1 ? 4 : 5)));
    } else {
        return (i == 0) ? (j == 0 ? 0 : (j == 1 ? 1 : -1))
             : (i == 1 ? (j == 0 ? 1 : (j == 1 ? 2 : -1)) : (j == 2 ? 3 : -1));
    }
}

template <int NC>
__device__ __forceinline__ constexpr bool is_diag(int k) {
    return NC == 6 ? (k == 0 || k == 3 || k == 5) : (k == 0 || k == 2 || k == 3);
}

template <int NC>
__device__ __forceinline__ constexpr int row_of(int k) {
    return NC == 6 ? (k <= 2 ? 0 : (k <= 4 ? 1 : 2)) : (k <= 1 ? 0 : (k == 2 ? 1 : 2));
}

template <int NC>
__device__ __forceinline__ constexpr int col_of(int k) {
    return NC == 6 ? (k == 0 ? 0 : (k == 1 ? 1 : (k == 2 ? 2 : (k == 3 ? 1 : 2)))) : (k == 0 ? 0 : (k <= 2 ? 1 : 2));
}

// Cholesky scheme (Sec. 2): sigma_P = f(r_P) C = L L^T with L lower
// triangular.  For the right-hand side dC/dt of the direct scheme,
//   d sigma_P/dt = f dC/dt + sigma_P f tr(dC/dt) / (L^2 - 3),
//   dL/dt = L Phi(L^-1 (d sigma_P/dt) L^-T),  Phi = lower triangle, diagonal halved,
// and AB2 advances lambda = (ln l_ii, l_ij for i > j) with the history of its
// rates.  The new C = L L^T / f with f = (L^2 - 3 + tr L L^T)/L^2 is SPD with
// tr C < L^2 whenever lambda is finite.  c and cnew hold C - I; Rk is dC/dt;
// Rprev and Rnew the lambda rates, in the stored component slots.
template <int NC>
__device__ __forceinline__ void chol_step(const float c[NC], const float Rk[NC], const float Rprev[NC], int have_prev,
                                          float L2m3, float cnew[NC], float Rnew[NC]) {
    float C[3][3], Cd[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int k = tidx<NC>(a, b);
            C[a][b] = (k < 0 ? 0.0f : c[k]) + (a == b ? 1.0f : 0.0f);
            Cd[a][b] = k < 0 ? 0.0f : Rk[k];
        }
    const float trt = NC == 6 ? c[0] + c[3] + c[5] : c[0] + c[2] + c[3];
    const float f = L2m3 / (L2m3 - trt);
    const float trd = Cd[0][0] + Cd[1][1] + Cd[2][2];
    const float g = f * trd / L2m3;
    float S[3][3], Sd[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            S[a][b] = f * C[a][b];
            Sd[a][b] = f * Cd[a][b] + S[a][b] * g;
        }
    // S = L L^T and the inverse of L
    float L[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j <= i; ++j) {
            float v = S[i][j];
#pragma unroll
            for (int k = 0; k < j; ++k) v -= L[i][k] * L[j][k];
            L[i][j] = (i == j) ? sqrtf(v) : v / L[j][j];
        }
    float Li[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        Li[j][j] = 1.0f / L[j][j];
#pragma unroll
        for (int i = j + 1; i < 3; ++i) {
            float v = 0.0f;
#pragma unroll
            for (int k = j; k < i; ++k) v -= L[i][k] * Li[k][j];
            Li[i][j] = v / L[i][i];
        }
    }
    // A = L^-1 Sd L^-T (symmetric; lower triangle), Phi(A), dL/dt = L Phi(A)
    float T[3][3], P[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            float v = 0.0f;
#pragma unroll
            for (int k = 0; k <= i; ++k) v += Li[i][k] * Sd[k][j];
            T[i][j] = v;
        }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            float v = 0.0f;
            if (j <= i) {
#pragma unroll
                for (int k = 0; k <= j; ++k) v += T[i][k] * Li[j][k];
                if (i == j) v *= 0.5f;
            }
            P[i][j] = v;
        }
    float Ln[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        const int i = col_of<NC>(k), j = row_of<NC>(k);  // lower-triangle entry (i >= j)
        float ld = 0.0f;
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (q >= j && q <= i) ld += L[i][q] * P[q][j];
        const float lam = (i == j) ? logf(L[i][i]) : L[i][j];
        const float rl = (i == j) ? ld / L[i][i] : ld;
        const float lamn = lam + (have_prev ? 1.5f * rl - 0.5f * Rprev[k] : rl);
        Ln[i][j] = (i == j) ? expf(lamn) : lamn;
        Rnew[k] = rl;
    }
    float Sn[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            float v = 0.0f;
#pragma unroll
            for (int q = 0; q < 3; ++q) v += Ln[a][q] * Ln[b][q];
            Sn[a][b] = v;
        }
    const float inv_fn = (L2m3 + 3.0f) / (L2m3 + Sn[0][0] + Sn[1][1] + Sn[2][2]);
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        const int a = row_of<NC>(k), b = col_of<NC>(k);
        cnew[k] = Sn[a][b] * inv_fn - (a == b ? 1.0f : 0.0f);
    }
}

// FENE-P update at one node from its gathered stencil.  v(k, d) returns field
// k (0..NC-1: C - I components, NC..NC+D-1: velocity components) at stencil
// point d (0 centre, 1 -x, 2 +x, 3 -y, 4 +y, 5 -z, 6 +z); hy1 and hy2 are the
// y weights of the first and second differences (1/2 and 1 inside, 1 and 0
// at a wall row, where the -y or +y point is the node itself).  Writes the new
// C - I to cnew, the right-hand side to Rnew, and returns the guard bits.
template <int D, int NC, class V>
__device__ __forceinline__ unsigned fenep_compute(V v, float hy1, float hy2, const float Rprev[NC], const StepParams& p,
                                                  float cnew[NC], float Rnew[NC]) {
    // velocity gradient Gu[a][b] = d_a u_b and the local velocity
    float Gu[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
    float uu[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int b = 0; b < D; ++b) {
        uu[b] = v(NC + b, 0);
        Gu[0][b] = 0.5f * (v(NC + b, 2) - v(NC + b, 1));
        Gu[1][b] = hy1 * (v(NC + b, 4) - v(NC + b, 3));
        if (D == 3) Gu[2][b] = 0.5f * (v(NC + b, 6) - v(NC + b, 5));
    }
    float c[NC], adv[NC], lap[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        const float c0 = v(k, 0);
        const float cxm = v(k, 1), cxp = v(k, 2), cym = v(k, 3), cyp = v(k, 4);
        c[k] = c0;
        float a = uu[0] * 0.5f * (cxp - cxm) + uu[1] * hy1 * (cyp - cym);
        float l = (cxp - 2.0f * c0 + cxm) + hy2 * (cyp - 2.0f * c0 + cym);
        if (D == 3) {
            const float czm = v(k, 5), czp = v(k, 6);
            a += uu[2] * 0.5f * (czp - czm);
            l += czp - 2.0f * c0 + czm;
        }
        adv[k] = a;
        lap[k] = l;
    }
    const float tr = NC == 6 ? c[0] + c[3] + c[5] : c[0] + c[2] + c[3];
    const float fm1 = tr / (p.L2m3 - tr);
    const float f = 1.0f + fm1;
    // full C = Ct + I as a 3x3 matrix
    float Cm[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int k = tidx<NC>(a, b);
            Cm[a][b] = (k < 0 ? 0.0f : c[k]) + (a == b ? 1.0f : 0.0f);
        }
    float Rc[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        const int a = row_of<NC>(k), b = col_of<NC>(k);
        float up = 0.0f;
#pragma unroll
        for (int e = 0; e < D; ++e) up += Cm[a][e] * Gu[e][b] + Gu[e][a] * Cm[e][b];
        const float relax = (f * c[k] + (is_diag<NC>(k) ? fm1 : 0.0f)) * p.inv_tau_p;
        Rc[k] = -adv[k] + up - relax + p.kappa * lap[k];
    }
    if (p.chol) {
        chol_step<NC>(c, Rc, Rprev, p.have_prev, p.L2m3, cnew, Rnew);
    } else {
        // Compensated AB2: the sum c + inc is rounded to FP32, and its exact
        // rounding error e (Knuth's TwoSum) is carried into the next step's
        // increment through the stored history, R~ = R - 2e, so that
        // 3/2 R' - 1/2 R~ = 3/2 R' - 1/2 R + e.  Near steady state the increment
        // falls below half an ulp of C - I; without the carry it would be lost
        // and C would stall up to (tau_P / f) ulp short of the fixed point.
        // The history then stays within FP32 rounding of max(|R|, |e|).
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const float inc = p.have_prev ? 1.5f * Rc[k] - 0.5f * Rprev[k] : Rc[k];
            const float sum = c[k] + inc;
            const float inc_kept = sum - c[k];
            const float err = (c[k] - (sum - inc_kept)) + (inc - inc_kept);
            cnew[k] = sum;
            Rnew[k] = fmaf(-2.0f, err, Rc[k]);
        }
    }
    float trn = 0.0f;
    bool bad = false;
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        if (is_diag<NC>(k)) trn += cnew[k];
        bad |= isnan(cnew[k]);
    }
    if (bad || isnan(tr)) return kStNan;
    if (trn >= p.L2m3 || tr >= p.L2m3) return kStTrace;
    return 0u;
}

// Feedback stress at one node, Q = (f C - I) m(phi) = (f Ct + (f - 1) I) m(phi)
// with f - 1 = tr Ct / (L^2 - 3 - tr Ct) and m = 1, f_+(phi) or f_-(phi)
// (Eq. NS and the last equation of Sec. 2); stored as the NQ components
// xx xy xz yy yz zz (3D) or xx xy yy (2D) that the divergence needs.
template <class L, int NCOMP>
__device__ __forceinline__ void store_feedback(const float c[L::NC], const float d[NCOMP], const StepParams& p,
                                               float* __restrict__ Q, long long N, long long i) {
    const float tr = L::NC == 6 ? c[0] + c[3] + c[5] : c[0] + c[2] + c[3];
    const float fm1 = tr / (p.L2m3 - tr);
    const float f = 1.0f + fm1;
    float m = 1.0f;
    if (p.phase != 0) {
        float phi = 1.0f;  // one component: phi = 1 everywhere
        if (NCOMP == 2) {
            const float ra = p.rho_ref[0] + d[0], rb = p.rho_ref[1] + d[NCOMP - 1];
            phi = (ra - rb) / (ra + rb);
        }
        const float t = tanhf(phi * p.inv_delta);
        m = p.phase > 0 ? 0.5f * (1.0f + t) : 0.5f * (1.0f - t);
    }
    if (L::NC == 6) {
#pragma unroll
        for (int k = 0; k < 6; ++k) Q[k * N + i] = (f * c[k] + (is_diag<6>(k) ? fm1 : 0.0f)) * m;
    } else {
        Q[i] = (f * c[0] + fm1) * m;          // xx
        Q[N + i] = (f * c[1]) * m;            // xy
        Q[2 * N + i] = (f * c[2] + fm1) * m;  // yy
    }
}

}  // namespace
}  // namespace vefd
