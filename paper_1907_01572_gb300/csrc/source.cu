// Right-hand side of eq. (equationFh2) with Dirichlet data:
//   F_alpha = int_e g psi_alpha  - int_{Gamma_D} g_D n . grad psi_alpha + int_{Gamma_D} sigma g_D psi_alpha,
// volume part by GL quadrature with the interpolation matrix I (Sec. II.A.5),
// boundary part at the boundary mortars' GL points with the side's metric
// factors c = (J^-1) n (so n . grad psi = c . grad_xi psi).
#include "source.h"

namespace dg {
namespace {

__device__ inline void tangential(int d, int& t1, int& t2) {
    t1 = d == 0 ? 1 : 0;
    t2 = d == 2 ? 1 : 2;
}

__global__ void rhs_kernel(RhsArgs a, const double* g, const double* gD, double* F) {
    const int e = blockIdx.x;
    if (e >= a.n_elems) return;
    const int n = a.p[e] + 1, n2 = n * n, n3 = n2 * n;
    __shared__ double b0[kMaxN * kMaxN * kMaxN], b1[kMaxN * kMaxN * kMaxN], Fe[kMaxN * kMaxN * kMaxN];
    __shared__ double P[4 * kMaxN * kMaxN], X[3 * kMaxN * kMaxN];
    const double* I = a.tab + tab_n(TabIndex::I, n);
    const long long vo = a.vqp_off[e];
    for (int k = threadIdx.x; k < n3; k += blockDim.x) b0[k] = g ? a.wdetJ[vo + k] * g[vo + k] : 0.0;
    __syncthreads();
    // F = (I^T x I^T x I^T) b0, one axis at a time
    for (int k = threadIdx.x; k < n3; k += blockDim.x) {
        const int i = k % n, r = k / n;
        double s = 0.0;
        for (int m = 0; m < n; ++m) s += I[m * n + i] * b0[m + n * r];
        b1[k] = s;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < n3; k += blockDim.x) {
        const int i = k % n, j = (k / n) % n, l = k / n2;
        double s = 0.0;
        for (int m = 0; m < n; ++m) s += I[m * n + j] * b1[i + n * (m + n * l)];
        b0[k] = s;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < n3; k += blockDim.x) {
        const int ij = k % n2, l = k / n2;
        double s = 0.0;
        for (int m = 0; m < n; ++m) s += I[m * n + l] * b0[ij + n2 * m];
        Fe[k] = s;
    }
    __syncthreads();
    if (gD) {
        const int st[3] = {1, n, n2};
        const double* DL = a.tab + tab_n(TabIndex::DL, n);
        for (int s = a.slot_off[e]; s < a.slot_off[e + 1]; ++s) {
            const Mortar M = a.mortars[a.slot_mortar[s]];
            if (M.eB >= 0) continue;
            const int f = a.slot_face[s], d = f >> 1, fn = (f & 1) ? n - 1 : 0;
            int t1, t2;
            tangential(d, t1, t2);
            const int q = M.q, q2 = q * q;
            const double* Im = a.tab + tab_m(TabIndex::Im, n, q, 0);
            const double* Dm = a.tab + tab_m(TabIndex::Dm, n, q, 0);
            const double* mg = a.mg + 7 * M.goff;
            const double sig = a.sigma[a.slot_mortar[s]];
            // flux factors at the mortar points, then lifted direction by direction (FP64 arithmetic bounds
            // the kernel: 7 q n^2 multiply-adds a face instead of 10 q^2 n^2 point by point)
            double *PA = P, *P1 = PA + q2, *P2 = P1 + q2, *Pn = P2 + q2;
            for (int pt = threadIdx.x; pt < q2; pt += blockDim.x) {
                const double v = mg[pt] * gD[M.bnd_off + pt];
                PA[pt] = sig * v;
                P1[pt] = -v * mg[(1 + t1) * q2 + pt];
                P2[pt] = -v * mg[(1 + t2) * q2 + pt];
                Pn[pt] = -v * mg[(1 + d) * q2 + pt];
            }
            __syncthreads();
            double *X1 = X, *X2 = X1 + q * n, *X3 = X2 + q * n;
            for (int k = threadIdx.x; k < q * n; k += blockDim.x) {
                const int i1 = k % q, bb = k / q;
                double x1 = 0.0, x2 = 0.0, x3 = 0.0;
                for (int i2 = 0; i2 < q; ++i2) {
                    const double iv = Im[i2 * n + bb], dv = Dm[i2 * n + bb];
                    const int pt = i1 + q * i2;
                    x1 += iv * PA[pt] + dv * P2[pt];
                    x2 += iv * P1[pt];
                    x3 += iv * Pn[pt];
                }
                X1[k] = x1;
                X2[k] = x2;
                X3[k] = x3;
            }
            __syncthreads();
            for (int k = threadIdx.x; k < n2; k += blockDim.x) {
                const int aa = k % n, bb = k / n;
                double fu = 0.0, fd = 0.0;
                for (int i1 = 0; i1 < q; ++i1) {
                    const double iv = Im[i1 * n + aa], dv = Dm[i1 * n + aa];
                    fu += iv * X1[i1 + q * bb] + dv * X2[i1 + q * bb];
                    fd += iv * X3[i1 + q * bb];
                }
                const int base = aa * st[t1] + bb * st[t2];
                Fe[base + fn * st[d]] += fu;
                for (int c = 0; c < n; ++c) Fe[base + c * st[d]] += DL[fn * n + c] * fd;
            }
            __syncthreads();
        }
    }
    for (int k = threadIdx.x; k < n3; k += blockDim.x) F[a.dof_off[e] + k] = Fe[k];
}

__global__ void scale_coef_kernel(const double* wdetJ, const double* coef, double* c64, float* c32, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double v = wdetJ[i] * coef[i];
        c64[i] = v;
        c32[i] = (float)v;
    }
}

}  // namespace

cudaError_t launch_rhs(const RhsArgs& a, const double* g_qp, const double* gD_qp, double* F, cudaStream_t st) {
    rhs_kernel<<<a.n_elems, 128, 0, st>>>(a, g_qp, gD_qp, F);
    return cudaGetLastError();
}

cudaError_t launch_scale_coef(const double* wdetJ, const double* coef, double* c64, float* c32, long long n,
                              cudaStream_t st) {
    long long g = (n + 255) / 256;
    if (g > 2432) g = 2432;
    if (g < 1) g = 1;
    scale_coef_kernel<<<(int)g, 256, 0, st>>>(wdetJ, coef, c64, c32, n);
    return cudaGetLastError();
}

}  // namespace dg
