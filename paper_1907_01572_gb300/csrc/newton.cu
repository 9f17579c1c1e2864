// Zeroth-order term and the puncture equation (Sec. II.E.6 eq. operator_oh,
// Sec. III.B nonlinear terms at GL points, Sec. III.D puncture data).
//
// * Finest level: int f u v is evaluated at the volume GL points with the
//   coefficient c0 = w det J f folded into the apply kernel.
// * Coarse levels: the Galerkin form O^H = (I_h^H)^T O^h I_h^H.  Because the
//   prolongation interpolates exactly (coarse spaces are nested in the fine
//   ones), O^H_ab = sum over the finest descendants' GL points x_q of
//   c0_q phi(x_q) with phi = psi^H_a psi^H_b, a polynomial of degree 2p per
//   direction, which its values at the m = 2p + 1 GL points y_k of the coarse
//   element determine: phi(x_q) = sum_k L_k(x_q) phi(y_k).  So the coarse
//   coefficient c_k = sum_q c0_q L_k(x_q) carries the whole term, and (spaces
//   nested level by level) it follows from the next finer level's coefficient
//   by one transposed interpolation per child.  The dense block is then
//   O^H_ab = sum_k c_k psi_a(y_k) psi_b(y_k), summed direction by direction over
//   the pairs (c, c'), (b, b'), (a, a') with c <= c' and so on.  Work per
//   element at n = 7: 0.3 M multiply-adds and 0.1 M per child (summing every
//   entry over every finest point: 6.6 M per finest descendant).
// * Puncture: 1/alpha = sum_I m_I / (2 r_I); A_ij = sum_I 3/(2 r_I^2)
//   [P_i n_j + P_j n_i - (delta_ij - n_i n_j) P.n] + 3/r_I^3 [n_i w_j + n_j w_i],
//   w = S_I x n (the spin term of eq. Two_Punctures_Aij, its symmetrisation
//   taken as t_(ij) = (t_ij + t_ji) / 2); beta = alpha^7 A_ij A_ij / 8.  Source s(u) = beta (1 + alpha (1 + u))^-7,
//   Jacobian coefficient f(u) = 7 alpha beta (1 + alpha (1 + u))^-8.
// * Power-law source (the constant-density star of Sec. III.C,
//   Lap psi + 2 pi rho psi^5 = 0): s(u) = c u^k, f(u) = -k c u^(k-1), with c
//   given at the GL points; the nonlinear term is evaluated at the GL points
//   after interpolating u there, as the paper describes for that problem.
#include "newton.h"

namespace dg {
namespace {

__global__ void puncture_kernel(const double* vxyz, long long n, PunctureDev P, double* alpha, double* beta) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double x[3] = {vxyz[i], vxyz[n + i], vxyz[2 * n + i]};
        double inv_a = 0.0, A[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
        for (int I = 0; I < P.n; ++I) {
            double dx[3], r2 = 0.0;
            for (int k = 0; k < 3; ++k) {
                dx[k] = x[k] - P.c[I][k];
                r2 += dx[k] * dx[k];
            }
            const double r = sqrt(r2);
            double nv[3];
            for (int k = 0; k < 3; ++k) nv[k] = dx[k] / r;
            const double Pn = P.P[I][0] * nv[0] + P.P[I][1] * nv[1] + P.P[I][2] * nv[2];
            const double f = 1.5 / r2, fs = 3.0 / (r2 * r);
            const double w[3] = {P.S[I][1] * nv[2] - P.S[I][2] * nv[1], P.S[I][2] * nv[0] - P.S[I][0] * nv[2],
                                 P.S[I][0] * nv[1] - P.S[I][1] * nv[0]};   // S x n
            for (int a = 0; a < 3; ++a)
                for (int b = 0; b < 3; ++b)
                    A[a][b] += f * (P.P[I][a] * nv[b] + P.P[I][b] * nv[a] - ((a == b ? 1.0 : 0.0) - nv[a] * nv[b]) * Pn) +
                               fs * (nv[a] * w[b] + nv[b] * w[a]);
            inv_a += P.m[I] / (2.0 * r);
        }
        double AA = 0.0;
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b) AA += A[a][b] * A[a][b];
        const double al = 1.0 / inv_a;
        const double a2 = al * al, a4 = a2 * a2;
        alpha[i] = al;
        beta[i] = a4 * a2 * al * AA / 8.0;
    }
}

// per element: S = I^T (w det J s(u~)), optional jac = w det J f(u~) at GL points
__global__ void nl_kernel(NlArgs a, const double* u, double* S, double* jac64, float* jac32) {
    const int e = blockIdx.x;
    if (e >= a.n_elems) return;
    const int n = a.p[e] + 1, n2 = n * n, n3 = n2 * n;
    __shared__ double b0[kMaxN * kMaxN * kMaxN], b1[kMaxN * kMaxN * kMaxN];
    const double* I = a.tab + tab_n(TabIndex::I, n);
    const long long vo = a.vqp_off[e], dofo = a.dof_off[e];
    if (n < kMinN || n > kMaxN || vo < 0 || vo + n3 > a.n_vqp) {
        if (threadIdx.x == 0) atomicExch(a.chk, 2);
        return;
    }
    for (int k = threadIdx.x; k < n3; k += blockDim.x) b0[k] = u[dofo + k];
    __syncthreads();
    // u at GL points: three forward passes (x, y, z)
    for (int k = threadIdx.x; k < n3; k += blockDim.x) {
        const int i = k % n, r = k / n;
        double s = 0.0;
        for (int m = 0; m < n; ++m) s += I[i * n + m] * b0[m + n * r];
        b1[k] = s;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < n3; k += blockDim.x) {
        const int i = k % n, j = (k / n) % n, l = k / n2;
        double s = 0.0;
        for (int m = 0; m < n; ++m) s += I[j * n + m] * b1[i + n * (m + n * l)];
        b0[k] = s;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < n3; k += blockDim.x) {
        const int ij = k % n2, l = k / n2;
        double s = 0.0;
        for (int m = 0; m < n; ++m) s += I[l * n + m] * b0[ij + n2 * m];
        b1[k] = s;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < n3; k += blockDim.x) {
        const double wd = a.wdetJ[vo + k];
        double s, jc;
        if (a.kind == kNlPower) {
            const double c = a.alpha[vo + k], uq = b1[k];
            double pk1 = 1.0;                   // u^(k-1)
            for (int q = 1; q < a.power; ++q) pk1 *= uq;
            s = c * pk1 * uq;
            jc = -a.power * c * pk1;            // d(-s)/du: the source grows with u
        } else {
            const double al = a.alpha[vo + k], be = a.beta[vo + k];
            const double base = 1.0 + al * (1.0 + b1[k]);
            const double b2 = base * base, b4 = b2 * b2, b8 = b4 * b4;
            s = be * base / b8;                 // beta base^-7
            jc = 7.0 * al * be / b8;
        }
        if (jac64) {
            jac64[vo + k] = wd * jc;
            jac32[vo + k] = (float)(wd * jc);
        }
        b0[k] = wd * s;
    }
    __syncthreads();
    // lift: three transposed passes
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
        if (S) S[dofo + k] = s;
    }
}

// R = Lu - S - F
__global__ void sub_kernel(const double* Lu, const double* S, const double* F, double* R, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        R[i] = Lu[i] - S[i] - (F ? F[i] : 0.0);
}

// out (= or +=) sum_j W[k][j] in[.. j ..]: one direction of a transposed interpolation, of a cube with
// dims (d0, d1, d2) to m points along `dir`.
__device__ void interp_pass(const double* in, double* out, const double* W, int dir, int d0, int d1, int d2, int m,
                            bool add) {
    const int q = dir == 0 ? d0 : (dir == 1 ? d1 : d2);
    const int e0 = dir == 0 ? m : d0, e1 = dir == 1 ? m : d1, e2 = dir == 2 ? m : d2;
    const int si = dir == 0 ? 1 : (dir == 1 ? d0 : d0 * d1);
    for (int idx = threadIdx.x; idx < e0 * e1 * e2; idx += blockDim.x) {
        const int a = idx % e0, b = (idx / e0) % e1, c = idx / (e0 * e1);
        const int k = dir == 0 ? a : (dir == 1 ? b : c);
        const double* v = in + (dir == 0 ? 0 : a) + d0 * ((dir == 1 ? 0 : b) + d1 * (dir == 2 ? 0 : c));
        const double* w = W + k * kGalM;
        double s = 0.0;
        for (int j = 0; j < q; ++j) s += w[j] * v[j * si];
        out[idx] = add ? out[idx] + s : s;
    }
}

// Coefficients of one coarse level (block per element, its children in turn).
__global__ void galerkin_coef_kernel(GalerkinArgs g, const double* __restrict__ cf, double* __restrict__ coef) {
    extern __shared__ double gal_smem[];
    constexpr int M3 = kGalM * kGalM * kGalM;
    double *b0 = gal_smem, *b1 = b0 + M3, *acc = b1 + M3;
    const int H = blockIdx.x;
    const int n = g.pH[H] + 1, m = 2 * n - 1, m3 = m * m * m;
    const long long off = g.off[H];
    if (n < kMinN || n > kMaxN || off < 0 || off + m3 > g.n_coef) {
        if (threadIdx.x == 0) atomicExch(g.chk, 3);
        return;
    }
    for (int k = threadIdx.x; k < m3; k += blockDim.x) acc[k] = 0.0;
    for (int ci = g.child_off[H]; ci < g.child_off[H + 1]; ++ci) {
        const int f = g.child_id[ci], bits = g.child_bits[ci];
        const int nf = g.pf[f] + 1, q = g.fine_is_finest ? nf : 2 * nf - 1, q3 = q * q * q;
        const long long of = g.off_f[f];
        if (nf < kMinN || nf > kMaxN || of < 0 || of + q3 > g.n_coef_f) {
            if (threadIdx.x == 0) atomicExch(g.chk, 4);
            break;
        }
        for (int k = threadIdx.x; k < q3; k += blockDim.x) b0[k] = cf[of + k];
        __syncthreads();
        const double* W[3];
        for (int d = 0; d < 3; ++d) W[d] = g.tab + GalerkinTab::w(n, q, bits == 0xFF ? 2 : (bits >> d) & 1);
        interp_pass(b0, b1, W[0], 0, q, q, q, m, false);
        __syncthreads();
        interp_pass(b1, b0, W[1], 1, m, q, q, m, false);
        __syncthreads();
        interp_pass(b0, acc, W[2], 2, m, m, q, m, true);
        __syncthreads();
    }
    __syncthreads();
    for (int k = threadIdx.x; k < m3; k += blockDim.x) coef[off + k] = acc[k];
}

// Entries of one element's block with z indices (c, c') or (c', c): a CTA per pair.
__global__ void galerkin_block_kernel(GalerkinArgs g, const double* __restrict__ coef, double* __restrict__ O64,
                                      float* __restrict__ O32) {
    constexpr int NP = kMaxN * (kMaxN + 1) / 2;
    __shared__ double E[kGalM][kMaxN], ez[kGalM], T1[kGalM * kGalM], T2[NP][kGalM], S[NP][NP];
    __shared__ unsigned char pa[NP], pb[NP];
    const int H = blockIdx.x, n = g.pH[H] + 1, n3 = n * n * n, m = 2 * n - 1, np = n * (n + 1) / 2;
    if ((int)blockIdx.y >= np) return;
    const long long off = g.off[H], oo = g.Ob_off[H];
    if (n < kMinN || n > kMaxN || off < 0 || off + m * m * m > g.n_coef || oo < 0 || oo + (long long)n3 * n3 > g.ob_total) {
        if (threadIdx.x == 0) atomicExch(g.chk, 5);
        return;
    }
    for (int k = threadIdx.x; k < m * n; k += blockDim.x) E[k / n][k % n] = g.tab[GalerkinTab::e(n) + (k / n) * kGalM + k % n];
    for (int k = threadIdx.x; k < n * n; k += blockDim.x) {
        const int a = k % n, b = k / n;
        if (a <= b) {
            pa[b * (b + 1) / 2 + a] = a;
            pb[b * (b + 1) / 2 + a] = b;
        }
    }
    __syncthreads();
    const int c = pa[blockIdx.y], c2 = pb[blockIdx.y];
    if (threadIdx.x < m) ez[threadIdx.x] = E[threadIdx.x][c] * E[threadIdx.x][c2];
    __syncthreads();
    for (int ij = threadIdx.x; ij < m * m; ij += blockDim.x) {
        double s = 0.0;
        for (int k = 0; k < m; ++k) s += coef[off + ij + m * m * k] * ez[k];
        T1[ij] = s;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < np * m; k += blockDim.x) {
        const int i = k % m, b = k / m;
        double s = 0.0;
        for (int j = 0; j < m; ++j) s += T1[i + m * j] * (E[j][pa[b]] * E[j][pb[b]]);
        T2[b][i] = s;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < np * np; k += blockDim.x) {
        const int a = k % np, b = k / np;
        double s = 0.0;
        for (int i = 0; i < m; ++i) s += T2[b][i] * (E[i][pa[a]] * E[i][pb[a]]);
        S[b][a] = s;
    }
    __syncthreads();
    const int n2 = n * n;
    for (int k = threadIdx.x; k < n2 * n2; k += blockDim.x) {   // rows (a', b') fastest: runs of n^2 values
        const int r = k % n2, l = k / n2;
        const int a2 = r % n, b2 = r / n, a = l % n, b = l / n;
        const int ia = a < a2 ? a2 * (a2 + 1) / 2 + a : a * (a + 1) / 2 + a2;
        const int ib = b < b2 ? b2 * (b2 + 1) / 2 + b : b * (b + 1) / 2 + b2;
        const double v = S[ib][ia];
        const long long p0 = oo + (long long)(l + n2 * c) * n3 + r + n2 * c2;
        const long long p1 = oo + (long long)(l + n2 * c2) * n3 + r + n2 * c;
        O64[p0] = v;
        O64[p1] = v;
        O32[p0] = (float)v;
        O32[p1] = (float)v;
    }
}

inline int grid_for(long long n) {
    long long g = (n + 255) / 256;
    return (int)(g < 1 ? 1 : (g > 2432 ? 2432 : g));
}

}  // namespace

cudaError_t launch_puncture(const double* vxyz, long long n, const PunctureDev& P, double* alpha, double* beta,
                            cudaStream_t st) {
    puncture_kernel<<<grid_for(n), 256, 0, st>>>(vxyz, n, P, alpha, beta);
    return cudaGetLastError();
}

cudaError_t launch_nl(const NlArgs& a, const double* u, double* S, double* jac64, float* jac32, cudaStream_t st) {
    nl_kernel<<<a.n_elems, 128, 0, st>>>(a, u, S, jac64, jac32);
    return cudaGetLastError();
}

cudaError_t launch_sub(const double* Lu, const double* S, const double* F, double* R, long long n, cudaStream_t st) {
    sub_kernel<<<grid_for(n), 256, 0, st>>>(Lu, S, F, R, n);
    return cudaGetLastError();
}

cudaError_t launch_galerkin(const GalerkinArgs& g, int max_n, const double* coef_f, double* coef, double* O64,
                            float* O32, cudaStream_t st) {
    const size_t smem = sizeof(double) * 3 * kGalM * kGalM * kGalM;
    static const cudaError_t attr =   // once per process, thread-safe initialisation
        cudaFuncSetAttribute(galerkin_coef_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (attr != cudaSuccess) return attr;
    galerkin_coef_kernel<<<g.n_coarse, 512, smem, st>>>(g, coef_f, coef);
    galerkin_block_kernel<<<dim3(g.n_coarse, max_n * (max_n + 1) / 2), 128, 0, st>>>(g, coef, O64, O32);
    return cudaGetLastError();
}

}  // namespace dg
