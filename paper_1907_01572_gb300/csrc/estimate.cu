// A-posteriori error estimator (Sec. II.D): eta^2(e) of eq. (Eta2_Local) with
// the ingredients of eq. (Eta2_Ingredients) and the weights of eq.
// (Eta2_Integrals), for -Lap u + f u = g with Dirichlet data g_D.
//
// One CTA per element, one volume GL point per thread.  The element residual
// R = f u - g - Lap u needs the exact Laplacian of the mapped polynomial:
// with J = dx/dxi, H the reference Hessian of u and X^k the reference Hessian
// of the coordinate x_k (all polynomials of the element's LGL basis),
//   Hess_x u = J^-T (H - sum_k (du/dx_k) X^k) J^-1.
// Each reference derivative of a nodal field at the GL points is three
// sum-factorised passes with the 1-D matrices of the LGL basis at the GL
// points: values I, first derivatives, and second derivatives (the first
// derivative matrix times the LGL-node derivative matrix, exact because the
// derivative of a degree-p polynomial is held by its LGL values).
// On multi-block meshes the geometry is the exact block map (as in the
// operator): J and X^k come from the map's first and second derivatives at
// the GL points (blocks.h), composed with the element's linear map into its
// block.  With a fiducial grid the integrands stay those of the physical grid
// and the weights (w det J, w S), h_e, h_m and sigma are the fiducial grid's.
// The mortar terms read the trace buffer that an FP64 apply of u leaves
// behind: u and n_A . grad u of both sides at the mortar's GL points; each
// element sums the mortars of its own slots, so every interior mortar counts
// in full for both of its elements and the result needs no atomics.
#include "blocks.h"
#include "estimate.h"

namespace dg {
namespace {

constexpr int kEstThreads = 768;   // >= kMaxN^3 = 729
constexpr int kNV = kMaxN * kMaxN * kMaxN;
constexpr int kEstMaxSlots = 24;   // four mortars on each of six faces

// The kernel is bound by FP64 arithmetic (two operations per clock and SM), so
// it shares the partial passes of the derivatives (19 n^4 multiply-adds for the
// value, gradient and Hessian of u instead of 30 n^4), contracts the block
// map's second derivatives with the gradient before expanding them, divides
// once per point and length, and leaves the mortar sums to one warp per slot.
// 1,056 elements of the cubed sphere, n = 5..9: 1.75 -> 0.43 ms.

struct Derivs {            // value, first and second reference derivatives (00, 11, 22, 01, 02, 12) at a point
    double v, d[3], h[6];
};

// Derivatives of the nodal field F (n^3 values, x fastest) at GL point k of
// this thread (0 when k >= n^3): value and gradient (LOW), Hessian (HIGH).
// Every thread of the CTA calls it.
template <bool LOW, bool HIGH>
__device__ void eval_derivs(const double* F, double* T1, double* T2, const double* const* M, int n, int k, Derivs& o) {
    const int n2 = n * n, n3 = n2 * n, ij = k % n2, l = k / n2;
    auto zdot = [&](const double* T, const double* Z) {
        double v = 0.0;
        if (k < n3)
            for (int m = 0; m < n; ++m) v += Z[l * n + m] * T[ij + n2 * m];
        return v;
    };
    for (int d0 = 0; d0 < (HIGH ? 3 : 2); ++d0) {
        const double* A = M[d0];
        for (int t = threadIdx.x; t < n3; t += blockDim.x) {
            const int i = t % n, r = t / n;
            double s = 0.0;
            for (int m = 0; m < n; ++m) s += A[i * n + m] * F[m + n * r];
            T1[t] = s;
        }
        __syncthreads();
        const int ny = (HIGH ? 3 : 2) - d0;   // derivatives along y: 0 .. ny - 1
        for (int t = threadIdx.x; t < n3; t += blockDim.x) {
            const int i = t % n, j = (t / n) % n, c = t / n2;
            double s0 = 0.0, s1 = 0.0, s2 = 0.0;
            for (int m = 0; m < n; ++m) {
                const double v = T1[i + n * (m + n * c)];
                s0 += M[0][j * n + m] * v;
                if (ny > 1) s1 += M[1][j * n + m] * v;
                if (ny > 2) s2 += M[2][j * n + m] * v;
            }
            T2[t] = s0;
            if (ny > 1) T2[kNV + t] = s1;
            if (ny > 2) T2[2 * kNV + t] = s2;
        }
        __syncthreads();
        if (d0 == 0) {
            if (LOW) {
                o.v = zdot(T2, M[0]);
                o.d[1] = zdot(T2 + kNV, M[0]);
                o.d[2] = zdot(T2, M[1]);
            }
            if (HIGH) {
                o.h[1] = zdot(T2 + 2 * kNV, M[0]);
                o.h[2] = zdot(T2, M[2]);
                o.h[5] = zdot(T2 + kNV, M[1]);
            }
        } else if (d0 == 1) {
            if (LOW) o.d[0] = zdot(T2, M[0]);
            if (HIGH) {
                o.h[3] = zdot(T2 + kNV, M[0]);
                o.h[4] = zdot(T2, M[1]);
            }
        } else {
            o.h[0] = zdot(T2, M[0]);
        }
        __syncthreads();
    }
}

// Block map at xi (the formulas of blocks.h with one division per length): J,
// and what map_second needs for sum_i g_i d^2 x_i / dxi_l dxi_m.
struct MapPoint {
    double u[3], du[2][3], il, t, R, dR, ddR;
    int t1, t2;
};

__device__ void map_first(const dg_block& B, const double xi[3], double J[3][3], MapPoint& p) {
    if (B.kind == DG_BLOCK_HEX8) {
        double x[3];
        block_jacobian(B, xi, J, x);
        return;
    }
    int d;
    double sg, v[3];
    wedge_frame(B.face, d, sg, p.t1, p.t2);
    for (int i = 0; i < 3; ++i) v[i] = i == d ? sg : (i == p.t1 ? xi[0] : xi[1]);
    p.il = 1.0 / sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    for (int i = 0; i < 3; ++i) p.u[i] = v[i] * p.il;
    const double ua = (p.t1 == 0 ? p.u[0] : (p.t1 == 1 ? p.u[1] : p.u[2])), ub = (p.t2 == 0 ? p.u[0] : (p.t2 == 1 ? p.u[1] : p.u[2]));
    for (int i = 0; i < 3; ++i) {
        p.du[0][i] = ((i == p.t1 ? 1.0 : 0.0) - p.u[i] * ua) * p.il;
        p.du[1][i] = ((i == p.t2 ? 1.0 : 0.0) - p.u[i] * ub) * p.il;
    }
    p.t = 0.5 * (xi[2] + 1.0);
    if (B.kind == DG_BLOCK_WEDGE) {
        const double s = (1.0 - p.t) * B.a, r = p.t * B.r;
        for (int i = 0; i < 3; ++i) {
            J[i][0] = (i == p.t1 ? s : 0.0) + r * p.du[0][i];
            J[i][1] = (i == p.t2 ? s : 0.0) + r * p.du[1][i];
            J[i][2] = 0.5 * (B.r * p.u[i] - B.a * v[i]);
        }
    } else {
        const double i1 = 1.0 / B.r1, i2 = 1.0 / B.r2, k = i1 - i2;
        p.R = 1.0 / ((1.0 - p.t) * i1 + p.t * i2);
        p.dR = p.R * p.R * k;
        p.ddR = 2.0 * p.R * p.dR * k;
        for (int i = 0; i < 3; ++i) {
            J[i][0] = p.R * p.du[0][i];
            J[i][1] = p.R * p.du[1][i];
            J[i][2] = 0.5 * p.dR * p.u[i];
        }
    }
}

// S[c] = sum_i g_i d^2 x_i / dxi_l dxi_m, pairs in the order of Derivs::h: the
// second derivatives of the formulas in block_point, for the exact Laplacian of
// mapped polynomials.  Wedge and shell, with v linear in xi_0, xi_1, u = v / |v|,
// t = (xi_2 + 1) / 2 and a, b in {0, 1} along e_ta:
//   d_a u_i = (delta_i,ta - u_i u_ta) / |v|,
//   d_a d_b u_i = -[(d_b u_i) u_ta + u_i (d_b u_ta) + (d_a u_i) u_tb] / |v|;
//   wedge x = (1 - t) a v + t r u: d_a d_b x = t r d_a d_b u,
//     d_a d_2 x = (r d_a u - a e_ta) / 2, d_2 d_2 x = 0;
//   shell x = R(t) u: d_a d_b x = R d_a d_b u, d_a d_2 x = R' d_a u / 2,
//     d_2 d_2 x = R'' u / 4, R' = R^2 (1/r1 - 1/r2), R'' = 2 R R' (1/r1 - 1/r2).
__device__ void map_second(const dg_block& B, const double xi[3], const MapPoint& p, const double g[3], double S[6]) {
    if (B.kind == DG_BLOCK_HEX8) {
        double s01 = 0.0, s02 = 0.0, s12 = 0.0;
        for (int c = 0; c < 8; ++c) {
            const double q = g[0] * B.corners[c][0] + g[1] * B.corners[c][1] + g[2] * B.corners[c][2];
            double f[3], df[3];
            for (int k = 0; k < 3; ++k) {
                const bool hi = (c >> k) & 1;
                f[k] = hi ? 0.5 * (1.0 + xi[k]) : 0.5 * (1.0 - xi[k]);
                df[k] = hi ? 0.5 : -0.5;
            }
            s01 += df[0] * df[1] * f[2] * q;
            s02 += df[0] * f[1] * df[2] * q;
            s12 += f[0] * df[1] * df[2] * q;
        }
        S[0] = S[1] = S[2] = 0.0;
        S[3] = s01;
        S[4] = s02;
        S[5] = s12;
        return;
    }
    auto at = [&](const double* w, int i) { return i == 0 ? w[0] : (i == 1 ? w[1] : w[2]); };
    auto dot = [&](const double* w) { return g[0] * w[0] + g[1] * w[1] + g[2] * w[2]; };
    const double gu = dot(p.u), g0 = dot(p.du[0]), g1 = dot(p.du[1]);
    const double ua = at(p.u, p.t1), ub = at(p.u, p.t2);
    const double s00 = -(2.0 * g0 * ua + gu * at(p.du[0], p.t1)) * p.il;   // g . d_a d_b u
    const double s11 = -(2.0 * g1 * ub + gu * at(p.du[1], p.t2)) * p.il;
    const double s01 = -(g1 * ua + gu * at(p.du[1], p.t1) + g0 * ub) * p.il;
    if (B.kind == DG_BLOCK_WEDGE) {
        const double r = p.t * B.r;
        S[0] = r * s00;
        S[1] = r * s11;
        S[2] = 0.0;
        S[3] = r * s01;
        S[4] = 0.5 * (B.r * g0 - B.a * at(g, p.t1));
        S[5] = 0.5 * (B.r * g1 - B.a * at(g, p.t2));
    } else {
        S[0] = p.R * s00;
        S[1] = p.R * s11;
        S[2] = 0.25 * p.ddR * gu;
        S[3] = p.R * s01;
        S[4] = 0.5 * p.dR * g0;
        S[5] = 0.5 * p.dR * g1;
    }
}

__device__ double det3(const double (&J)[3][3]) {
    return J[0][0] * (J[1][1] * J[2][2] - J[1][2] * J[2][1]) - J[0][1] * (J[1][0] * J[2][2] - J[1][2] * J[2][0]) +
           J[0][2] * (J[1][0] * J[2][1] - J[1][1] * J[2][0]);
}

__device__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum over the CTA, in a fixed order; the result is valid in warp 0.
__device__ double block_sum(double v, double* red) {
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    return threadIdx.x < 32 ? warp_sum(threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0) : 0.0;
}

__global__ void __launch_bounds__(kEstThreads) estimate_kernel(EstimateArgs a, const double* u, const double* g,
                                                               const double* f, const double* gD, double* eta2) {
    const int e = blockIdx.x;
    if (e >= a.n_elems) return;
    const int n = a.p[e] + 1, n2 = n * n, n3 = n2 * n;
    const int k = threadIdx.x;
    __shared__ double F[kNV], T1[kNV], T2[3 * kNV];
    __shared__ double Mx[3][kMaxN * kMaxN];
    __shared__ double red[32], mort[kEstMaxSlots], V[8][3];
    const double* I = a.tab + tab_n(TabIndex::I, n);
    const double* D1 = a.tab + tab_n(TabIndex::IDg, n);
    const double* DL = a.tab + tab_n(TabIndex::DL, n);
    const double* wg = a.tab + tab_n(TabIndex::GLw, n);
    for (int t = threadIdx.x; t < n2; t += blockDim.x) {
        const int i = t / n, c = t % n;
        Mx[0][t] = I[t];
        Mx[1][t] = D1[t];
        double s = 0.0;
        for (int b = 0; b < n; ++b) s += D1[i * n + b] * DL[b * n + c];
        Mx[2][t] = s;
    }
    const double* M[3] = {Mx[0], Mx[1], Mx[2]};
    const double* Xe = a.n_blocks > 0 ? nullptr : a.X + 3 * a.dof_off[e];
    const double* ue = u + a.dof_off[e];
    const bool blk = a.n_blocks > 0;

    // element diameter: largest distance between two of the eight vertices (a lane per vertex, then per pair)
    double he2 = 0.0;
    double binv = 1.0, bxi0[3] = {0.0, 0.0, 0.0};   // block meshes: xi_block = bxi0 + binv (xi + 1)
    if (blk) {
        const int* lf = a.leaves + 4 * e;
        binv = 1.0 / (double)(1 << lf[0]);
        for (int dd = 0; dd < 3; ++dd) bxi0[dd] = -1.0 + 2.0 * lf[1 + dd] * binv;
    }
    if (threadIdx.x < 32) {
        const int c = threadIdx.x & 7;
        double x[3];
        if (blk) {
            double xb[3];
            for (int dd = 0; dd < 3; ++dd) xb[dd] = bxi0[dd] + binv * (((c >> dd) & 1) ? 2.0 : 0.0);
            block_point(a.fblocks[a.block[e]], xb, x);
        } else {
            const int idx = ((c & 1) ? n - 1 : 0) + n * (((c >> 1) & 1) ? n - 1 : 0) + n2 * (((c >> 2) & 1) ? n - 1 : 0);
            for (int i = 0; i < 3; ++i) x[i] = Xe[i * n3 + idx];
        }
        if (threadIdx.x < 8)
            for (int i = 0; i < 3; ++i) V[c][i] = x[i];
        __syncwarp();
        for (int p = threadIdx.x; p < 64; p += 32) {
            const double dx = V[p & 7][0] - V[p >> 3][0], dy = V[p & 7][1] - V[p >> 3][1], dz = V[p & 7][2] - V[p >> 3][2];
            he2 = fmax(he2, dx * dx + dy * dy + dz * dz);
        }
        for (int o = 16; o > 0; o >>= 1) he2 = fmax(he2, __shfl_xor_sync(0xffffffffu, he2, o));
    }
    __syncthreads();

    // J_il = d x_i / d xi_l (block meshes: the exact map's) and the fiducial Jacobian
    // determinant of the volume weight
    double J[3][3], xb[3] = {0.0, 0.0, 0.0}, detW = 0.0;
    MapPoint mp;
    Derivs D;
    if (blk) {
        const double* xg = a.tab + tab_n(TabIndex::GLx, n);
        if (k < n3) {
            const int ii[3] = {k % n, (k / n) % n, k / n2};
            for (int dd = 0; dd < 3; ++dd) xb[dd] = bxi0[dd] + binv * (xg[ii[dd]] + 1.0);
            if (a.fblocks != a.blocks) {
                map_first(a.fblocks[a.block[e]], xb, J, mp);
                detW = det3(J) * (binv * binv * binv);
            }
            map_first(a.blocks[a.block[e]], xb, J, mp);
            for (int i = 0; i < 3; ++i)
                for (int l = 0; l < 3; ++l) J[i][l] *= binv;
        }
    } else {
        for (int i = 0; i < 3; ++i) {
            for (int t = threadIdx.x; t < n3; t += blockDim.x) F[t] = Xe[i * n3 + t];
            __syncthreads();
            eval_derivs<true, false>(F, T1, T2, M, n, k, D);
            for (int l = 0; l < 3; ++l) J[i][l] = D.d[l];
        }
    }
    double Ji[3][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}}, det = 1.0;
    if (k < n3) {
        det = det3(J);
        if (!blk || a.fblocks == a.blocks) detW = det;
        const double r = 1.0 / det;
        Ji[0][0] = (J[1][1] * J[2][2] - J[1][2] * J[2][1]) * r;
        Ji[0][1] = (J[0][2] * J[2][1] - J[0][1] * J[2][2]) * r;
        Ji[0][2] = (J[0][1] * J[1][2] - J[0][2] * J[1][1]) * r;
        Ji[1][0] = (J[1][2] * J[2][0] - J[1][0] * J[2][2]) * r;
        Ji[1][1] = (J[0][0] * J[2][2] - J[0][2] * J[2][0]) * r;
        Ji[1][2] = (J[0][2] * J[1][0] - J[0][0] * J[1][2]) * r;
        Ji[2][0] = (J[1][0] * J[2][1] - J[1][1] * J[2][0]) * r;
        Ji[2][1] = (J[0][1] * J[2][0] - J[0][0] * J[2][1]) * r;
        Ji[2][2] = (J[0][0] * J[1][1] - J[0][1] * J[1][0]) * r;
    }

    // u, its physical gradient and the reference Hessian
    for (int t = threadIdx.x; t < n3; t += blockDim.x) F[t] = ue[t];
    __syncthreads();
    eval_derivs<true, true>(F, T1, T2, M, n, k, D);
    const double uv = D.v;
    double ux[3], H[6];
    for (int i = 0; i < 3; ++i) ux[i] = Ji[0][i] * D.d[0] + Ji[1][i] * D.d[1] + Ji[2][i] * D.d[2];
    for (int c = 0; c < 6; ++c) H[c] = D.h[c];
    // minus sum_k (du/dx_k) X^k
    if (blk) {
        if (k < n3) {
            double S[6];
            map_second(a.blocks[a.block[e]], xb, mp, ux, S);
            for (int c = 0; c < 6; ++c) H[c] -= S[c] * (binv * binv);
        }
    } else {
        for (int i = 0; i < 3; ++i) {
            for (int t = threadIdx.x; t < n3; t += blockDim.x) F[t] = Xe[i * n3 + t];
            __syncthreads();
            eval_derivs<false, true>(F, T1, T2, M, n, k, D);
            for (int c = 0; c < 6; ++c) H[c] -= ux[i] * D.h[c];
        }
    }
    double vol = 0.0;
    if (k < n3) {
        double G[3][3];
        for (int l = 0; l < 3; ++l)
            for (int m = 0; m < 3; ++m) G[l][m] = Ji[l][0] * Ji[m][0] + Ji[l][1] * Ji[m][1] + Ji[l][2] * Ji[m][2];
        const double lap = G[0][0] * H[0] + G[1][1] * H[1] + G[2][2] * H[2] +
                           2.0 * (G[0][1] * H[3] + G[0][2] * H[4] + G[1][2] * H[5]);
        const long long vo = a.vqp_off[e];
        const double R = (f ? f[vo + k] : 0.0) * uv - (g ? g[vo + k] : 0.0) - lap;
        const double w = wg[k % n] * wg[(k / n) % n] * wg[k / n2];
        vol = w * detW * R * R;
    }
    vol = block_sum(vol, red);

    // mortar terms of the element's slots, a warp per slot, summed in slot order
    const int s0 = a.slot_off[e], ns = a.slot_off[e + 1] - s0, lane = threadIdx.x & 31;
    if (ns > kEstMaxSlots && threadIdx.x == 0) atomicExch(a.chk, 6);
    for (int s = threadIdx.x >> 5; s < ns && s < kEstMaxSlots; s += blockDim.x >> 5) {
        const int mi = a.slot_mortar[s0 + s];
        const Mortar Mo = a.mortars[mi];
        const int q2 = Mo.q * Mo.q;
        const double* mg = a.mgW + 7 * Mo.goff;   // w S of the weighting grid
        const double* mt = a.mt + 4 * Mo.goff;
        double s1 = 0.0, s2 = 0.0;
        for (int pt = lane; pt < q2; pt += 32) {
            const double wS = mg[pt];
            if (Mo.eB >= 0) {
                const double j1 = mt[q2 + pt] - mt[3 * q2 + pt];
                const double j2 = mt[pt] - mt[2 * q2 + pt];
                s1 += wS * j1 * j1;
                s2 += wS * j2 * j2;
            } else {
                const double j3 = mt[pt] - (gD ? gD[Mo.bnd_off + pt] : 0.0);
                s2 += wS * j3 * j3;
            }
        }
        s1 = warp_sum(s1);
        s2 = warp_sum(s2);
        if (lane == 0) {
            const double pm = Mo.q - 1, sig = a.sigW[mi];
            const double hm = a.C * pm * pm / sig;
            mort[s] = (Mo.eB >= 0 ? hm / pm * s1 : 0.0) + sig / hm * pm * pm * s2;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const double pe = n - 1;
        double m = 0.0;
        for (int s = 0; s < ns && s < kEstMaxSlots; ++s) m += mort[s];
        eta2[e] = he2 * pe * pe * vol + m;
    }
}

}  // namespace

cudaError_t launch_estimate(const EstimateArgs& a, const double* u, const double* g, const double* f,
                            const double* gD, double* eta2, cudaStream_t st) {
    if (a.n_elems == 0) return cudaSuccess;
    estimate_kernel<<<a.n_elems, kEstThreads, 0, st>>>(a, u, g, f, gD, eta2);
    return cudaGetLastError();
}

}  // namespace dg
