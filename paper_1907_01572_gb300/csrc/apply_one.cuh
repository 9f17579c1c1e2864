// FP32 operator apply in one launch, for small levels (included by
// apply_impl.cuh, which describes the operator).
//
// A level of a few hundred elements is bound by latency: of the two launches
// (trace, element) each waits for its tables, its records and its input, and
// the second for the first.  Here one CTA per element computes the traces of
// both sides of its mortars itself -- the neighbour's straight from the input
// vector, so that no CTA waits for another -- while four warps run the volume
// passes; then the warps lift the mortars' fluxes, each into arrays of its own,
// and the nodes gather volume and face parts in slot order.  The traces are computed twice (once
// on either side), which costs nothing where the chip is not full.
// Measured (FP32, two launches -> one): 64 elements of p = 5 14.8 -> 8.8 us, 216
// elements, p 4..6, hanging faces, 18.6 -> 13.0 us, 512 elements of p = 5 25.4 ->
// 19.1 us.  What bounds it is the chain of one element: input and records, seven
// to twelve dependent passes, the gather.
#pragma once

namespace dg {
namespace apply_detail {

constexpr int kOneVolWarps = 4, kOneFaceWarps = 8, kOneWarps = kOneVolWarps + kOneFaceWarps;
constexpr int kOneMaxSlots = 24;   // four mortars on each of six faces
constexpr int kOneTrace = 4 * kQ * kQ, kOneScratch = 4 * kQ * kQ + 3 * kQ * kMaxN;

template <int N>
struct OneLayout {         // in values of T
    static constexpr int NR = r4(Strides<N>::SIZE);
    static constexpr int TAB = vol_vals(N), VOL = 6 * NR;
    static constexpr int SIZE = TAB + VOL + kOneMaxSlots * kOneTrace + kOneWarps * kOneScratch;
};

__device__ __forceinline__ int one_point(int o, int Q, int j1, int j2) {   // MortarMap with a run-time Q
    const int b1 = (o & 2) ? Q - 1 - j1 : j1, b2 = (o & 4) ? Q - 1 - j2 : j2;
    return (o & 1) ? b2 + Q * b1 : b1 + Q * b2;
}

// Trace (u and c . grad u) of one side of a mortar at its Q x Q points, from the
// element's values in the input vector (see trace_slot), by one warp.
template <int N, typename T, typename TX>
__device__ __noinline__ void one_trace(const T* __restrict__ tab, const T* __restrict__ ftab, const TX* __restrict__ x,
                                       int f, int p0, int p1, int Q, int o, const T* __restrict__ co, T* F, T* out,
                                       int lane) {
    constexpr int N2 = N * N;
    const int d = f >> 1, fn = (f & 1) ? N - 1 : 0, Q2 = Q * Q;
    int t1, t2;
    tangential(d, t1, t2);
    auto st = [](int k) { return k == 0 ? 1 : (k == 1 ? N : N * N); };
    const int sd = st(d), st1 = st(t1), st2 = st(t2);
    const T* DL = tab + tab_n(TabIndex::DL, N) + fn * N;
    const T* ft = ftab + face_seg_off(N);
    const T* M1 = ft + face_tab_off(N, Q, p0);
    const T* M2 = ft + face_tab_off(N, Q, p1);
    T *uf = F, *df = uf + N2, *U1 = df + N2, *DU1 = U1 + Q * N, *N1 = DU1 + Q * N;
    T dl[N];
#pragma unroll
    for (int c = 0; c < N; ++c) dl[c] = DL[c];
#pragma unroll
    for (int k0 = 0; k0 < N2; k0 += 32) {
        const int k = k0 + lane;
        if (k >= N2) continue;
        const TX* p = x + (k % N) * st1 + (k / N) * st2;
        T v[N], s = 0;
#pragma unroll
        for (int c = 0; c < N; ++c) v[c] = ld<T>(p + c * sd);
#pragma unroll
        for (int c = 0; c < N; ++c) s += dl[c] * v[c];
        uf[k] = fn ? v[N - 1] : v[0];
        df[k] = s;
    }
    __syncwarp();
    for (int k = lane; k < Q * N; k += 32) {
        const int i1 = k % Q, b = k / Q;
        T su = 0, sd1 = 0, sn = 0;
#pragma unroll
        for (int a = 0; a < N; ++a) {
            T iv, dv;
            ld2(M1 + 2 * (i1 * N + a), iv, dv);
            su += iv * uf[a + N * b];
            sd1 += dv * uf[a + N * b];
            sn += iv * df[a + N * b];
        }
        U1[k] = su;
        DU1[k] = sd1;
        N1[k] = sn;
    }
    __syncwarp();
    for (int k = lane; k < Q2; k += 32) {
        const int i1 = k % Q, i2 = k / Q, kA = one_point(o, Q, i1, i2);
        const T c1 = co[t1 * Q2 + kA], c2 = co[t2 * Q2 + kA], cn = co[d * Q2 + kA];
        T u = 0, g1 = 0, g2 = 0, gn = 0;
#pragma unroll
        for (int b = 0; b < N; ++b) {
            T iv, dv;
            ld2(M2 + 2 * (i2 * N + b), iv, dv);
            const T ub = U1[i1 + Q * b];
            u += iv * ub;
            g1 += iv * DU1[i1 + Q * b];
            g2 += dv * ub;
            gn += iv * N1[i1 + Q * b];
        }
        out[kA] = u;
        out[Q2 + kA] = c1 * g1 + c2 * g2 + cn * gn;
    }
    __syncwarp();
}

// Flux and lift of one mortar (see lift_slot, lift_apply) by one warp: fu (values
// on the face) and fd (times the face-normal row of DL), N^2 each, take the place
// of the mortar's traces m.
template <int N, typename T>
__device__ __noinline__ void one_lift(const T* __restrict__ ftab, int f, int side, int p0, int p1, int Q, int o, bool interior,
                                      T sig, const T* __restrict__ wSp, const T* __restrict__ co, T* m, T* F,
                                      int lane) {
    const int d = f >> 1, Q2 = Q * Q;
    int t1, t2;
    tangential(d, t1, t2);
    const T* ft = ftab + face_seg_off(N);
    const T* M1 = ft + face_tab_off(N, Q, p0);
    const T* M2 = ft + face_tab_off(N, Q, p1);
    T *PA = F, *P1 = PA + Q2, *P2 = P1 + Q2, *Pn = P2 + Q2, *X1 = F + 4 * Q2, *X2 = X1 + Q * N, *X3 = X2 + Q * N;
    const T half = interior ? T(0.5) : T(1), sgn = side == 0 ? T(1) : T(-1);
    for (int k = lane; k < Q2; k += 32) {
        const int kA = one_point(o, Q, k % Q, k / Q);
        const T wS = wSp[kA];
        T j = m[kA], a = m[Q2 + kA];
        if (interior) {
            j -= m[2 * Q2 + kA];
            a += m[3 * Q2 + kA];
        }
        const T b = -half * wS * j;
        PA[k] = sgn * (wS * (sig * j - half * a));
        P1[k] = b * co[t1 * Q2 + kA];
        P2[k] = b * co[t2 * Q2 + kA];
        Pn[k] = b * co[d * Q2 + kA];
    }
    __syncwarp();
    for (int k = lane; k < Q * N; k += 32) {
        const int i1 = k % Q, b = k / Q;
        T a1 = 0, a2 = 0, a3 = 0;
#pragma unroll 4
        for (int i2 = 0; i2 < Q; ++i2) {
            T iv, dv;
            ld2(M2 + 2 * (i2 * N + b), iv, dv);
            const int p = i1 + Q * i2;
            a1 += iv * PA[p] + dv * P2[p];
            a2 += iv * P1[p];
            a3 += iv * Pn[p];
        }
        X1[k] = a1;
        X2[k] = a2;
        X3[k] = a3;
    }
    __syncwarp();
    for (int k = lane; k < N * N; k += 32) {
        const int a = k % N, b = k / N;
        T fu = 0, fd = 0;
#pragma unroll 4
        for (int i1 = 0; i1 < Q; ++i1) {
            T iv, dv;
            ld2(M1 + 2 * (i1 * N + a), iv, dv);
            fu += iv * X1[i1 + Q * b] + dv * X2[i1 + Q * b];
            fd += iv * X3[i1 + Q * b];
        }
        m[k] = fu;
        m[N * N + k] = fd;
    }
    __syncwarp();
}

__device__ __forceinline__ void one_vol_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(32 * kOneVolWarps) : "memory"); }

// Volume terms into Y, by the first kOneVolWarps warps.
template <int N, typename T, typename TX>
__device__ __forceinline__ void one_volume(const LevelView<T>& L, const TX* __restrict__ x, long long vo, T* sV, T* Y) {
    constexpr int NP = r4(N), N3 = N * N * N, NR = OneLayout<N>::NR, nt = 32 * kOneVolWarps;
    const int tid = threadIdx.x;
    const T* tI = L.tab + tab_n(TabIndex::I, N);
    const T* tD = L.tab + tab_n(TabIndex::Dg, N);
    T *U = Y + NR, *A = U + NR, *B = A + NR, *G1 = B + NR, *G3 = G1 + NR, *G2 = Y;
    const T* Ge = L.G + 6 * vo;
    const bool mass = L.c0 != nullptr;
    for (int k = tid; k < N3; k += nt) U[sidx<N>(k)] = ld<T>(x + k);
    prefetch_l2(Ge, 6 * N3, tid, nt);
    for (int k = tid; k < N * NP; k += nt) {
        const int i = k / NP, m = k % NP;
        const bool in = m < N;
        sV[k] = in ? tI[i * N + m] : T(0);
        sV[N * NP + k] = in ? tI[m * N + i] : T(0);
        sV[2 * N * NP + k] = in ? tD[i * N + m] : T(0);
        sV[3 * N * NP + k] = in ? tD[m * N + i] : T(0);
    }
    const T *sI = sV, *sDg = sV + 2 * N * NP;
    one_vol_barrier();
    wpass<N, 0, false, false>(U, A, sI, tid, nt);
    one_vol_barrier();
    wpass<N, 1, false, false>(A, B, sI, tid, nt);
    one_vol_barrier();
    wpass<N, 2, false, false>(B, A, sI, tid, nt);
    one_vol_barrier();
    wpass<N, 0, false, false>(A, G1, sDg, tid, nt);
    wpass<N, 1, false, false>(A, G2, sDg, tid, nt);
    wpass<N, 2, false, false>(A, G3, sDg, tid, nt);
    one_vol_barrier();
    for (int k = tid; k < N3; k += nt) {
        const int s = sidx<N>(k);
        const T g0 = G1[s], g1 = G2[s], g2 = G3[s];
        const T m00 = Ge[k], m01 = Ge[N3 + k], m02 = Ge[2 * N3 + k];
        const T m11 = Ge[3 * N3 + k], m12 = Ge[4 * N3 + k], m22 = Ge[5 * N3 + k];
        G1[s] = m00 * g0 + m01 * g1 + m02 * g2;
        G2[s] = m01 * g0 + m11 * g1 + m12 * g2;
        G3[s] = m02 * g0 + m12 * g1 + m22 * g2;
        if (mass) B[s] = L.c0[vo + k] * A[s];
    }
    one_vol_barrier();
    if (mass) wpass<N, 0, true, true>(G1, B, sDg, tid, nt);
    else wpass<N, 0, true, false>(G1, B, sDg, tid, nt);
    one_vol_barrier();
    wpass<N, 1, true, true>(G2, B, sDg, tid, nt);
    one_vol_barrier();
    wpass<N, 2, true, true>(G3, B, sDg, tid, nt);
    one_vol_barrier();
    wpass<N, 0, true, false>(B, A, sI, tid, nt);
    one_vol_barrier();
    wpass<N, 1, true, false>(A, B, sI, tid, nt);
    one_vol_barrier();
    wpass<N, 2, true, false>(B, Y, sI, tid, nt);
}

template <int N, typename T, typename TX>
__device__ __forceinline__ void one_body(const LevelView<T>& L, const ElemDesc& de, const TX* __restrict__ x,
                                         T* __restrict__ y) {
    using Ly = OneLayout<N>;
    constexpr int N2 = N * N, N3 = N2 * N;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sV = reinterpret_cast<T*>(smem_raw);
    T* Y = sV + Ly::TAB;
    T* TR = Y + Ly::VOL;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    T* F = TR + kOneMaxSlots * kOneTrace + warp * kOneScratch;
    __shared__ int next_task, face_start[7];
    const int ns = min(de.s1 - de.s0, kOneMaxSlots);
    if (tid == 0) {
        next_task = 0;
        if (de.s1 - de.s0 > kOneMaxSlots) atomicExch(L.chk, 7);
    }
    __syncthreads();
    if (warp < kOneVolWarps) one_volume<N, T, TX>(L, x + de.dofo, de.vo, sV, Y);
    if (warp == kOneWarps - 1) {   // first slot of each face (slots come face by face)
        const int f = lane < ns ? L.spack[de.s0 + lane].info & 7 : 6;
        for (int k = 0; k < 7; ++k) {
            const unsigned before = __ballot_sync(0xffffffffu, f < k);
            if (lane == 0) face_start[k] = __popc(before);
        }
    }
    // tasks: the own side of every slot, then the neighbours' (whichever warp is free: each writes its own array)
    for (;;) {
        int k = 0;
        if (lane == 0) k = atomicAdd(&next_task, 1);
        k = __shfl_sync(0xffffffffu, k, 0);
        if (k >= 2 * ns) break;
        {
            const int s = k % ns;
            const SlotPack<T> sp = L.spack[de.s0 + s];
            const SlotNb nb = L.snb[de.s0 + s];
            const bool own = k < ns;
            if (!own && nb.n == 0) continue;   // boundary
            const int side = ((sp.info >> 3) & 1) ^ (own ? 0 : 1), q = (sp.info >> 8) & 15;
            T* out = TR + s * kOneTrace + 2 * side * q * q;
            if (!own && L.bdiag) {             // element diagonal block: the other side's trace is zero
                for (int i = lane; i < 2 * q * q; i += 32) out[i] = T(0);
                continue;
            }
            const int info = own ? sp.info : nb.info, n = own ? N : nb.n;
            const TX* xe = x + (own ? de.dofo : nb.dofo);
            const T* co = L.mg + 7 * sp.goff + (side == 0 ? 1 : 4) * q * q;
            DG_BODY_SWITCH(n, (one_trace<NN, T, TX>(L.tab, L.ftab, xe, info & 7, (info >> 4) & 3, (info >> 6) & 3, q,
                                                    (info >> 13) & 7, co, F, out, lane)))
        }
    }
    __syncthreads();
    for (int s = warp; s < ns; s += kOneWarps) {
        const SlotPack<T> sp = L.spack[de.s0 + s];
        const int q = (sp.info >> 8) & 15, side = (sp.info >> 3) & 1;
        const T* mg = L.mg + 7 * sp.goff;
        one_lift<N, T>(L.ftab, sp.info & 7, side, (sp.info >> 4) & 3, (sp.info >> 6) & 3, q, (sp.info >> 13) & 7,
                       (sp.info >> 12) & 1, sp.sig, mg, mg + (side == 0 ? 1 : 4) * q * q, TR + s * kOneTrace, F, lane);
    }
    __syncthreads();
    const T* DL = L.tab + tab_n(TabIndex::DL, N);
    for (int k = tid; k < N3; k += 32 * kOneWarps) {
        const int c[3] = {k % N, (k / N) % N, k / N2};
        T v = Y[sidx<N>(k)];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int i = (d == 0 ? c[1] : c[0]) + N * (d == 2 ? c[1] : c[2]);
            for (int h = 0; h < 2; ++h) {
                const T w = DL[h * (N - 1) * N + c[d]];
                const bool on = c[d] == h * (N - 1);
                for (int s = face_start[2 * d + h]; s < face_start[2 * d + h + 1]; ++s) {
                    const T* m = TR + s * kOneTrace + i;
                    v += w * m[N2];
                    if (on) v += m[0];
                }
            }
        }
        if (L.Ob != nullptr) v += y[de.dofo + k];   // the Galerkin blocks' part (galerkin_apply_kernel)
        y[de.dofo + k] = v;
    }
}

template <typename T, typename TX>
__global__ void __launch_bounds__(32 * kOneWarps, 2)
    one_kernel(LevelView<T> L, FusedBuckets fb, const TX* __restrict__ x, T* __restrict__ y) {
    const int b = fused_bucket(fb);
    const ElemDesc de = fb.desc[b][blockIdx.x - fb.cta_start[b]];
    DG_BODY_SWITCH(fb.n[b], (one_body<NN, T, TX>(L, de, x, y)))
}

template <typename T, typename TX>
cudaError_t launch_one(const LevelView<T>& L, const BucketInfo* buckets, const TX* x, T* y, cudaStream_t st,
                       int* launches) {
    size_t smem = 0;
    FusedBuckets fb{};
    int ctas = 0;
    for (int n = kMaxN; n >= kMinN; --n) {   // the longest elements first
        const BucketInfo& b = buckets[n];
        if (b.count == 0) continue;
        DG_N_SWITCH(n, (smem = std::max(smem, OneLayout<NN>::SIZE * sizeof(T))))
        fb.n[fb.nb] = n;
        fb.desc[fb.nb] = b.desc;
        fb.count[fb.nb] = b.count;
        fb.cta_start[fb.nb] = ctas;
        ctas += b.count;
        ++fb.nb;
    }
    fb.cta_start[fb.nb] = ctas;
    if (ctas == 0) return cudaSuccess;
    static const cudaError_t attr = cudaFuncSetAttribute(one_kernel<T, TX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                         (int)(OneLayout<kMaxN>::SIZE * sizeof(T)));
    if (attr != cudaSuccess) return attr;
    one_kernel<T, TX><<<ctas, 32 * kOneWarps, smem, st>>>(L, fb, x, y);
    if (launches) ++*launches;
    return cudaGetLastError();
}

}  // namespace apply_detail
}  // namespace dg
