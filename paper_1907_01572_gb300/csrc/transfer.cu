// Inter-mesh operators of Sec. II.E.6.
// Prolongation (eq. psi-interpolation): the coarse polynomial is evaluated at
// the children's LGL nodes, child half b along each axis mapping the child
// coordinate xi to (xi + 2b - 1)/2 of the parent; the 3-D operator is the
// tensor product of three 1-D (n_h x n_H) matrices.  Restriction of weak
// residuals is its transpose (eq. temp-G), summed over the children.
// Elements carried over unchanged between levels are copied.
#include "transfer.h"

namespace dg {
namespace {

// out has dims dout (x fastest), in has dims din; contraction along `dir`, by nt threads (t of them).
template <typename T>
__device__ void rect_pass(const T* in, T* out, const T* M, int dir, int n_in, const int din[3], const int dout[3],
                          bool trans, int m_cols, int t, int nt) {
    const int total = dout[0] * dout[1] * dout[2];
    for (int idx = t; idx < total; idx += nt) {
        int o[3] = {idx % dout[0], (idx / dout[0]) % dout[1], idx / (dout[0] * dout[1])};
        T s = 0;
        for (int m = 0; m < n_in; ++m) {
            int ii[3] = {o[0], o[1], o[2]};
            ii[dir] = m;
            const T mv = trans ? M[m * m_cols + o[dir]] : M[o[dir] * m_cols + m];
            s += mv * in[ii[0] + din[0] * (ii[1] + din[1] * ii[2])];
        }
        out[idx] = s;
    }
}

template <typename T>
__global__ void prolong_kernel(TransferView<T> t, const T* __restrict__ vH, T* __restrict__ vh) {
    const int c = blockIdx.x;
    if (c >= t.n_fine) return;
    __shared__ T buf[3][kMaxN * kMaxN * kMaxN];
    const int H = t.fine_parent[c];
    const int bits = t.fine_bits[c];
    const int nH = t.pH[H] + 1, nh = t.ph[c] + 1;
    const T* src = vH + t.dofH[H];
    T* dst = vh + t.dofh[c];
    if (bits == 0xFF) {
        for (int k = threadIdx.x; k < nh * nh * nh; k += blockDim.x) dst[k] += src[k];
        return;
    }
    for (int k = threadIdx.x; k < nH * nH * nH; k += blockDim.x) buf[0][k] = src[k];
    __syncthreads();
    const T* Cx = t.tab + tab_ci(nH, nh, bits & 1);
    const T* Cy = t.tab + tab_ci(nH, nh, (bits >> 1) & 1);
    const T* Cz = t.tab + tab_ci(nH, nh, (bits >> 2) & 1);
    int d0[3] = {nH, nH, nH}, d1[3] = {nh, nH, nH}, d2[3] = {nh, nh, nH}, d3[3] = {nh, nh, nh};
    rect_pass(buf[0], buf[1], Cx, 0, nH, d0, d1, false, nH, threadIdx.x, blockDim.x);
    __syncthreads();
    rect_pass(buf[1], buf[2], Cy, 1, nH, d1, d2, false, nH, threadIdx.x, blockDim.x);
    __syncthreads();
    rect_pass(buf[2], buf[0], Cz, 2, nH, d2, d3, false, nH, threadIdx.x, blockDim.x);
    __syncthreads();
    for (int k = threadIdx.x; k < nh * nh * nh; k += blockDim.x) dst[k] += buf[0][k];
}

// One block per coarse element, 128 threads per child: the children's transposed
// interpolations run side by side (they are a chain of dependent passes, bound by
// latency: 216 -> 27 elements, n <= 7, FP32, took 41 us one child after the other,
// 13 us now) and are summed in child order.
// Levels of up to kSideBySideMax coarse elements (7,680 -> 960: 39 and 27 us).
constexpr int kChildThreads = 128, kMaxChildren = 8, kSideBySideMax = 2048;

template <typename T>
__global__ void __launch_bounds__(kChildThreads* kMaxChildren) restrict_kernel(TransferView<T> t, const T* __restrict__ rh,
                                                                               T* __restrict__ fH) {
    constexpr int N3 = kMaxN * kMaxN * kMaxN;
    extern __shared__ __align__(16) unsigned char restrict_smem[];
    const int H = blockIdx.x;
    const int nH = t.pH[H] + 1, n3H = nH * nH * nH, c0 = t.child_off[H], nc = t.child_off[H + 1] - c0;
    const int ch = threadIdx.x / kChildThreads, tid = threadIdx.x % kChildThreads;
    T* b0 = reinterpret_cast<T*>(restrict_smem) + 2 * N3 * ch;
    T* b1 = b0 + N3;
    const bool on = ch < nc;
    const int bits = on ? t.child_bits[c0 + ch] : 0xFF, c = on ? t.child_id[c0 + ch] : 0, nh = on ? t.ph[c] + 1 : 0;
    if (on) {
        const T* src = rh + t.dofh[c];
        for (int k = tid; k < nh * nh * nh; k += kChildThreads) b0[k] = src[k];
    }
    __syncthreads();
    const bool go = on && bits != 0xFF;   // a carried-over element's values are copied
    int d0[3] = {nh, nh, nh}, d1[3] = {nH, nh, nh}, d2[3] = {nH, nH, nh}, d3[3] = {nH, nH, nH};
    if (go) rect_pass(b0, b1, t.tab + tab_ci(nH, nh, bits & 1), 0, nh, d0, d1, true, nH, tid, kChildThreads);
    __syncthreads();
    if (go) rect_pass(b1, b0, t.tab + tab_ci(nH, nh, (bits >> 1) & 1), 1, nh, d1, d2, true, nH, tid, kChildThreads);
    __syncthreads();
    if (go) rect_pass(b0, b1, t.tab + tab_ci(nH, nh, (bits >> 2) & 1), 2, nh, d2, d3, true, nH, tid, kChildThreads);
    __syncthreads();
    T* dst = fH + t.dofH[H];
    for (int k = threadIdx.x; k < n3H; k += blockDim.x) {
        T s = 0;
        for (int j = 0; j < nc; ++j)
            s += reinterpret_cast<const T*>(restrict_smem)[2 * N3 * j + (t.child_bits[c0 + j] == 0xFF ? 0 : N3) + k];
        dst[k] = s;
    }
}

// The same, one child after the other, in 128 threads: more coarse elements fill
// the chip by themselves, and eight children's 47 KB (FP32) or 93 KB (FP64), with
// threads that wait where an element was carried over and has one child, cost more
// than they give (FP32, side by side and in turn: 61,440 -> 7,680 elements 161 and
// 127 us, 32,768 -> 4,096 of p = 2 60 and 39 us).
template <typename T>
__global__ void __launch_bounds__(kChildThreads) restrict_in_turn_kernel(TransferView<T> t, const T* __restrict__ rh,
                                                                         T* __restrict__ fH) {
    constexpr int N3 = kMaxN * kMaxN * kMaxN;
    __shared__ T b0[N3], b1[N3], acc[N3];
    const int H = blockIdx.x, tid = threadIdx.x;
    const int nH = t.pH[H] + 1, n3H = nH * nH * nH;
    for (int k = tid; k < n3H; k += kChildThreads) acc[k] = 0;
    for (int ci = t.child_off[H]; ci < t.child_off[H + 1]; ++ci) {
        const int c = t.child_id[ci], bits = t.child_bits[ci], nh = t.ph[c] + 1;
        const T *src = rh + t.dofh[c], *res = src;   // a carried-over element's values are copied
        if (bits != 0xFF) {
            for (int k = tid; k < nh * nh * nh; k += kChildThreads) b0[k] = src[k];
            __syncthreads();
            int d0[3] = {nh, nh, nh}, d1[3] = {nH, nh, nh}, d2[3] = {nH, nH, nh}, d3[3] = {nH, nH, nH};
            rect_pass(b0, b1, t.tab + tab_ci(nH, nh, bits & 1), 0, nh, d0, d1, true, nH, tid, kChildThreads);
            __syncthreads();
            rect_pass(b1, b0, t.tab + tab_ci(nH, nh, (bits >> 1) & 1), 1, nh, d1, d2, true, nH, tid, kChildThreads);
            __syncthreads();
            rect_pass(b0, b1, t.tab + tab_ci(nH, nh, (bits >> 2) & 1), 2, nh, d2, d3, true, nH, tid, kChildThreads);
            res = b1;
        }
        for (int k = tid; k < n3H; k += kChildThreads) acc[k] += res[k];   // (each thread its own values throughout)
        __syncthreads();
    }
    for (int k = tid; k < n3H; k += kChildThreads) fH[t.dofH[H] + k] = acc[k];
}

}  // namespace

template <typename T>
cudaError_t launch_prolong_add(const TransferView<T>& t, const T* vH, T* vh, cudaStream_t st) {
    prolong_kernel<T><<<t.n_fine, 128, 0, st>>>(t, vH, vh);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_restrict(const TransferView<T>& t, const T* rh, T* fH, cudaStream_t st) {
    if (t.n_coarse > kSideBySideMax) {
        restrict_in_turn_kernel<T><<<t.n_coarse, kChildThreads, 0, st>>>(t, rh, fH);
        return cudaGetLastError();
    }
    constexpr size_t smem = sizeof(T) * 2 * kMaxChildren * kMaxN * kMaxN * kMaxN;
    static const cudaError_t attr = cudaFuncSetAttribute(restrict_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (attr != cudaSuccess) return attr;
    restrict_kernel<T><<<t.n_coarse, kChildThreads * kMaxChildren, smem, st>>>(t, rh, fH);
    return cudaGetLastError();
}
template cudaError_t launch_prolong_add<double>(const TransferView<double>&, const double*, double*, cudaStream_t);
template cudaError_t launch_prolong_add<float>(const TransferView<float>&, const float*, float*, cudaStream_t);
template cudaError_t launch_restrict<double>(const TransferView<double>&, const double*, double*, cudaStream_t);
template cudaError_t launch_restrict<float>(const TransferView<float>&, const float*, float*, cudaStream_t);

}  // namespace dg
