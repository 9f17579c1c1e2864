// Zeroth-order / Galerkin and puncture kernels.
#pragma once
#include "internal.h"

namespace dg {

struct PunctureDev {
    int n;
    double m[16];
    double c[16][3];
    double P[16][3];
    double S[16][3];
};

enum NlKind { kNlNone = 0, kNlPuncture = 1, kNlPower = 2 };

struct NlArgs {
    int n_elems;
    int kind;                  // kNlPuncture: s = beta (1 + alpha (1 + u))^-7; kNlPower: s = coef u^power
    int power;
    const int* p;
    const long long* dof_off;
    const long long* vqp_off;
    const double* wdetJ;
    const double* alpha;       // puncture: alpha; power: coef
    const double* beta;
    const double* tab;
    long long n_vqp;   // bounds check
    int* chk;
};

// Zeroth-order term on a coarse level (see newton.cu): its coefficient at the
// m^3 = (2p + 1)^3 GL points of every element, and the dense blocks.
struct GalerkinArgs {
    int n_coarse;
    const int* pH;             // coarse degrees
    const int* pf;             // degrees of the next finer level
    int fine_is_finest;        // its coefficients sit at n = p + 1 points per direction (else at 2p + 1)
    const int* child_off;      // n_coarse + 1
    const int* child_id;
    const unsigned char* child_bits;
    const long long* off_f;    // per finer element: offset of its coefficients
    const long long* off;      // per coarse element: offset of its coefficients
    const long long* Ob_off;   // per coarse element: offset of its (n^3 x n^3) block
    const double* tab;         // GalerkinTab
    long long n_coef_f, n_coef, ob_total;   // bounds checks
    int* chk;
};

// Tables of the coarse zeroth-order term, each matrix padded to kGalM x kGalM:
//   W[n][q][b]: W[k][j] = L_k(map_b(x^q_j)), L_k the Lagrange basis of the
//     2n - 1 GL points, x^q the q GL points, map_b: b = 0, 1 the child halves, 2 the identity
//   E[n]:       E[k][a] = l_a(x^(2n-1)_k), l_a the LGL basis of n points
constexpr int kGalM = 2 * kMaxN - 1;
struct GalerkinTab {
    static constexpr int Stride = kGalM * kGalM;
    static constexpr int E = kNumN * (kGalM + 1) * 3;
    static constexpr int Count = E + kNumN;
    __host__ __device__ static int w(int n, int q, int b) { return (((n - kMinN) * (kGalM + 1) + q) * 3 + b) * Stride; }
    __host__ __device__ static int e(int n) { return (E + n - kMinN) * Stride; }
};
void build_galerkin_tables(std::vector<double>& tab);

cudaError_t launch_puncture(const double* vxyz, long long n, const PunctureDev& P, double* alpha, double* beta,
                            cudaStream_t st);
// S = I^T (w det J beta (1 + alpha (1 + u))^-7); jac (optional) = w det J 7 alpha beta (...)^-8
cudaError_t launch_nl(const NlArgs& a, const double* u, double* S, double* jac64, float* jac32, cudaStream_t st);
// R = Lu - S - F (F may be NULL)
cudaError_t launch_sub(const double* Lu, const double* S, const double* F, double* R, long long n, cudaStream_t st);
// coef = the level's coefficients from the finer level's; O64, O32 = its dense blocks.  max_n: largest n of the level.
cudaError_t launch_galerkin(const GalerkinArgs& g, int max_n, const double* coef_f, double* coef, double* O64,
                            float* O32, cudaStream_t st);

}  // namespace dg
