// FP64 contractions by exact digit products on the tensor cores (k_dg.cu).
#pragma once
#include "common.cuh"

struct DgLeft;    // digits of a static left operand per batch entry
struct DgGemm;    // C (+)= A X per batch entry
struct DgSeries;  // the Chebyshev series

// element (r, k) of a left operand: src[r rs + k cs], conjugated when conj
struct DgMat {
    const zd* src;
    size_t rs, cs;
    int conj, M, K;
};
struct DgRight {
    const zd* X;  // K x ncol, column-major
    int ldx, K;   // K at most the left operand's
    zd* C;
    int ldc;
    const zd* X2 = nullptr;          // rows K1 .. K - 1 of X from here, or null
    int ldx2 = 0, K1 = 0;
    const double* scale = nullptr;   // device factor on the product, or null
};

DgLeft* dg_left_create(int nk, const DgMat* m, cudaStream_t s);
int launch_dg_left(const DgLeft* l, cudaStream_t s);  // cut the operand anew; returns its launches
void dg_left_destroy(DgLeft* l);
size_t dg_left_bytes(int M, int K);
// null where the device memory does not suffice; lmod > 0: entry k takes the left operand k % lmod
DgGemm* dg_gemm_create(const DgLeft* l, int nk, const DgRight* r, int ncol, int* flag, int lmod = 0);
void dg_gemm_destroy(DgGemm* g);
int launch_dg_gemm(const DgGemm* g, int kofs, int nk, int beta, cudaStream_t s, bool packed = false);  // returns its launches

// the interstitial sum with the left operand generated from the table
struct DgToep;
DgToep* dg_toep_create(int nk, const DgRight* r, const int* const* glin, int ncol, const DgGemm* x, int nvt, int center, int* flag);
void dg_toep_destroy(DgToep* t);
// which: 0 V~, 1 the step's V~ + s dV~
int launch_dg_table(const DgToep* t, int which, const zd* tab, cudaStream_t s);
int launch_dg_toep(const DgToep* t, int which, int kofs, int nk, cudaStream_t s);

struct StepArgs;
DgSeries* dg_series_create(int nk, int n, int ns, const zd* const* coef);  // coef: the c_n of every k-point (device)
void dg_series_destroy(DgSeries* g);
int launch_dg_series(const DgSeries* g, const StepArgs& a, cudaStream_t s);       // returns its launches
