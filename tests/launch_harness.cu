// C entry points to launchers of the library that its public calls reach only through a solve, for the GPU tests.
#include "kernels.h"

using namespace wmg;

// Level-0 stencil with fused dots: out = a in + b Hop(in), <out|in> and ||out||^2 of right-hand side r at result[4 r].
extern "C" int t_wilson_dots(int prec, const void* in, void* out, const void* links, const int* L, double a, double b,
                             int nrhs, double* partials, unsigned* tickets, double* result, int variant) {
  DslashCall d;
  d.prec = prec;
  d.in = in;
  d.out = out;
  d.y = nullptr;
  d.z = in;
  d.links = links;
  for (int m = 0; m < 4; ++m) d.L[m] = L[m];
  d.a = a;
  d.b = b;
  d.c = 0.0;
  d.nrhs = nrhs;
  d.red = {partials, tickets, result, 4};
  d.adiag = nullptr;
  d.variant = variant;
  return launch_wilson(d, nullptr);
}
extern "C" int t_pack_links(int prec, const void* ext, void* out, int V) { return launch_pack_links(prec, ext, out, V, nullptr); }
extern "C" int t_wilson_variants(int prec, int nrhs, int V) { return wilson_variants(prec, true, nrhs, V); }

// Tensor-core coarse stencil of a packed operator, FP32 vectors, waits of `spins` tries.
extern "C" int t_coarse_mma(const void* C, void* packed, const void* in, void* out, const int* L, int n, int R, int variant,
                            void* scratch, int spins) {
  const int V = L[0] * L[1] * L[2] * L[3];
  if (launch_mma_pack((const double2*)C, n, V, packed, nullptr)) return -1;
  return launch_coarse_mma(1, packed, in, out, nullptr, L, n, R, 1.0, 0.0, nullptr, variant, nullptr, scratch, spins);
}
extern "C" size_t t_mma_pack_bytes(int n, int V) { return mma_pack_bytes(n, V); }
extern "C" size_t t_mma_scratch_bytes(int n, int V, int R) { return coarse_mma_scratch_bytes(n, V, R); }

// Coarsest product y = inv x, row form or tiled (scratch zeroed).
extern "C" int t_matvec(int pm, int pin, int pout, int N, const void* inv, const void* x, void* y, int nrhs, int acc,
                        void* scratch) {
  return launch_dense_matvec(pm, pin, pout, N, inv, x, y, nrhs, acc, nullptr, scratch, nullptr);
}
extern "C" size_t t_matvec_scratch_bytes(int N) { return dense_matvec_scratch_bytes(N); }

// Overlaps <W_j|w> of right-hand side r at result[(r kmax + j) 2]; W holds a multiple of eight vectors.
extern "C" int t_multidot(int prec, size_t n, int nrhs, int k, int kmax, const void* W, const void* w, double* partials,
                          unsigned* tickets, double* result) {
  const RedArgs red = {partials, tickets, result, 0};
  return launch_multidot(prec, n, nrhs, k, kmax, W, n * nrhs, w, red, nullptr);
}
