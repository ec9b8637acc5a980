// Shared device helpers: complex arithmetic, storage precisions, deterministic reductions.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>
#include <utility>

namespace wmg {

// Launch checks: a launcher reads (and so clears) the thread's last CUDA error
// right after its launch; the error is kept here so that the caller's message
// names it.
inline thread_local cudaError_t tl_launch_error = cudaSuccess;
inline bool launch_ok() {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) tl_launch_error = e;
  return e == cudaSuccess;
}
inline cudaError_t take_launch_error() {
  const cudaError_t e = tl_launch_error;
  tl_launch_error = cudaSuccess;
  return e;
}

// Dynamic shared memory above 48 KB needs a per-kernel opt-in.  The attribute
// is global to the kernel, so a value chosen per launch would race between
// host threads launching the same kernel with different sizes; every caller
// sets the device's maximum instead, the same value from any thread (the
// amount a launch really uses still sets its occupancy).
inline int smem_optin_bytes() {
  static const int v = [] {
    int d = 0, x = 48 * 1024;
    if (cudaGetDevice(&d) != cudaSuccess || cudaDeviceGetAttribute(&x, cudaDevAttrMaxSharedMemoryPerBlockOptin, d) !=
                                                 cudaSuccess) {
      cudaGetLastError();
      x = 48 * 1024;
    }
    return x;
  }();
  return v;
}
// Streaming multiprocessors of the current device (queried once; 152 on GB300).
inline int sm_count() {
  static const int v = [] {
    int d = 0, x = 152;
    if (cudaGetDevice(&d) != cudaSuccess || cudaDeviceGetAttribute(&x, cudaDevAttrMultiProcessorCount, d) != cudaSuccess ||
        x < 1) {
      cudaGetLastError();
      x = 152;
    }
    return x;
  }();
  return v;
}

// Chains of dependent launches.  A kernel of the solver's loops begins with
// chain_begin(): it waits there until the launches before it on its stream
// have completed, and lets the next one be launched meanwhile.  Launched with
// launch_chain it may then start (its blocks take their places, its
// instructions are fetched) while its predecessor still runs, so a dependent
// launch costs less than a full drain and start: 18 x 14 x 10 x 21, two MR
// steps in BF16 (six launches): 49 -> 41 us; 360 launches of a Gauss-Jordan
// inverse: 6.7 -> 5.9 ms.  Everything after chain_begin() sees its
// predecessors' memory; a kernel without it is launched with <<<>>>.
// An early grid takes the places that its predecessor leaves, so where CTAs run
// long and few, some SMs get more of them than others: chain_fits (launch_rules.h)
// keeps FP64 launches and the coarsest product from that, ChainOff the cases below.
// Off in the library's own captures (a graph's edges cost little by themselves,
// and the twelve-source solve took 333 ms with early starts, 309 without), among
// the solves of mg_solve_many (four on 8^3 x 16: 17.1 and 16.7 ms), for FP64
// transfers inside a cycle, and for one-wave launches of the fused setup step (14.6
// and 13.4 ms of setup).  On in a caller's capture (20 FP16 stencils on 8^3 x 16: 51
// us, 59 without; two BF16 MR steps gain 4 %, the tile transfers lose 2 %) and in
// solves on a caller's threads (mg_solve_masses on two threads: one right-hand side
// 8.2 ms, 8.6 without; eight 20.6 and 20.3).
__device__ __forceinline__ void chain_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
inline thread_local bool tl_chain_off = false;  // set by ChainOff
// While alive (and `off`), this thread's launch_chain launches wait for their predecessor's end.
struct ChainOff {
  const bool prev = tl_chain_off;
  explicit ChainOff(bool off) { tl_chain_off = prev || off; }
  ~ChainOff() { tl_chain_off = prev; }
  ChainOff(const ChainOff&) = delete;
};
// CTAs of a kernel that an SM holds at once (0: not to be had).
template <typename K>
inline int ctas_per_sm(K kern, int threads, size_t smem) {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads, smem) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  return n;
}
// The same through a word that keeps the last answer: shared memory in the upper bits, CTAs + 1 in the low byte.
template <typename K>
inline int ctas_held(std::atomic<unsigned long long>& last, K kern, int threads, size_t smem) {
  const unsigned long long v = last.load(std::memory_order_relaxed);
  if ((v & 255) && v >> 8 == smem) return (int)(v & 255) - 1;
  const int n = ctas_per_sm(kern, threads, smem);
  last.store((unsigned long long)smem << 8 | (unsigned)(n + 1), std::memory_order_relaxed);
  return n;
}
template <typename... P, typename... A>
inline void launch_chain(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = tl_chain_off ? 0 : 1;
  cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);  // an error stays for launch_ok()
}

template <typename K>
inline void allow_big_smem(K kern) {
  cudaFuncAttributes fa;
  int bytes = smem_optin_bytes();
  if (cudaFuncGetAttributes(&fa, kern) == cudaSuccess)
    bytes -= (int)fa.sharedSizeBytes;  // the opt-in limit covers static plus dynamic shared memory
  else
    cudaGetLastError();
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess)
    cudaGetLastError();
}


// ------------------------------------------------------------------ complex
template <typename R>
struct cx {
  R re, im;
};

template <typename R>
__host__ __device__ __forceinline__ cx<R> mk(R a, R b) {
  cx<R> z;
  z.re = a;
  z.im = b;
  return z;
}
template <typename R>
__host__ __device__ __forceinline__ cx<R> zero() {
  return mk<R>(R(0), R(0));
}
template <typename R>
__host__ __device__ __forceinline__ cx<R> operator+(cx<R> a, cx<R> b) {
  return mk<R>(a.re + b.re, a.im + b.im);
}
template <typename R>
__host__ __device__ __forceinline__ cx<R> operator-(cx<R> a, cx<R> b) {
  return mk<R>(a.re - b.re, a.im - b.im);
}
template <typename R>
__host__ __device__ __forceinline__ cx<R> operator*(cx<R> a, cx<R> b) {
  return mk<R>(a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re);
}
template <typename R>
__host__ __device__ __forceinline__ cx<R> operator*(R s, cx<R> a) {
  return mk<R>(s * a.re, s * a.im);
}
template <typename R>
__host__ __device__ __forceinline__ cx<R> conj(cx<R> a) {
  return mk<R>(a.re, -a.im);
}
// conj(a) * b
template <typename R>
__host__ __device__ __forceinline__ cx<R> cmul_conj(cx<R> a, cx<R> b) {
  return mk<R>(a.re * b.re + a.im * b.im, a.re * b.im - a.im * b.re);
}
// acc + a * b
template <typename R>
__host__ __device__ __forceinline__ cx<R> cfma(cx<R> a, cx<R> b, cx<R> acc) {
  acc.re = fma(a.re, b.re, acc.re);
  acc.re = fma(-a.im, b.im, acc.re);
  acc.im = fma(a.re, b.im, acc.im);
  acc.im = fma(a.im, b.re, acc.im);
  return acc;
}
// acc + conj(a) * b
template <typename R>
__host__ __device__ __forceinline__ cx<R> cfma_conj(cx<R> a, cx<R> b, cx<R> acc) {
  acc.re = fma(a.re, b.re, acc.re);
  acc.re = fma(a.im, b.im, acc.re);
  acc.im = fma(a.re, b.im, acc.im);
  acc.im = fma(-a.im, b.re, acc.im);
  return acc;
}
template <typename R>
__host__ __device__ __forceinline__ cx<R> times_i(cx<R> a) {
  return mk<R>(-a.im, a.re);
}
template <typename R>
__host__ __device__ __forceinline__ cx<R> times_minus_i(cx<R> a) {
  return mk<R>(a.im, -a.re);
}
template <typename R>
__host__ __device__ __forceinline__ R norm2(cx<R> a) {
  return a.re * a.re + a.im * a.im;
}

// ------------------------------------------------------------------ storage
// A complex element stored as two reals of type T; arithmetic type R.
template <typename T>
struct Store;

template <>
struct Store<double2> {
  typedef double R;
  static __device__ __forceinline__ cx<double> ld(const double2* p, size_t i) {
    double2 v = p[i];
    return mk<double>(v.x, v.y);
  }
  static __device__ __forceinline__ void st(double2* p, size_t i, cx<double> v) {
    p[i] = make_double2(v.re, v.im);
  }
};
template <>
struct Store<float2> {
  typedef float R;
  static __device__ __forceinline__ cx<float> ld(const float2* p, size_t i) {
    float2 v = p[i];
    return mk<float>(v.x, v.y);
  }
  static __device__ __forceinline__ void st(float2* p, size_t i, cx<float> v) {
    p[i] = make_float2(v.re, v.im);
  }
};
template <>
struct Store<__half2> {
  typedef float R;
  static __device__ __forceinline__ cx<float> ld(const __half2* p, size_t i) {
    float2 v = __half22float2(p[i]);
    return mk<float>(v.x, v.y);
  }
  static __device__ __forceinline__ void st(__half2* p, size_t i, cx<float> v) {
    p[i] = __floats2half2_rn(v.re, v.im);
  }
};
template <>
struct Store<__nv_bfloat162> {
  typedef float R;
  static __device__ __forceinline__ cx<float> ld(const __nv_bfloat162* p, size_t i) {
    float2 v = __bfloat1622float2(p[i]);
    return mk<float>(v.x, v.y);
  }
  static __device__ __forceinline__ void st(__nv_bfloat162* p, size_t i, cx<float> v) {
    p[i] = __floats2bfloat162_rn(v.re, v.im);
  }
};

// The value a complex number has after a round trip through storage T.
template <typename T>
__device__ __forceinline__ cx<typename Store<T>::R> as_stored(cx<typename Store<T>::R> v);
template <>
__device__ __forceinline__ cx<double> as_stored<double2>(cx<double> v) { return v; }
template <>
__device__ __forceinline__ cx<float> as_stored<float2>(cx<float> v) { return v; }
template <>
__device__ __forceinline__ cx<float> as_stored<__half2>(cx<float> v) {
  float2 f = __half22float2(__floats2half2_rn(v.re, v.im));
  return mk<float>(f.x, f.y);
}
template <>
__device__ __forceinline__ cx<float> as_stored<__nv_bfloat162>(cx<float> v) {
  float2 f = __bfloat1622float2(__floats2bfloat162_rn(v.re, v.im));
  return mk<float>(f.x, f.y);
}

// Read a complex value of any storage into arithmetic type R2.
template <typename R2, typename T>
__device__ __forceinline__ cx<R2> ldc(const T* p, size_t i) {
  cx<typename Store<T>::R> v = Store<T>::ld(p, i);
  return mk<R2>((R2)v.re, (R2)v.im);
}
template <typename T, typename R2>
__device__ __forceinline__ void stc(T* p, size_t i, cx<R2> v) {
  typedef typename Store<T>::R R;
  Store<T>::st(p, i, mk<R>((R)v.re, (R)v.im));
}

// Bytes of one stored complex element per precision code (0 f64, 1 f32, 2 f16, 3 bf16).
__host__ __device__ inline size_t cx_bytes(int prec) { return prec == 0 ? 16 : (prec == 1 ? 8 : 4); }

// ------------------------------------------------------------------ lattice geometry
// Sites are lexicographic with x fastest; directions d = 0 (self),
// 1 + 2 mu (n + mu), 2 + 2 mu (n - mu); periodic boundaries.
__host__ __device__ __forceinline__ void site_coords(int s, const int (&L)[4], int (&c)[4]) {
  c[0] = s % L[0];
  s /= L[0];
  c[1] = s % L[1];
  s /= L[1];
  c[2] = s % L[2];
  c[3] = s / L[2];
}
__host__ __device__ __forceinline__ int site_index(const int (&c)[4], const int (&L)[4]) {
  return c[0] + L[0] * (c[1] + L[1] * (c[2] + L[2] * c[3]));
}
__host__ __device__ __forceinline__ int neighbor(const int (&c)[4], const int (&L)[4], int d) {
  int n[4] = {c[0], c[1], c[2], c[3]};
  if (d > 0) {
    const int mu = (d - 1) >> 1;
    if (d & 1)
      n[mu] = (n[mu] + 1 == L[mu]) ? 0 : n[mu] + 1;
    else
      n[mu] = (n[mu] == 0) ? L[mu] - 1 : n[mu] - 1;
  }
  return site_index(n, L);
}

// ------------------------------------------------------------------ field layouts
// Level-0 fields (12 complex components c = spin * 3 + colour per site) are
// stored in three chunks of four components, each chunk site-major:
// component c of site s at complex index ((c / 4) V + s) 4 + c % 4 (per
// right-hand side; wilson_hop.cuh gives the reason).  Coarse-level fields
// are component-major, [ncomp][V].  The chunk q of a field is 4 or 1.
__host__ __device__ __forceinline__ size_t fidx(int c, size_t s, size_t V) {
  return (((size_t)(c >> 2) * V + s) << 2) + (c & 3);
}
__host__ __device__ __forceinline__ size_t fidx_q(int c, size_t s, size_t V, int q) {
  return q == 4 ? fidx(c, s, V) : (size_t)c * V + s;
}

// ------------------------------------------------------------------ reductions
// Deterministic grid reductions: every block writes NV partial doubles, then
// the last block to finish (atomic ticket after a fence) sums the partials of
// all blocks in block order and writes the result.  Summation order is fixed
// by the launch shape, never by scheduling.  Each reduction "lane" (one per
// right-hand side) owns a ticket counter that the last block resets to 0.
struct RedArgs {
  double* partials;   // [nlanes][gridDim.x][NV]
  unsigned* tickets;  // [nlanes]
  double* result;     // [nlanes][stride]
  int stride;         // doubles between lanes in result
};

template <int NV, int NT, typename T>
__device__ __forceinline__ void block_sum(T (&v)[NV], T* smem /* NV * NT/32 */) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    T s = v[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) smem[k * (NT / 32) + warp] = s;
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      T s = lane < NT / 32 ? smem[k * (NT / 32) + lane] : (T)0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
      v[k] = s;  // valid in thread 0
    }
  }
  __syncthreads();
}

// The two halves of a grid reduction for lane `ln`: every tile of NT threads'
// values is summed within its CTA into its own partial (grid_partial), and the
// last CTA to finish adds the `ntiles` partials in tile order (grid_finish).
// Call from every thread of every CTA; NT = blockDim.x (a multiple of 32,
// <= 1024).  The tree inside a tile runs in T (FP32 for the FP32 / 16-bit
// kernels: FP64 arithmetic is scarce on this part); the sum over tiles runs in
// FP64.  A CTA may take several tiles before it finishes: the result depends
// on the tiles alone, not on how CTAs share them.
template <int NV, int NT, typename T>
__device__ __forceinline__ void grid_partial(T (&v)[NV], const RedArgs& ra, int ln, int tile, int ntiles) {
  __shared__ T smem_t[NV * (NT / 32)];
  block_sum<NV, NT, T>(v, smem_t);
  if (threadIdx.x == 0) {
    double* dst = ra.partials + ((size_t)ln * ntiles + tile) * NV;
#pragma unroll
    for (int k = 0; k < NV; ++k) dst[k] = (double)v[k];
  }
}
// Sums of lane ln's `ntiles` partials, valid in thread 0: thread t takes the
// partials t, t + NT, ..., and the threads' sums are added in the tree of
// block_sum, but level by level through shared memory with every lane at work.
// A warp's FP64 addition occupies this part's FP64 unit whether one lane needs
// it or 32: the shuffle tree issues 135 of them for three values and 256
// threads, this about 25, and the last block of a reduction waits for them
// (18 x 14 x 10 x 21, two BF16 MR steps: 41 -> 39 us).  The same bits.
template <int NV, int NT>
__device__ __forceinline__ void sum_partials(double (&w)[NV], const double* partials, int ln, int ntiles,
                                             double* smem /* NV * NT */) {
  static_assert((NT & (NT - 1)) == 0 && NT >= 32, "the tree halves NT");
#pragma unroll
  for (int k = 0; k < NV; ++k) w[k] = 0.0;
  for (int b = threadIdx.x; b < ntiles; b += NT) {
    const double* src = partials + ((size_t)ln * ntiles + b) * NV;
#pragma unroll
    for (int k = 0; k < NV; ++k) w[k] += __ldcg(src + k);
  }
#pragma unroll
  for (int k = 0; k < NV; ++k) smem[k * NT + threadIdx.x] = w[k];
  __syncthreads();
  // within groups of 32: element i of a group takes element i + o
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    for (int e = threadIdx.x; e < NV * (NT / 32) * o; e += NT) {
      double* q = smem + (e / o) * 32 + e % o;
      *q += q[o];
    }
    __syncthreads();
  }
  // the groups' sums
#pragma unroll
  for (int o = NT / 64; o > 0; o >>= 1) {
    if ((int)threadIdx.x < NV * o) {
      double* q = smem + (threadIdx.x / o) * NT + (threadIdx.x % o) * 32;
      *q += q[o * 32];
    }
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < NV; ++k) w[k] = smem[k * NT];
}
// Next ticket of a counter, releasing this thread's earlier writes (and those it
// has seen through a barrier) and acquiring those of the earlier tickets.  One
// instruction, and weaker than the two sequentially consistent fences around a
// plain atomic.
__device__ __forceinline__ unsigned take_ticket(unsigned* t) {
  unsigned v;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(v) : "l"(t) : "memory");
  return v;
}
template <int NV, int NT>
__device__ __forceinline__ void grid_finish(const RedArgs& ra, int ln, int ntiles) {
  __shared__ double smem_d[NV * NT];
  // the barrier carries the flag: a CTA may finish several lanes in turn, and a
  // flag in shared memory could be overwritten before every warp has read it
  const bool mine = threadIdx.x == 0 && take_ticket(ra.tickets + ln) == gridDim.x - 1;
  if (!__syncthreads_or(mine)) return;
  double w[NV];
  sum_partials<NV, NT>(w, ra.partials, ln, ntiles, smem_d);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) ra.result[(size_t)ln * ra.stride + k] = w[k];
    ra.tickets[ln] = 0u;
  }
}
// One tile per CTA.
template <int NV, int NT, typename T>
__device__ __forceinline__ void grid_reduce(T (&v)[NV], const RedArgs& ra, int ln) {
  grid_partial<NV, NT, T>(v, ra, ln, blockIdx.x, gridDim.x);
  grid_finish<NV, NT>(ra, ln, gridDim.x);
}

}  // namespace wmg
