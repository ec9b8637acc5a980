// Restriction R = P^+ and prolongation P (Sec. 3, Eq. 3.2 and the text
// after it) for many right-hand sides on tensor cores.
//
// Per aggregate B and chirality chi both are dense complex products with the
// aggregate's block of P, P_B (nv x len, len = ncomp/2 * |B| components):
//   restriction   out (nv x R)  = conj(P_B) (nv x len) * v (len x R)
//   prolongation  out (len x R) = P_B^T (len x nv) * x_c (nv x R)
// The kernels on CUDA cores read P_B once per right-hand side; here one CTA
// per (B, chi) reads it once for all R (R <= 64), which is what bounds the
// multi-right-hand-side transfer: at nv = 24 and 16-bit storage P is 1152 B
// per fine site, as much as 24 right-hand sides of the vectors themselves.
//
// Arithmetic: mma.sync m16n8k16 with 16-bit inputs (FP16 or BF16, the
// storage type of the fine vectors and of P) and FP32 accumulation, in the
// real embedding of the complex product: with P = Pr + i Pi,
//   conj(P) v : re = Pr vr + Pi vi,  im = Pr vi - Pi vr
//   P x       : re = Pr xr - Pi xi,  im = Pr xi + Pi xr
// so each 16 x 16 fragment pair of P feeds four MMAs (-Pi is Pi with the
// sign bits flipped).  Operands are staged in shared memory as separate real
// and imaginary planes, K contiguous, so every fragment register is one
// 32-bit shared load.  Summation order is fixed (K ascending per warp slice,
// slices added in order), so results are deterministic.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "common.cuh"
#include "kernels.h"
#include "wilson_hop.cuh"

namespace wmg {

static inline bool launched() { return launch_ok(); }

template <typename T>
struct MmaT;
template <>
struct MmaT<__half> {
  typedef __half2 T2;
  static __device__ __forceinline__ __half from(float x) { return __float2half_rn(x); }
  static __device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
  }
};
template <>
struct MmaT<__nv_bfloat16> {
  typedef __nv_bfloat162 T2;
  static __device__ __forceinline__ __nv_bfloat16 from(float x) { return __float2bfloat16_rn(x); }
  static __device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
  }
};

__device__ __forceinline__ uint32_t ld32(const void* p) { return *(const uint32_t*)p; }

// A stored complex value as its two 16-bit planes: a bit move when the
// storage type is the MMA type, a rounding when it is FP32.
template <typename T>
__device__ __forceinline__ void planes(const typename MmaT<T>::T2 v, T& re, T& im) {
  re = v.x;
  im = v.y;
}
template <typename T>
__device__ __forceinline__ void planes(const float2 v, T& re, T& im) {
  re = MmaT<T>::from(v.x);
  im = MmaT<T>::from(v.y);
}
__device__ __forceinline__ uint32_t neg2(uint32_t v) { return v ^ 0x80008000u; }

// Fine site of aggregate B, aggregate-local site s (x fastest in both).
__device__ __forceinline__ int agg_site_t(const Agg& g, int B, int s) {
  int cb[4], cl[4], cf[4];
  site_coords(B, g.Lc, cb);
  site_coords(s, g.blk, cl);
#pragma unroll
  for (int m = 0; m < 4; ++m) cf[m] = cb[m] * g.blk[m] + cl[m];
  return site_index(cf, g.L);
}

constexpr int kTThreads = 256;  // 8 warps
constexpr int kTK = 128;        // K (restriction) or M (prolongation) chunk staged per step
constexpr int kTKs = kTK + 8;   // row stride of a staged plane: rows gid = 0..7 of a fragment fall in distinct banks

// ------------------------------------------------------------------ restriction
// CTA (B, chi).  Warp w owns M tile mt = w % MT (rows k of P) and the K steps
// ks = w / MT, w / MT + 8 / MT, ... of every chunk; the 8 / MT slices are
// added through shared memory at the end.
template <typename T, typename SI, typename SO, int NT8>
__global__ void __launch_bounds__(kTThreads)
    restrict_mma_kernel(const Agg g, const typename MmaT<T>::T2* P, const SI* in, SO* out, int R, int sidx_off) {
  chain_begin();
  typedef typename MmaT<T>::T2 T2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int MT = (g.nv + 15) / 16, Mp = MT * 16, NS = 8 / MT;
  const int Rp = NT8 * 8;
  T* Ps = (T*)smem_raw;          // [2][Mp][kTKs]
  T* Vs = Ps + 2 * Mp * kTKs;    // [2][Rp][kTKs]
  int* sidx = (int*)(smem_raw + sidx_off);  // fine site of each aggregate-local site
  const int B = blockIdx.x, chi = blockIdx.y;
  const int r0 = blockIdx.z * Rp;  // first right-hand side of this CTA (launch-shape split)
  const int len = g.nhalf * g.bsites;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
  const int mt = warp % MT, ks0 = warp / MT;
  const T2* Pb = P + ((size_t)B * 2 + chi) * g.nv * len;
  for (int s = threadIdx.x; s < g.bsites; s += kTThreads) sidx[s] = agg_site_t(g, B, s);
  float accr[NT8][4], acci[NT8][4];
#pragma unroll
  for (int q = 0; q < NT8; ++q)
#pragma unroll
    for (int e = 0; e < 4; ++e) accr[q][e] = acci[q][e] = 0.f;
  for (int e0 = 0; e0 < len; e0 += kTK) {
    __syncthreads();
    // staging: thread t owns column el = t % kTK of the chunk and the rows
    // t / kTK, t / kTK + 2, ... (the aggregate site of el is looked up once)
    {
      const int el = threadIdx.x % kTK, rr = threadIdx.x / kTK, e = e0 + el;
      const bool live = e < len;
      const T zero16 = MmaT<T>::from(0.f);
#pragma unroll 4
      for (int k = rr; k < Mp; k += kTThreads / kTK) {
        T re = zero16, im = zero16;
        if (live && k < g.nv) planes<T>(Pb[(size_t)k * len + e], re, im);
        Ps[(size_t)k * kTKs + el] = re;
        Ps[(size_t)(Mp + k) * kTKs + el] = im;
      }
      size_t base = 0;
      if (live) {
        const int c = e / g.bsites, s = e - c * g.bsites;
        base = fidx_q(chi * g.nhalf + c, sidx[s], g.V, g.q);
      }
      const size_t rstride = (size_t)g.ncomp * g.V;
#pragma unroll 4
      for (int r = rr; r < Rp; r += kTThreads / kTK) {
        T re = zero16, im = zero16;
        if (live && r0 + r < R) planes<T>(in[(size_t)(r0 + r) * rstride + base], re, im);
        Vs[(size_t)r * kTKs + el] = re;
        Vs[(size_t)(Rp + r) * kTKs + el] = im;
      }
    }
    __syncthreads();
    for (int ks = ks0; ks < kTK / 16; ks += NS) {
      const int kc = ks * 16 + 2 * tig;
      const T* pr0 = Ps + (size_t)(mt * 16 + gid) * kTKs + kc;
      const T* pi0 = Ps + (size_t)(Mp + mt * 16 + gid) * kTKs + kc;
      const uint32_t Ar[4] = {ld32(pr0), ld32(pr0 + 8 * kTKs), ld32(pr0 + 8), ld32(pr0 + 8 * kTKs + 8)};
      const uint32_t Ai[4] = {ld32(pi0), ld32(pi0 + 8 * kTKs), ld32(pi0 + 8), ld32(pi0 + 8 * kTKs + 8)};
      const uint32_t An[4] = {neg2(Ai[0]), neg2(Ai[1]), neg2(Ai[2]), neg2(Ai[3])};
#pragma unroll
      for (int q = 0; q < NT8; ++q) {
        const T* vr = Vs + (size_t)(q * 8 + gid) * kTKs + kc;
        const T* vi = Vs + (size_t)(Rp + q * 8 + gid) * kTKs + kc;
        const uint32_t br0 = ld32(vr), br1 = ld32(vr + 8), bi0 = ld32(vi), bi1 = ld32(vi + 8);
        MmaT<T>::mma(accr[q], Ar, br0, br1);  // Pr vr
        MmaT<T>::mma(accr[q], Ai, bi0, bi1);  // + Pi vi
        MmaT<T>::mma(acci[q], Ar, bi0, bi1);  // Pr vi
        MmaT<T>::mma(acci[q], An, br0, br1);  // - Pi vr
      }
    }
  }
  // add the K slices: slice ks0 > 0 parks its tile, slice 0 sums in slice order
  __syncthreads();
  float* red = (float*)smem_raw;  // [8 warps][NT8][2][4][32]
  if (ks0 > 0) {
#pragma unroll
    for (int q = 0; q < NT8; ++q)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        red[((((size_t)warp * NT8 + q) * 2 + 0) * 4 + e) * 32 + lane] = accr[q][e];
        red[((((size_t)warp * NT8 + q) * 2 + 1) * 4 + e) * 32 + lane] = acci[q][e];
      }
  }
  __syncthreads();
  if (ks0 != 0) return;
  for (int sl = 1; sl < NS; ++sl) {
    const int w2 = sl * MT + mt;
#pragma unroll
    for (int q = 0; q < NT8; ++q)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        accr[q][e] += red[((((size_t)w2 * NT8 + q) * 2 + 0) * 4 + e) * 32 + lane];
        acci[q][e] += red[((((size_t)w2 * NT8 + q) * 2 + 1) * 4 + e) * 32 + lane];
      }
  }
#pragma unroll
  for (int q = 0; q < NT8; ++q)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int k = mt * 16 + gid + (e >= 2 ? 8 : 0);
      const int r = r0 + q * 8 + 2 * tig + (e & 1);
      if (k < g.nv && r < R)
        stc(out, ((size_t)r * 2 * g.nv + chi * g.nv + k) * g.Vc + B, mk<float>(accr[q][e], acci[q][e]));
    }
}

// ------------------------------------------------------------------ prolongation
// CTA (B, chi); chunks of kTK rows e of P_B^T, warp w the 16 rows w * 16.. of
// the chunk, all of K = nv (padded to KT * 16) and all right-hand sides.
template <typename T, typename SI, typename SO, int NT8>
__global__ void __launch_bounds__(kTThreads)
    prolong_mma_kernel(const Agg g, const typename MmaT<T>::T2* P, const SI* in, SO* out, int R, int sidx_off) {
  chain_begin();
  typedef typename MmaT<T>::T2 T2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int KT = (g.nv + 15) / 16, Kp = KT * 16, Kps = Kp + 8;  // Kps: bank-spread row stride
  const int Rp = NT8 * 8;
  T* Xs = (T*)smem_raw;          // [2][Rp][Kps]
  T* Pt = Xs + 2 * Rp * Kps;     // [2][kTK][Kps]
  int* sidx = (int*)(smem_raw + sidx_off);
  const int B = blockIdx.x, chi = blockIdx.y;
  const int r0 = blockIdx.z * Rp;  // first right-hand side of this CTA (launch-shape split)
  const int len = g.nhalf * g.bsites;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
  const T2* Pb = P + ((size_t)B * 2 + chi) * g.nv * len;
  for (int s = threadIdx.x; s < g.bsites; s += kTThreads) sidx[s] = agg_site_t(g, B, s);
  for (int t = threadIdx.x; t < Rp * Kp; t += kTThreads) {
    const int r = t / Kp, k = t % Kp;
    T re = MmaT<T>::from(0.f), im = re;
    if (r0 + r < R && k < g.nv) planes<T>(in[((size_t)(r0 + r) * 2 * g.nv + chi * g.nv + k) * g.Vc + B], re, im);
    Xs[(size_t)r * Kps + k] = re;
    Xs[(size_t)(Rp + r) * Kps + k] = im;
  }
  for (int e0 = 0; e0 < len; e0 += kTK) {
    __syncthreads();
    {
      const int el = threadIdx.x % kTK, rr = threadIdx.x / kTK, e = e0 + el;
      const T zero16 = MmaT<T>::from(0.f);
#pragma unroll 4
      for (int k = rr; k < Kp; k += kTThreads / kTK) {
        T re = zero16, im = zero16;
        if (e < len && k < g.nv) planes<T>(Pb[(size_t)k * len + e], re, im);
        Pt[(size_t)el * Kps + k] = re;
        Pt[(size_t)(kTK + el) * Kps + k] = im;
      }
    }
    __syncthreads();
    float accr[NT8][4], acci[NT8][4];
#pragma unroll
    for (int q = 0; q < NT8; ++q)
#pragma unroll
      for (int e = 0; e < 4; ++e) accr[q][e] = acci[q][e] = 0.f;
    for (int ks = 0; ks < KT; ++ks) {
      const int kc = ks * 16 + 2 * tig;
      const T* pr0 = Pt + (size_t)(warp * 16 + gid) * Kps + kc;
      const T* pi0 = Pt + (size_t)(kTK + warp * 16 + gid) * Kps + kc;
      const uint32_t Ar[4] = {ld32(pr0), ld32(pr0 + 8 * Kps), ld32(pr0 + 8), ld32(pr0 + 8 * Kps + 8)};
      const uint32_t Ai[4] = {ld32(pi0), ld32(pi0 + 8 * Kps), ld32(pi0 + 8), ld32(pi0 + 8 * Kps + 8)};
      const uint32_t An[4] = {neg2(Ai[0]), neg2(Ai[1]), neg2(Ai[2]), neg2(Ai[3])};
#pragma unroll
      for (int q = 0; q < NT8; ++q) {
        const T* xr = Xs + (size_t)(q * 8 + gid) * Kps + kc;
        const T* xi = Xs + (size_t)(Rp + q * 8 + gid) * Kps + kc;
        const uint32_t br0 = ld32(xr), br1 = ld32(xr + 8), bi0 = ld32(xi), bi1 = ld32(xi + 8);
        MmaT<T>::mma(accr[q], Ar, br0, br1);  // Pr xr
        MmaT<T>::mma(accr[q], An, bi0, bi1);  // - Pi xi
        MmaT<T>::mma(acci[q], Ar, bi0, bi1);  // Pr xi
        MmaT<T>::mma(acci[q], Ai, br0, br1);  // + Pi xr
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = e0 + warp * 16 + gid + 8 * h;
      if (e >= len) continue;
      const int c = e / g.bsites, s = e - c * g.bsites;
      const size_t o = fidx_q(chi * g.nhalf + c, sidx[s], g.V, g.q);
#pragma unroll
      for (int q = 0; q < NT8; ++q)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int r = r0 + q * 8 + 2 * tig + j;
          if (r < R) stc(out, (size_t)r * g.ncomp * g.V + o, mk<float>(accr[q][2 * h + j], acci[q][2 * h + j]));
        }
    }
  }
}

// ------------------------------------------------------------------ level 0: pipelined tiles
// The same two products on level-0 fields (chunked layout, a site's chunk of
// four components is 16 bytes), aggregates of a multiple of four sites.  What
// bounds them is HBM: at nv = 24 and 24 right-hand sides P and the vectors
// are 302 MB on 16^3 x 32, 24 flop per byte.  The kernels above stage both
// operands with 4-byte loads, split into planes, and wait for each chunk; here
// everything moves as 16-byte asynchronous copies of raw storage, the next
// stage's in flight while one is multiplied (16 sites per stage, 37 KB at
// nv = R = 24, two CTAs per SM).
//
// No planes: the operands stay interleaved (re, im), a 32-bit register of an
// MMA operand is one complex number, and K runs over the real numbers
// (k16 = 8 complex).  With v = (vr, vi) pairs as the A operand (rows = right-
// hand sides), conj(P) v is v . (Pr, Pi) and v . (-Pi, Pr): the second B
// operand is the first with halves swapped and one sign flipped.  Likewise
// P x is x . (Pr, -Pi) and x . (Pi, Pr).  The sum over k is free in its order,
// so a fragment's eight complex numbers are taken as two components of four
// consecutive aggregate sites, which is how they lie in memory: a lane reads
// a site's two components as 8 bytes, and writes a site's chunk as 16.
//
// 16^3 x 32, nv = 24, 24 right-hand sides, FP16: restriction 212 -> 64 us,
// prolongation 226 -> 64.5 us (4.8 TB/s; 45 us is the floor).
constexpr int kTileE = 16;                     // sites per stage
constexpr int kTilePRow = 6 * kTileE * 4 + 16;  // bytes of a staged row of P (4 mod 32 words: no bank conflicts)
// ... and of a staged (right-hand side, chunk): nch = 3 or 2 of them per right-hand side are 64 mod 128
__host__ __device__ constexpr int tile_vrow(int nch) { return kTileE * 16 + (nch == 3 ? 64 : 32); }
constexpr int kProlongThreads = 384;                       // 12 warps: one (four sites, chunk) each per stage

// dst: shared-memory address
__device__ __forceinline__ void cp_async16(unsigned dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
// Waits until at most `left` (0 or 1) of the committed stages are in flight.
__device__ __forceinline__ void cp_async_wait(int left) {
  if (left)
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
  else
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}
__device__ __forceinline__ uint32_t swap16(uint32_t v) { return __byte_perm(v, 0u, 0x1032u); }

// Copies of P into a stage: rows (chi, k) of NCHI chiralities, row chi np + k
// of the stage, 24 pieces of 16 bytes each (six components x four).  A thread
// keeps its piece and steps over rows, so a copy costs two additions.
template <int NCHI, typename T2>
struct StageP {
  const T2* src;  // piece of row 0 at site 0; null for a thread with none
  int off, row0, step, p4, nv, np, bs;
  __device__ __forceinline__ void init(const T2* Pb, int nv_, int np_, int bs_) {
    constexpr int PC = 6 * (kTileE / 4);
    nv = nv_;
    np = np_;
    bs = bs_;
    step = blockDim.x / PC;
    row0 = threadIdx.x / PC;
    const int piece = threadIdx.x - row0 * PC, c = piece / (kTileE / 4);
    p4 = 4 * (piece - c * (kTileE / 4));
    src = row0 < step ? Pb + c * bs + p4 : nullptr;
    off = (c * kTileE + p4) * 4;
  }
  __device__ __forceinline__ void issue(unsigned dst, int s0, int ns) const {
    if (!src || p4 >= ns) return;
    const int qs = step * 6 * bs, ds = step * kTilePRow;
#pragma unroll
    for (int chi = 0; chi < NCHI; ++chi) {
      const T2* q = src + s0 + (chi * nv + row0) * 6 * bs;
      unsigned d = dst + off + (chi * np + row0) * kTilePRow;
      int k = row0;
      for (; k + step < nv; k += 2 * step, q += 2 * qs, d += 2 * ds) {
        cp_async16(d, q);
        cp_async16(d + ds, q + qs);
      }
      if (k < nv) cp_async16(d, q);
    }
  }
};

// CTA = (aggregate, chiralities [one or both], 16 MT right-hand sides).  Four
// warps per chirality: groups of NG n-tiles (8 vectors each) times slices of
// the sites, whose sums are added in slice order.  NG = 1..4 is all of nv <= 32
// (one group, every offset a constant: the inner loop is bound by issue slots);
// NG = 0 is nv > 32, two groups of up to four.
template <typename T, typename SO, int MT, int NCHI, int NGT>
__global__ void __launch_bounds__(128 * NCHI, 4 / NCHI)
    restrict_tile_kernel(const Agg g, const typename MmaT<T>::T2* P, const typename MmaT<T>::T2* in, SO* out, int R,
                         int nsplit, int vrows, int sidx_off) {
  chain_begin();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int NCH = NCHI + 1, kVRow = tile_vrow(NCH), VROW = NCH * kVRow, NG = NGT ? NGT : 4;
  const int B = blockIdx.x / nsplit, r0 = (blockIdx.x % nsplit) * MT * 16;
  const int Rc = min(R - r0, MT * 16);
  const int bs = g.bsites, nv = g.nv, NT = (nv + 7) / 8;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
  const int chi = NCHI == 2 ? (warp & 1) : blockIdx.y, rest = NCHI == 2 ? warp >> 1 : warp;
  constexpr int ngroups = NGT ? 1 : 2, KS = 4 / ngroups;
  const int n0 = (rest % ngroups) * NG, slice = rest / ngroups;
  const int jb = NCHI == 2 ? 0 : (int)blockIdx.y;  // first chunk staged
  int* sidx = (int*)(smem_raw + sidx_off);
  for (int s = threadIdx.x; s < bs; s += blockDim.x) sidx[s] = agg_site_t(g, B, s);
  const int vbytes = vrows * VROW, stage_bytes = vbytes + NCHI * NT * 8 * kTilePRow;
  const int nst = (bs + kTileE - 1) / kTileE;
  StageP<NCHI, typename MmaT<T>::T2> cp;
  cp.init(P + ((size_t)B * 2 + (NCHI == 2 ? 0 : blockIdx.y)) * nv * 6 * bs, nv, NT * 8, bs);
  // copies of the field: row (r, chunk) = 3 r + chunk of the CTA's right-hand
  // sides, thread t always site t % 16 of the stage, rows t / 16, + blockDim / 16, ...
  const int vs = threadIdx.x % kTileE, vr = threadIdx.x / kTileE, vstep = blockDim.x / kTileE;
  // (vstep is even, so with two chunks staged a thread's rows are all of one chunk)
  const int vrow0 = NCHI == 2 ? vr : 3 * (vr >> 1) + jb + (vr & 1);
  const size_t vinc = (size_t)(NCHI == 2 ? vstep : 3 * (vstep >> 1)) * g.V * 4;
  const typename MmaT<T>::T2* vin = in + ((size_t)r0 * 3 + vrow0) * g.V * 4;
  const unsigned smem0 = (unsigned)__cvta_generic_to_shared(smem_raw);
  const int vn = Rc * NCH;
  __syncthreads();
  auto issue = [&](int i) {
    const unsigned buf = smem0 + (i & 1) * stage_bytes;
    const int s0 = i * kTileE, ns = min(kTileE, bs - s0);
    if (vs < ns) {
      const typename MmaT<T>::T2* src = vin + ((size_t)sidx[s0 + vs] << 2);
      unsigned d = buf + vr * kVRow + vs * 16;
      int q = vr;
      for (; q + vstep < vn; q += 2 * vstep, src += 2 * vinc, d += 2 * vstep * kVRow) {
        cp_async16(d, src);
        cp_async16(d + vstep * kVRow, src + vinc);
      }
      if (q < vn) cp_async16(d, src);
    }
    cp.issue(buf + vbytes, s0, ns);
  };
  float accr[MT][NG][4], acci[MT][NG][4];
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int t = 0; t < NG; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) accr[m][t][e] = acci[m][t][e] = 0.f;
  // rows past the CTA's right-hand sides repeat the last one and columns past nv hold anything: neither is stored
  int vro[MT][2], vok[3];
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int h = 0; h < 2; ++h) vro[m][h] = min(m * 16 + 8 * h + gid, Rc - 1) * VROW;
  // component pair kst of the chirality is half (3 chi + kst) & 1 of chunk (3 chi + kst) >> 1
#pragma unroll
  for (int kst = 0; kst < 3; ++kst)
    vok[kst] = (((3 * chi + kst) >> 1) - jb) * kVRow + tig * 16 + ((3 * chi + kst) & 1) * 8;
  const int pro = ((NCHI == 2 ? chi * NT * 8 : 0) + n0 * 8 + gid) * kTilePRow + tig * 4;
  issue(0);
  cp_async_commit();
  for (int i = 0; i < nst; ++i) {
    cp_async_wait(0);
    __syncthreads();  // stage i is complete for every warp, and every warp is done with stage i - 1
    if (i + 1 < nst) issue(i + 1);
    cp_async_commit();
    const unsigned char* sv = smem_raw + (i & 1) * stage_bytes;
    const unsigned char* sp = sv + vbytes;
    const int ngr = min(kTileE, bs - i * kTileE) / 4;
    for (int sg = slice; sg < ngr; sg += KS) {
#pragma unroll
      for (int kst = 0; kst < 3; ++kst) {  // components 2 kst, 2 kst + 1 of the chirality
        uint32_t a[MT][4];
#pragma unroll
        for (int m = 0; m < MT; ++m) {
          const uint2 lo = *(const uint2*)(sv + vro[m][0] + vok[kst] + sg * 64);
          const uint2 hi = *(const uint2*)(sv + vro[m][1] + vok[kst] + sg * 64);
          a[m][0] = lo.x;
          a[m][1] = hi.x;
          a[m][2] = lo.y;
          a[m][3] = hi.y;
        }
        const unsigned char* pk = sp + pro + sg * 16 + 2 * kst * kTileE * 4;
#pragma unroll
        for (int t = 0; t < NG; ++t) {
          if (NGT == 0 && n0 + t >= NT) break;
          const uint32_t b0 = ld32(pk + t * 8 * kTilePRow), b1 = ld32(pk + t * 8 * kTilePRow + kTileE * 4);
          const uint32_t c0 = swap16(b0) ^ 0x00008000u, c1 = swap16(b1) ^ 0x00008000u;  // (-Pi, Pr)
#pragma unroll
          for (int m = 0; m < MT; ++m) {
            MmaT<T>::mma(accr[m][t], a[m], b0, b1);
            MmaT<T>::mma(acci[m][t], a[m], c0, c1);
          }
        }
      }
    }
  }
  // add the slices: slices > 0 park their tiles, slice 0 sums in slice order
  __syncthreads();
  float* red = (float*)smem_raw;  // [warp][MT][NG][2][4][32]
  auto slot = [&](int w, int m, int t, int ri, int e) {
    return ((((size_t)(w * MT + m) * NG + t) * 2 + ri) * 4 + e) * 32 + lane;
  };
  if (slice > 0) {
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int t = 0; t < NG; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          red[slot(warp, m, t, 0, e)] = accr[m][t][e];
          red[slot(warp, m, t, 1, e)] = acci[m][t][e];
        }
  }
  __syncthreads();
  if (slice > 0) return;
  for (int sl = 1; sl < KS; ++sl) {
    const int w2 = warp + sl * ngroups * NCHI;
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int t = 0; t < NG; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          accr[m][t][e] += red[slot(w2, m, t, 0, e)];
          acci[m][t][e] += red[slot(w2, m, t, 1, e)];
        }
  }
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int t = 0; t < NG; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int k = (n0 + t) * 8 + 2 * tig + (e & 1), r = m * 16 + gid + (e >= 2 ? 8 : 0);
        if (k < nv && r < Rc)
          stc(out, ((size_t)(r0 + r) * 2 * nv + chi * nv + k) * g.Vc + B, mk<float>(accr[m][t][e], acci[m][t][e]));
      }
}

// CTA = (aggregate, part of its stages, 16 MT right-hand sides).  The coarse
// values of both chiralities sit in shared memory as the A operand (rows =
// right-hand sides, ldmatrix), P comes in stages of 16 sites.  A warp's unit is
// a chunk (components 4 j .. 4 j + 3) of four sites: n-tile t holds components
// 4 j + 2 t, 4 j + 2 t + 1 of the four sites, so a lane ends up with the whole
// chunk of one site for each of its right-hand sides.  NTC = 1..4 K tiles of 8
// vectors are nv <= 32, with constant offsets; NTC = 0 is nv > 32.  A warp's j
// never changes, so with one row tile its A fragments stay in registers; with
// two they would cost the second CTA per SM (72 -> 84 us) and are read back.
template <typename T, typename SI, int MT, int NTC>
__global__ void __launch_bounds__(kProlongThreads, 2)
    prolong_tile_kernel(const Agg g, const typename MmaT<T>::T2* P, const SI* in, typename MmaT<T>::T2* out, int R,
                        int nsplit, int stages, int bufs, int sidx_off) {
  chain_begin();
  typedef typename MmaT<T>::T2 T2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int B = blockIdx.x / nsplit, r0 = (blockIdx.x % nsplit) * MT * 16;
  const int Rc = min(R - r0, MT * 16);
  const int bs = g.bsites, nv = g.nv, NT = NTC ? NTC : (nv + 7) / 8;
  const int XROW = 64 * NT + 16;  // bytes of a row of coarse values, 16 mod 64: conflict-free ldmatrix
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
  unsigned char* xs = smem_raw;
  unsigned char* pst = smem_raw + MT * 16 * XROW;
  int* sidx = (int*)(smem_raw + sidx_off);
  StageP<2, T2> cp;
  cp.init(P + (size_t)B * 2 * nv * 6 * bs, nv, NT * 8, bs);
  const int nst_all = (bs + kTileE - 1) / kTileE;
  const int st0 = (int)((long)blockIdx.y * nst_all / gridDim.y), st1 = (int)((long)(blockIdx.y + 1) * nst_all / gridDim.y);
  const int stage_bytes = 2 * NT * 8 * kTilePRow;
  const unsigned pst0 = (unsigned)__cvta_generic_to_shared(pst);
  int wr = 0, rd = 0;  // ring positions of the next stage to load and to use
  auto issue = [&](int i) {
    const int s0 = i * kTileE;
    cp.issue(pst0 + wr * stage_bytes, s0, min(kTileE, bs - s0));
    wr = wr + 1 == stages ? 0 : wr + 1;
  };
  // rows past nv multiply zeros: they have to be finite, and no copy writes them
  for (int q = threadIdx.x; q < (NT * 8 - nv) * 2 * bufs * (kTilePRow / 4); q += kProlongThreads) {
    const int w = q % (kTilePRow / 4), row = q / (kTilePRow / 4), k = row % (NT * 8 - nv), cb = row / (NT * 8 - nv);
    *(uint32_t*)(pst + (cb >> 1) * stage_bytes + ((cb & 1) * NT * 8 + nv + k) * kTilePRow + w * 4) = 0u;
  }
  for (int i = st0; i < st0 + stages - 1; ++i) {
    if (i < st1) issue(i);
    cp_async_commit();
  }
  for (int s = threadIdx.x; s < bs; s += blockDim.x) sidx[s] = agg_site_t(g, B, s);
  for (int q = threadIdx.x; q < MT * 16 * 2 * NT * 8; q += blockDim.x) {
    const int k = q % (NT * 8), chi = (q / (NT * 8)) & 1, r = q / (NT * 16);
    T re = MmaT<T>::from(0.f), im = re;
    if (r < Rc && k < nv) planes<T>(in[((size_t)(r0 + r) * 2 * nv + chi * nv + k) * g.Vc + B], re, im);
    T* d = (T*)(xs + (size_t)r * XROW + (chi * NT * 8 + k) * 4);
    d[0] = re;
    d[1] = im;
  }
  // this lane's row address for ldmatrix: matrices (rows 0-7, 8-15) x (first, second four complex numbers)
  const unsigned xaddr =
      (unsigned)__cvta_generic_to_shared(xs) + ((lane & 7) + ((lane >> 3) & 1) * 8) * XROW + (lane >> 4) * 16;
  const int sg = warp / 3, j = warp - sg * 3;  // 12 warps: every (four sites, chunk) of a stage once
  int xo[2], po[2];                            // of n-tile t's chirality in xs, and of its components in a stage of P
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    const int gp = 2 * j + t, chi = gp >= 3 ? 1 : 0, c = 2 * (gp - 3 * chi) + (gid & 1);
    xo[t] = chi * NT * 32;
    po[t] = (c * kTileE + sg * 4 + (gid >> 1)) * 4 + (chi * NT * 8 + tig) * kTilePRow;
  }
  auto ld_a = [&](uint32_t (&a)[4], int t, int m, int kk) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"(xaddr + m * 16 * XROW + xo[t] + kk * 32)
                 : "memory");
  };
  constexpr bool keep = NTC > 0 && MT == 1;
  constexpr int KA = keep ? NTC : 1;
  uint32_t a[2][KA][MT][4];
  for (int i = st0; i < st1; ++i) {
    cp_async_wait(stages - 2);
    __syncthreads();  // stage i (and before the first, xs and sidx) complete; every warp is done with stage i - 1
    if (i + stages - 1 < st1) issue(i + stages - 1);
    cp_async_commit();
    if (keep && i == st0) {
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int kk = 0; kk < KA; ++kk)
#pragma unroll
          for (int m = 0; m < MT; ++m) ld_a(a[t][kk][m], t, m, kk);
    }
    const unsigned char* sp = pst + rd * stage_bytes;
    rd = rd + 1 == stages ? 0 : rd + 1;
    const int s0 = i * kTileE;
    if (sg * 4 < bs - s0) {
      float acc[2][2][MT][4];  // [n-tile][re, im]
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int ri = 0; ri < 2; ++ri)
#pragma unroll
          for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[t][ri][m][e] = 0.f;
      auto step = [&](int kk, int ka) {
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const unsigned char* pc = sp + po[t] + kk * 8 * kTilePRow;
          const uint32_t b0 = ld32(pc), b1 = ld32(pc + 4 * kTilePRow);
          const uint32_t r0_ = b0 ^ 0x80000000u, r1_ = b1 ^ 0x80000000u;  // (Pr, -Pi)
          const uint32_t i0_ = swap16(b0), i1_ = swap16(b1);              // (Pi, Pr)
#pragma unroll
          for (int m = 0; m < MT; ++m) {
            if (!keep) ld_a(a[t][0][m], t, m, kk);
            MmaT<T>::mma(acc[t][0][m], a[t][ka][m], r0_, r1_);
            MmaT<T>::mma(acc[t][1][m], a[t][ka][m], i0_, i1_);
          }
        }
      };
      if constexpr (NTC > 0) {
#pragma unroll
        for (int kk = 0; kk < NTC; ++kk) step(kk, keep ? kk : 0);
      } else {
        for (int kk = 0; kk < NT; ++kk) step(kk, 0);
      }
      const size_t so = ((size_t)j * g.V + sidx[s0 + sg * 4 + tig]) << 2;
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = m * 16 + 8 * h + gid;
          if (r >= Rc) continue;
          cx<float> v[4];
#pragma unroll
          for (int q = 0; q < 4; ++q)
            v[q] = mk<float>(acc[q >> 1][0][m][2 * h + (q & 1)], acc[q >> 1][1][m][2 * h + (q & 1)]);
          st_chunk<T2, float>(out, (size_t)(r0 + r) * 12 * g.V + so, v);
        }
    }
  }
}

// ------------------------------------------------------------------ launchers
// Dynamic shared memory: the staged operands (or, in the restriction, the
// K-slice partial sums that reuse them), then the aggregate's site table at
// the returned offset.
static size_t restrict_smem(const Agg& g, int NT8, size_t* sidx_off) {
  const int MT = (g.nv + 15) / 16;
  const size_t stage = (size_t)2 * (MT * 16 + NT8 * 8) * kTKs * 2;
  const size_t red = (size_t)8 * NT8 * 2 * 4 * 32 * 4;
  *sidx_off = ((stage > red ? stage : red) + 15) / 16 * 16;
  return *sidx_off + (size_t)g.bsites * 4;
}

static size_t prolong_smem(const Agg& g, int NT8, size_t* sidx_off) {
  const int Kps = (g.nv + 15) / 16 * 16 + 8;
  *sidx_off = ((size_t)2 * (NT8 * 8 + kTK) * Kps * 2 + 15) / 16 * 16;
  return *sidx_off + (size_t)g.bsites * 4;
}

bool transfer_mma_ok(const Agg& g, int nrhs) {
  const int MT = (g.nv + 15) / 16;
  return nrhs >= 2 && nrhs <= 64 && (MT == 1 || MT == 2 || MT == 4) && g.ncomp % 2 == 0 && g.bsites <= 8192;
}

// Launch shapes: variant v puts kXTiles[v] tiles of 8 right-hand sides in a CTA
// (the admissible ones for nrhs, in this order); the default holds them all.
static const int kXTiles[] = {8, 4, 2, 1, 3, 6};
constexpr int kXVariants = 6;

static int tiles_of(int nrhs, int variant) {
  const int all = (nrhs + 7) / 8;
  if (variant < 0) return all;
  int seen = -1;
  for (int v = 0; v < kXVariants; ++v)
    if (kXTiles[v] <= all && ++seen == variant) return kXTiles[v];
  return all;
}

// Shared memory a tile kernel may use: the opt-in limit less the reserved KB.
static size_t tile_smem_max() { return (size_t)smem_optin_bytes() - 1024; }

// Geometry the tile kernels take: level-0 fields, whole groups of four sites.
// Everything else (16-bit coarse fields, coarse levels in 16-bit storage, odd
// aggregates) stays on the plane kernels.
static bool tile_geom(const Agg& g) {
  return g.q == 4 && g.ncomp == 12 && g.bsites % 4 == 0;
}
// ... and 16-byte accesses to the fine field.
static bool tile_ok(const Agg& g, const void* P, const void* fine) {
  return tile_geom(g) && ((uintptr_t)P & 15u) == 0 && ((uintptr_t)fine & 15u) == 0;
}

// Launch shapes of the tile kernels, bit-identical results: restriction
// {chiralities per CTA}, prolongation {parts of the aggregate, stages}, and
// both again with one m-tile of 16 right-hand sides per CTA instead of two.
struct PTile {
  int parts, stages;
};
// Measured at 16^3 x 32, nv = 24, FP16 (512 aggregates): both chiralities in a
// CTA 66.8 us against 68.7, whole aggregates 67.5 against 71.9 in halves, two
// m-tiles 67 against 81-86 (24 right-hand sides); at 8^3 x 16 (32 aggregates,
// 12 right-hand sides) 13.2 us against 16.4, quarters 9.1 against 17.3.
static const int kRTiles[] = {2, 1};
static const PTile kPTiles[] = {{1, 3}, {2, 2}, {4, 2}, {16, 2}};
constexpr int kRShapes = 2, kPShapes = 4;

int transfer_mma_variants(const Agg& g, int nrhs, bool prolong, int coarse_prec) {
  if (tile_geom(g) && cx_bytes(coarse_prec) == 8) return (prolong ? kPShapes : kRShapes) * (nrhs > 16 ? 2 : 1);
  const int NT8 = (nrhs + 7) / 8;
  int nv = 0;
  for (int v = 0; v < kXVariants; ++v) nv += kXTiles[v] <= NT8 ? 1 : 0;
  return nv;
}

template <typename T, typename SO>
static int restrict_tile_t(const Agg& g, const void* P, const void* in, void* out, int nrhs, cudaStream_t st,
                           int variant) {
  typedef typename MmaT<T>::T2 T2;
  const int mt = nrhs > 16 && variant < kRShapes ? 2 : 1, nsplit = (nrhs + 16 * mt - 1) / (16 * mt);
  // untuned: both chiralities in a CTA read the field's lines once; two CTAs where that leaves SMs idle
  const int nchi = variant >= 0 ? kRTiles[variant % kRShapes] : (g.Vc * nsplit >= sm_count() ? 2 : 1);
  const int vrows = nrhs < 16 * mt ? nrhs : 16 * mt;
  const int nst = (g.bsites + kTileE - 1) / kTileE;
  const size_t stage = (size_t)vrows * (nchi + 1) * tile_vrow(nchi + 1) + (size_t)nchi * ((g.nv + 7) / 8 * 8) * kTilePRow;
  const int have = nst < 2 ? nst : 2;  // buffers that a short aggregate really uses
  const size_t red = (size_t)4 * nchi * mt * 4 * 2 * 4 * 32 * 4;
  const size_t so = ((have * stage > red ? have * stage : red) + 15) / 16 * 16;
  const size_t sm = so + (size_t)g.bsites * 4;
  if (sm > tile_smem_max()) return 1;
  const dim3 grid((unsigned)(g.Vc * nsplit), nchi == 2 ? 1 : 2);
  const int ng = g.nv <= 32 ? (g.nv + 7) / 8 : 0;
#define WMG_RT(M, C, N)                                                                                     \
  case (M) * 100 + (C) * 10 + (N): {                                                                        \
    auto kern = restrict_tile_kernel<T, SO, M, C, N>;                                                       \
    if (sm > 48 * 1024) allow_big_smem(kern);                                                               \
    launch_chain(kern, grid, 128 * C, sm, st, g, (const T2*)P, (const T2*)in, (SO*)out, nrhs, nsplit, vrows, (int)so); \
    break;                                                                                                  \
  }
#define WMG_RTN(M, C) WMG_RT(M, C, 0) WMG_RT(M, C, 1) WMG_RT(M, C, 2) WMG_RT(M, C, 3) WMG_RT(M, C, 4)
  switch (mt * 100 + nchi * 10 + ng) {
    WMG_RTN(1, 1)
    WMG_RTN(1, 2)
    WMG_RTN(2, 1)
    WMG_RTN(2, 2)
  }
#undef WMG_RTN
#undef WMG_RT
  return launched() ? 0 : -1;
}

template <typename T, typename SI>
static int prolong_tile_t(const Agg& g, const void* P, const void* in, void* out, int nrhs, cudaStream_t st,
                          int variant) {
  typedef typename MmaT<T>::T2 T2;
  const int mt = nrhs > 16 && variant < kPShapes ? 2 : 1, nsplit = (nrhs + 16 * mt - 1) / (16 * mt);
  PTile sh = kPTiles[variant < 0 ? 0 : variant % kPShapes];
  if (variant < 0)  // untuned: parts only as far as whole aggregates leave SMs idle (each part reads the coarse values)
    while (sh.parts < 16 && g.Vc * nsplit * sh.parts < sm_count()) sh = PTile{sh.parts * 2, 2};
  const int nst = (g.bsites + kTileE - 1) / kTileE;
  const int parts = sh.parts < nst ? sh.parts : nst;
  const int per = (nst + parts - 1) / parts, have = per < sh.stages ? per : sh.stages;
  const size_t xb = (size_t)mt * 16 * (64 * ((g.nv + 7) / 8) + 16);
  const size_t so = (xb + (size_t)have * 2 * ((g.nv + 7) / 8 * 8) * kTilePRow + 15) / 16 * 16;
  const size_t sm = so + (size_t)g.bsites * 4;
  if (sm > tile_smem_max()) return 1;
  const dim3 grid((unsigned)(g.Vc * nsplit), (unsigned)parts);
  const int nt = g.nv <= 32 ? (g.nv + 7) / 8 : 0;
#define WMG_PT(M, N)                                                                                              \
  case (M) * 10 + (N): {                                                                                          \
    auto kern = prolong_tile_kernel<T, SI, M, N>;                                                                 \
    if (sm > 48 * 1024) allow_big_smem(kern);                                                                     \
    launch_chain(kern, grid, kProlongThreads, sm, st, g, (const T2*)P, (const SI*)in, (T2*)out, nrhs, nsplit, sh.stages, have, \
                                            (int)so);                                                             \
    break;                                                                                                        \
  }
#define WMG_PTN(M) WMG_PT(M, 0) WMG_PT(M, 1) WMG_PT(M, 2) WMG_PT(M, 3) WMG_PT(M, 4)
  switch (mt * 10 + nt) {
    WMG_PTN(1)
    WMG_PTN(2)
  }
#undef WMG_PTN
#undef WMG_PT
  return launched() ? 0 : -1;
}

template <typename T, typename SI, typename SO>
static int restrict_mma_t(const Agg& g, const void* P, const void* in, void* out, int nrhs, cudaStream_t st,
                          int variant) {
  if constexpr (sizeof(SO) == 8) {
    if (tile_ok(g, P, in)) {
      const int rc = restrict_tile_t<T, SO>(g, P, in, out, nrhs, st, variant);
      if (rc <= 0) return rc;
    }
  }
  const int NT8 = tiles_of(nrhs, variant);
  size_t so = 0;
  const size_t sm = restrict_smem(g, NT8, &so);
  const dim3 grid(g.Vc, 2, ((nrhs + 7) / 8 + NT8 - 1) / NT8);
#define WMG_RM(K)                                                                                              \
  {                                                                                                            \
    auto kern = restrict_mma_kernel<T, SI, SO, K>;                                                             \
    if (sm > 48 * 1024) allow_big_smem(kern);                                                                  \
    launch_chain(kern, grid, kTThreads, sm, st, g, (const typename MmaT<T>::T2*)P, (const SI*)in, (SO*)out, nrhs, (int)so); \
  }
  switch (NT8) {
    case 1: WMG_RM(1); break;
    case 2: WMG_RM(2); break;
    case 3: WMG_RM(3); break;
    case 4: WMG_RM(4); break;
    case 5: WMG_RM(5); break;
    case 6: WMG_RM(6); break;
    case 7: WMG_RM(7); break;
    case 8: WMG_RM(8); break;
    default: return -1;
  }
#undef WMG_RM
  return launched() ? 0 : -1;
}

template <typename T, typename SI, typename SO>
static int prolong_mma_t(const Agg& g, const void* P, const void* in, void* out, int nrhs, cudaStream_t st,
                         int variant) {
  if constexpr (sizeof(SI) == 8) {
    if (tile_ok(g, P, out)) {
      const int rc = prolong_tile_t<T, SI>(g, P, in, out, nrhs, st, variant);
      if (rc <= 0) return rc;
    }
  }
  const int NT8 = tiles_of(nrhs, variant);
  size_t so = 0;
  const size_t sm = prolong_smem(g, NT8, &so);
  const dim3 grid(g.Vc, 2, ((nrhs + 7) / 8 + NT8 - 1) / NT8);
#define WMG_PM(K)                                                                                              \
  {                                                                                                            \
    auto kern = prolong_mma_kernel<T, SI, SO, K>;                                                              \
    if (sm > 48 * 1024) allow_big_smem(kern);                                                                  \
    launch_chain(kern, grid, kTThreads, sm, st, g, (const typename MmaT<T>::T2*)P, (const SI*)in, (SO*)out, nrhs, (int)so); \
  }
  switch (NT8) {
    case 1: WMG_PM(1); break;
    case 2: WMG_PM(2); break;
    case 3: WMG_PM(3); break;
    case 4: WMG_PM(4); break;
    case 5: WMG_PM(5); break;
    case 6: WMG_PM(6); break;
    case 7: WMG_PM(7); break;
    case 8: WMG_PM(8); break;
    default: return -1;
  }
#undef WMG_PM
  return launched() ? 0 : -1;
}

// (vector-in, P, vector-out) precision triples with 16-bit P: 2 = FP16, 3 = BF16, 1 = FP32.
int launch_restrict_mma(int pin, int pP, int pout, const Agg& g, const void* P, const void* in, void* out, int nrhs,
                        cudaStream_t st, int variant) {
  if (pin == 2 && pP == 2 && pout == 1)
    return restrict_mma_t<__half, __half2, float2>(g, P, in, out, nrhs, st, variant);
  if (pin == 3 && pP == 3 && pout == 1)
    return restrict_mma_t<__nv_bfloat16, __nv_bfloat162, float2>(g, P, in, out, nrhs, st, variant);
  if (pin == 2 && pP == 2 && pout == 2)
    return restrict_mma_t<__half, __half2, __half2>(g, P, in, out, nrhs, st, variant);
  if (pin == 3 && pP == 3 && pout == 3)
    return restrict_mma_t<__nv_bfloat16, __nv_bfloat162, __nv_bfloat162>(g, P, in, out, nrhs, st, variant);
  return -1;
}

int launch_prolong_mma(int pin, int pP, int pout, const Agg& g, const void* P, const void* in, void* out, int nrhs,
                       cudaStream_t st, int variant) {
  if (pin == 1 && pP == 2 && pout == 2)
    return prolong_mma_t<__half, float2, __half2>(g, P, in, out, nrhs, st, variant);
  if (pin == 1 && pP == 3 && pout == 3)
    return prolong_mma_t<__nv_bfloat16, float2, __nv_bfloat162>(g, P, in, out, nrhs, st, variant);
  if (pin == 2 && pP == 2 && pout == 2)
    return prolong_mma_t<__half, __half2, __half2>(g, P, in, out, nrhs, st, variant);
  if (pin == 3 && pP == 3 && pout == 3)
    return prolong_mma_t<__nv_bfloat16, __nv_bfloat162, __nv_bfloat162>(g, P, in, out, nrhs, st, variant);
  return -1;
}

}  // namespace wmg
