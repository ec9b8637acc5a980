// Coarse 9-point stencil on tensor cores for many right-hand sides.
//
// (A_c y)(B) = sum_d C_d(B) y(B + d)  (A_c = P^+ A P, Sec. 2) is, per coarse
// site B, one dense contraction O (n x R) = [C_0 .. C_8](B) (n x 9n) * Y (9n x R)
// over the R right-hand sides.  In the real embedding
//   [O_re; O_im] = [[C_re, -C_im], [C_im, C_re]] [Y_re; Y_im]
// it runs as BF16 mma.sync m16n8k16 with FP32 accumulation.  One warp owns
// a pair of 16-row tiles (the real rows and the imaginary rows of the same
// 16 components), so each 16x16 block of C_re and C_im is loaded once and
// used by four MMAs (C_re Y_re, -C_im Y_im into the real tile; C_im Y_re,
// C_re Y_im into the imaginary tile; -C_im is C_im with the sign bits
// flipped).  The operator is stored at setup in MMA fragment order,
// [B][d][tile][kstep][re|im][lane][8 x bf16], so a warp reads 512 contiguous
// bytes per fragment; the right-hand sides are first rounded to BF16 rows
// [site][r][re..., im...] and those of the 9 neighbours staged in shared
// memory.  n is padded to a multiple of
// 16 and R to a multiple of 8 with zeros.
#include <cuda_bf16.h>

#include "common.cuh"
#include "kernels.h"

namespace wmg {

static inline bool launched() { return launch_ok(); }

// ------------------------------------------------------------------ operator in fragment order
// One thread per (B, d, tile, kstep, part, lane): 8 bf16 of the A fragment
// of m16n8k16 (rows gid, gid + 8; columns 2 tig, 2 tig + 1, and + 8).
__global__ void mma_pack_kernel(const double2* C, int n, int npad, int V, uint4* out) {
  const int T = npad / 16;  // row tiles = k steps per half
  const size_t per_site = (size_t)9 * T * T * 2 * 32;
  const size_t tot = per_site * V;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (size_t)gridDim.x * blockDim.x) {
    size_t q = e;
    const int lane = (int)(q % 32);
    q /= 32;
    const int part = (int)(q % 2);
    q /= 2;
    const int s = (int)(q % T);
    q /= T;
    const int t = (int)(q % T);
    q /= T;
    const int d = (int)(q % 9);
    const int B = (int)(q / 9);
    const int gid = lane >> 2, tig = lane & 3;
    const int rows[2] = {t * 16 + gid, t * 16 + gid + 8};
    const int cols[4] = {s * 16 + 2 * tig, s * 16 + 2 * tig + 1, s * 16 + 2 * tig + 8, s * 16 + 2 * tig + 9};
    // a0 a1: (r0, c0 c1); a2 a3: (r1, c0 c1); a4 a5: (r0, c2 c3); a6 a7: (r1, c2 c3)
    const int ri[8] = {0, 0, 1, 1, 0, 0, 1, 1};
    const int ci[8] = {0, 1, 0, 1, 2, 3, 2, 3};
    __nv_bfloat16 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int i = rows[ri[k]], j = cols[ci[k]];
      double x = 0.0;
      if (i < n && j < n) {
        const double2 c = C[((size_t)(d * n + i) * n + j) * V + B];
        x = part ? c.y : c.x;
      }
      v[k] = __float2bfloat16_rn((float)x);
    }
    uint4 w;
    w.x = (uint32_t)__bfloat16_as_ushort(v[0]) | ((uint32_t)__bfloat16_as_ushort(v[1]) << 16);
    w.y = (uint32_t)__bfloat16_as_ushort(v[2]) | ((uint32_t)__bfloat16_as_ushort(v[3]) << 16);
    w.z = (uint32_t)__bfloat16_as_ushort(v[4]) | ((uint32_t)__bfloat16_as_ushort(v[5]) << 16);
    w.w = (uint32_t)__bfloat16_as_ushort(v[6]) | ((uint32_t)__bfloat16_as_ushort(v[7]) << 16);
    out[e] = w;
  }
}

size_t mma_pack_bytes(int n, int V) {
  const int npad = (n + 15) / 16 * 16, T = npad / 16;
  return (size_t)9 * T * T * 2 * 32 * 16 * V;
}

int launch_mma_pack(const double2* C, int n, int V, void* out, cudaStream_t st) {
  const int npad = (n + 15) / 16 * 16, T = npad / 16;
  const size_t tot = (size_t)9 * T * T * 2 * 32 * V;
  size_t b = (tot + 255) / 256;
  if (b > 8192) b = 8192;
  mma_pack_kernel<<<(unsigned)b, 256, 0, st>>>(C, n, npad, V, (uint4*)out);
  return launched() ? 0 : -1;
}

// ------------------------------------------------------------------ apply
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Bytes from one (site, right-hand side) row of BF16 planes (re then im, npad
// each) to the next: an odd number of 16-byte units, so that eight rows of an
// ldmatrix fall on distinct banks, in global memory as in shared.
__host__ __device__ constexpr int row_pitch(int npad) { return 4 * npad + 16; }

// Component-major vectors [R][n][V] -> rows [V][R][re npad | im npad] of BF16.
// A site's vector is strided by V in memory; gathering it in every CTA that
// needs it (nine of them) moved each 32-byte sector for 8 bytes, nine times:
// here each value is read once, coalesced, and the stencil reads whole rows.
// CTA = 32 sites of one right-hand side, transposed through shared memory.
template <typename S>
__global__ void __launch_bounds__(256) coarse_rows_kernel(const S* in, unsigned char* rows, int n, int npad, int V, int R) {
  chain_begin();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int r = blockIdx.y, B0 = blockIdx.x * 32, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int pitch = 4 * npad + 4;  // one bank further per site
  const S* v = in + (size_t)r * n * V;
  for (int j = warp; j < npad; j += 8) {
    cx<float> x = zero<float>();
    if (j < n && B0 + lane < V) x = ldc<float>(v, (size_t)j * V + B0 + lane);
    __nv_bfloat16* d = (__nv_bfloat16*)(smem_raw + lane * pitch);
    d[j] = __float2bfloat16_rn(x.re);
    d[npad + j] = __float2bfloat16_rn(x.im);
  }
  __syncthreads();
  const int words = npad;  // 4-byte words of a row
  const int ns = min(32, V - B0);
  for (int b = warp; b < ns; b += 8) {
    uint32_t* o = (uint32_t*)(rows + ((size_t)(B0 + b) * R + r) * row_pitch(npad));
    for (int w = lane; w < words; w += 32) o[w] = *(const uint32_t*)(smem_raw + b * pitch + 4 * w);
  }
}

// Direct form, for a few right-hand sides (it gathers the nine neighbours'
// vectors itself: no rows, no second launch) and for stencils whose directions
// do not fit the ring of the streaming form below.  CTA = one coarse site and
// NT8 tiles of 8 right-hand sides; warp = row tile t; kAhead operator
// fragments in flight per warp (two, three, five and nine measured: three).
constexpr int kAhead = 3;
// Threads a CTA may have at NT8 (32 T of the launches that fit shared memory): bounds the registers.
constexpr int mma_threads(int NT8) { return NT8 == 1 ? 1024 : (NT8 == 2 ? 704 : 448); }

// One kstep of a warp's row tile: 16 x 16 of the operator (re, im fragments)
// times the staged rows at `ya` (this lane's ldmatrix row; matrices re 0-7,
// re 8-15, im 0-7, im 8-15).
template <int NT8>
__device__ __forceinline__ void mma_kstep(float (&accr)[NT8][4], float (&acci)[NT8][4], const uint4& fr, const uint4& fi,
                                          unsigned ya, int pitch) {
  const uint32_t Ar[4] = {fr.x, fr.y, fr.z, fr.w};
  const uint32_t Ai[4] = {fi.x, fi.y, fi.z, fi.w};
  const uint32_t An[4] = {fi.x ^ 0x80008000u, fi.y ^ 0x80008000u, fi.z ^ 0x80008000u, fi.w ^ 0x80008000u};
  // groups of four tiles, each product of the group before the next product: an
  // accumulator's second MMA would otherwise wait out its first one's latency
  constexpr int QG = NT8 < 4 ? NT8 : 4;
#pragma unroll
  for (int q0 = 0; q0 < NT8; q0 += QG) {
    uint32_t y[QG][4];  // re 0-7, re 8-15, im 0-7, im 8-15
#pragma unroll
    for (int u = 0; u < QG; ++u)
      if (q0 + u < NT8)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                     : "=r"(y[u][0]), "=r"(y[u][1]), "=r"(y[u][2]), "=r"(y[u][3])
                     : "r"(ya + (q0 + u) * 8 * pitch)
                     : "memory");
#pragma unroll
    for (int u = 0; u < QG; ++u)
      if (q0 + u < NT8) mma_bf16(accr[q0 + u], Ar, y[u][0], y[u][1]);  // C_re Y_re
#pragma unroll
    for (int u = 0; u < QG; ++u)
      if (q0 + u < NT8) mma_bf16(acci[q0 + u], Ai, y[u][0], y[u][1]);  // C_im Y_re
#pragma unroll
    for (int u = 0; u < QG; ++u)
      if (q0 + u < NT8) mma_bf16(accr[q0 + u], An, y[u][2], y[u][3]);  // -C_im Y_im
#pragma unroll
    for (int u = 0; u < QG; ++u)
      if (q0 + u < NT8) mma_bf16(acci[q0 + u], Ar, y[u][2], y[u][3]);  // C_re Y_im
  }
}

template <int NT8>
__device__ __forceinline__ void mma_zero(float (&accr)[NT8][4], float (&acci)[NT8][4]) {
#pragma unroll
  for (int q = 0; q < NT8; ++q)
#pragma unroll
    for (int k = 0; k < 4; ++k) accr[q][k] = acci[q][k] = 0.f;
}

// Rows t*16 + gid (+8), right-hand sides r0 + q*8 + 2 tig (+1) of site B.
template <typename S, int NT8>
__device__ __forceinline__ void mma_store(const float (&accr)[NT8][4], const float (&acci)[NT8][4], const S* in, S* out,
                                          const S* y2, const double* shift, int B, int V, int t, int r0, int n, int R,
                                          float a, float c) {
  const int lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
#pragma unroll
  for (int q = 0; q < NT8; ++q)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = t * 16 + gid + (k >= 2 ? 8 : 0);
      const int r = r0 + q * 8 + 2 * tig + (k & 1);
      if (i < n && r < R) {
        const size_t o = ((size_t)r * n + i) * V + B;
        cx<float> acc = mk<float>(accr[q][k], acci[q][k]);
        if (shift) acc = cfma(mk<float>((float)shift[r], 0.f), ldc<float>(in, o), acc);
        cx<float> v = mk<float>(a * acc.re, a * acc.im);
        if (y2) v = v + c * ldc<float>(y2, o);
        stc(out, o, v);
      }
    }
}

template <typename S, int NT8>
__global__ void __launch_bounds__(mma_threads(NT8))
    coarse_mma_kernel(const uint4* Cf, const S* in, S* out, const S* y2, int L0, int L1, int L2, int L3, int n, int npad,
                      int R, float a, float c, const double* shift) {
  chain_begin();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int nbs[9];
  const int V = L0 * L1 * L2 * L3;
  const int B = blockIdx.x;
  const int r0 = blockIdx.y * NT8 * 8, Rc = min(R - r0, NT8 * 8);  // this CTA's right-hand sides
  const int T = npad / 16;
  const int pitch = row_pitch(npad);
  const int t = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int KS = 9 * T, dskip = (T - 1) * T * 64;  // from a direction's last kstep to the next direction's first
  uint4 fr[kAhead], fi[kAhead];
  int ld_s = 0, ld_k = 0;  // position of the next fragment to load
  const uint4* cp = Cf + (((size_t)B * 9 * T + t) * T * 2) * 32 + lane;
  auto load = [&](int u) {
    if (ld_k < KS) {
      fr[u] = __ldg(cp);
      fi[u] = __ldg(cp + 32);
      cp += 64;
      ++ld_k;
      if (++ld_s == T) {
        ld_s = 0;
        cp += dskip;
      }
    }
  };
#pragma unroll
  for (int u = 0; u < kAhead; ++u) load(u);
  if (threadIdx.x < 9) {
    const int L[4] = {L0, L1, L2, L3};
    int cB[4];
    site_coords(B, L, cB);
    nbs[threadIdx.x] = neighbor(cB, L, threadIdx.x);
  }
  __syncthreads();
  for (int row = t; row < 9 * Rc; row += T) {
    const int d = row / Rc, r = row - d * Rc;
    __nv_bfloat16* o = (__nv_bfloat16*)(smem_raw + (d * NT8 * 8 + r) * pitch);
    for (int j = lane; j < npad; j += 32) {
      cx<float> v = zero<float>();
      if (j < n) v = ldc<float>(in, ((size_t)(r0 + r) * n + j) * V + nbs[d]);
      o[j] = __float2bfloat16_rn(v.re);
      o[npad + j] = __float2bfloat16_rn(v.im);
    }
  }
  __syncthreads();
  float accr[NT8][4], acci[NT8][4];
  mma_zero<NT8>(accr, acci);
  unsigned ya = (unsigned)__cvta_generic_to_shared(smem_raw) + (lane & 7) * pitch + ((lane >> 3) & 1) * 16 +
                (lane >> 4) * 2 * npad;
  int s = 0;
  for (int k = 0; k < KS; k += kAhead) {
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      if (k + u >= KS) break;
      const uint4 Ar = fr[u], Ai = fi[u];
      load(u);
      mma_kstep<NT8>(accr, acci, Ar, Ai, ya, pitch);
      ya += 32;
      if (++s == T) {
        s = 0;
        ya += NT8 * 8 * pitch - 32 * T;
      }
    }
  }
  mma_store<S, NT8>(accr, acci, in, out, y2, shift, B, V, t, r0, n, R, a, c);
}

// ------------------------------------------------------------------ streaming form
// A persistent CTA takes (site, group of right-hand sides) items.  Its last
// warp's first thread streams each item's nine directions -- 9 KB of operator
// and 5 KB of a neighbour's rows at n = 48 and 24 right-hand sides -- as two
// bulk copies into a ring of `ns` stages, on into the next items while the T
// consumer warps (one row tile each) multiply; full and empty are mbarriers
// per stage.  Bound by the latency of a site's chain of ksteps and its strided
// 8-byte stores (a component's sites are contiguous, its CTA has one of them),
// not yet by the 42 MB of operator that 512 sites read.  Directions and ksteps
// in the direct form's order: the same bits.
//
// 16^3 x 32, level 1 (512 sites, n = 48), rows included: 24 right-hand sides
// 55 -> 19 us, 12 34 -> 14 us.
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_copy(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// Wait for the phase of the given parity, at most `spins` tries; false when they ran out.
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, int spins) {
  for (int i = 0; i < spins; ++i) {
    unsigned ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

constexpr int kMaxStages = 8;

template <typename S, int NT8>
__global__ void __launch_bounds__(224)
    coarse_stream_kernel(const unsigned char* Cf, const S* in, const unsigned char* rows, S* out, const S* y2, int L0,
                         int L1, int L2, int L3, int n, int npad, int R, float a, float c, const double* shift,
                         int splits, int items, int ns, int spins) {
  chain_begin();
  extern __shared__ __align__(128) unsigned char smem_ring[];
  __shared__ __align__(8) unsigned long long bars[2 * kMaxStages];  // full, empty
  const int V = L0 * L1 * L2 * L3;
  const int T = npad / 16, pitch = row_pitch(npad);
  const unsigned abytes = T * T * 1024, stage = abytes + NT8 * 8 * pitch;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned ring = (unsigned)__cvta_generic_to_shared(smem_ring);
  const unsigned full = (unsigned)__cvta_generic_to_shared(bars), empty = full + 8 * kMaxStages;
  if (threadIdx.x == 0) {
    for (int i = 0; i < ns; ++i) {
      mbar_init(full + 8 * i, 1);
      mbar_init(empty + 8 * i, T);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  int slot = 0;
  unsigned ph = 0;
  if (warp == T) {  // producer
    if (lane != 0) return;
    const int L[4] = {L0, L1, L2, L3};
    int issued = 0;
    bool ok = true;
    for (int w = blockIdx.x; w < items && ok; w += gridDim.x) {
      const int B = w / splits, r0 = (w - B * splits) * NT8 * 8, Rc = min(R - r0, NT8 * 8);
      int cB[4];
      site_coords(B, L, cB);
      const unsigned rbytes = Rc * pitch;
#pragma unroll
      for (int d = 0; d < 9; ++d) {
        ok = ok && mbar_wait(empty + 8 * slot, ph ^ 1u, spins);
        if (!ok) break;
        const unsigned bar = full + 8 * slot, dst = ring + slot * stage;
        mbar_expect(bar, abytes + rbytes);
        bulk_copy(dst, Cf + ((size_t)B * 9 + d) * abytes, abytes, bar);
        bulk_copy(dst + abytes, rows + ((size_t)neighbor(cB, L, d) * R + r0) * pitch, rbytes, bar);
        ++issued;
        if (++slot == ns) {
          slot = 0;
          ph ^= 1u;
        }
      }
    }
    // a ring that stopped: its copies land before the CTA's shared memory goes (the consumers report it)
    if (!ok)
      for (int i = 0; i < (issued < ns ? issued : ns); ++i) {
        slot = slot == 0 ? ns - 1 : slot - 1;
        if (slot == ns - 1) ph ^= 1u;
        mbar_wait(full + 8 * slot, ph, spins);
      }
    return;
  }
  const unsigned ya0 = ring + abytes + (lane & 7) * pitch + ((lane >> 3) & 1) * 16 + (lane >> 4) * 2 * npad;
  const unsigned char* af0 = smem_ring + (size_t)warp * T * 1024 + lane * 16;
  bool ok = true;
  for (int w = blockIdx.x; w < items; w += gridDim.x) {
    const int B = w / splits, r0 = (w - B * splits) * NT8 * 8;
    float accr[NT8][4], acci[NT8][4];
    mma_zero<NT8>(accr, acci);
    for (int d = 0; d < 9 && ok; ++d) {
      // a warp whose wait runs out reads and arrives no more: the others' stages stay theirs until their waits run out too
      ok = __all_sync(0xffffffffu, mbar_wait(full + 8 * slot, ph, spins));
      if (!ok) break;
      unsigned ya = ya0 + slot * stage;
      const unsigned char* af = af0 + (size_t)slot * stage;
#pragma unroll 3
      for (int s = 0; s < T; ++s) {
        const uint4 fr = *(const uint4*)af, fi = *(const uint4*)(af + 512);
        mma_kstep<NT8>(accr, acci, fr, fi, ya, pitch);
        af += 1024;
        ya += 32;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty + 8 * slot);
      if (++slot == ns) {
        slot = 0;
        ph ^= 1u;
      }
    }
    if (!ok) {  // every output of this item and the next ones: the solver refuses NaN
#pragma unroll
      for (int q = 0; q < NT8; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) accr[q][k] = acci[q][k] = __int_as_float(0x7fc00000);
    }
    mma_store<S, NT8>(accr, acci, in, out, y2, shift, B, V, warp, r0, n, R, a, c);
  }
}

// The streaming form takes stencils of up to kStreamT row tiles: three stages
// of any group of right-hand sides then fit one CTA's shared memory.
constexpr int kStreamT = 6;
// Stages of the ring: what 48 KB hold, at least three.  More CTAs per SM gain
// more than deeper rings (512 sites, n = 48, 24 right-hand sides: four CTAs of
// three stages 13.1 us, two of seven 15.4).
static int stream_stages(int T, int NT8, size_t* stage) {
  *stage = (size_t)T * T * 1024 + (size_t)NT8 * 8 * row_pitch(16 * T);
  const int ns = (int)(48 * 1024 / *stage);
  return ns < 3 ? 3 : (ns > kMaxStages ? kMaxStages : ns);
}

// Scratch of launch_coarse_mma for R right-hand sides (0: the direct form runs).
// Below four the gathers cost less than the extra launch.
constexpr int kRowsFrom = 4;
size_t coarse_mma_scratch_bytes(int n, int V, int R) {
  const int T = (n + 15) / 16;
  return R < kRowsFrom || T > kStreamT ? 0 : (size_t)V * R * row_pitch(16 * T);
}

// Launch shapes: variant v splits the right-hand sides over CTAs in groups of
// kMmaTiles[v] tiles of 8 (each output's arithmetic is the same in every shape).
static const int kMmaTiles[] = {8, 4, 2, 1, 3, 6};
constexpr int kMmaVariants = 6;

int coarse_mma_variants(int R) {
  const int NT8 = (R + 7) / 8;
  int nv = 0;
  for (int v = 0; v < kMmaVariants; ++v) nv += kMmaTiles[v] <= NT8 ? 1 : 0;
  return nv;
}

int launch_coarse_mma(int prec, const void* Cf, const void* in, void* out, const void* y2, const int L[4], int n, int R,
                      double a, double c, cudaStream_t st, int variant, const double* shift, void* scratch, int spins) {
  if (prec != 1 && prec != 3) return -1;
  const int npad = (n + 15) / 16 * 16, T = npad / 16;
  const int V = L[0] * L[1] * L[2] * L[3];
  const int NT8all = (R + 7) / 8;
  int NT8 = NT8all;  // default: one CTA per coarse site holds every right-hand side, if they fit
  if (variant >= 0) {
    int seen = -1;
    for (int v = 0; v < kMmaVariants; ++v)
      if (kMmaTiles[v] <= NT8all && ++seen == variant) NT8 = kMmaTiles[v];
  }
  if (T > 32) return -1;
  size_t stage = 0;
  const int ns = stream_stages(T, NT8, &stage);
  unsigned char* rows = coarse_mma_scratch_bytes(n, V, R) ? (unsigned char*)scratch : nullptr;
  if (ns * stage + 2048 > (size_t)smem_optin_bytes()) rows = nullptr;
  if (!rows) {  // the direct form holds the nine directions: as many tiles as fit, in even groups
    const int most = (int)(200 * 1024 / ((size_t)9 * 8 * 4 * npad));
    if (most < 1) return -1;
    const int groups = (NT8all + most - 1) / most;
    if (NT8 > most) NT8 = (NT8all + groups - 1) / groups;
  }
  const int splits = (NT8all + NT8 - 1) / NT8;
  const size_t sm = (size_t)9 * NT8 * 8 * row_pitch(npad);
  if (rows) {
    const size_t smr = (size_t)32 * (4 * npad + 4);
    const dim3 g((unsigned)((V + 31) / 32), (unsigned)R);
    if (prec == 1)
      launch_chain(coarse_rows_kernel<float2>, g, 256, smr, st, (const float2*)in, rows, n, npad, V, R);
    else
      launch_chain(coarse_rows_kernel<__nv_bfloat162>, g, 256, smr, st, (const __nv_bfloat162*)in, rows, n, npad, V, R);
    if (!launched()) return -1;
  }
  const int items = V * splits;
  const size_t ring = (size_t)ns * stage;
  int ctas = rows ? (int)(224 * 1024 / (ring + 2048)) : 0;  // that shared memory lets an SM hold
  ctas = (ctas < 1 ? 1 : (ctas > 8 ? 8 : ctas)) * sm_count();
  if (ctas > items) ctas = items;
#define WMG_MMA(S, K)                                                                                       \
  if (rows) {                                                                                               \
    auto kern = coarse_stream_kernel<S, K>;                                                                 \
    allow_big_smem(kern);                                                                                   \
    launch_chain(kern, ctas, 32 * (T + 1), ring, st, (const unsigned char*)Cf, (const S*)in, rows, (S*)out, (const S*)y2, L[0], \
                                           L[1], L[2], L[3], n, npad, R, (float)a, (float)c, shift, splits, items, ns, spins); \
  } else {                                                                                                  \
    auto kern = coarse_mma_kernel<S, K>;                                                                    \
    if (sm > 40 * 1024) allow_big_smem(kern);                                                               \
    launch_chain(kern, dim3(V, splits), 32 * T, sm, st, (const uint4*)Cf, (const S*)in, (S*)out, (const S*)y2, L[0], L[1], L[2], \
                                              L[3], n, npad, R, (float)a, (float)c, shift);                 \
  }
#define WMG_MMA_R(S)                       \
  switch (NT8) {                           \
    case 1: WMG_MMA(S, 1); break;          \
    case 2: WMG_MMA(S, 2); break;          \
    case 3: WMG_MMA(S, 3); break;          \
    case 4: WMG_MMA(S, 4); break;          \
    case 5: WMG_MMA(S, 5); break;          \
    case 6: WMG_MMA(S, 6); break;          \
    case 7: WMG_MMA(S, 7); break;          \
    case 8: WMG_MMA(S, 8); break;          \
    default: return -1;                    \
  }
  if (prec == 1) {
    WMG_MMA_R(float2)
  } else {
    WMG_MMA_R(__nv_bfloat162)
  }
#undef WMG_MMA_R
#undef WMG_MMA
  return launched() ? 0 : -1;
}

}  // namespace wmg
