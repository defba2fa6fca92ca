// chi0_overlap_tc.cu -- |M_mn(k,q)|^2 (the Eq. 1 matrix elements in the tight-binding form
// of the Sec. III footnote) on the 5th-generation tensor cores: tcgen05.mma with shared-memory
// operands and an FP32 accumulator in tensor memory.
//
// Per k corner c the overlap O = A^H B, A = C[c][:, lo:hi] (norb x w, complex), B the same
// block at k+q, is one real GEMM with K = 2 norb, real and imaginary parts interleaved along K
// (K index 2o: real part of orbital o, 2o + 1: imaginary part):
//   row m of the A operand:        (Re A[o][m], Im A[o][m])  for o = 0 .. norb-1
//   row n of the B operand (Re):   (Re B[o][n], Im B[o][n])          -> Re O[m][n]
//   row NW + n (Im):               (Im B[o][n], -Re B[o][n])         -> Im O[m][n]
// so that one accumulator row (one tensor-memory lane) holds both Re O[m][:] and Im O[m][:]
// and the epilogue forms |O|^2 without exchanging data between lanes.  Several corners share
// one MMA round: corner g's A rows sit at g*w .. g*w + w - 1 of the M = 128 tile and its B
// rows at g*2NW .. of the N <= 256 tile; the off-diagonal corner blocks of the product are
// computed and never read.
//
// Accumulation.  The tensor core adds each MMA's products to its FP32 accumulator with
// truncation, so every MMA accumulated into one place moves the result toward zero by a
// fraction of an ulp: measured on chi0, 6e-8 relative per MMA (3.2e-7 with 6 MMAs per
// element, 1.8e-6 with 30), a bias that the sum over k does not average away.  The K steps
// are therefore spread over NACC accumulators (tensor-memory column blocks of N: round-robin
// when all of K is staged at once, one contiguous chunk each otherwise), each accumulator
// takes its smallest products first and the leading piece product last, and the epilogue
// adds the NACC partial results on the CUDA cores (round to nearest).  With NACC equal to
// the number of K steps each accumulator sees one leading-order MMA.
//
// Precision forms (FP32 accumulation in all):
//   TF32    one product of round-to-nearest TF32 operands
//   BF16X3  x = p0 + p1 with p0 = bf16(x), p1 = bf16(x - p0); products p0 p0 + p0 p1 + p1 p0
//   BF16X6  x = p0 + p1 + p2 (p2 = bf16(x - p0 - p1)); the six products pa pb with a + b <= 2
//
// K chunks.  When the whole K extent of every piece does not fit in shared memory (the
// three-piece split at 80 orbitals: 3 (128 + 160) 320 bytes = 276 KB), K is cut into chunks of
// kc K steps, staged into two buffers in turn: the threads convert chunk j + 1 while the
// tensor core multiplies chunk j.  Each chunk goes to its own accumulator (chunks are
// contiguous runs of K steps), smallest products first, so that the truncation bias stays
// that of kc leading-order MMAs per accumulator.
//
// Operands are staged by the CTA's threads (conversion to TF32/BF16 and the real form above)
// into the K-major, non-swizzled tcgen05 layout: core matrices of 8 rows x 16 bytes stored as
// 128 contiguous bytes, core matrix (row group rb, 16-byte column kb) at (rb * KB + kb) * 128
// bytes (KB = 16-byte columns per row), so the descriptor strides are 128 bytes along K and
// KB * 128 bytes along M/N.  One thread issues the MMAs and commits them to an mbarrier; every
// wait on it is bounded (the plan's wait budget, in clock cycles) and a wait that runs out
// sets the error word, frees the tensor memory and ends the kernel.
//
// Bound: the round's serial chain of staging, MMAs and epilogue in each CTA (the floor is HBM:
// 32^3 corners of 40 bands read and write 1.05 GB, 0.16 ms; 80 bands 4.3 GB, 0.64 ms).  Measured
// before (two-byte staging stores, no loads ahead, the issuing thread's index arithmetic between
// MMAs) and now, 32^3 corners: 40 bands BF16X3 2.9 -> 0.86 ms, 20 of 40 bands 1.5 -> 0.46 ms,
// 80 bands BF16X6 5.7 -> 2.8 ms.  Results are bitwise the same.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "chi0_grid.cuh"
#include "chi0_internal.h"

namespace chi0int {
namespace {

constexpr int kTcThreads = 256;  // 8 warps: warp i reads tensor-memory lanes 32(i%4) .. +31
constexpr int kTcM = 128;        // MMA rows (cta_group::1)
constexpr int kTcMaxN = 256;     // MMA columns
constexpr int kTcCols = 512;           // tensor-memory columns of an SM
constexpr int kTcMinSmem = 80 * 1024;  // at most 2 CTAs per SM when a CTA takes <= 256 columns
constexpr int kTcOneSmem = 116 * 1024; // one CTA per SM when it takes all 512 columns

struct TcShape {
  int w, NW, G, N, Kpad, Kbytes, ES, P, nks, NACC, ncols;
  int kc, nch, chunked;  // K steps per staged chunk, chunks per round, double-buffered chunks
  size_t smem;
};

// gcap > 0 caps the corners per round (the autotuner's candidates)
__host__ __device__ inline TcShape tc_shape(int w, int norb, int mode, int gcap) {
  TcShape s{};
  s.w = w;
  s.NW = (w + 7) & ~7;
  s.ES = mode == TC_TF32 ? 4 : 2;
  s.P = mode == TC_TF32 ? 1 : (mode == TC_BF16X3 ? 2 : 3);
  const int kstep = 32 / s.ES;  // K elements per MMA instruction (32 bytes of K)
  s.Kpad = (2 * norb + kstep - 1) / kstep * kstep;
  s.Kbytes = s.Kpad * s.ES;
  s.nks = s.Kbytes / 32;
  const int g1 = kTcM / (w > 0 ? w : 1), g2 = kTcMaxN / (2 * s.NW);
  s.G = g1 < g2 ? g1 : g2;
  if (s.G < 1) s.G = 0;  // window too wide for one tile
  if (gcap > 0 && s.G > gcap) s.G = gcap;
  if (mode != TC_TF32 && s.G > 1) {
    // fewer corners per round when that lets every K step have its own accumulator
    const int g3 = kTcCols / (2 * s.NW * s.nks);
    s.G = g3 < 1 ? 1 : (g3 < s.G ? g3 : s.G);
  }
  s.N = s.G * 2 * s.NW;
  s.NACC = mode == TC_TF32 ? 1 : (s.N > 0 ? kTcCols / s.N : 1);
  if (s.NACC > s.nks) s.NACC = s.nks;
  if (s.NACC < 1) s.NACC = 1;
  s.kc = s.nks;
  s.nch = 1;
  s.chunked = 0;
  s.smem = (size_t)s.P * (kTcM + s.N) * s.Kbytes + 64;
  if (s.G >= 1 && s.smem > kTcSmemMax) {
    // two chunk buffers; one accumulator per chunk where the tensor memory allows
    s.chunked = 1;
    s.kc = (s.nks + s.NACC - 1) / s.NACC;
    while (s.kc > 1 && 2 * (size_t)s.P * (kTcM + s.N) * s.kc * 32 + 64 > kTcSmemMax) --s.kc;
    s.nch = (s.nks + s.kc - 1) / s.kc;
    if (s.NACC > s.nch) s.NACC = s.nch;
    s.smem = 2 * (size_t)s.P * (kTcM + s.N) * s.kc * 32 + 64;
    if (s.smem > kTcSmemMax) s.G = 0;  // even one K step per chunk does not fit
  }
  int nc = 32;
  while (nc < s.NACC * s.N) nc <<= 1;
  s.ncols = nc;
  return s;
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: start address, leading (K) and stride (M/N) byte offsets,
// descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
         (1ull << 46);
}

// instruction descriptor: FP32 accumulator, TF32 or BF16 operands, both K-major, M = 128
__device__ __forceinline__ uint32_t idesc(int mode, int N) {
  const uint32_t ab = mode == TC_TF32 ? 2u : 1u;
  return (1u << 4) | (ab << 7) | (ab << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kTcM >> 4) << 24);
}

__device__ __forceinline__ void mma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t id, uint32_t acc, int mode) {
  if (mode == TC_TF32)
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(a), "l"(b), "r"(id), "r"(acc));
  else
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(a), "l"(b), "r"(id), "r"(acc));
}

// 8 consecutive FP32 columns at each of two addresses of this thread's tensor-memory lane (both
// loads in flight together; loads and wait in one block)
__device__ __forceinline__ void tmem_ld8x2(uint32_t ta, uint32_t tb, float v[8], float u[8]) {
  uint32_t r[8], q[8];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%16];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8, %9, %10, %11, %12, %13, %14, %15}, [%17];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(q[0]),
        "=r"(q[1]), "=r"(q[2]), "=r"(q[3]), "=r"(q[4]), "=r"(q[5]), "=r"(q[6]), "=r"(q[7])
      : "r"(ta), "r"(tb)
      : "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    v[i] = __uint_as_float(r[i]);
    u[i] = __uint_as_float(q[i]);
  }
}

__device__ __forceinline__ uint32_t tf32_rn(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}

// byte offset of element (row r, column k) in a K-major core-matrix tile
__device__ __forceinline__ uint32_t tile_off(int r, int k, int ES, int KB) {
  const int kb = k * ES;
  return (uint32_t)(((r >> 3) * KB + (kb >> 4)) * 128 + (r & 7) * 16 + (kb & 15));
}

// store x at (r, k) of every piece of a tile (pieces are `stride` bytes apart)
template <int MODE>
__device__ __forceinline__ void put(unsigned char *base, size_t stride, int r, int k, int KB, float x) {
  if constexpr (MODE == TC_TF32) {
    *(uint32_t *)(base + tile_off(r, k, 4, KB)) = tf32_rn(x);
  } else {
    const uint32_t off = tile_off(r, k, 2, KB);
    constexpr int P = MODE == TC_BF16X3 ? 2 : 3;
    float rem = x;
#pragma unroll
    for (int p = 0; p < P; ++p) {
      const __nv_bfloat16 h = __float2bfloat16_rn(rem);
      *(unsigned short *)(base + p * stride + off) = __bfloat16_as_ushort(h);
      rem -= __bfloat162float(h);
    }
  }
}

// Bounded wait on an mbarrier phase; false when the budget (clock cycles) ran out.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, long long budget) {
  const long long t0 = clock64();
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (clock64() - t0 > budget) return false;
  }
}

// Staging moves one 16-byte column of K at a time: kOrb orbitals of one band of one corner (4 in
// the BF16 forms, 2 in TF32), which is one 16-byte store per piece into each of the three operand
// rows that the band fills (A row gg*w + m; B rows gg*2NW + n and gg*2NW + NW + n).  Threads of a
// warp take neighbouring bands: their loads are contiguous and their stores fall on different
// rows of a core matrix (no bank conflicts).  Two-byte stores, element by element, took 2 P x 6
// stores where this takes 3 P / 4.
template <int MODE> struct TcItem {
  static constexpr int kOrb = MODE == TC_TF32 ? 2 : 4;
};
constexpr int kAhead = 3;  // items per thread whose loads are issued a step ahead

__device__ __forceinline__ float2 as_float2(float2 v) { return v; }
__device__ __forceinline__ float2 as_float2(double2 v) { return make_float2(grid::d2f_int(v.x), grid::d2f_int(v.y)); }

// one item's loads (zeros past the last orbital of the chunk); row < 0: no such item
template <int MODE, typename CTq> struct Staged {
  float2 x[TcItem<MODE>::kOrb];
  CTq y[TcItem<MODE>::kOrb];
  int ra, rb, kb;
};

template <int MODE, typename CTq>
__device__ __forceinline__ void load_item(const Grid &g, const float2 *__restrict__ C, const CTq *__restrict__ Cb,
                                          int explicit_q, const Q &q, const TcShape &sh, long long c0, int o0, int o1,
                                          int i, Staged<MODE, CTq> &t) {
  constexpr int kOrb = TcItem<MODE>::kOrb;
  const int w = sh.w, no = g.norb, nob = (o1 - o0 + kOrb - 1) / kOrb, per = nob * w;
  const int gg = i / per, rem = i - gg * per;
  const long long c = c0 + gg;
  t.ra = -1;
  if (gg >= sh.G || c >= g.nc) return;
  const int ob = rem / w, mm = rem - ob * w, o = o0 + ob * kOrb;
  const long long ck = explicit_q ? c : shift_corner(g, c, q.shift);
  const float2 *px = C + (c * no + o) * g.nb + q.lo + mm;
  const CTq *py = Cb + (ck * no + o) * g.nb + q.lo + mm;
#pragma unroll
  for (int j = 0; j < kOrb; ++j) {
    const bool in = o + j < o1;
    t.x[j] = in ? px[(long long)j * g.nb] : make_float2(0.f, 0.f);
    t.y[j] = CTq{};
    if (in) t.y[j] = py[(long long)j * g.nb];
  }
  t.ra = gg * w + mm;
  t.rb = gg * 2 * sh.NW + mm;
  t.kb = ob;
}

// 16 bytes of K at (row r, 16-byte column kb) of every piece: (re, im) pairs of the item's orbitals
__device__ __forceinline__ uint32_t row_off(int r, int kb, int KB) {
  return (uint32_t)(((r >> 3) * KB + kb) * 128 + (r & 7) * 16);
}
__device__ __forceinline__ uint32_t bf16_pair(float2 v) {  // low half: v.x
  const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
  return *reinterpret_cast<const uint32_t *>(&h);
}

template <int MODE, typename CTq>
__device__ __forceinline__ void store_item(const TcShape &sh, const Staged<MODE, CTq> &t, unsigned char *sA,
                                           unsigned char *sB, size_t a_piece, size_t b_piece, int KB) {
  if (t.ra < 0) return;
  const uint32_t oa = row_off(t.ra, t.kb, KB), ob = row_off(t.rb, t.kb, KB), oi = row_off(t.rb + sh.NW, t.kb, KB);
  if constexpr (MODE == TC_TF32) {
    const float2 y0 = as_float2(t.y[0]), y1 = as_float2(t.y[1]);
    *(uint4 *)(sA + oa) = make_uint4(tf32_rn(t.x[0].x), tf32_rn(t.x[0].y), tf32_rn(t.x[1].x), tf32_rn(t.x[1].y));
    *(uint4 *)(sB + ob) = make_uint4(tf32_rn(y0.x), tf32_rn(y0.y), tf32_rn(y1.x), tf32_rn(y1.y));
    *(uint4 *)(sB + oi) = make_uint4(tf32_rn(y0.y), tf32_rn(-y0.x), tf32_rn(y1.y), tf32_rn(-y1.x));
  } else {
    constexpr int P = MODE == TC_BF16X3 ? 2 : 3;
    float2 x[4], y[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      x[j] = t.x[j];
      y[j] = as_float2(t.y[j]);
    }
#pragma unroll
    for (int p = 0; p < P; ++p) {
      uint32_t hx[4], hy[4], hi[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        hx[j] = bf16_pair(x[j]);
        hy[j] = bf16_pair(y[j]);
        hi[j] = __byte_perm(hy[j], 0u, 0x1032) ^ 0x80000000u;  // (im, -re)
        if (p + 1 < P) {  // the rest, for the next piece
          x[j].x -= __uint_as_float(hx[j] << 16);
          x[j].y -= __uint_as_float(hx[j] & 0xFFFF0000u);
          y[j].x -= __uint_as_float(hy[j] << 16);
          y[j].y -= __uint_as_float(hy[j] & 0xFFFF0000u);
        }
      }
      *(uint4 *)(sA + p * a_piece + oa) = make_uint4(hx[0], hx[1], hx[2], hx[3]);
      *(uint4 *)(sB + p * b_piece + ob) = make_uint4(hy[0], hy[1], hy[2], hy[3]);
      *(uint4 *)(sB + p * b_piece + oi) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    }
  }
}

// Zeroes K columns [k0, k1) of the rows a round uses (a chunk buffer that held a longer chunk
// before: its K padding must read as zero).
template <int MODE>
__device__ __forceinline__ void zero_columns(const TcShape &sh, int k0, int k1, unsigned char *sA,
                                             unsigned char *sB, size_t a_piece, size_t b_piece, int KB) {
  const int na = sh.G * sh.w, nbr = sh.N, nk = k1 - k0;
  const int tot = (na + nbr) * nk;
  for (int i = threadIdx.x; i < tot; i += kTcThreads) {
    const int r = i / nk, k = k0 + (i - r * nk);
    if (r < na) put<MODE>(sA, a_piece, r, k, KB, 0.0f);
    else put<MODE>(sB, b_piece, r - na, k, KB, 0.0f);
  }
}

template <int MODE, typename CTq>
__global__ void __launch_bounds__(kTcThreads, sizeof(CTq) == 8 ? 2 : 1)
    k_overlap_tc(Grid g, const float2 *__restrict__ C, const CTq *__restrict__ Cb, int explicit_q, Q q,
                 float *__restrict__ W2, long long budget, int test_stall, int gcap, int *__restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const TcShape sh = tc_shape(q.hi - q.lo, g.norb, MODE, gcap);
  const int w = sh.w, NW = sh.NW, G = sh.G;
  // operand buffers: one holding all of K, or two holding one chunk of kc K steps each
  const int cbytes = sh.chunked ? sh.kc * 32 : sh.Kbytes;  // K bytes per row of a buffer
  const int KB = cbytes / 16;
  const size_t a_piece = (size_t)kTcM * cbytes, b_piece = (size_t)sh.N * cbytes;
  const size_t buf_bytes = sh.P * (a_piece + b_piece);
  const int nbuf = sh.chunked ? 2 : 1;
  unsigned char *tail = smem + nbuf * buf_bytes;
  uint64_t *bar = (uint64_t *)tail;
  uint32_t *tslot = (uint32_t *)(tail + 16);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int kOrbStep = MODE == TC_TF32 ? 4 : 8;  // orbitals per K step (32 bytes of K)
  const int ostep = kOrbStep * sh.kc;                 // orbitals per chunk

  // operand memory starts at zero: padding rows and K columns are never written again
  // (except a chunk buffer's K padding, cleared where a longer chunk used the buffer before)
  const size_t nz = (nbuf * buf_bytes) / 16;
  for (size_t i = tid; i < nz; i += blockDim.x) ((uint4 *)smem)[i] = make_uint4(0, 0, 0, 0);
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(sh.ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  const uint32_t id = idesc(MODE, sh.N);
  const bool vec = (w & 3) == 0 && ((size_t)W2 & 15) == 0;  // every row of W2 starts on 16 bytes
  const long long nround = (g.nc + G - 1) / G;
  uint32_t parity = 0;
  bool ok = true;
  constexpr int kOrb = TcItem<MODE>::kOrb;
  // Chunk j of the round at corner c0 goes to buffer j % nbuf.  The loads of a thread's first
  // kAhead items are issued a chunk ahead (fetch), before the wait for the MMAs and the epilogue,
  // and stored here; the rest are loaded here.
  Staged<MODE, CTq> ahead[kAhead];
  auto fetch = [&](long long c0, int j) {
    const int o0 = j * ostep, o1 = min(g.norb, o0 + ostep);
#pragma unroll
    for (int k = 0; k < kAhead; ++k)
      load_item<MODE, CTq>(g, C, Cb, explicit_q, q, sh, c0, o0, o1, tid + k * kTcThreads, ahead[k]);
  };
  auto stage = [&](long long c0, int j) {
    unsigned char *sA = smem + (j % nbuf) * buf_bytes;
    unsigned char *sB = sA + sh.P * a_piece;
    const int o0 = j * ostep, o1 = min(g.norb, o0 + ostep);
#pragma unroll
    for (int k = 0; k < kAhead; ++k) store_item<MODE, CTq>(sh, ahead[k], sA, sB, a_piece, b_piece, KB);
    const int tot = G * ((o1 - o0 + kOrb - 1) / kOrb) * w;
#pragma unroll 1
    for (int i = tid + kAhead * kTcThreads; i < tot; i += kAhead * kTcThreads) {
#pragma unroll
      for (int k = 0; k < kAhead; ++k)
        load_item<MODE, CTq>(g, C, Cb, explicit_q, q, sh, c0, o0, o1, i + k * kTcThreads, ahead[k]);
#pragma unroll
      for (int k = 0; k < kAhead; ++k) store_item<MODE, CTq>(sh, ahead[k], sA, sB, a_piece, b_piece, KB);
    }
    // the last chunk of three or more may sit in a buffer whose K padding (inside its last K
    // step) an earlier, longer chunk filled (an item writes whole 16-byte columns)
    if (sh.chunked && sh.nch >= 3 && j == sh.nch - 1) {
      const int kstep = 32 / sh.ES, kcol = 16 / sh.ES, kused = (2 * (o1 - o0) + kcol - 1) / kcol * kcol;
      const int kpad = (kused + kstep - 1) / kstep * kstep;
      if (kused < kpad) zero_columns<MODE>(sh, kused, kpad, sA, sB, a_piece, b_piece, KB);
    }
    // generic-proxy stores must be visible to the tensor core's (async-proxy) reads
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  };
  // One thread issues chunk j's MMAs and commits them to the mbarrier.  The loops below are that
  // thread's serial chain, so they hold nothing but the MMAs and descriptor sums (a K step is 256
  // bytes further on: 16 in the descriptor's address field): with a modulo per K step to find the
  // accumulator and descriptors built anew, the chain took 0.65 us per MMA, four fifths of the
  // kernel at 40 bands.
  constexpr int P = MODE == TC_TF32 ? 1 : (MODE == TC_BF16X3 ? 2 : 3);
  auto issue = [&](int j) {
    if (tid != 0 || test_stall) return;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned char *sA = smem + (j % nbuf) * buf_bytes;
    const unsigned char *sB = sA + P * a_piece;
    uint64_t da[P], db[P];
#pragma unroll
    for (int k = 0; k < P; ++k) {
      da[k] = sdesc(smem_u32(sA + k * a_piece), 128, KB * 128);
      db[k] = sdesc(smem_u32(sB + k * b_piece), 128, KB * 128);
    }
    const int s0 = j * sh.kc, ns = min(sh.nks, s0 + sh.kc) - s0;  // K steps of the chunk
    // unchunked: K step s goes to accumulator s % NACC; chunked: chunk j to j * NACC / nch
    const int ia0 = sh.chunked ? j * sh.NACC / sh.nch : 0, ia1 = sh.chunked ? ia0 + 1 : sh.NACC;
    const int sstep = sh.chunked ? 1 : sh.NACC;
    // the first MMA into an accumulator in this round overwrites it
    const uint32_t first = (sh.chunked && j > 0 && (j - 1) * sh.NACC / sh.nch == ia0) ? 1u : 0u;
#pragma unroll 1
    for (int ia = ia0; ia < ia1; ++ia) {
      uint32_t acc = first;
      const uint32_t at = tmem + (uint32_t)(ia * sh.N);
      // products of pieces a, b with a + b = lvl < P, smallest level first
#pragma unroll
      for (int lvl = P - 1; lvl >= 0; --lvl)
#pragma unroll
        for (int pa = 0; pa <= lvl; ++pa)
#pragma unroll 1
          for (int s = sh.chunked ? 0 : ia; s < ns; s += sstep) {
            mma(at, da[pa] + 16u * (uint32_t)s, db[lvl - pa] + 16u * (uint32_t)s, id, acc, MODE);
            acc = 1;
          }
    }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
  };
  if (blockIdx.x < nround) fetch((long long)blockIdx.x * G, 0);
  for (long long rd = blockIdx.x; rd < nround && ok; rd += gridDim.x) {
    const long long c0 = rd * G;
    stage(c0, 0);
    if (sh.nch > 1) fetch(c0, 1);
    __syncthreads();
    for (int j = 0; j < sh.nch; ++j) {
      issue(j);
      if (j + 1 < sh.nch) stage(c0, j + 1);  // the other buffer: chunk j - 1's MMAs are done
      if (j + 2 < sh.nch) fetch(c0, j + 2);
      else if (j + 1 == sh.nch && rd + gridDim.x < nround) fetch((rd + gridDim.x) * G, 0);
      // test_stall: nothing arrives, so the bounded wait below runs out (error path test).  The
      // CTA agrees on the outcome before any warp-wide tensor-memory load or buffer reuse.
      const int got = mbar_wait(smem_u32(bar), parity, budget) ? 1 : 0;
      if (!__syncthreads_and(got)) {
        ok = false;
        if (tid == 0) atomicExch(err, 1);
        break;
      }
      parity ^= 1u;
    }
    if (!ok) break;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // epilogue: lane r = gg*w + m of the tile holds Re O (columns gg*2NW + n) and Im O (+ NW);
    // warps i and i + 4 share lane quarter i%4 and split the 8-column chunks between them
    const int quarter = warp & 3, half = warp >> 2;
    const int r = quarter * 32 + lane;
    const int gg = r / (w > 0 ? w : 1), m = r - gg * w;
    const long long c = c0 + gg;
    const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16);
    // (the corner blocks that this warp's 32 rows belong to; rows past G*w belong to none)
    const int blk0 = quarter * 32 / w, blk1 = min(G - 1, (quarter * 32 + 31) / w);
    for (int blk = blk0; blk <= blk1; ++blk) {  // warp-uniform loops: every lane takes part in tcgen05.ld
      for (int n0 = half * 8; n0 < NW; n0 += 16) {
        float re[8], im[8];
        tmem_ld8x2(trow + blk * 2 * NW + n0, trow + blk * 2 * NW + NW + n0, re, im);
        for (int ia = 1; ia < sh.NACC; ++ia) {  // partial accumulators, added in FP32
          float r2[8], i2[8];
          tmem_ld8x2(trow + ia * sh.N + blk * 2 * NW + n0, trow + ia * sh.N + blk * 2 * NW + NW + n0, r2, i2);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            re[j] += r2[j];
            im[j] += i2[j];
          }
        }
        if (blk == gg && c < g.nc) {
          float *out = W2 + (c * w + m) * w + n0;
#pragma unroll
          for (int j = 0; j < 8; ++j) re[j] = re[j] * re[j] + im[j] * im[j];
          if (vec) {
            *(float4 *)out = make_float4(re[0], re[1], re[2], re[3]);
            if (n0 + 4 < w) *(float4 *)(out + 4) = make_float4(re[4], re[5], re[6], re[7]);
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if (n0 + j < w) out[j] = re[j];
          }
        }
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
  }
  if (!ok) {
    // the MMAs this CTA issued (if any) may still be running: wait for them once more,
    // bounded, before the tensor memory is released.  (The error-path test issues no MMA, so
    // there the second wait runs out as well and nothing is in flight.)
    mbar_wait(smem_u32(bar), parity, budget);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(sh.ncols) : "memory");
}

template <int MODE, typename CTq>
cudaError_t launch_tc(const Grid &g, const float2 *Ck, const CTq *Cb, int explicit_q, const Q &q, float *W2,
                      long long budget, int test_stall, int gcap, int *err, cudaStream_t s) {
  const TcShape sh = tc_shape(q.hi - q.lo, g.norb, MODE, gcap);
  const size_t floor_smem = sh.ncols > 256 ? (size_t)kTcOneSmem : (size_t)kTcMinSmem;
  const size_t smem = sh.smem < floor_smem ? floor_smem : sh.smem;
  cudaError_t e = cudaFuncSetAttribute(k_overlap_tc<MODE, CTq>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long long nround = (g.nc + sh.G - 1) / sh.G;
  const int per_sm = smem > (size_t)113 * 1024 ? 1 : 2;
  long long blocks = (long long)sms * per_sm;
  if (blocks > nround) blocks = nround;
  k_overlap_tc<MODE, CTq><<<(int)blocks, kTcThreads, smem, s>>>(g, Ck, Cb, explicit_q, q, W2, budget, test_stall,
                                                                gcap, err);
  return cudaGetLastError();
}

// Tensor-core throughput: one CTA per SM issues `iters` MMAs (M = 128, N = 256, one K step of
// 32 bytes) from fixed zeroed shared-memory operands into one tensor-memory accumulator, then
// commits them and waits (bounded).  The large shared-memory request keeps one CTA per SM.
constexpr int kPeakSmem = 160 * 1024;
__global__ void __launch_bounds__(128, 1) k_tc_peak(int mode, int iters, long long budget, int *err) {
  extern __shared__ __align__(1024) unsigned char smem[];
  constexpr int kN = 256;
  unsigned char *sA = smem, *sB = smem + kTcM * 32;
  uint64_t *bar = (uint64_t *)(sB + kN * 32);
  uint32_t *tslot = (uint32_t *)(sB + kN * 32 + 16);
  const int tid = threadIdx.x, warp = tid >> 5;
  for (int i = tid; i < (kTcM + kN) * 32 / 16; i += blockDim.x) ((uint4 *)smem)[i] = make_uint4(0, 0, 0, 0);
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(kN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  if (tid == 0) {
    const uint64_t da = sdesc(smem_u32(sA), 128, 2 * 128), db = sdesc(smem_u32(sB), 128, 2 * 128);
    const uint32_t id = idesc(mode, kN);
    for (int i = 0; i < iters; ++i) mma(tmem, da, db, id, i > 0 ? 1u : 0u, mode);
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
  }
  const int got = mbar_wait(smem_u32(bar), 0, budget) ? 1 : 0;
  if (!__syncthreads_and(got)) {
    if (tid == 0) atomicExch(err, 1);
    mbar_wait(smem_u32(bar), 0, budget);  // the MMAs may still run: wait once more, bounded
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kN) : "memory");
}

}  // namespace

cudaError_t tc_peak(int mode, int iters, double *tflops, double *ms_out) {
  int *err = nullptr;
  cudaError_t e = cudaMalloc(&err, sizeof(int));
  if (e != cudaSuccess) return e;
  cudaMemset(err, 0, sizeof(int));
  e = cudaFuncSetAttribute(k_tc_peak, cudaFuncAttributeMaxDynamicSharedMemorySize, kPeakSmem);
  if (e != cudaSuccess) {
    cudaFree(err);
    return e;
  }
  const int sms = device_sms();
  const long long budget = 1LL << 32;  // about two seconds: far above the run's length
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  k_tc_peak<<<sms, 128, kPeakSmem>>>(mode, iters / 8 + 1, budget, err);  // warm-up
  cudaEventRecord(e0);
  k_tc_peak<<<sms, 128, kPeakSmem>>>(mode, iters, budget, err);
  cudaEventRecord(e1);
  e = cudaEventSynchronize(e1);
  float ms = 0.f;
  cudaEventElapsedTime(&ms, e0, e1);
  int herr = 0;
  if (e == cudaSuccess) e = cudaMemcpy(&herr, err, sizeof(int), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaGetLastError();
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(err);
  if (e != cudaSuccess) return e;
  if (herr) return cudaErrorTimeout;
  const double kel = mode == TC_TF32 ? 8.0 : 16.0;  // K elements of one 32-byte K step
  const double flops = 2.0 * kTcM * 256.0 * kel * (double)iters * sms;
  *tflops = flops / (ms * 1e-3) / 1e12;
  *ms_out = ms;
  return cudaSuccess;
}

size_t overlap_tc_smem(int w, int norb, int mode) {
  const TcShape sh = tc_shape(w, norb, mode, 0);
  if (sh.G < 1) return (size_t)-1;
  return sh.smem;
}

int overlap_tc_max_corners(int w, int norb, int mode) { return tc_shape(w, norb, mode, 0).G; }

cudaError_t launch_overlap_tc(const Grid &g, const void *C32, int dtype, const Q &q, float *W2, int mode,
                              long long budget, int test_stall, int gcap, int *err, cudaStream_t s) {
  const int w = q.hi - q.lo;
  if (w < 1 || overlap_tc_smem(w, g.norb, mode) > kTcSmemMax || !err) return cudaErrorInvalidValue;
  const float2 *Ck = (const float2 *)C32;
  if (budget <= 0) budget = 1LL << 31;
  if (mode == TC_BF16X6) {
    if (q.Cq && dtype == DT_C128)
      return launch_tc<TC_BF16X6, double2>(g, Ck, (const double2 *)q.Cq, 1, q, W2, budget, test_stall, gcap, err, s);
    if (q.Cq)
      return launch_tc<TC_BF16X6, float2>(g, Ck, (const float2 *)q.Cq, 1, q, W2, budget, test_stall, gcap, err, s);
    return launch_tc<TC_BF16X6, float2>(g, Ck, Ck, 0, q, W2, budget, test_stall, gcap, err, s);
  }
  if (mode == TC_TF32) {
    if (q.Cq && dtype == DT_C128)
      return launch_tc<TC_TF32, double2>(g, Ck, (const double2 *)q.Cq, 1, q, W2, budget, test_stall, gcap, err, s);
    if (q.Cq) return launch_tc<TC_TF32, float2>(g, Ck, (const float2 *)q.Cq, 1, q, W2, budget, test_stall, gcap, err, s);
    return launch_tc<TC_TF32, float2>(g, Ck, Ck, 0, q, W2, budget, test_stall, gcap, err, s);
  }
  if (q.Cq && dtype == DT_C128)
    return launch_tc<TC_BF16X3, double2>(g, Ck, (const double2 *)q.Cq, 1, q, W2, budget, test_stall, gcap, err, s);
  if (q.Cq) return launch_tc<TC_BF16X3, float2>(g, Ck, (const float2 *)q.Cq, 1, q, W2, budget, test_stall, gcap, err, s);
  return launch_tc<TC_BF16X3, float2>(g, Ck, Ck, 0, q, W2, budget, test_stall, gcap, err, s);
}

}  // namespace chi0int
