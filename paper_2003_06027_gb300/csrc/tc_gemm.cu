// tc_gemm.cu - BF16 x BF16 -> FP32 GEMM on the 5th-generation tensor cores
// (tcgen05.mma, accumulator in tensor memory), operands staged by TMA.
//
// One CTA computes a 128 x BN tile of D = A . B^T (BN <= 256, a multiple of 16)
// over its run of K:
//   * warp 0 allocates BN (rounded up to a power of two, >= 32) TMEM columns;
//   * one thread of warp 0 is the producer: per 64-wide k-block it loads the
//     128 x 64 tile of A and the BN x 64 tile of B into one of STAGES shared
//     memory slots with cp.async.bulk.tensor (128-byte swizzle, zero fill beyond
//     the matrix edges), completing on the slot's "full" mbarrier;
//   * one thread of warp 1 issues the MMAs: 4 x tcgen05.mma (K = 16 each) per
//     k-block into the TMEM accumulator, then tcgen05.commit onto the slot's
//     "empty" mbarrier, which frees the slot for the producer once the MMAs
//     that read it have completed; a last commit signals "accumulator ready";
//   * all four warps drain the accumulator: warp w reads TMEM lanes 32w..32w+31
//     (tile rows m) with tcgen05.ld, adds the bias, applies the ReLU and writes
//     out[n][m]: for each column n the 32 lanes of a warp store 32 consecutive
//     m, so the transposed write is coalesced.
// The convolution variant (CONV) gathers A instead of loading it: 256 threads
// build each 128 x 64 A stage from the FP32 activations of a 3x3 layer in the
// same swizzled layout, fence their shared-memory writes for the tensor core
// and arrive on the stage's second "full" barrier, which the MMA thread also
// waits for; warp 8 loads B by TMA, warp 9 issues the MMAs.
// Every mbarrier wait is bounded (2^24 polls or 1 s); a wait that gives up
// records a timeout in the status word, the tile is written as NaN, and the
// CTA waits (again bounded) for its own TMA copies and MMAs still in flight,
// frees its TMEM and exits (drain).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "fwi_internal.cuh"
#include "tc_gemm.h"
#include "tma.cuh"

namespace fwi {
namespace {

constexpr int TC_BM = 128;
constexpr int TC_BK = 64;  // one 128-byte swizzle row of BF16
constexpr int TC_STAGES = 4;
constexpr int TC_THREADS = 128;
constexpr int A_STAGE = TC_BM * TC_BK * 2;  // 16 KB
constexpr int TC_WG_ROWS = 9 * TC_WG_CH;
constexpr int SM_SMEM = 228 * 1024;  // shared memory of an SM (a CTA takes 1 KB more than it asks for)

struct TcArgs {
  long long M;
  int N, BN, nkb, kbps;
  float* out;
  long long ldo, split_stride;
  const float* bias;
  int relu;
  int* status;
  uint32_t idesc;
  uint32_t tmem_cols;
  int stages;  // of the shared-memory ring: fewer than TC_STAGES if all k-blocks fit (CONV 0)
  uint32_t issue_limit;  // k-blocks after which a CTA's MMA issuer gives up (self-test; no limit: 2^32 - 1)
};

// Shared-memory matrix descriptor of a K-major operand tile written by TMA with
// the 128-byte swizzle: rows of 128 bytes, 8-row groups 1024 bytes apart.
//   bits  0-13 start address >> 4      bits 16-29 leading byte offset >> 4 (unused here)
//   bits 32-45 stride byte offset >> 4 bits 46-47 descriptor version (1)
//   bits 61-63 layout: 2 = 128-byte swizzle
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// The same for an operand kept with its M index contiguous (M-major): per k, 64
// values of M in 128 swizzled bytes; 8 values of k 1024 bytes apart (stride byte
// offset), the next 64 of M at the leading byte offset.
__device__ __forceinline__ uint64_t sdesc_sw128_mn(uint32_t saddr, uint32_t lbo) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(lbo >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t r[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_n(uint64_t* bar, uint32_t n) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(n) : "memory");
}
// After a wait that ran out, once every role of the CTA has left its loop: bounded waits
// for what the CTA may still have in flight, so that no copy or MMA writes after it has
// exited or freed its TMEM. The MMA issuer commits what it has issued onto a barrier of
// its own; of the `armed` k-blocks that the TMA producer asked for, each stage's last
// one completes that stage's phase (armed - 1 - s) / TC_STAGES.
__device__ __forceinline__ void drain(bool issuer, bool producer, uint64_t* full, int armed, uint64_t* issued) {
  if (issuer) {
    tc_commit(issued);
    mbar_wait(issued, 0);
  }
  if (producer)
    for (int s = 0; s < TC_STAGES && s < armed; s++) mbar_wait(&full[s], (uint32_t)((armed - 1 - s) / TC_STAGES) & 1u);
  __syncwarp();
}
// Row m of a tile whose product is not to be had, whatever the bias and the ReLU (a
// maximum with 0 would drop a NaN). A loop of its own: one selection per element in the
// epilogue cost the products of 96 to 256 columns 2.5 %.
__device__ __forceinline__ void nan_rows(const TcArgs& a, float* out, long long m, int n0) {
  for (int n = n0; n < a.N && n < n0 + a.BN; n++) out[(long long)n * a.ldo + m] = __int_as_float(0x7fc00000);
}
__device__ __forceinline__ uint32_t mulhi_div(uint32_t n, unsigned long long m, uint32_t s) {
  return (uint32_t)(((unsigned long long)n * m) >> s);
}

// The threads of a CTA: 128 (warp 0: TMEM and the TMA producer, warp 1: the
// MMA issuer, all four: the epilogue); with a gathered A operand (CONV) 320:
// warps 0-7 gather A (two threads per tile row, 32 taps each; warps 0-3 also
// run the epilogue), warp 8 loads B by TMA, warp 9 issues the MMAs. Up to two
// CONV CTAs share an SM, so that one's gather covers the other's load latency.
// CONV: 0 A by TMA, 1 gathered tap by tap through a table (any layer), 2 and 3 the
// weight gradient's A (rows = taps, K = pixels) gathered by pixel pairs (layers of
// horizontal stride 1 and 2; their forward and data-gradient products have a kernel
// of their own, k_conv_pairs).
template <int CONV>
struct TcRoles {
  static constexpr bool WG = CONV >= 2;
  static constexpr int BM = WG ? TC_WG_ROWS : TC_BM;  // rows of D per tile
  static constexpr int ARRIVE = WG ? 2 : 2 * TC_BM / 32;  // gathering warps of one stage
  static constexpr int THREADS = CONV ? 320 : TC_THREADS;
  static constexpr int GATHER = 2 * TC_BM;  // gathering threads (CONV)
  static constexpr int B_WARP = CONV ? 8 : 0;
  static constexpr int MMA_WARP = CONV ? 9 : 1;
  static constexpr int CTAS = CONV ? 2 : 1;
};

// Gathered A rows (CONV): threads r and r + 128 build row r of every 128 x 64
// stage tile, pixel m0 + r, each 32 of its taps (half h: k0 + 32 h .. k0 + 32 h
// + 31), read from x (zero outside the image and beyond 9 C), rounded to BF16 as
// the im2col kernels round them, and stored as four 16-byte chunks in the
// layout TMA's 128-byte swizzle gives a K-major tile (chunk c of row r at
// 16 (c ^ (r % 8)) within its 128-byte row).
struct GatherRow {
  long long base;  // x offset of (b, r0, s0) relative to channel 0, if m is a pixel
  uint32_t mask;   // bit 3p + q: tap (p, q) inside the image (0 if m is not a pixel)
};
__device__ __forceinline__ GatherRow gather_row(const TcConvA& c, long long m, long long M) {
  GatherRow g{0, 0u};
  if (m >= M) return g;
  const uint32_t bi = mulhi_div((uint32_t)m, c.wo_m, c.wo_s);
  const int j = (int)((uint32_t)m - bi * (uint32_t)c.Wo);
  const uint32_t b = mulhi_div(bi, c.ho_m, c.ho_s);
  const int i = (int)(bi - b * (uint32_t)c.Ho);
  const int r0 = c.sh * i - 1, s0 = c.sw * j - 1;
  g.base = ((long long)b * c.H + r0) * c.W + s0;
#pragma unroll
  for (int p = 0; p < 3; p++)
#pragma unroll
    for (int q = 0; q < 3; q++)
      if (r0 + p >= 0 && r0 + p < c.H && s0 + q >= 0 && s0 + q < c.W) g.mask |= 1u << (3 * p + q);
  return g;
}
constexpr int GATHER_K = TC_BK / 2;  // taps of a row built by one gathering thread per stage
// Tap table of a CONV CTA (shared memory, built once, one entry per tap of every
// k-block): for tap k < 9 C the x offset of (channel c, tap row p, tap column q)
// relative to a pixel's base, c B H W + p W + q, and the mask bit of its tap,
// 1 << (3 p + q); beyond 9 C, offset 0 and bit 1 << 9 (a bit no mask has).
// Loads (into registers) the GATHER_K taps of half `half` of k-block kb for the thread's row.
__device__ __forceinline__ void gather_load(const TcConvA& c, const GatherRow& g, const int2* tab, int kb, int half,
                                            float v[GATHER_K]) {
  const int2* t = tab + kb * TC_BK + GATHER_K * half;
  const float* xb = c.x + g.base;
#pragma unroll
  for (int kk = 0; kk < GATHER_K; kk++) {
    const int2 e = t[kk];
    v[kk] = (g.mask & (uint32_t)e.y) ? __ldg(xb + e.x) : 0.f;
  }
}
// Rounds them to BF16 and stores them as chunks 4 half .. 4 half + 3 of the row.
__device__ __forceinline__ void gather_store(const float v[GATHER_K], int row, int half, unsigned char* dst) {
  unsigned char* rowp = dst + row * 128;
#pragma unroll
  for (int cl = 0; cl < 4; cl++) {
    const int cc = 4 * half + cl;  // 16-byte chunk of the row
    uint32_t w[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(v[8 * cl + 2 * u], v[8 * cl + 2 * u + 1]);
      w[u] = *reinterpret_cast<const uint32_t*>(&h);
    }
    *reinterpret_cast<uint4*>(rowp + ((cc ^ (row & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// The input window of a pair of output pixels (m, m + 1): its corner in channel 0
// and which of its rows and columns are inside the image (none if m is no pixel).
template <int SW>
struct PairWin {
  const float* base;
  bool rok[3], left, right;
  __device__ __forceinline__ PairWin(const TcConvA& c, long long m, long long M) {
    base = c.x;
    rok[0] = rok[1] = rok[2] = left = right = false;
    if (m < M) {  // the pair's pixels are both inside: Wo is even
      const uint32_t bi = mulhi_div((uint32_t)m, c.wo_m, c.wo_s);
      const int j = (int)((uint32_t)m - bi * (uint32_t)c.Wo);
      const uint32_t b = mulhi_div(bi, c.ho_m, c.ho_s);
      const int i = (int)(bi - b * (uint32_t)c.Ho), r0 = c.sh * i - 1;
      base += ((long long)b * c.H + r0) * c.W + SW * j;
#pragma unroll
      for (int p = 0; p < 3; p++) rok[p] = r0 + p >= 0 && r0 + p < c.H;
      left = SW * j - 1 >= 0;
      right = SW == 2 || j + 2 < c.W;
    }
  }
  // BF16 words of NB channels' 9 NB taps for both pixels; channel u of them exists if cok(u)
  template <int NB, typename F>
  __device__ __forceinline__ void words(const TcConvA& c, int ch0, F cok, uint32_t* w0, uint32_t* w1) const {
    constexpr int NV = SW + 3;  // input columns SW j - 1 .. SW j + SW + 1 of a pair
    const long long plane = (long long)c.B * c.H * c.W;
    float v[NB][3][NV];
#pragma unroll
    for (int u = 0; u < NB; u++) {
      const float* xc = base + (long long)(ch0 + u) * plane;
      const bool ck = cok(u);
#pragma unroll
      for (int p = 0; p < 3; p++) {
        const float* q = xc + p * c.W;
        const bool ok = ck && rok[p];
        v[u][p][0] = ok && left ? __ldg(q - 1) : 0.f;
        if (SW == 1) {
          const float2 t = ok ? __ldg(reinterpret_cast<const float2*>(q)) : make_float2(0.f, 0.f);
          v[u][p][1] = t.x;
          v[u][p][2] = t.y;
          v[u][p][3] = ok && right ? __ldg(q + 2) : 0.f;
        } else {
          const float4 t = ok ? __ldg(reinterpret_cast<const float4*>(q)) : make_float4(0.f, 0.f, 0.f, 0.f);
          v[u][p][1] = t.x;
          v[u][p][2] = t.y;
          v[u][p][3] = t.z;
          v[u][p][NV - 1] = t.w;
        }
      }
    }
    // tap e of the channels: (channel e / 9, row e % 9 / 3, column e % 3)
#pragma unroll
    for (int k = 0; k < 9 * NB / 2; k++) {
      const int e = 2 * k, f = 2 * k + 1;
      const __nv_bfloat162 h0 = __floats2bfloat162_rn(v[e / 9][e % 9 / 3][e % 3], v[f / 9][f % 9 / 3][f % 3]);
      const __nv_bfloat162 h1 =
          __floats2bfloat162_rn(v[e / 9][e % 9 / 3][e % 3 + SW], v[f / 9][f % 9 / 3][f % 3 + SW]);
      w0[k] = *reinterpret_cast<const uint32_t*>(&h0);
      w1[k] = *reinterpret_cast<const uint32_t*>(&h1);
    }
  }
};

// Gathers the A tile of pixels m0 .. m0 + 127 by pairs: thread (pair, sub) of 64 x
// SUBS builds two rows of every stage tile, two neighbouring output pixels of one
// image row, taking every SUBS-th run of 8 channels. The 72 taps of 8 channels are 9
// whole 16-byte chunks of a row, so a run's values go from registers to shared
// memory without a table: per channel a thread reads the 3 x (2 SW + 2) input
// values of its pair once (9 loads for 18 operand elements at SW = 1), and each
// BF16 word is one packed conversion of two of them: about 1.6 instructions per
// element against 6 for the table (each tap decoded, tested and loaded by itself).
// Within 16 pixels the even ones take the first 8 rows and the odd ones the next 8:
// the 8 lanes of a 16-byte store phase then write 8 different rows mod 8, which the
// swizzle sends to different banks (even and odd rows in turn would meet two by two).
// Run r of a tile fills chunks 9 r .. 9 r + 8: a stage of 8 chunks belongs to one or two
// runs, and only their warps wait for it and arrive on it (one warp of a lone run for
// two), so that no warp spends instructions on stages that it has nothing for. The
// runs of all tiles go round the SUBS groups in turn: few channels keep all of them
// busy, and a group's next run starts at most 9 SUBS chunks after its last one's start:
// with SUBS <= TC_STAGES its wait for a stage is at most one phase ahead, as the parity needs.
// Against every thread of every group waiting for and arriving on every stage, tile by
// tile (batch 32): 16 channels at 500 x 64, 107 -> 81 us, 32 at 128 x 256, 195 -> 143, 64 at
// 128 x 256, 256 -> 229; the step's 18 products 1782 -> 1650. With the next run's lines
// asked for ahead 1744 -> 1650.
__device__ __forceinline__ int pair_row(int pair) { return ((pair & ~7) << 1) | (pair & 7); }  // and + 8
__device__ __forceinline__ int row_pixel(int row) { return 2 * (((row >> 4) << 3) | (row & 7)) + ((row >> 3) & 1); }
// The whole warp waits for a stage (and agrees on a wait that ran out), and leaves it
// by one arrival of weight n.
__device__ __forceinline__ bool warp_enter(uint64_t* empty, uint32_t ph) {
  return __all_sync(0xffffffffu, mbar_wait(empty, ph));
}
__device__ __forceinline__ void warp_leave(uint64_t* fulla, uint32_t n) {
  fence_proxy_async();  // the generic-proxy writes before the tensor core reads them
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive_n(fulla, n);
}
template <int SW, int SUBS>
__device__ __forceinline__ bool gather_pairs(const TcConvA& c, long long M, int nk, int ntn, int ntiles,
                                             unsigned char* smA, uint64_t* empty, uint64_t* fulla) {
  static_assert(SUBS <= TC_STAGES, "stage waits at most one phase ahead");
  const int pair = threadIdx.x & 63;
  const int nchunk = nk * (TC_BK / 8), nrun = (nchunk + 8) / 9;
  int t = blockIdx.x, kb0 = 0, r = threadIdx.x >> 6;  // tile, its first k-block in this CTA's sequence, run
  for (; r >= nrun; r -= nrun, kb0 += nk) t += gridDim.x;
  unsigned char* rows = smA + pair_row(pair) * 128;
  int wt = -1;
  PairWin<SW> win(c, M, M);
  for (; t < ntiles;) {
    if (wt != t) win = PairWin<SW>(c, (long long)(t / ntn) * TC_BM + 2 * pair, M);
    wt = t;
    const int g0 = 9 * r, ch0 = 8 * r;
    // the next run's lines into L1, which its loads need in four dependent rounds: lane
    // l asks for channel l % 8 at the window of lane l & 24, 16 pixels apart
    const int lane = threadIdx.x & 31, ca = ch0 + 8 * SUBS + (lane & 7);
    const float* ahead = reinterpret_cast<const float*>(
        __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(win.base), lane & 24));
    const int ar = __shfl_sync(0xffffffffu, (int)win.rok[0] | (int)win.rok[1] << 1 | (int)win.rok[2] << 2, lane & 24);
    if (ca < c.C) {
#pragma unroll
      for (int p = 0; p < 3; p++)
        if (ar >> p & 1) prefetch_l1(ahead + (long long)ca * c.B * c.H * c.W + p * c.W);
    }
    int kb = -1;  // k-block of the tile whose stage this warp has entered
    uint32_t w0[12], w1[12];  // BF16 words of the two rows: up to three carried over, 9 of two channels
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const int ch = ch0 + 2 * u;
      win.template words<2>(c, ch, [&](int k) { return ch + k < c.C; }, w0 + u, w1 + u);
      const int nc = u < 3 ? 2 : 3;  // whole chunks in hand
#pragma unroll
      for (int k = 0; k < nc; k++) {
        const int g = g0 + 2 * u + k;
        if (g < nchunk) {
          if (kb != g >> 3) {
            if (kb >= 0) warp_leave(&fulla[(kb0 + kb) % TC_STAGES], 8 * kb % 9 <= 1 ? 2 : 1);
            kb = g >> 3;
            const uint32_t n = (uint32_t)(kb0 + kb);
            if (!warp_enter(&empty[n % TC_STAGES], (n / TC_STAGES & 1u) ^ 1u)) return false;
          }
          unsigned char* rp = rows + ((kb0 + kb) % TC_STAGES) * A_STAGE + (((g & 7) ^ (pair & 7)) << 4);
          *reinterpret_cast<uint4*>(rp) = make_uint4(w0[4 * k], w0[4 * k + 1], w0[4 * k + 2], w0[4 * k + 3]);
          *reinterpret_cast<uint4*>(rp + 1024) = make_uint4(w1[4 * k], w1[4 * k + 1], w1[4 * k + 2], w1[4 * k + 3]);
        }
      }
#pragma unroll
      for (int k = 0; k < u + 1 && u < 3; k++) {
        w0[k] = w0[8 + k];
        w1[k] = w1[8 + k];
      }
    }
    warp_leave(&fulla[(kb0 + kb) % TC_STAGES], 8 * kb % 9 <= 1 ? 2 : 1);
    for (r += SUBS; r >= nrun; r -= nrun, kb0 += nk) t += gridDim.x;
  }
  return true;
}

// Gathers the weight gradient's A (M = taps, K = pixels): tile `blockIdx.x` holds
// the 126 taps of 14 channels, a stage 64 pixels of them, M-major (a pixel's taps
// are contiguous, as gather_pairs builds them). Warps 2 q and 2 q + 1 build the
// stages of slot q for 32 pixel pairs: the first 8 channels (chunks 0-8) and the
// last 6 (chunks 9-15, two zero rows). This replaces an im2col matrix that was
// written to and read back from memory (2 x 2 x 9 C bytes per pixel) before a
// TMA-staged GEMM: 64 channels at 128 x 256, batch 32, 372 + 249 -> 293 us.
template <int SW>
__device__ __forceinline__ bool gather_wgrad(const TcConvA& c, int kb0, int nk, unsigned char* smA, uint64_t* empty,
                                             uint64_t* fulla) {
  const int pair = threadIdx.x & 31, grp = (threadIdx.x >> 5) & 1, slot = threadIdx.x >> 6;
  const int row = 2 * pair, ch0 = TC_WG_CH * (int)blockIdx.x + 8 * grp;
  const int nch = min(grp ? TC_WG_CH - 8 : 8, c.C - ch0);
  const long long npix = (long long)c.B * c.Ho * c.Wo;
  static_assert(TC_STAGES == 4, "stage slots and warp pairs");
  for (int i = slot; i < nk; i += TC_STAGES) {
    const PairWin<SW> win(c, (long long)(kb0 + i) * TC_BK + row, npix);
    unsigned char* dst = smA + slot * A_STAGE + row * 128;
    uint32_t w0[20], w1[20];  // as in gather_pairs
#pragma unroll
    for (int half = 0; half < 2; half++) {
      win.template words<4>(c, ch0 + 4 * half, [&](int u) { return 4 * half + u < nch; }, w0 + 2 * half, w1 + 2 * half);
      if (half == 0 && !warp_enter(&empty[slot], ((uint32_t)(i / TC_STAGES) & 1u) ^ 1u)) return false;
#pragma unroll
      for (int k = 0; k < 4 + half; k++) {
        const int g = 9 * grp + 4 * half + k;  // chunk of the pixel's 16
        if (g < 16) {
          unsigned char* rp = dst + (g >> 3) * (A_STAGE / 2);
          *reinterpret_cast<uint4*>(rp + (((g & 7) ^ (row & 7)) << 4)) =
              make_uint4(w0[4 * k], w0[4 * k + 1], w0[4 * k + 2], w0[4 * k + 3]);
          *reinterpret_cast<uint4*>(rp + 128 + (((g & 7) ^ ((row & 7) + 1)) << 4)) =
              make_uint4(w1[4 * k], w1[4 * k + 1], w1[4 * k + 2], w1[4 * k + 3]);
        }
      }
      if (half == 0) {  // words 16, 17 open the fifth chunk
        w0[0] = w0[16];
        w0[1] = w0[17];
        w1[0] = w1[16];
        w1[1] = w1[17];
      }
    }
    warp_leave(&fulla[slot], 1);
  }
  return true;
}

template <int CONV>
__global__ void __launch_bounds__(TcRoles<CONV>::THREADS, TcRoles<CONV>::CTAS)
    k_tc_gemm(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, const TcArgs a,
              const TcConvA conv) {
  using R = TcRoles<CONV>;
  extern __shared__ unsigned char tc_smem_raw[];
  __shared__ uint64_t full[TC_STAGES], empty[TC_STAGES], fulla[TC_STAGES], accb, issued;
  __shared__ uint32_t tmem_slot;
  __shared__ int err, armed;
  // the swizzled tiles need 1024-byte alignment
  const uint32_t raw = smem_u32(tc_smem_raw);
  unsigned char* smA = tc_smem_raw + ((1024u - (raw & 1023u)) & 1023u);
  const int B_STAGE = a.BN * TC_BK * 2;
  unsigned char* smB = smA + (CONV ? TC_STAGES : a.stages) * A_STAGE;
  int2* tab = nullptr;
  if (CONV == 1) {  // after the stages: a.nkb k-blocks of (offset, tap bit) entries
    const int K9 = 9 * conv.C, len = a.nkb * TC_BK;
    tab = reinterpret_cast<int2*>(smB + TC_STAGES * a.BN * TC_BK * 2);
    const int plane = conv.B * conv.H * conv.W;
    for (int k = threadIdx.x; k < len; k += blockDim.x) {
      const int ch = k / 9, t = k - 9 * ch, p = t / 3, q = t - 3 * p;
      tab[k] = k < K9 ? make_int2(ch * plane + p * conv.W + q, 1 << t) : make_int2(0, 1 << 9);
    }
  }

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long m0 = (long long)blockIdx.x * R::BM;
  const int n0 = blockIdx.y * a.BN;
  const int kb0 = blockIdx.z * a.kbps;
  const int nk = min(a.nkb - kb0, a.kbps);

  if (threadIdx.x == 0) {
    for (int s = 0; s < TC_STAGES; s++) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
      mbar_init(&fulla[s], R::ARRIVE);  // CONV: one arrival per gathering warp of the stage
    }
    mbar_init(&accb, 1);
    mbar_init(&issued, 1);
    err = armed = 0;
    fence_mbar_init();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(a.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp == R::B_WARP && lane == 0) {
    // TMA producer: A and B, or B alone when A is gathered
    int i = 0;
    for (; i < nk; i++) {
      const int s = i % TC_STAGES;
      const uint32_t ph = (uint32_t)(i / TC_STAGES) & 1u;
      if (!mbar_wait(&empty[s], ph ^ 1u)) {
        err = 1;
        break;
      }
      mbar_expect_tx(&full[s], (uint32_t)((CONV ? 0 : A_STAGE) + B_STAGE));
      if (!CONV) tma_2d(smA + s * A_STAGE, &ta, (kb0 + i) * TC_BK, (int)m0, &full[s]);
      tma_2d(smB + s * B_STAGE, &tb, (kb0 + i) * TC_BK, n0, &full[s]);
    }
    armed = i;
  } else if (warp == R::MMA_WARP && lane == 0) {
    // MMA issuer
    const int ni = (int)min((uint32_t)nk, a.issue_limit);
    int i = 0;
    for (; i < ni; i++) {
      const int s = i % TC_STAGES;
      const uint32_t ph = (uint32_t)(i / TC_STAGES) & 1u;
      if (!mbar_wait(&full[s], ph) || (CONV && !mbar_wait(&fulla[s], ph))) break;
      tc_fence_after();
      const uint64_t ad = R::WG ? sdesc_sw128_mn(smem_u32(smA + s * A_STAGE), A_STAGE / 2)
                                : sdesc_sw128(smem_u32(smA + s * A_STAGE));
      const uint64_t bd = sdesc_sw128(smem_u32(smB + s * B_STAGE));
#pragma unroll
      for (int kk = 0; kk < TC_BK / 16; kk++)  // 16 values of K per MMA: 32 bytes, or 16 rows of an M-major A
        tc_mma(tmem, ad + (R::WG ? 128 : 2) * kk, bd + 2 * kk, a.idesc, (uint32_t)(i | kk));
      tc_commit(&empty[s]);
    }
    if (i < nk) {
      err = 1;
      __threadfence_block();  // seen by the epilogue with the commit
    }
    tc_commit(&accb);
  } else if (R::WG && (int)threadIdx.x < R::GATHER) {
    if (!gather_wgrad<CONV == 3 ? 2 : 1>(conv, kb0, nk, smA, empty, fulla)) err = 1;
  } else if (CONV == 1 && (int)threadIdx.x < R::GATHER) {
    // A gatherers: half threadIdx.x / 128 of row threadIdx.x % 128 of every stage tile
    const int row = threadIdx.x % TC_BM, half = threadIdx.x / TC_BM;
    const GatherRow g = gather_row(conv, m0 + row, a.M);
    // the loads of k-block i + 1 are issued before block i is converted and stored
    float vn[GATHER_K];
    if (nk > 0) gather_load(conv, g, tab, kb0, half, vn);
    for (int i = 0; i < nk; i++) {
      const int s = i % TC_STAGES;
      const uint32_t ph = (uint32_t)(i / TC_STAGES) & 1u;
      float v[GATHER_K];
#pragma unroll
      for (int kk = 0; kk < GATHER_K; kk++) v[kk] = vn[kk];
      if (i + 1 < nk) gather_load(conv, g, tab, kb0 + i + 1, half, vn);
      if (!warp_enter(&empty[s], ph ^ 1u)) {
        err = 1;
        break;
      }
      gather_store(v, row, half, smA + s * A_STAGE);
      warp_leave(&fulla[s], 1);
    }
  }
  __syncwarp();

  // epilogue (warps 0-3): TMEM lane = tile row m, column = n
  if (warp < 4) {
    const bool ok = mbar_wait(&accb, 0);
    tc_fence_after();
    __syncwarp();
    if (!ok) err = 1;
    const int row = warp * 32 + lane;
    const long long m = m0 + row;
    float* outp = a.out + (long long)blockIdx.z * a.split_stride;
    const bool mine = row < R::BM && m < a.M;
    const bool bad = __any_sync(0xffffffffu, !ok || err);
    if (bad && mine) nan_rows(a, outp, m, n0);
    for (int c0 = 0; c0 < (bad ? 0 : a.BN); c0 += 16) {
      uint32_t r[16];
      tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, r);
      if (mine) {
#pragma unroll
        for (int j = 0; j < 16; j++) {
          const int n = n0 + c0 + j;
          if (n < a.N) {
            float v = __uint_as_float(r[j]);
            if (a.bias) v += a.bias[n];
            if (a.relu) v = fmaxf(v, 0.f);
            outp[(long long)n * a.ldo + m] = v;
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (err) {
    if (threadIdx.x == 0) atomicOr(a.status, ST_TIMEOUT);
    drain(warp == R::MMA_WARP && lane == 0, warp == R::B_WARP && lane == 0, full, armed, &issued);
    __syncthreads();
  }
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.tmem_cols) : "memory");
}

// The forward and stride-1 data-gradient products of a layer whose outputs come in
// pairs: persistent CTAs walk the 128-pixel tiles, and each role runs ahead through
// the stage ring and two TMEM accumulators without waiting for the others' tiles:
//   warps 0-7 gather A, warp 8 loads B by TMA, warp 9 issues the MMAs, warps 10-13
//   drain the accumulator of the tile before (TMEM lane quarter = warp mod 4).
// One tile per CTA (8192 of them for 32 images of 128 x 256) paid the set-up, the
// last MMAs and the epilogue with its gather warps idle.
constexpr int CP_SUBS = 4;  // groups of two gathering warps
template <int SW>
__global__ void __launch_bounds__(64 * CP_SUBS + 192, 2)
    k_conv_pairs(const __grid_constant__ CUtensorMap tb, const TcArgs a, const TcConvA conv, int ntn, int ntiles) {
  constexpr int GW = 2 * CP_SUBS;  // gathering warps
  extern __shared__ unsigned char tc_smem_raw[];
  __shared__ uint64_t full[TC_STAGES], empty[TC_STAGES], fulla[TC_STAGES], accf[2], acce[2], issued;
  __shared__ uint32_t tmem_slot;
  __shared__ int err, armed;
  const uint32_t raw = smem_u32(tc_smem_raw);
  unsigned char* smA = tc_smem_raw + ((1024u - (raw & 1023u)) & 1023u);
  const int B_STAGE = a.BN * TC_BK * 2;
  unsigned char* smB = smA + TC_STAGES * A_STAGE;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nk = a.nkb;
  if (threadIdx.x == 0) {
    for (int s = 0; s < TC_STAGES; s++) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
      mbar_init(&fulla[s], 4);  // two warps of two runs
    }
    for (int s = 0; s < 2; s++) {
      mbar_init(&accf[s], 1);
      mbar_init(&acce[s], 4);  // one arrival per epilogue warp
    }
    mbar_init(&issued, 1);
    err = armed = 0;
    fence_mbar_init();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(a.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot, acc_stride = a.tmem_cols / 2;
  volatile int* verr = &err;

  if (warp < GW) {
    if (!gather_pairs<SW, CP_SUBS>(conv, a.M, nk, ntn, ntiles, smA, empty, fulla)) *verr = 1;
  } else if (warp == GW) {
    if (lane == 0) {
      int kb = 0;
      for (int t = blockIdx.x; t < ntiles && !*verr; t += gridDim.x)
        for (int i = 0; i < nk; i++, kb++) {
          const int s = kb % TC_STAGES;
          if (!mbar_wait(&empty[s], ((uint32_t)(kb / TC_STAGES) & 1u) ^ 1u)) {
            *verr = 1;
            break;
          }
          mbar_expect_tx(&full[s], (uint32_t)B_STAGE);
          tma_2d(smB + s * B_STAGE, &tb, i * TC_BK, (t % ntn) * a.BN, &full[s]);
        }
      armed = kb;
    }
  } else if (warp == GW + 1) {
    if (lane == 0) {
      int kb = 0, it = 0;
      for (int t = blockIdx.x; t < ntiles && !*verr; t += gridDim.x, it++) {
        const int b = it & 1;
        if (!mbar_wait(&acce[b], ((uint32_t)(it >> 1) & 1u) ^ 1u)) {
          *verr = 1;
          break;
        }
        tc_fence_after();
        const int ni = (int)min((uint32_t)nk, a.issue_limit - (uint32_t)kb);
        int i = 0;
        for (; i < ni; i++, kb++) {
          const int s = kb % TC_STAGES;
          const uint32_t ph = (uint32_t)(kb / TC_STAGES) & 1u;
          if (!mbar_wait(&full[s], ph) || !mbar_wait(&fulla[s], ph)) break;
          tc_fence_after();
          const uint64_t ad = sdesc_sw128(smem_u32(smA + s * A_STAGE));
          const uint64_t bd = sdesc_sw128(smem_u32(smB + s * B_STAGE));
#pragma unroll
          for (int kk = 0; kk < TC_BK / 16; kk++)
            tc_mma(tmem + b * acc_stride, ad + 2 * kk, bd + 2 * kk, a.idesc, (uint32_t)(i | kk));
          tc_commit(&empty[s]);
        }
        if (i < nk) {
          *verr = 1;
          __threadfence_block();  // seen by the epilogue with the commit
        }
        tc_commit(&accf[b]);
      }
    }
  } else {
    // epilogue: TMEM lane = tile row, column = n
    const int quarter = warp & 3, row = quarter * 32 + lane;
    int it = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, it++) {
      const int b = it & 1;
      const bool ok = !*verr && mbar_wait(&accf[b], (uint32_t)(it >> 1) & 1u);
      tc_fence_after();
      __syncwarp();
      if (!ok) *verr = 1;
      const bool bad = __any_sync(0xffffffffu, !ok || *verr);
      const long long m = (long long)(t / ntn) * TC_BM + row_pixel(row);
      const int n0 = (t % ntn) * a.BN;
      if (bad && m < a.M) nan_rows(a, a.out, m, n0);
      for (int c0 = 0; c0 < (bad ? 0 : a.BN); c0 += 16) {
        uint32_t r[16];
        tmem_ld16(tmem + b * acc_stride + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c0, r);
        if (m < a.M) {
#pragma unroll
          for (int j = 0; j < 16; j++) {
            const int n = n0 + c0 + j;
            if (n < a.N) {
              float v = __uint_as_float(r[j]);
              if (a.bias) v += a.bias[n];
              if (a.relu) v = fmaxf(v, 0.f);
                a.out[(long long)n * a.ldo + m] = v;
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acce[b]);
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (err) {
    if (threadIdx.x == 0) atomicOr(a.status, ST_TIMEOUT);
    drain(warp == GW + 1 && lane == 0, warp == GW && lane == 0, full, armed, &issued);
    __syncthreads();
  }
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.tmem_cols) : "memory");
}

bool encode_bf16_sw128(CUtensorMap* map, const void* base, long long inner, long long rows, long long ld_elems,
                       int box_rows) {
  tma_host::EncodeTiled fn = tma_host::encoder();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld_elems * 2};
  const cuuint32_t box[2] = {(cuuint32_t)TC_BK, (cuuint32_t)box_rows};
  const cuuint32_t es[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// Multiply-shift constants for floor(n / d), n < 2^31 (Granlund & Montgomery,
// "Division by invariant integers using multiplication", 1994): l = ceil(log2 d),
// m = ceil(2^(32+l) / d), floor(n / d) = (n m) >> (32 + l).
static void div_consts(uint32_t d, unsigned long long* m, uint32_t* s) {
  uint32_t l = 0;
  while ((1ull << l) < d) l++;
  *s = 32 + l;
  *m = ((1ull << *s) + d - 1) / d;
}

TcConvA tc_conv_a(const float* x, int C, int B, int H, int W, int sh, int sw) {
  TcConvA c;
  c.x = x;
  c.C = C;
  c.B = B;
  c.H = H;
  c.W = W;
  c.sh = sh;
  c.sw = sw;
  c.Ho = (H - 1) / sh + 1;
  c.Wo = (W - 1) / sw + 1;
  div_consts((uint32_t)c.Wo, &c.wo_m, &c.wo_s);
  div_consts((uint32_t)c.Ho, &c.ho_m, &c.ho_s);
  return c;
}

int tc_conv_pairs(const TcConvA& c) {
  if (c.sw == 1 && c.W % 2 == 0 && (uintptr_t)c.x % 8 == 0) return 1;
  if (c.sw == 2 && c.W % 4 == 0 && (uintptr_t)c.x % 16 == 0) return 2;
  return 0;
}

int tc_split_count(long long K, int want) {
  const long long nkb = tc_kblocks(K);
  if (want < 1) want = 1;
  const long long kbps = (nkb + want - 1) / want;
  return (int)((nkb + kbps - 1) / kbps);
}

namespace {
// Per device: the SM count, and the dynamic shared memory that each kernel may be
// launched with, raised once to all that a CTA can have. The attribute belongs to the
// kernel, not to a launch: set to each launch's own size, one thread's smaller product
// lowers it between another thread's set and launch, which then fails.
enum { K_TMA, K_TABLE, K_WG1, K_WG2, K_PAIRS1, K_PAIRS2, TC_KERNELS };
struct TcDev {
  bool ready = false;
  int sms = 0, smem[TC_KERNELS];
};
std::mutex g_tc_mu;
TcDev g_tc[64];

template <typename K>
cudaError_t tc_setup(K kern, int optin, int* smem) {
  cudaFuncAttributes at;
  cudaError_t e = cudaFuncGetAttributes(&at, kern);
  if (e != cudaSuccess) return e;
  *smem = optin - (int)at.sharedSizeBytes;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, *smem);
}

// The current device's entry, set up at its first use; `again` repeats that (a new
// handle: the device may have been reset since).
cudaError_t tc_device(const TcDev** out, bool again = false) {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_tc_mu);
  *out = &g_tc[dev];
  if (g_tc[dev].ready && !again) return cudaSuccess;
  TcDev d;
  if ((e = cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
  if ((e = tc_setup(k_tc_gemm<0>, optin, &d.smem[K_TMA])) != cudaSuccess) return e;
  if ((e = tc_setup(k_tc_gemm<1>, optin, &d.smem[K_TABLE])) != cudaSuccess) return e;
  if ((e = tc_setup(k_tc_gemm<2>, optin, &d.smem[K_WG1])) != cudaSuccess) return e;
  if ((e = tc_setup(k_tc_gemm<3>, optin, &d.smem[K_WG2])) != cudaSuccess) return e;
  if ((e = tc_setup(k_conv_pairs<1>, optin, &d.smem[K_PAIRS1])) != cudaSuccess) return e;
  if ((e = tc_setup(k_conv_pairs<2>, optin, &d.smem[K_PAIRS2])) != cudaSuccess) return e;
  d.ready = true;
  if (!g_tc[dev].ready) g_tc[dev] = d;  // others may be reading it
  return cudaSuccess;
}

// Launch of k_conv_pairs: its tiles, and two CTAs per SM while two stage rings fit in
// shared memory (227 KB) and four accumulators in TMEM (512 columns), else one.
int pairs_smem(const TcArgs& a) { return TC_STAGES * (A_STAGE + a.BN * TC_BK * 2) + 1024; }
int pairs_per_sm(const TcArgs& a) { return pairs_smem(a) <= 112 * 1024 && a.tmem_cols <= 128 ? 2 : 1; }
long long pairs_tiles(const TcArgs& a) { return (a.M + TC_BM - 1) / TC_BM * ((a.N + a.BN - 1) / a.BN); }

// Whether a layer of C channels whose outputs come in pairs goes to k_conv_pairs rather
// than to the tap table. A run of 8 channels is four load rounds one after the other in two
// warps, so the persistent kernel pays where a CTA has several tiles, whose runs the warp
// groups share, or a tile has enough runs; with one tile a CTA the table, all of whose
// threads load all taps of a k-block at once, has the shorter chain. us, pairs / table:
//   100 tiles, 16 columns (96): 8 channels 6.3 / 5.5 (10.6 / 10.0), 9: 8.0 / 7.5 (12.4 / 11.7),
//     24: 7.3 / 7.3 (11.7 / 11.6), 40: 8.7 / 8.7 (12.7 / 12.7); 64 tiles of 64 columns, 128 channels: 17.2 / 20.3
//   280 tiles, 16 columns, two CTAs an SM: 8: 7.5 / 7.1, 9: 10.0 / 9.3, 12: 8.1 / 8.4, 24: 8.3 / 9.8
//   380 tiles, 144 columns: 8: 28.1 / 30.9, 9: 30.7 / 33.0, 24: 29.7 / 36.5
// With fewer than 8 channels most of a run would be padding.
bool pairs_pay(const TcArgs& a, int C, int sms) {
  const long long t = pairs_tiles(a);
  if (t <= sms) return C >= 32;
  return C >= (t <= (long long)sms * pairs_per_sm(a) ? 12 : 8);
}

cudaError_t conv_pairs(const TcConvA& c, const CUtensorMap& tb, TcArgs a, int pairs, const TcDev* dev, cudaStream_t st) {
  const int smem = pairs_smem(a), per_sm = pairs_per_sm(a);
  const long long ntn = (a.N + a.BN - 1) / a.BN, ntiles = pairs_tiles(a);
  a.tmem_cols *= 2;
  if (ntiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  if (smem > dev->smem[pairs == 1 ? K_PAIRS1 : K_PAIRS2]) return cudaErrorInvalidValue;
  auto kern = pairs == 1 ? k_conv_pairs<1> : k_conv_pairs<2>;
  const int grid = (int)std::min<long long>(ntiles, (long long)dev->sms * per_sm);
  kern<<<grid, 64 * CP_SUBS + 192, smem, st>>>(tb, a, c, (int)ntn, (int)ntiles);
  return cudaGetLastError();
}
}  // namespace

cudaError_t tc_gemm_init() {
  const TcDev* dev;
  return tc_device(&dev, true);
}

cudaError_t tc_gemm(const TcGemm& g, cudaStream_t st) {
  const bool conv = g.conv != nullptr;
  if ((!conv && !g.A) || !g.B || !g.out || !g.status || g.M < 1 || g.N < 1 || g.K < 1 || g.splits < 1)
    return cudaErrorInvalidValue;
  if (g.ldb % 8 || g.ldb < g.K || ((uintptr_t)g.B & 15)) return cudaErrorInvalidValue;
  if (!conv && (g.lda % 8 || g.lda < g.K || ((uintptr_t)g.A & 15))) return cudaErrorInvalidValue;
  if (conv) {  // the gathered operand must be the one the sizes describe
    const TcConvA& c = *g.conv;
    const long long npix = (long long)c.B * c.Ho * c.Wo, k9 = 9LL * c.C;
    if (!c.x || (g.wgrad ? npix != g.K || k9 != g.M : npix != g.M || k9 != g.K)) return cudaErrorInvalidValue;
    if (g.wgrad && !tc_conv_pairs(c)) return cudaErrorInvalidValue;
  }
  if (g.M > 0x7fffff00LL || g.N > 0x7fffff00) return cudaErrorInvalidValue;
  // columns shared evenly between the fewest tiles of at most 256 (288 as 2 x 144)
  const int ntn = (g.N + 255) / 256, BN = ((g.N + ntn - 1) / ntn + 15) / 16 * 16;
  const long long nkb = tc_kblocks(g.K);
  const long long kbps = (nkb + g.splits - 1) / g.splits;
  const int splits = (int)((nkb + kbps - 1) / kbps);
  uint32_t cols = 32;
  while ((int)cols < BN) cols <<= 1;
  TcArgs a;
  a.M = g.M;
  a.N = g.N;
  a.BN = BN;
  a.nkb = (int)nkb;
  a.kbps = (int)kbps;
  a.out = g.out;
  a.ldo = g.ldo;
  a.split_stride = g.split_stride;
  a.bias = g.bias;
  a.relu = g.relu;
  a.status = g.status;
  a.issue_limit = g.issue_limit < 0 ? ~0u : (uint32_t)g.issue_limit;
  // instruction descriptor, kind::f16: D FP32 (bits 4-5 = 1), A and B BF16
  // (bits 7-9 = 1, 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at bit 24
  a.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(TC_BM >> 4) << 24);
  a.tmem_cols = cols;
  CUtensorMap ta, tb;
  if (!encode_bf16_sw128(&tb, g.B, g.K, g.N, g.ldb, BN)) return cudaErrorInvalidValue;
  if (conv) ta = tb;  // unused: A is gathered
  else if (!encode_bf16_sw128(&ta, g.A, g.K, g.M, g.lda, TC_BM)) return cudaErrorInvalidValue;
  const TcDev* dev;
  const cudaError_t e = tc_device(&dev);
  if (e != cudaSuccess) return e;
  int kind = 0, bm = TC_BM;
  if (conv) {
    const int pairs = tc_conv_pairs(*g.conv);
    kind = 1;
    if (g.wgrad) {
      kind = 1 + pairs;
      bm = TC_WG_ROWS;
      a.idesc |= 1u << 15;  // A is M-major
    } else if (pairs && splits == 1 && pairs_pay(a, g.conv->C, dev->sms)) {
      return conv_pairs(*g.conv, tb, a, pairs, dev, st);
    }
  }
  // Products of few k-blocks (a strided layer's data gradient has one to four) are bound
  // by their epilogue: with no more stages than k-blocks several CTAs share an SM and one
  // tile's epilogue covers another's loads; as many as TMEM's 512 columns hold, so that
  // no allocation waits. Batch of 32, four strided layers (288 columns also as 2 x 144
  // instead of 256 + 32): 360 -> 258 us.
  a.stages = kind == 0 ? (int)std::min<long long>(TC_STAGES, a.kbps) : TC_STAGES;
  int smem = a.stages * (A_STAGE + BN * TC_BK * 2) + 1024 + (kind == 1 ? (int)nkb * TC_BK * 8 : 0);
  if (kind == 0) smem = std::max(smem, (int)(SM_SMEM / (512 / a.tmem_cols + 1)));
  const dim3 grid((unsigned)((g.M + bm - 1) / bm), (unsigned)((g.N + BN - 1) / BN), (unsigned)splits);
  TcConvA c{};
  if (conv) c = *g.conv;
  auto kern = kind == 0 ? k_tc_gemm<0> : kind == 1 ? k_tc_gemm<1> : kind == 2 ? k_tc_gemm<2> : k_tc_gemm<3>;
  if (smem > dev->smem[K_TMA + kind]) return cudaErrorInvalidValue;
  kern<<<grid, conv ? TcRoles<1>::THREADS : TcRoles<0>::THREADS, smem, st>>>(ta, tb, a, c);
  return cudaGetLastError();
}

}  // namespace fwi
