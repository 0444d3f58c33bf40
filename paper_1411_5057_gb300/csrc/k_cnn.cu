// Learned warm start: a 6-layer 3x3 CNN (3 -> 32 -> 32 -> 32 -> 32 -> 32 -> 2,
// ReLU between layers) that maps [Re A^H b, Im A^H b, mask] to a correction,
// x1 = A^H b + CNN(.).  BF16 weights and activations (NHWC), FP32 accumulation
// on the tensor cores, FP32 master weights and Adam.
//
// Forward and data-gradient convolutions run on tcgen05 (TMEM accumulators,
// k_conv3x3_tc) when n is a multiple of 128; otherwise, and for the weight
// gradient, on mma.m16n8k16.  The mma.sync form is an implicit GEMM per tile
// of 8 x 32 output pixels: the input
// tile with a one-pixel halo sits in shared memory; each of the 9 taps is a
// shifted view of it (the A operand, pixels x input channels) times the tap's
// weights (input x output channels).  The same kernel runs the backward data
// pass with the taps flipped and the channel roles swapped; the weight
// gradient sums X[p + tap]^T dZ[p] over all pixels with per-CTA partials and a
// fixed-order reduction (deterministic).
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include <cuda_bf16.h>

#include "cnn_index.h"
#include "firls.h"
#include "firls_common.cuh"
#include "per_device.h"

using namespace firls;

namespace {

constexpr int NL = 6;
constexpr int CH[NL + 1] = {3, 32, 32, 32, 32, 32, 2};
constexpr int CINP[NL] = {16, 32, 32, 32, 32, 32};   // padded input channels
constexpr int COUTP[NL] = {32, 32, 32, 32, 32, 16};  // padded output channels
constexpr int TH = 8, TW = 32;                       // output tile
constexpr int HH = TH + 2, HW = TW + 2;              // halo tile
constexpr int CONV_THREADS = 256;
constexpr int WG_CTAS = 304;                         // weight-gradient partials: two CTAs per SM

FI uint32_t ld_u32(const __nv_bfloat16* p) { return *reinterpret_cast<const uint32_t*>(p); }

FI void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

enum { MODE_HIDDEN = 0, MODE_LAST = 1, MODE_DGRAD = 2 };

// in:  bf16 [B][n][n][CIN]; wt: bf16 [9][COUT][CIN] (tap, out, in); bias f32 [COUT]
// HIDDEN: out bf16 [B][n][n][COUT] = relu(conv + bias)
// LAST:   x1 complex64 = atb + (conv + bias)[0..1]
// DGRAD:  out bf16 [B][n][n][COUT] = conv (no bias) * (gate > 0), gate bf16 [..][COUT]
template <int CIN, int COUT, int MODE>
__global__ void __launch_bounds__(CONV_THREADS) k_conv3x3(int n, const __nv_bfloat16* __restrict__ in,
                                                          const __nv_bfloat16* __restrict__ wt,
                                                          const float* __restrict__ bias,
                                                          __nv_bfloat16* __restrict__ out,
                                                          const __nv_bfloat16* __restrict__ gate,
                                                          const float2* __restrict__ atb, float2* __restrict__ x1) {
  constexpr int PS = CIN + 8;   // padded pixel stride (bf16) in shared memory
  constexpr int WS = CIN + 8;   // padded weight row stride
  constexpr int NT = COUT / 8;  // n-tiles
  extern __shared__ __align__(16) unsigned char smem[];
  __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(smem);  // [HH*HW][PS]
  __nv_bfloat16* ws = xs + HH * HW * PS;                        // [9*COUT][WS]
  const int tiles_x = n / TW;
  const int ty0 = (blockIdx.x / tiles_x) * TH, tx0 = (blockIdx.x % tiles_x) * TW;
  const int img = blockIdx.y;
  const size_t ibase = (size_t)img * n * n;
  // halo tile, 16-byte chunks
  constexpr int CPP = CIN / 8;
  for (int idx = threadIdx.x; idx < HH * HW * CPP; idx += blockDim.x) {
    const int px = idx / CPP, ch = idx % CPP;
    const int y = ty0 - 1 + px / HW, x = tx0 - 1 + px % HW;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (y >= 0 && y < n && x >= 0 && x < n)
      v = reinterpret_cast<const uint4*>(in + (ibase + (size_t)y * n + x) * CIN)[ch];
    *reinterpret_cast<uint4*>(xs + px * PS + ch * 8) = v;
  }
  for (int idx = threadIdx.x; idx < 9 * COUT * CPP; idx += blockDim.x) {
    const int row = idx / CPP, ch = idx % CPP;
    *reinterpret_cast<uint4*>(ws + row * WS + ch * 8) = reinterpret_cast<const uint4*>(wt + (size_t)row * CIN)[ch];
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, tg = lane & 3;
  float acc[2][NT][4];
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[mt][j][e] = 0.f;
#pragma unroll
  for (int t = 0; t < 9; ++t) {
    const int dy = t / 3, dx = t % 3;
#pragma unroll
    for (int kc = 0; kc < CIN / 16; ++kc) {
      const int c0 = kc * 16 + 2 * tg;
      uint32_t a[2][4];
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        const int p0 = (warp + dy) * HW + mt * 16 + g + dx;
        a[mt][0] = ld_u32(xs + p0 * PS + c0);
        a[mt][1] = ld_u32(xs + (p0 + 8) * PS + c0);
        a[mt][2] = ld_u32(xs + p0 * PS + c0 + 8);
        a[mt][3] = ld_u32(xs + (p0 + 8) * PS + c0 + 8);
      }
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const __nv_bfloat16* wr = ws + (t * COUT + j * 8 + g) * WS + c0;
        const uint32_t b0 = ld_u32(wr), b1 = ld_u32(wr + 8);
        mma_bf16(acc[0][j], a[0], b0, b1);
        mma_bf16(acc[1][j], a[1], b0, b1);
      }
    }
  }
  // epilogue: acc[mt][j][e] -> pixel (warp, mt*16 + g + 8*(e>>1)), channel j*8 + 2*tg + (e&1)
#pragma unroll
  for (int mt = 0; mt < 2; ++mt) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int y = ty0 + warp, x = tx0 + mt * 16 + g + 8 * h;
      const size_t p = ibase + (size_t)y * n + x;
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const int co = j * 8 + 2 * tg;
        float v0 = acc[mt][j][2 * h], v1 = acc[mt][j][2 * h + 1];
        if (MODE == MODE_LAST) {
          if (j == 0 && tg == 0) {  // channels 0, 1 = Re, Im of the correction
            const float2 ab = atb[p];
            x1[p] = make_float2(ab.x + v0 + bias[0], ab.y + v1 + bias[1]);
          }
        } else {
          if (MODE == MODE_HIDDEN) {
            v0 = fmaxf(v0 + bias[co], 0.f);
            v1 = fmaxf(v1 + bias[co + 1], 0.f);
          } else {
            const __nv_bfloat162 gt = *reinterpret_cast<const __nv_bfloat162*>(gate + p * COUT + co);
            if (!(__bfloat162float(gt.x) > 0.f)) v0 = 0.f;
            if (!(__bfloat162float(gt.y) > 0.f)) v1 = 0.f;
          }
          *reinterpret_cast<__nv_bfloat162*>(out + p * COUT + co) = __floats2bfloat162_rn(v0, v1);
        }
      }
    }
  }
}

template <int CIN, int COUT> constexpr int conv_smem() { return (HH * HW * (CIN + 8) + 9 * COUT * (CIN + 8)) * 2; }

// ---- the same convolution on the 5th-generation tensor cores (tcgen05) ----
// Tiles of TC_R image rows x TC_W pixels.  Per output row r the GEMM
// D_r[pixel][co] = sum_tap sum_ci X[row r + dy][pixel + dx][ci] W[tap][co][ci]
// runs as 9 * CIN/16 tcgen05.mma (M = 128 pixels, N = COUT, K = 16) with its
// FP32 accumulator in TMEM (columns 32 r ..).  Operands sit in shared memory
// in the canonical K-major layout without swizzle: 8-channel planes of
// 16-byte pixel (or weight-row) records, so the A operand of tap (dy, dx) is
// the halo row r + dy starting at pixel dx: core matrices 128 bytes apart
// along M (SBO), planes one plane apart along K (LBO).
//
// One persistent CTA per SM walks the tiles with the weights resident, its
// warps in three roles, so that a tile's copies, the next one's products and
// the one's before it results run at the same time:
//   warps 5-8   fill a ring of TC_STAGES tiles (asynchronous 16-byte copies),
//   warp 4     one thread issues a tile's MMAs into one of TC_BUFS TMEM buffers,
//   warps 0-3  read a finished buffer (tcgen05.ld), apply bias and ReLU, the last
//              layer's correction or the ReLU gate (both fetched before the
//              products are done), and store: a warp's 32 pixels of a row are
//              2 KB in a row of the image, staged in shared memory and sent as
//              one bulk copy (16-byte stores 64 bytes apart write every sector
//              twice and took longer than the products).
// Handover by mbarriers, every wait bounded.  A CTA per tile that filled,
// multiplied and stored in series took 258 us for 32 x 32 channels at 64 images of
// 256^2 (three CTAs per SM; the weights fetched for each tile); this takes 139 us
// (537 MB read and written: 3.9 TB/s; 168 us with 16-byte stores from registers),
// 16 x 32: 169 -> 127 us, 32 x 16 with the correction: 191 -> 105 us, and at 16
// images 70 -> 41 us (hidden), 80 -> 55 us (gated).  What is left is the chain of
// a tile's four epilogue rows per warp: TMEM read, conversion, staging.
constexpr int TC_W = 128, TC_R = 4, TC_HW = TC_W + 2, TC_HR = TC_R + 2;
constexpr int TC_STAGES = 3, TC_PRODUCERS = 128, TC_THREADS = 128 + 32 + TC_PRODUCERS;
constexpr int TC_BUFS = 4, TC_TMEM = TC_BUFS * TC_R * 32;  // columns

FI unsigned cnn_su32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// tcgen05 shared-memory matrix descriptor: start, leading (K) and stride (M/N)
// byte offsets, fixed version bits 46-48 = 1, no swizzle.  Its low word is the
// start / 16 plus the leading offset, so a shifted operand is an addition to it.
FI uint32_t umma_lo(unsigned addr, unsigned lbo) { return ((addr & 0x3FFFF) >> 4) | ((lbo >> 4) << 16); }
__host__ __device__ constexpr uint32_t umma_hi(unsigned sbo) { return (sbo >> 4) | (1u << 14); }

FI void cnn_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(cnn_su32(bar)) : "memory");
}
// Bounded wait (about a second) for the phase of that parity; every wait of a
// CTA whose waits have run out once gives up after one poll.
FI bool cnn_wait(uint64_t* bar, unsigned parity, const volatile int* abort_flag) {
  for (int it = 0; it < 10000; ++it) {
    unsigned ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok)
                 : "r"(cnn_su32(bar)), "r"(parity), "r"(100000u)
                 : "memory");
    if (ok) return true;
    if (*abort_flag) return false;
  }
  return false;
}

template <int CIN> constexpr int tc_stage_bytes() { return TC_HR * TC_HW * CIN * 2; }
template <int COUT> __host__ __device__ constexpr int tc_row_bytes() { return 32 * COUT * 2; }  // of a warp
template <int CIN, int COUT> constexpr int tc_smem() {
  return TC_STAGES * tc_stage_bytes<CIN>() + 9 * COUT * CIN * 2 + 4 * 2 * tc_row_bytes<COUT>();
}

template <int CIN, int COUT, int MODE>
__global__ void __launch_bounds__(TC_THREADS, 1) k_conv3x3_tc(int n, int tiles, const __nv_bfloat16* __restrict__ in,
                                                              const __nv_bfloat16* __restrict__ wt,
                                                              const float* __restrict__ bias,
                                                              __nv_bfloat16* __restrict__ out,
                                                              const __nv_bfloat16* __restrict__ gate,
                                                              const float2* __restrict__ atb, float2* __restrict__ x1,
                                                              int* __restrict__ err) {
  constexpr int KP = CIN / 8;                  // 8-channel planes
  constexpr int XPL = TC_HR * TC_HW * 16;      // bytes per activation plane
  constexpr int WPL = COUT * 16;               // bytes per weight plane
  constexpr int STAGE = TC_HR * TC_HW * CIN * 2;
  static_assert(COUT % 16 == 0 && COUT <= 32 && CIN % 16 == 0, "tcgen05 conv shape");
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* wsm = smem + TC_STAGES * STAGE;  // [9][KP][COUT][16 B]
  __shared__ uint32_t tmem_base;
  // full: a stage has landed; empty: its MMAs are done; ready: a TMEM buffer
  // holds a tile; drained: it has been read
  __shared__ __align__(8) uint64_t full[TC_STAGES], empty[TC_STAGES], ready[TC_BUFS], drained[TC_BUFS];
  __shared__ volatile int abort_flag;
  const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t >> 5, 0), lane = t & 31;
  const int segs = n / TC_W, per_img = segs * (n / TC_R);
  const int count = ((int)blockIdx.x < tiles) ? (tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  // the tile's image, first row and first pixel
  auto where = [&](int i, int& img, int& y0, int& x0) {
    const int tile = blockIdx.x + i * gridDim.x, r = tile % per_img;
    img = tile / per_img;
    y0 = r / segs * TC_R;
    x0 = r % segs * TC_W;
  };
  for (int idx = t; idx < 9 * COUT * KP; idx += TC_THREADS) {
    const int row = idx / KP, ch = idx % KP;  // row = tap * COUT + co
    const int tap = row / COUT, co = row % COUT;
    *reinterpret_cast<uint4*>(wsm + ((size_t)(tap * KP + ch) * COUT + co) * 16) =
        reinterpret_cast<const uint4*>(wt + (size_t)row * CIN)[ch];
  }
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");  // generic writes -> tensor core reads
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(cnn_su32(&tmem_base)),
                 "r"(TC_TMEM)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  if (t == 0) {
    auto init = [](uint64_t* b, unsigned c) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(cnn_su32(b)), "r"(c) : "memory");
    };
    for (int i = 0; i < TC_STAGES; ++i) {
      init(full + i, TC_PRODUCERS);
      init(empty + i, 1);
    }
    for (int i = 0; i < TC_BUFS; ++i) {
      init(ready + i, 1);
      init(drained + i, 128);
    }
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = tmem_base;
  bool ok = true;

  if (warp > 4) {
    // ============================================================ producers
    const int pt = t - 160;
    // halo rows y0-1 .. y0+TC_R, pixels x0-1 .. x0+TC_W, zero outside the image.
    // A thread copies one 8-channel plane of every (TC_PRODUCERS / KP)-th pixel
    // and steps its coordinates from one to the next.
    constexpr int STEP = TC_PRODUCERS / KP;
    static_assert(STEP < TC_HW, "one row crossed per step");
    const int ch = pt % KP, px0 = pt / KP;
    auto fill = [&](int i) {
      int img, y0, x0;
      where(i, img, y0, x0);
      unsigned dst = cnn_su32(smem + (i % TC_STAGES) * STAGE + ch * XPL + px0 * 16);
      const __nv_bfloat16* src = in + (size_t)img * n * n * CIN + ch * 8;
      int x = x0 - 1 + px0, y = y0 - 1;
      const int xe = x0 - 1 + TC_HW;
#pragma unroll 4
      for (int px = px0; px < TC_HR * TC_HW; px += STEP) {
        const bool inside = (unsigned)y < (unsigned)n && (unsigned)x < (unsigned)n;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst),
                     "l"(src + (inside ? cnn_pixel(y, x, n, CIN) : 0)), "r"(inside ? 16 : 0)
                     : "memory");
        dst += STEP * 16;
        x += STEP;
        if (x >= xe) {
          x -= TC_HW;
          ++y;
        }
      }
    };
    // tile i - 1 is handed over once its copies have landed, tile i's in flight
    for (int i = 0; i <= count && ok; ++i) {
      if (i < count) {
        if (i >= TC_STAGES) ok = cnn_wait(empty + i % TC_STAGES, (i / TC_STAGES - 1) & 1, &abort_flag);
        if (ok) fill(i);
      }
      asm volatile("cp.async.commit_group;\n" ::: "memory");
      if (i > 0) {
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        cnn_arrive(full + (i - 1) % TC_STAGES);
      }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
  } else if (warp == 4) {
    // ============================================================== products
    // D f32, A and B bf16, both K-major, N >> 3 at bit 17, M >> 4 at bit 24
    constexpr uint32_t idesc =
        (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(COUT >> 3) << 17) | ((uint32_t)(TC_W >> 4) << 24);
    // The whole warp runs the loop, so that the descriptors are computed in the
    // uniform datapath, and one elected thread issues: computed by one diverged
    // thread, they took longer than the products.
    uint32_t leader;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(leader));
    const uint32_t bl = umma_lo(cnn_su32(wsm), WPL);
    for (int i = 0; i < count; ++i) {
      const int buf = i % TC_BUFS;
      ok = cnn_wait(full + i % TC_STAGES, (i / TC_STAGES) & 1, &abort_flag);
      if (ok && i >= TC_BUFS) ok = cnn_wait(drained + buf, (i / TC_BUFS - 1) & 1, &abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      const uint32_t al = umma_lo(cnn_su32(smem + (i % TC_STAGES) * STAGE), XPL);
      const uint32_t d0 = tmem + (uint32_t)(buf * TC_R * 32);
#pragma unroll
      for (int r = 0; r < TC_R; ++r) {
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
          const int dy = tap / 3, dx = tap % 3;
#pragma unroll
          for (int kk = 0; kk < CIN / 16; ++kk) {
            asm volatile(
                "{\n .reg .pred p, q;\n .reg .b64 a, b;\n setp.ne.u32 p, %5, 0;\n setp.ne.u32 q, %6, 0;\n"
                " mov.b64 a, {%1, %3};\n mov.b64 b, {%2, %4};\n"
                " @q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %7, p;\n}\n" ::"r"(d0 + r * 32),
                "r"(al + (uint32_t)(2 * kk * XPL + ((r + dy) * TC_HW + dx) * 16) / 16),
                "r"(bl + (uint32_t)((tap * KP + 2 * kk) * WPL) / 16), "r"(umma_hi(128)), "r"(umma_hi(128)),
                "r"(tap + kk > 0 ? 1u : 0u), "r"(leader), "r"(idesc)
                : "memory");
          }
        }
      }
      auto commit = [&](uint64_t* b) {
        asm volatile(
            "{\n .reg .pred q;\n setp.ne.u32 q, %1, 0;\n"
            " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(cnn_su32(b)),
            "r"(leader)
            : "memory");
      };
      commit(empty + i % TC_STAGES);
      commit(ready + buf);
    }
  } else {
    // =============================================================== results
    unsigned char* stage_out = wsm + 9 * COUT * CIN * 2 + warp * 2 * tc_row_bytes<COUT>();
    float bv[COUT];
    if (MODE == MODE_HIDDEN) {
#pragma unroll
      for (int j = 0; j < COUT; ++j) bv[j] = bias[j];
    }
    for (int i = 0; i < count; ++i) {
      int img, y0, x0;
      where(i, img, y0, x0);
      const int buf = i % TC_BUFS;
      // this thread's pixel: row y0 + r, column x0 + 32 warp + lane
      const size_t p0 = (size_t)img * n * n + (size_t)y0 * n + x0 + warp * 32 + lane;
      uint4 gt[TC_R][COUT / 8];
      float2 ab[TC_R];
#pragma unroll
      for (int r = 0; r < TC_R; ++r) {
        if (MODE == MODE_DGRAD) {
#pragma unroll
          for (int q = 0; q < COUT / 8; ++q)
            gt[r][q] = reinterpret_cast<const uint4*>(gate + (p0 + (size_t)r * n) * COUT)[q];
        }
        if (MODE == MODE_LAST) ab[r] = atb[p0 + (size_t)r * n];
      }
      ok = __all_sync(0xffffffffu, cnn_wait(ready + buf, (i / TC_BUFS) & 1, &abort_flag));
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
      for (int r = 0; r < TC_R; ++r) {
        const size_t p = p0 + (size_t)r * n;
        uint32_t v[32];
        const uint32_t ta = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(buf * TC_R * 32 + r * 32);
        if (COUT == 32) {
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,"
              "%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
              : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]),
                "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]),
                "=r"(v[30]), "=r"(v[31])
              : "r"(ta));
        } else {
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
              : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
              : "r"(ta));
        }
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
        if (r + 1 == TC_R) {  // the buffer has been read
          asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
          cnn_arrive(drained + buf);
        }
        if (MODE == MODE_LAST) {
          x1[p] = make_float2(ab[r].x + __uint_as_float(v[0]) + bias[0], ab[r].y + __uint_as_float(v[1]) + bias[1]);
        } else {
          uint32_t pk[COUT / 2];
#pragma unroll
          for (int j = 0; j < COUT / 2; ++j) {
            float a = __uint_as_float(v[2 * j]), b = __uint_as_float(v[2 * j + 1]);
            if (MODE == MODE_HIDDEN) {
              a = fmaxf(a + bv[2 * j], 0.f);
              b = fmaxf(b + bv[2 * j + 1], 0.f);
            } else {  // the gate's BF16 values as FP32
              const uint4 g4 = gt[r][j / 4];
              const uint32_t gw = j % 4 == 0 ? g4.x : j % 4 == 1 ? g4.y : j % 4 == 2 ? g4.z : g4.w;
              if (!(__uint_as_float(gw << 16) > 0.f)) a = 0.f;
              if (!(__uint_as_float(gw & 0xffff0000u) > 0.f)) b = 0.f;
            }
            const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
            pk[j] = *reinterpret_cast<const uint32_t*>(&h);
          }
          // two staging rows per warp: the copy of the row before last has left
          // this one
          unsigned char* row = stage_out + (r & 1) * tc_row_bytes<COUT>();
          if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;\n" ::: "memory");
          __syncwarp();
          uint4* o = reinterpret_cast<uint4*>(row + lane * COUT * 2);
#pragma unroll
          for (int q = 0; q < COUT / 8; ++q) o[q] = make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
          asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n cp.async.bulk.commit_group;\n" ::"l"(
                             out + p * COUT),
                         "r"(cnn_su32(row)), "r"(tc_row_bytes<COUT>())
                         : "memory");
          }
        }
      }
    }
  }
  if (warp < 4 && MODE != MODE_LAST && lane == 0) asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");
  if (!ok) {
    abort_flag = 1;
    if (lane == 0) atomicExch(err, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TC_TMEM) : "memory");
}

// dW[t][ci][co] = sum_p X[p + off(t)][ci] dZ[p][co]; db[co] = sum_p dZ[p][co].
// Per-CTA partials over a strided set of 8 x 32 tiles: pw [cta][9][CIN][COUT],
// pb [cta][COUT].  Pixels are the K dimension of mma.m16n8k16, and both operands
// lie pixel-major in memory: the tiles go to shared memory as they are (16-byte
// asynchronous copies, the next tile's in flight under this one's products), and
// ldmatrix.trans turns them.  A warp owns 16 input and 16 output channels and
// every KS-th group of 16 pixels, for all nine taps: a B fragment serves nine
// taps, an A fragment two products.  db is a product with ones.  Bound by the
// shared-memory reads, about one ldmatrix per two products.  Measured, 16 images
// of 256^2, 32 x 32 channels: 67 us; the form before (element-wise transposed
// copies, operands packed from single values) took 414.
constexpr int WG_THREADS = 256;

FI unsigned wg_su32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
FI void ldsm_x4_trans(uint32_t (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}

template <int CIN, int COUT> struct WgShape {
  static constexpr int XS = CIN * 2 + 16, ZS = COUT * 2 + 16;  // bytes per pixel: rows of a fragment on distinct banks
  static constexpr int STAGE = HH * HW * XS + TH * TW * ZS;
  static constexpr int WM = CIN / 16, WN = COUT / 16, KS = 8 / (WM * WN);
  static constexpr int SUMS = 9 * CIN * COUT * 4;  // reuses the stages
  static constexpr int SMEM = 2 * STAGE > SUMS ? 2 * STAGE : SUMS;
};

template <int CIN, int COUT>
__global__ void __launch_bounds__(WG_THREADS, 2) k_wgrad(int n, int batch, const __nv_bfloat16* __restrict__ x,
                                                         const __nv_bfloat16* __restrict__ dz,
                                                         float* __restrict__ pw, float* __restrict__ pb) {
  using S = WgShape<CIN, COUT>;
  extern __shared__ __align__(16) unsigned char smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int mt = warp % S::WM, nt = warp / S::WM % S::WN, ks = warp / (S::WM * S::WN);
  const int tiles_x = n / TW, per_img = tiles_x * (n / TH), tiles = per_img * batch;
  auto fill = [&](int stage, int tile) {
    if (tile < tiles) {
      unsigned char* xs = smem + stage * S::STAGE;
      unsigned char* zs = xs + HH * HW * S::XS;
      const int img = tile / per_img, r = tile % per_img;
      const int ty0 = (r / tiles_x) * TH, tx0 = (r % tiles_x) * TW;
      const size_t ibase = (size_t)img * n * n;
      for (int i = threadIdx.x; i < HH * HW * (CIN / 8); i += WG_THREADS) {
        const int px = i / (CIN / 8), ch = i % (CIN / 8);
        const int yy = ty0 - 1 + px / HW, xx = tx0 - 1 + px % HW;
        const bool in = yy >= 0 && yy < n && xx >= 0 && xx < n;  // zeros outside the image
        const __nv_bfloat16* src = x + (in ? (ibase + (size_t)yy * n + xx) * CIN + ch * 8 : 0);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(wg_su32(xs + px * S::XS + ch * 16)),
                     "l"(src), "r"(in ? 16 : 0)
                     : "memory");
      }
      for (int i = threadIdx.x; i < TH * TW * (COUT / 8); i += WG_THREADS) {
        const int px = i / (COUT / 8), ch = i % (COUT / 8);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(wg_su32(zs + px * S::ZS + ch * 16)),
                     "l"(dz + (ibase + (size_t)(ty0 + px / TW) * n + tx0 + px % TW) * COUT + ch * 8)
                     : "memory");
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  float acc[9][2][4], bacc[2][4];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      bacc[h][e] = 0.f;
#pragma unroll
      for (int t = 0; t < 9; ++t) acc[t][h][e] = 0.f;
    }
  // this lane's address in an A fragment: matrices 0 and 1 are pixels 0..7 of
  // channels 0..7 and 8..15, matrices 2 and 3 the same of pixels 8..15
  const int fpx = (lane & 7) + ((lane >> 4) & 1) * 8, fch = (lane >> 3) & 1;
  fill(0, blockIdx.x);
  int stage = 0;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, stage ^= 1) {
    fill(stage ^ 1, tile + gridDim.x);
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();
    const unsigned xb = wg_su32(smem + stage * S::STAGE) + mt * 32 + fch * 16;
    // B: matrices 0, 1 are pixels 0..7, 8..15 of the first 8 output channels
    const unsigned zb = wg_su32(smem + stage * S::STAGE + HH * HW * S::XS) + nt * 32 + (lane >> 4) * 16;
    const int bpx = lane & 15;
    for (int kc = ks; kc < TH * TW / 16; kc += S::KS) {
      const int py = kc / (TW / 16), px = kc % (TW / 16) * 16;  // 16 pixels of one tile row
      uint32_t b[4];
      ldsm_x4_trans(b, zb + (py * TW + px + bpx) * S::ZS);
#pragma unroll
      for (int t = 0; t < 9; ++t) {
        uint32_t a[4];
        ldsm_x4_trans(a, xb + ((py + t / 3) * HW + px + t % 3 + fpx) * S::XS);
        mma_bf16(acc[t][0], a, b[0], b[1]);
        mma_bf16(acc[t][1], a, b[2], b[3]);
      }
      if (mt == 0) {
        const uint32_t ones[4] = {0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u};
        mma_bf16(bacc[0], ones, b[0], b[1]);
        mma_bf16(bacc[1], ones, b[2], b[3]);
      }
    }
    __syncthreads();  // the stage may be filled again
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  // the KS pixel groups of each channel block, added in order
  float* sums = reinterpret_cast<float*>(smem);
  __shared__ float bsum[COUT];
  const int g = lane >> 2, tg = lane & 3;
  for (int k = 0; k < S::KS; ++k) {
    if (ks == k) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int ci = mt * 16 + g + 8 * (e >> 1), co = nt * 16 + h * 8 + 2 * tg + (e & 1);
#pragma unroll
          for (int t = 0; t < 9; ++t) {
            float* d = sums + (t * CIN + ci) * COUT + co;
            *d = k == 0 ? acc[t][h][e] : *d + acc[t][h][e];
          }
          if (mt == 0 && g == 0 && e < 2) bsum[co] = k == 0 ? bacc[h][e] : bsum[co] + bacc[h][e];
        }
    }
    __syncthreads();
  }
  float* pwc = pw + (size_t)blockIdx.x * 9 * CIN * COUT;
  for (int i = threadIdx.x; i < 9 * CIN * COUT; i += WG_THREADS) pwc[i] = sums[i];
  if (threadIdx.x < COUT) pb[(size_t)blockIdx.x * COUT + threadIdx.x] = bsum[threadIdx.x];
}

// NHWC bf16 input [B][n][n][16]: Re A^H b, Im A^H b, mask, zeros.
__global__ void k_cnn_input(int total, const float2* __restrict__ atb, const uint8_t* __restrict__ mask,
                            __nv_bfloat16* __restrict__ in) {
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < total; p += gridDim.x * blockDim.x) {
    const float2 a = atb[p];
    __nv_bfloat16 v[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) v[c] = __float2bfloat16(0.f);
    v[0] = __float2bfloat16(a.x);
    v[1] = __float2bfloat16(a.y);
    v[2] = __float2bfloat16(mask[p] ? 1.f : 0.f);
    uint4* o = reinterpret_cast<uint4*>(in + (size_t)p * 16);
    o[0] = *reinterpret_cast<uint4*>(v);
    o[1] = *reinterpret_cast<uint4*>(v + 8);
  }
}

// dOut = 2 (x1 - target) as bf16 [B][n][n][16] (channels 0, 1) and partial
// sums of |x1 - target|^2.
__global__ void k_cnn_loss(int total, const float2* __restrict__ x1, const float2* __restrict__ tgt,
                           __nv_bfloat16* __restrict__ dout, double* __restrict__ part) {
  __shared__ double red[32];
  float acc = 0.f;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < total; p += gridDim.x * blockDim.x) {
    const float2 r = make_float2(x1[p].x - tgt[p].x, x1[p].y - tgt[p].y);
    acc += r.x * r.x + r.y * r.y;
    __nv_bfloat16 v[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) v[c] = __float2bfloat16(0.f);
    v[0] = __float2bfloat16(2.f * r.x);
    v[1] = __float2bfloat16(2.f * r.y);
    uint4* o = reinterpret_cast<uint4*>(dout + (size_t)p * 16);
    o[0] = *reinterpret_cast<uint4*>(v);
    o[1] = *reinterpret_cast<uint4*>(v + 8);
  }
  const double tot = block_sum((double)acc, red);
  if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

// One layer's parameters, gradients and partials, as the update kernel sees them.
struct CnnLayer {
  float *w, *mw, *vw, *gw, *b, *mb, *vb, *gb, *bp;
  __nv_bfloat16 *wf, *wd;
  const float *pw, *pb;
  int cin, cout, cinp, coutp, first;  // first: the layer's first CTA
};
struct CnnLayers {
  CnnLayer l[NL];
};

// The end of a training step for every layer: the gradients (fixed-order sums
// of the per-CTA partials, carried in three floats), Adam (Kingma & Ba) on the
// FP32 masters and the packed BF16 copies.  A CTA takes 32 parameters, 8 threads
// each to fetch and add the partials (coalesced over the parameters).  One launch
// instead of 30, and the sums no longer 296 loads in a row per thread (107 us per
// layer); 43 MB of partials, 49 us with FP64 sums, 21 us with these.
constexpr int UP_PARAMS = 32, UP_PARTS = 8;
__global__ void __launch_bounds__(UP_PARAMS* UP_PARTS) k_cnn_update(CnnLayers layers, int ctas, float lr, float b1,
                                                                    float b2, float eps, float c1, float c2) {
  __shared__ Sum3 red[UP_PARTS][UP_PARAMS];
  int li = NL - 1;
  while (li > 0 && (int)blockIdx.x < layers.l[li].first) --li;
  const CnnLayer& L = layers.l[li];
  const int nw = 9 * L.cin * L.cout;
  const int u = threadIdx.x % UP_PARAMS, k = threadIdx.x / UP_PARAMS;
  const int i = (blockIdx.x - L.first) * UP_PARAMS + u;
  const int t = i / (L.cin * L.cout), ci = (i / L.cout) % L.cin, co = i % L.cout;
  const bool weight = i < nw;
  const size_t stride = weight ? (size_t)9 * L.cinp * L.coutp : (size_t)L.coutp;
  const float* parts = weight ? L.pw + ((size_t)t * L.cinp + ci) * L.coutp + co : L.pb + (i - nw);
  Sum3 s{0.f, 0.f, 0.f};
  if (i < nw + L.cout) {
#pragma unroll 8
    for (int c = k; c < ctas; c += UP_PARTS) s.add(__ldcs(parts + c * stride));
  }
  red[k][u] = s;
  __syncthreads();
  if (k != 0 || i >= nw + L.cout) return;
#pragma unroll
  for (int c = 1; c < UP_PARTS; ++c) s.add(red[c][u]);
  const int q = weight ? i : i - nw;
  float gi = (float)s.value();
  if (!isfinite(gi)) {  // the floats overflowed on the way, or the gradient is not finite: FP64 decides
    double wide = 0.0;
    for (int c = 0; c < ctas; ++c) wide += parts[c * stride];
    gi = (float)wide;
  }
  (weight ? L.gw : L.gb)[q] = gi;
  float* m = weight ? L.mw : L.mb;
  float* v = weight ? L.vw : L.vb;
  float* p = weight ? L.w : L.b;
  const float mi = b1 * m[q] + (1.f - b1) * gi;
  const float vi = b2 * v[q] + (1.f - b2) * gi * gi;
  m[q] = mi;
  v[q] = vi;
  float pi = p[q];
  pi -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  p[q] = pi;
  if (weight) {  // the padding of the packed copies stays zero
    const __nv_bfloat16 h = __float2bfloat16(pi);
    L.wf[((size_t)t * L.coutp + co) * L.cinp + ci] = h;
    L.wd[((size_t)(8 - t) * L.cinp + ci) * L.coutp + co] = h;
  } else {
    L.bp[q] = pi;
  }
}

// Pack FP32 master weights [9][cin][cout] into the bf16 forward layout
// [9][coutp][cinp] and the data-gradient layout [9][cinp][coutp] (taps flipped).
__global__ void k_pack(int cin, int cout, int cinp, int coutp, const float* __restrict__ w,
                       __nv_bfloat16* __restrict__ wf, __nv_bfloat16* __restrict__ wd) {
  const int total = 9 * cinp * coutp;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int t = i / (cinp * coutp), ci = (i / coutp) % cinp, co = i % coutp;
    const float v = (ci < cin && co < cout) ? w[((size_t)t * cin + ci) * cout + co] : 0.f;
    wf[((size_t)t * coutp + co) * cinp + ci] = __float2bfloat16(v);
    if (wd) wd[((size_t)(8 - t) * cinp + ci) * coutp + co] = __float2bfloat16(v);
  }
}

__global__ void k_pad_bias(int cout, int coutp, const float* __restrict__ b, float* __restrict__ bp) {
  const int i = threadIdx.x;
  if (i < coutp) bp[i] = i < cout ? b[i] : 0.f;
}

}  // namespace

struct firls_cnn {
  int n = 0, batch = 0;
  cudaStream_t stream = nullptr;
  std::vector<void*> allocs;
  float *w[NL] = {}, *b[NL] = {}, *bp[NL] = {};           // FP32 master, padded bias
  float *mw[NL] = {}, *vw[NL] = {}, *mb[NL] = {}, *vb[NL] = {};
  float *gw[NL] = {}, *gb[NL] = {};
  __nv_bfloat16 *wf[NL] = {}, *wd[NL] = {};
  __nv_bfloat16* act[NL] = {};  // act[0] input (16 ch), act[l] output of layer l (32 ch)
  __nv_bfloat16 *dza = nullptr, *dzb = nullptr;
  // weight-gradient partials of each layer; the FP32 parameters, gradients and
  // Adam moments of all layers lie in one block each (w, b of layer 0, of layer
  // 1, ...: `params` floats)
  float *pw[NL] = {}, *pb[NL] = {};
  float *pall = nullptr, *gall = nullptr, *mall = nullptr, *vall = nullptr;
  size_t params = 0;
  int wg_ctas = 0;
  int sms = 152;
  double* lpart = nullptr;
  int* err = nullptr;  // set by a tcgen05 convolution whose bounded wait ran out
  int adam_t = 0;
  bool params_set = false;
};

namespace {

template <typename T> firls_status cnn_alloc(firls_cnn* c, T** p, size_t count) {
  void* v = nullptr;
  if (cudaMalloc(&v, count * sizeof(T) + 16) != cudaSuccess) return FIRLS_E_NOMEM;
  c->allocs.push_back(v);
  *p = static_cast<T*>(v);
  return FIRLS_OK;
}

template <int CIN, int COUT, int MODE> void launch_conv(firls_cnn* c, const __nv_bfloat16* in, const __nv_bfloat16* wt,
                                                       const float* bias, __nv_bfloat16* out,
                                                       const __nv_bfloat16* gate, const float2* atb, float2* x1) {
  if (c->n % TC_W == 0 && c->n % TC_R == 0) {  // tcgen05 form
    static PerDeviceOnce tattr;
    tattr.run([] {
      return cudaFuncSetAttribute(k_conv3x3_tc<CIN, COUT, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  tc_smem<CIN, COUT>()) == cudaSuccess;
    });
    const int tiles = (c->n / TC_W) * (c->n / TC_R) * c->batch;
    const int grid = tiles < c->sms ? tiles : c->sms;
    k_conv3x3_tc<CIN, COUT, MODE><<<grid, TC_THREADS, tc_smem<CIN, COUT>(), c->stream>>>(c->n, tiles, in, wt, bias, out,
                                                                                          gate, atb, x1, c->err);
    return;
  }
  static PerDeviceOnce attr;
  attr.run([] {
    return cudaFuncSetAttribute(k_conv3x3<CIN, COUT, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                conv_smem<CIN, COUT>()) == cudaSuccess;
  });
  const dim3 grid((c->n / TW) * (c->n / TH), c->batch);
  k_conv3x3<CIN, COUT, MODE><<<grid, CONV_THREADS, conv_smem<CIN, COUT>(), c->stream>>>(c->n, in, wt, bias, out, gate,
                                                                                         atb, x1);
}

template <int CIN, int COUT> void launch_wgrad(firls_cnn* c, const __nv_bfloat16* x, const __nv_bfloat16* dz, int l) {
  static PerDeviceOnce attr;
  attr.run([] {
    return cudaFuncSetAttribute(k_wgrad<CIN, COUT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                WgShape<CIN, COUT>::SMEM) == cudaSuccess;
  });
  k_wgrad<CIN, COUT><<<c->wg_ctas, WG_THREADS, WgShape<CIN, COUT>::SMEM, c->stream>>>(c->n, c->batch, x, dz, c->pw[l],
                                                                                      c->pb[l]);
}

// Gradients of every layer from the partials, Adam, packed copies.
void update(firls_cnn* c, float lr) {
  CnnLayers layers;
  int ctas = 0;
  for (int l = 0; l < NL; ++l) {
    layers.l[l] = CnnLayer{c->w[l],  c->mw[l], c->vw[l], c->gw[l], c->b[l],  c->mb[l], c->vb[l],  c->gb[l], c->bp[l],
                           c->wf[l], c->wd[l], c->pw[l], c->pb[l], CH[l],    CH[l + 1], CINP[l], COUTP[l], ctas};
    ctas += (9 * CH[l] * CH[l + 1] + CH[l + 1] + UP_PARAMS - 1) / UP_PARAMS;
  }
  c->adam_t += 1;
  const float c1 = 1.f - (float)std::pow(0.9, c->adam_t), c2 = 1.f - (float)std::pow(0.999, c->adam_t);
  k_cnn_update<<<ctas, UP_PARAMS * UP_PARTS, 0, c->stream>>>(layers, c->wg_ctas, lr, 0.9f, 0.999f, 1e-8f, c1, c2);
}

void pack_all(firls_cnn* c) {
  for (int l = 0; l < NL; ++l) {
    k_pack<<<64, 256, 0, c->stream>>>(CH[l], CH[l + 1], CINP[l], COUTP[l], c->w[l], c->wf[l], c->wd[l]);
    k_pad_bias<<<1, 64, 0, c->stream>>>(CH[l + 1], COUTP[l], c->b[l], c->bp[l]);
  }
}

void forward(firls_cnn* c, const float2* atb, const uint8_t* mask, float2* x1) {
  const int total = c->batch * c->n * c->n;
  k_cnn_input<<<1024, 256, 0, c->stream>>>(total, atb, mask, c->act[0]);
  launch_conv<16, 32, MODE_HIDDEN>(c, c->act[0], c->wf[0], c->bp[0], c->act[1], nullptr, nullptr, nullptr);
  for (int l = 1; l < 5; ++l)
    launch_conv<32, 32, MODE_HIDDEN>(c, c->act[l], c->wf[l], c->bp[l], c->act[l + 1], nullptr, nullptr, nullptr);
  launch_conv<32, 16, MODE_LAST>(c, c->act[5], c->wf[5], c->bp[5], nullptr, nullptr, atb, x1);
}

}  // namespace

extern "C" firls_status firls_cnn_create(firls_cnn** out, int n, int batch, void* cuda_stream) {
  if (!out) return FIRLS_E_INVALID_ARG;
  *out = nullptr;
  if (n < TW || n % TW || n % TH || batch < 1 || batch > 65535) return FIRLS_E_SHAPE;
  firls_cnn* c = new firls_cnn();
  c->n = n;
  c->batch = batch;
  c->stream = static_cast<cudaStream_t>(cuda_stream);
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, dev);
  const size_t P = (size_t)batch * n * n;
  firls_status s = FIRLS_OK;
  auto A = [&](auto** p, size_t cnt) {
    if (s == FIRLS_OK) s = cnn_alloc(c, p, cnt);
  };
  for (int l = 0; l < NL; ++l) c->params += (9 * (size_t)CH[l] + 1) * CH[l + 1];
  for (float** v : {&c->pall, &c->gall, &c->mall, &c->vall}) A(v, c->params);
  const long tiles = (long)(n / TW) * (n / TH) * batch;
  c->wg_ctas = tiles < WG_CTAS ? (int)tiles : WG_CTAS;
  for (int l = 0; l < NL; ++l) {
    A(&c->pw[l], (size_t)c->wg_ctas * 9 * CINP[l] * COUTP[l]);
    A(&c->pb[l], (size_t)c->wg_ctas * COUTP[l]);
    A(&c->bp[l], (size_t)COUTP[l]);
    A(&c->wf[l], 9 * (size_t)CINP[l] * COUTP[l]);
    A(&c->wd[l], 9 * (size_t)CINP[l] * COUTP[l]);
    A(&c->act[l], P * (l == 0 ? 16 : 32));
  }
  A(&c->dza, P * 32);
  A(&c->dzb, P * 32);
  A(&c->lpart, 1024);
  A(&c->err, 1);
  if (s != FIRLS_OK) {
    firls_cnn_destroy(c);
    return s;
  }
  cudaMemset(c->err, 0, sizeof(int));
  cudaMemset(c->gall, 0, c->params * 4);
  size_t o = 0;
  for (int l = 0; l < NL; ++l) {
    const size_t nw = 9 * (size_t)CH[l] * CH[l + 1];
    c->w[l] = c->pall + o;
    c->gw[l] = c->gall + o;
    c->mw[l] = c->mall + o;
    c->vw[l] = c->vall + o;
    o += nw;
    c->b[l] = c->pall + o;
    c->gb[l] = c->gall + o;
    c->mb[l] = c->mall + o;
    c->vb[l] = c->vall + o;
    o += CH[l + 1];
  }
  *out = c;
  return FIRLS_OK;
}

extern "C" firls_status firls_cnn_set_params(firls_cnn* c, const float* const* w, const float* const* b) {
  if (!c || !w || !b) return FIRLS_E_INVALID_ARG;
  for (int l = 0; l < NL; ++l) {
    const size_t nw = 9 * (size_t)CH[l] * CH[l + 1];
    if (cudaMemcpyAsync(c->w[l], w[l], nw * 4, cudaMemcpyHostToDevice, c->stream) != cudaSuccess ||
        cudaMemcpyAsync(c->b[l], b[l], CH[l + 1] * 4, cudaMemcpyHostToDevice, c->stream) != cudaSuccess)
      return FIRLS_E_CUDA;
  }
  cudaMemsetAsync(c->mall, 0, c->params * 4, c->stream);
  cudaMemsetAsync(c->vall, 0, c->params * 4, c->stream);
  c->adam_t = 0;
  pack_all(c);
  if (cudaStreamSynchronize(c->stream) != cudaSuccess) return FIRLS_E_CUDA;
  c->params_set = true;
  return FIRLS_OK;
}

// One copy of the whole block, then each layer's part on the host.
static firls_status get_block(firls_cnn* c, const float* block, float* const* w, float* const* b) {
  std::vector<float> h(c->params);
  if (cudaMemcpyAsync(h.data(), block, c->params * 4, cudaMemcpyDeviceToHost, c->stream) != cudaSuccess ||
      cudaStreamSynchronize(c->stream) != cudaSuccess)
    return FIRLS_E_CUDA;
  const float* p = h.data();
  for (int l = 0; l < NL; ++l) {
    const size_t nw = 9 * (size_t)CH[l] * CH[l + 1];
    if (w[l]) std::memcpy(w[l], p, nw * 4);
    p += nw;
    if (b[l]) std::memcpy(b[l], p, CH[l + 1] * 4);
    p += CH[l + 1];
  }
  return FIRLS_OK;
}

extern "C" firls_status firls_cnn_get_params(firls_cnn* c, float* const* w, float* const* b) {
  if (!c || !w || !b) return FIRLS_E_INVALID_ARG;
  return get_block(c, c->pall, w, b);
}

extern "C" firls_status firls_cnn_get_grads(firls_cnn* c, float* const* gw, float* const* gb) {
  if (!c || !gw || !gb) return FIRLS_E_INVALID_ARG;
  return get_block(c, c->gall, gw, gb);
}

extern "C" firls_status firls_cnn_forward(firls_cnn* c, const void* atb, const uint8_t* mask, void* x1) {
  if (!c || !atb || !mask || !x1) return FIRLS_E_INVALID_ARG;
  if (!c->params_set) return FIRLS_E_STATE;
  forward(c, static_cast<const float2*>(atb), mask, static_cast<float2*>(x1));
  return cudaGetLastError() == cudaSuccess ? FIRLS_OK : FIRLS_E_CUDA;
}

extern "C" firls_status firls_cnn_train_step(firls_cnn* c, const void* atb, const uint8_t* mask, const void* target,
                                             void* x1, float lr, double* loss) {
  if (!c || !atb || !mask || !target || !x1) return FIRLS_E_INVALID_ARG;
  if (!c->params_set) return FIRLS_E_STATE;
  if (!(lr >= 0.f)) return FIRLS_E_INVALID_ARG;
  float2* xo = static_cast<float2*>(x1);
  forward(c, static_cast<const float2*>(atb), mask, xo);
  const int total = c->batch * c->n * c->n;
  const int lblocks = 1024;
  k_cnn_loss<<<lblocks, 256, 0, c->stream>>>(total, xo, static_cast<const float2*>(target), c->dza, c->lpart);
  // layer 6: dZ6 = dOut (16 channels)
  launch_wgrad<32, 16>(c, c->act[5], c->dza, 5);
  launch_conv<16, 32, MODE_DGRAD>(c, c->dza, c->wd[5], nullptr, c->dzb, c->act[5], nullptr, nullptr);
  __nv_bfloat16 *cur = c->dzb, *nxt = c->dza;
  for (int l = 4; l >= 1; --l) {
    launch_wgrad<32, 32>(c, c->act[l], cur, l);
    launch_conv<32, 32, MODE_DGRAD>(c, cur, c->wd[l], nullptr, nxt, c->act[l], nullptr, nullptr);
    __nv_bfloat16* t = cur;
    cur = nxt;
    nxt = t;
  }
  launch_wgrad<16, 32>(c, c->act[0], cur, 0);
  update(c, lr);
  if (loss) {
    std::vector<double> h(lblocks);
    if (cudaMemcpyAsync(h.data(), c->lpart, sizeof(double) * lblocks, cudaMemcpyDeviceToHost, c->stream) !=
            cudaSuccess ||
        cudaStreamSynchronize(c->stream) != cudaSuccess)
      return FIRLS_E_CUDA;
    double s = 0.0;
    for (double v : h) s += v;
    *loss = s;
    int e = 0;
    if (cudaMemcpy(&e, c->err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return FIRLS_E_CUDA;
    if (e) return FIRLS_E_DEVICE_TIMEOUT;
  }
  return cudaGetLastError() == cudaSuccess ? FIRLS_OK : FIRLS_E_CUDA;
}

extern "C" void firls_cnn_destroy(firls_cnn* c) {
  if (!c) return;
  if (c->stream) cudaStreamSynchronize(c->stream);
  else cudaDeviceSynchronize();
  for (void* p : c->allocs)
    if (p) cudaFree(p);
  delete c;
}
