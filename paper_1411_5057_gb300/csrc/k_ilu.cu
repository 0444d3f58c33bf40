// The TV preconditioner's solves z = U^{-1} L^{-1} r (Eq. ptv, Sec. 4.2) with
// the residual update of the PCG step, and the ILU(0) pivots.
//
// L = I + L_P diag(a)^{-1}, U = diag(a) + U_P, where P = diag(a) + L_P + U_P is
// the TV penta-diagonal matrix with off-diagonals -lam W_{i+1} (couples i, i+1;
// zero at a row end) and -lam W_{i+n} (couples i, i+n; zero in the last row).
// With ia = 1/a, v = ia y and p = lam W z the solves need no neighbour's
// coefficient:
//   forward   y_i = r_i + lam W_i (v_{i-1} + v_{i-n}),   v_i = ia_i y_i
//   backward  z_i = v_i + ia_i (p_{i+1} + p_{i+n}),      p_i = lam W_i z_i
// (l1 TV: the vertical terms use W2).  P is symmetric, so U = diag(a) L^T and
// Re<r, z> = sum_i Re<v_i, y_i>.
//
// Both sweeps are first-order recurrences in two directions, so what bounds one
// slice is a chain of dependent steps, and what bounds many is memory.  A slice
// is one CTA; warp b owns the band of rows 32 b .. 32 b + 31, a lane per row,
// and lane L runs L steps behind lane 0, so the value from the row above is the
// one its neighbour lane has just made: one shuffle.  A step is a pair of
// columns; its chain is a shuffle, two FMAs and a product.  The bands follow
// each other 32 steps and a hand-over apart through shared memory, so a 256^2
// sweep is about 450 steps.  A band's warp issues every instruction of its
// steps alone, so what counts is few instructions and no branches between
// them.  The form before this one went row by row with a 32-lane scan in each
// row, about 600 cycles, 256 rows in series.
//
// The lanes of a step touch 32 rows on a diagonal, which no natural row layout
// serves with wide copies.  So everything the sweeps read or write (r, q, y, z
// and the weights) lives in a skewed layout in which a step's 32 pairs are
// consecutive: pair c (columns 2c, 2c + 1) of row 32 b + L is float4
// (b K + c + L) 32 + L of the slice, K = n/2 + 31.  The row IFFT writes q and
// the row FFT reads z in that layout.
//
// What a step moves goes through the SM's one load/store path, about 28 cycles a
// step (backward 20), and the next chunk of CS steps is loaded straight into a
// second set of registers while this one is worked on.  (A ring in shared memory,
// filled by cp.async, costs that path twice as much; filled by bulk copies, its
// mbarriers and divergent issue cost the band's warp more than the steps.  One
// slot refilled per step does not work: its loads share the warp's few
// scoreboards with the shuffles, so every step waits for the newest load.)  A
// lane without a pair loads its nearest valid one again, with its coefficients
// set to 0, so no load is conditional.
//
// Measured, row scans before and this form now, 256^2: 1 slice 158 and 92 us, 76
// slices 160 and 105, 152 slices 174 and 132, 304 slices 289 and 250; 16 slices of
// 512^2 540 and 286, 64 of 320^2 230 and 179.  The row scans also updated dx, 24 of
// their 88 bytes a pixel, which the row FFT does now, and the row IFFT stores q skewed.
// So many slices gain nothing by the form itself: a step's row FFT, row IFFT and sweeps
// of 304 slices took 96 + 133 + 287 us and take 141 + 153 + 253, of 40 of 512^2 59 + 85 +
// 547 and 83 + 104 + 314.  One form serves every batch all the same: a served queue
// ends with few slices, where the sweeps are the step.
#include <algorithm>

#include "launch.h"
#include "per_device.h"

namespace firls {

namespace {

constexpr int WV_CHUNK = 4;  // steps between two hand-overs of a band

__host__ __device__ inline int wv_bands(int n) { return (n + 31) / 32; }
__host__ __device__ inline int wv_steps(int n) { return n / 2 + 31; }
// the rows the bands hand over
__host__ __device__ inline int wv_rows_bytes(int n) { return (wv_bands(n) + 2) * (n / 2) * 16; }

FI unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
FI int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.cta.shared.b32 %0, [%1];\n" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
FI void st_release(int* p, int v) {
  asm volatile("st.release.cta.shared.b32 [%0], %1;\n" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
// Bounded wait (about a second at most) of a whole warp until lane `src` sees
// *p >= want; returns the value it saw, or -1 when the wait ran out.  A warp
// whose wait ran out marks the slice faulted and finishes its sweep without
// waiting for its neighbour (on whatever that left: the results are invalid,
// every access stays in bounds); the others give up at their next wait.
FI int wv_wait(const int* p, int want, int src, int tries, const volatile int* abort_flag) {
  for (int it = 0; it < tries; ++it) {
    const int v = __shfl_sync(0xffffffffu, ld_acquire(p), src);
    if (v >= want) return v;
    if (it >= 64) {
      if (__any_sync(0xffffffffu, *abort_flag != 0)) return -1;
      __nanosleep(20);
    }
  }
  return -1;
}

// predicated stores without a branch; STREAM: not read again soon
template <bool STREAM> FI void st_global_if(bool p, float4* dst, float4 v) {
  if (STREAM)
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %5, 0;\n @p st.global.cs.v4.f32 [%0], {%1, %2, %3, %4};\n}\n" ::"l"(
                     dst),
                 "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"((unsigned)p)
                 : "memory");
  else
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %5, 0;\n @p st.global.v4.f32 [%0], {%1, %2, %3, %4};\n}\n" ::"l"(dst),
                 "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"((unsigned)p)
                 : "memory");
}
FI void st_shared_if(bool p, float4* dst, float4 v) {
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %5, 0;\n @p st.shared.v4.f32 [%0], {%1, %2, %3, %4};\n}\n" ::"r"(
                   smem_u32(dst)),
               "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"((unsigned)p)
               : "memory");
}

}  // namespace

size_t ilu_slice_elems(int n) { return (size_t)wv_bands(n) * wv_steps(n) * 64; }

// CS: steps per chunk.  MAXT, MINB: threads and CTAs per SM the registers are
// sized for.  PF: chunks fetched into L2 ahead of the loads (0: none).
template <int CS, int MAXT, int MINB, int PF, bool ANISO>
__global__ void __launch_bounds__(MAXT, MINB)
    k_ilu(int n, int mode_arg, SliceState* __restrict__ st, double* __restrict__ part, float4* r_all,
          const float4* __restrict__ q_all, float4* y_all, float4* __restrict__ z_all,
          const float4* __restrict__ wa_all, const float2* __restrict__ w2_all, int fuse, PcgSched ps,
          int wait_test, int alpha_np) {
  chained_start();
  const int s = blockIdx.x;
  if (!slice_running(st, s)) return;
  const int t = threadIdx.x, lane = t & 31, b = t >> 5;
  // ILU_PER_SLICE: the first residual for a slice at the start of its outer
  // step, a PCG step otherwise
  int ph = st[s].phase;
  if (alpha_np > 0 && mode_arg == ILU_PER_SLICE && ph == PH_PCG) {
    // alpha = rho / <d, S d> from the S apply's alpha_np partial sums, as the
    // scalar kernel forms it (same order); a slice that stops here (rho = 0
    // or a breakdown) does nothing more in this macro step
    __shared__ int ph_alpha;
    __shared__ double dqs[MAXPART];
    const double* pp = part + ((size_t)s * NSLOT + SLOT_DQ) * MAXPART;
    for (int i = t; i < alpha_np; i += blockDim.x) dqs[i] = pp[i];
    __syncthreads();
    if (t == 0) {
      double dq = 0.0;
      for (int i = 0; i < alpha_np; ++i) dq += dqs[i];
      pcg_alpha_from(st + s, dq);
      ph_alpha = st[s].done ? -1 : st[s].phase;
    }
    __syncthreads();
    if (ph_alpha < 0) return;
    ph = ph_alpha;
  }
  if (mode_arg == ILU_PER_SLICE && !slice_working(ph)) return;
  const bool init = mode_arg != ILU_PER_SLICE ? mode_arg == ILU_INIT : ph == PH_START;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ int prog_f[16], prog_b[16];  // pairs of a band's row handed over, per sweep
  __shared__ volatile int abort_flag;
  __shared__ double red[32];
  const int nb = wv_bands(n), H = n / 2, K = wv_steps(n);
  // nb + 2 rows of pairs that the bands hand over: forward, band b reads row b
  // and writes its last row's v to row b + 1; backward, it reads row b + 1 and
  // writes its first row's p to row b.  Rows 0 and nb + 1 (read by the last
  // band) start as zeros.
  float4* rows = reinterpret_cast<float4*>(smem);
  for (int i = t; i < 2 * H; i += blockDim.x)
    rows[i < H ? i : nb * H + i] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (t < 16) prog_f[t] = prog_b[t] = 0;
  if (t == 0) abort_flag = 0;
  __syncthreads();
  const float alpha = (float)st[s].alpha;
  float rr = 0.f, rho = 0.f;

  const int last = min(31, n - 1 - 32 * b);  // the band's last row
  const bool row_ok = lane <= last;
  const int Le = min(lane, last);  // a lane past the image repeats the last row's loads
  const size_t slice = ((size_t)s * nb + b) * K * 32;
  float4* r = r_all + slice;
  float4* y = y_all + slice;
  float4* z = z_all + slice;
  const float4* q = q_all + slice;
  const float4* wa = wa_all + slice;
  const float2* w2 = ANISO ? w2_all + slice : nullptr;
  const int NC = (K + CS - 1) / CS;
  // wait_test (failure-detection test only): every hand-over wait gives up at
  // once, so the slice is reported faulted
  const int tries = wait_test ? 0 : 1 << 22;
  bool ok = true;
  struct Chunk {
    float4 r[CS], q[CS], w[CS];
    float2 v[ANISO ? CS : 1];
  };
  // steps k0 .. k0 + CS - 1 (the lane's nearest pair where it has none)
  auto load = [&](Chunk& c, int k0, bool fwd) {
#pragma unroll
    for (int u = 0; u < CS; ++u) {
      const int o = min(max(k0 + u, Le), Le + H - 1) * 32 + Le;
      if (!fwd) c.r[u] = __ldcs(y + o);
      else if (!init) c.r[u] = __ldcs(r + o);
      if (fwd) c.q[u] = __ldcs(q + o);
      c.w[u] = fwd ? wa[o] : __ldcs(wa + o);
      if (ANISO) c.v[u] = w2[o];
    }
  };
  // The lines of chunk k0 .. into L2, PF chunks before it is loaded: a chunk is
  // CS x 512 contiguous bytes per array, four 128-byte lines per step, and a
  // warp's own loads cover only one chunk of latency.  Lines of the padding
  // (no valid lane in them) are left out.
  constexpr int LINES = CS * 4;
  auto prefetch = [&](int k0, bool fwd) {
    if (PF == 0) return;
    const char* a0 = reinterpret_cast<const char*>(fwd ? (init ? q : r) : y);
    const char* a1 = reinterpret_cast<const char*>(fwd ? q : wa);
    const char* a2 = reinterpret_cast<const char*>(wa);
    if (ANISO) {  // W2: two lines per step
#pragma unroll
      for (int i = 0; i < CS * 2; i += 32) {
        const int j = i + lane, k = k0 + j / 2, l16 = j % 2 * 16;
        const char* p = reinterpret_cast<const char*>(w2) + (ptrdiff_t)k * 256 + l16 * 8;
        if (j < CS * 2 && l16 <= min(last, k) && l16 + 15 > k - H) asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
      }
    }
#pragma unroll
    for (int i = 0; i < (fwd ? 3 : 2) * LINES; i += 32) {
      const int j = i + lane, a = j / LINES, k = k0 + (j % LINES) / 4, l8 = j % 4 * 8;
      const char* p = (a == 0 ? a0 : a == 1 ? a1 : a2) + (ptrdiff_t)k * 512 + l8 * 16;
      if (a < (fwd ? 3 : 2) && l8 <= min(last, k) && l8 + 7 > k - H) asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
    }
  };
  {  // ---- forward: lane L at step k holds pair k - L
    float2 v0 = make_float2(0.f, 0.f), v1 = v0;  // this row's last pair
    const float4* from = rows + b * H;
    float4* to = rows + (b + 1) * H - 31;
    int avail = b > 0 || wait_test ? 0 : H;
    auto steps = [&](const Chunk& c, int k0) {
#pragma unroll
      for (int u = 0; u < CS; ++u) {
        const int k = k0 + u;
        if (u % WV_CHUNK == 0 && avail < min(k + min(WV_CHUNK, CS - u), H)) {
          avail = wv_wait(prog_f + (b > 0 ? b - 1 : 15), min(k + min(WV_CHUNK, CS - u), H), 0, tries, &abort_flag);
          if (avail < 0) {
            ok = false;
            avail = H;
          }
        }
        const bool valid = row_ok && (unsigned)(k - lane) < (unsigned)H;
        const float4 hv = from[min(k, H - 1)];
        float4 up;
        up.x = __shfl_up_sync(0xffffffffu, v0.x, 1);
        up.y = __shfl_up_sync(0xffffffffu, v0.y, 1);
        up.z = __shfl_up_sync(0xffffffffu, v1.x, 1);
        up.w = __shfl_up_sync(0xffffffffu, v1.y, 1);
        if (lane == 0) up = hv;
        const float4 w = c.w[u];
        const float ia0 = valid ? w.y : 0.f, ia1 = valid ? w.w : 0.f;
        const float lv0 = ANISO ? c.v[u].x : w.x, lv1 = ANISO ? c.v[u].y : w.z;
        float4 rn = c.q[u];
        if (!init)
          rn = make_float4(fmaf(-alpha, rn.x, c.r[u].x), fmaf(-alpha, rn.y, c.r[u].y),
                           fmaf(-alpha, rn.z, c.r[u].z), fmaf(-alpha, rn.w, c.r[u].w));
        const float2 t0 = make_float2(fmaf(lv0, up.x, rn.x), fmaf(lv0, up.y, rn.y));
        const float2 t1 = make_float2(fmaf(lv1, up.z, rn.z), fmaf(lv1, up.w, rn.w));
        const float2 y0 = make_float2(fmaf(w.x, v1.x, t0.x), fmaf(w.x, v1.y, t0.y));
        v0 = make_float2(ia0 * y0.x, ia0 * y0.y);
        const float2 y1 = make_float2(fmaf(w.z, v0.x, t1.x), fmaf(w.z, v0.y, t1.y));
        v1 = make_float2(ia1 * y1.x, ia1 * y1.y);
        const float4 vv = make_float4(v0.x, v0.y, v1.x, v1.y);
        st_global_if<true>(valid, r + k * 32 + lane, rn);
        st_global_if<false>(valid, y + k * 32 + lane, vv);
        st_shared_if(valid && lane == 31, to + k, vv);
        if (valid) rr = fmaf(rn.x, rn.x, fmaf(rn.y, rn.y, fmaf(rn.z, rn.z, fmaf(rn.w, rn.w, rr))));
        rho = fmaf(v0.x, y0.x, fmaf(v0.y, y0.y, fmaf(v1.x, y1.x, fmaf(v1.y, y1.y, rho))));
        if ((u % WV_CHUNK == WV_CHUNK - 1 || u == CS - 1) && lane == 31 && k >= 31 && !wait_test)
          st_release(prog_f + b, min(k - 30, H));
      }
    };
    Chunk A, B;
    load(A, 0, true);
    for (int j = 1; j < PF; ++j) prefetch(j * CS, true);
    for (int j = 0; j < NC; j += 2) {
      load(B, (j + 1) * CS, true);
      prefetch((j + PF) * CS, true);
      steps(A, j * CS);
      load(A, (j + 2) * CS, true);
      prefetch((j + PF + 1) * CS, true);
      steps(B, (j + 1) * CS);  // past the end: no lane has a pair
    }
  }
  if (!ok) abort_flag = 1;
  // in a part band the lanes past the image read lane `last`'s y below; their
  // coefficients are 0, but the values have to be those it has just stored
  __syncwarp();
  {  // ---- backward: step m = K - 1 - k, from the last row and column
    float2 p0 = make_float2(0.f, 0.f);  // lam W z of this row's last pair, and its
    float4 pv = make_float4(0.f, 0.f, 0.f, 0.f);  // vertical one (W2 for l1 TV)
    const float4* from = rows + (b < nb - 1 ? b + 1 : nb + 1) * H;
    float4* to = rows + b * H;
    int avail = b < nb - 1 ? 0 : H;
    auto steps = [&](const Chunk& c, int m0) {
#pragma unroll
      for (int u = 0; u < CS; ++u) {
        const int m = m0 + u, k = K - 1 - m;
        if (u % WV_CHUNK == 0 && avail < min(m + min(WV_CHUNK, CS - u), H)) {
          avail = wv_wait(prog_b + b + 1, min(m + min(WV_CHUNK, CS - u), H), 31, tries, &abort_flag);
          if (avail < 0) {
            ok = false;
            avail = H;
          }
        }
        const bool valid = row_ok && (unsigned)(k - lane) < (unsigned)H;
        const float4 hv = from[max(H - 1 - m, 0)];
        float4 dn;
        dn.x = __shfl_down_sync(0xffffffffu, pv.x, 1);
        dn.y = __shfl_down_sync(0xffffffffu, pv.y, 1);
        dn.z = __shfl_down_sync(0xffffffffu, pv.z, 1);
        dn.w = __shfl_down_sync(0xffffffffu, pv.w, 1);
        if (lane == 31) dn = hv;
        const float4 w = c.w[CS - 1 - u], vv = c.r[CS - 1 - u];
        const float lw0 = valid ? w.x : 0.f, lw1 = valid ? w.z : 0.f;
        const float2 t0 = make_float2(fmaf(w.y, dn.x, vv.x), fmaf(w.y, dn.y, vv.y));
        const float2 t1 = make_float2(fmaf(w.w, dn.z, vv.z), fmaf(w.w, dn.w, vv.w));
        const float2 z1 = make_float2(fmaf(w.w, p0.x, t1.x), fmaf(w.w, p0.y, t1.y));
        const float2 p1 = make_float2(lw1 * z1.x, lw1 * z1.y);
        const float2 z0 = make_float2(fmaf(w.y, p1.x, t0.x), fmaf(w.y, p1.y, t0.y));
        p0 = make_float2(lw0 * z0.x, lw0 * z0.y);
        if (ANISO) {
          const float l0 = valid ? c.v[CS - 1 - u].x : 0.f, l1 = valid ? c.v[CS - 1 - u].y : 0.f;
          pv = make_float4(l0 * z0.x, l0 * z0.y, l1 * z1.x, l1 * z1.y);
        } else {
          pv = make_float4(p0.x, p0.y, p1.x, p1.y);
        }
        st_global_if<false>(valid, z + k * 32 + lane, make_float4(z0.x, z0.y, z1.x, z1.y));
        st_shared_if(valid && lane == 0, to + k, pv);
        if ((u % WV_CHUNK == WV_CHUNK - 1 || u == CS - 1) && lane == 0 && m >= 31)
          st_release(prog_b + b, min(m - 30, H));
      }
    };
    Chunk A, B;
    load(A, K - CS, false);
    for (int j = 1; j < PF; ++j) prefetch(K - (j + 1) * CS, false);
    for (int j = 0; j < NC; j += 2) {
      load(B, K - (j + 2) * CS, false);
      prefetch(K - (j + PF + 1) * CS, false);
      steps(A, j * CS);
      load(A, K - (j + 3) * CS, false);
      prefetch(K - (j + PF + 2) * CS, false);
      steps(B, (j + 1) * CS);
    }
  }
  if (!ok) {
    abort_flag = 1;
    st[s].fault = 1;
  }
  __syncthreads();
  const double trz = block_sum((double)rho, red);
  __syncthreads();
  const double trr = block_sum((double)rr, red);
  if (t == 0) {
    part[((size_t)s * NSLOT + SLOT_RZ) * MAXPART] = trz;
    part[((size_t)s * NSLOT + SLOT_RR) * MAXPART] = trr;
    if (fuse && !abort_flag) {
      if (init)
        pcg_rho_init_from(st + s, 0.0 + trz, 0.0 + trr);
      else
        pcg_beta_from(st + s, 0.0 + trz, 0.0 + trr, ps);
    }
  }
}

// ILU(0) pivots of the penta-diagonal P: d_i = a_i - (lam W1_i)^2 / d_{i-1}
// [col > 0] - (lam W2_i)^2 / d_{i-n} [row > 0] (the incomplete LU with zero
// fill of Sec. 4.2 with updated pivots; W1 = W2 = W for isotropic TV).  The
// same wavefront as the forward sweep, on the packed weights: 1/a in `wa`
// becomes 1/d, also in the natural array `ia`.  (One warp per slice scanning 2 x 2
// maps row by row took 1358 us at 320^2.)
template <bool ANISO>
__global__ void __launch_bounds__(512) k_ilu0_pivots(int n, SliceState* st_all, const SliceState* __restrict__ st,
                                                     float4* wa_all, const float2* __restrict__ w2_all,
                                                     float* __restrict__ ia) {
  const int s = blockIdx.x;
  if (!slice_running(st, s)) return;
  const int t = threadIdx.x, lane = t & 31, b = t >> 5;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int prog[16];
  __shared__ volatile int abort_flag;
  const int nb = wv_bands(n), H = n / 2, K = wv_steps(n);
  float2* rows = reinterpret_cast<float2*>(smem);  // 1/d of each band's last row
  if (t < 16) prog[t] = 0;
  if (t == 0) abort_flag = 0;
  __syncthreads();
  const size_t base = ((size_t)s * nb + b) * K * 32 + lane;
  float4* wa = wa_all + base;
  const float2* w2 = ANISO ? w2_all + base : nullptr;
  const int row = 32 * b + lane;
  const unsigned Hrow = row < n ? (unsigned)H : 0u;
  float2* ian = reinterpret_cast<float2*>(ia + (size_t)s * n * n + (size_t)row * n);
  constexpr int D = 8;
  const int Kr = (K + D - 1) / D * D;
  float4 fw[D];
  float2 fv[ANISO ? D : 1];
  auto fetch = [&](int u, int k) {
    fw[u] = make_float4(0.f, 1.f, 0.f, 1.f);
    if (ANISO) fv[u] = make_float2(0.f, 0.f);
    if ((unsigned)(k - lane) < Hrow) {
      fw[u] = wa[k * 32];
      if (ANISO) fv[u] = w2[k * 32];
    }
  };
#pragma unroll
  for (int u = 0; u < D; ++u) fetch(u, u);
  float i0 = 0.f, i1 = 0.f;  // 1/d of this row's last pair
  int avail = 0;
  bool ok = true;
  for (int k0 = 0; k0 < Kr; k0 += D) {
#pragma unroll
    for (int u = 0; u < D; ++u) {
      const int k = k0 + u;
      if (u % WV_CHUNK == 0 && b > 0 && avail < min(k + WV_CHUNK, H)) {
        avail = wv_wait(prog + b - 1, min(k + WV_CHUNK, H), 0, 1 << 22, &abort_flag);
        if (avail < 0) {
          ok = false;
          avail = H;
          abort_flag = 1;
        }
      }
      float2 up = make_float2(0.f, 0.f);
      if (b > 0 && lane == 0 && k < H) up = rows[(b - 1) * H + k];
      const float n0 = __shfl_up_sync(0xffffffffu, i0, 1), n1 = __shfl_up_sync(0xffffffffu, i1, 1);
      if (lane > 0) up = make_float2(n0, n1);
      const int c = k - lane;
      const float4 w = fw[u];
      const float kh0 = c > 0 ? w.x : 0.f, kh1 = w.z;
      const float kv0 = row > 0 ? (ANISO ? fv[u].x : w.x) : 0.f;
      const float kv1 = row > 0 ? (ANISO ? fv[u].y : w.z) : 0.f;
      const float al0 = 1.0f / w.y - kv0 * kv0 * up.x, al1 = 1.0f / w.w - kv1 * kv1 * up.y;
      i0 = 1.0f / (al0 - kh0 * kh0 * i1);
      i1 = 1.0f / (al1 - kh1 * kh1 * i0);
      if ((unsigned)c < Hrow) {
        wa[k * 32] = make_float4(w.x, i0, w.z, i1);
        ian[c] = make_float2(i0, i1);
        if (lane == 31) rows[b * H + c] = make_float2(i0, i1);
      }
      fetch(u, k + D);
      if (u % WV_CHUNK == WV_CHUNK - 1 && lane == 31 && k >= 31) st_release(prog + b, min(k - 30, H));
    }
  }
  if (!ok) st_all[s].fault = 1;
}

// The kernels that write the skewed layout run in its order: a warp takes a step of
// a band, lane L the pair of row L, and a CTA SK_STEPS consecutive steps, whose reads
// of a natural array are SK_STEPS consecutive pairs of each row.  (Scattered 16-byte
// stores from the natural order cost more than scattered loads: a complex array of 304
// slices of 256^2 76 us, this way 47.)
constexpr int SK_STEPS = 32;
static dim3 skew_grid(int n, int batch) { return dim3((wv_steps(n) + SK_STEPS - 1) / SK_STEPS, wv_bands(n), batch); }

// fn(row, c, index of the pair in the slice) for this thread's pairs
template <typename Fn> FI void skew_pairs(int n, Fn&& fn) {
  const int lane = threadIdx.x & 31, row = blockIdx.y * 32 + lane, K = wv_steps(n);
  if (row >= n) return;
#pragma unroll
  for (int u = 0; u < SK_STEPS; u += 8) {
    const int k = blockIdx.x * SK_STEPS + u + (threadIdx.x >> 5), c = k - lane;
    if ((unsigned)c < (unsigned)(n / 2)) fn(row, c, (blockIdx.y * K + k) * 32 + lane);
  }
}

// The set-up of the sweeps for the slices st shows running, in one pass over the
// weights: 1/a of P (Eq. ptv, k_penta's formula) in the natural order, (lam W, 1/a)
// and for l1 TV lam W2 skewed.  Bound by memory, 16 bytes a pixel (l1 24).  304 slices
// of 256^2 84 us, l1 110 (k_penta and a pack of its result took 127 and 161).
template <bool ANISO>
__global__ void __launch_bounds__(256) k_penta_pack(int n, const SliceState* __restrict__ st,
                                                    const float* __restrict__ wtv, const float* __restrict__ wtv2,
                                                    const float* __restrict__ wdiag, float* __restrict__ ia,
                                                    float4* __restrict__ wa, float2* __restrict__ w2s) {
  const int s = blockIdx.z;
  if (!slice_running(st, s)) return;
  const float abar = st[s].abar, lt = st[s].lam_tv, lw = st[s].lam;
  const size_t nat = (size_t)s * n * n, out = (size_t)s * wv_bands(n) * wv_steps(n) * 32;
  skew_pairs(n, [&](int row, int c, int at) {
    const size_t i = nat + (size_t)row * n + 2 * c;
    auto pair = [](const float* p) { return *reinterpret_cast<const float2*>(p); };
    const float* V = ANISO ? wtv2 : wtv;  // the vertical weights
    const float2 w = pair(wtv + i);
    const float2 v = ANISO ? pair(V + i) : w;
    const float2 below = row < n - 1 ? pair(V + i + n) : make_float2(0.f, 0.f);
    const float right = 2 * c + 2 < n ? wtv[i + 2] : 0.f;
    float a0 = penta_diag<ANISO>(abar, lt, w.x, w.y, v.x, below.x);
    float a1 = penta_diag<ANISO>(abar, lt, w.y, right, v.y, below.y);
    if (wdiag) {
      const float2 g = pair(wdiag + i);
      a0 = fmaf(lw, g.x, a0);
      a1 = fmaf(lw, g.y, a1);
    }
    const float2 r = make_float2(1.0f / a0, 1.0f / a1);
    *reinterpret_cast<float2*>(ia + i) = r;
    wa[out + at] = make_float4(lt * w.x, r.x, lt * w.y, r.y);
    if (ANISO) w2s[out + at] = make_float2(lt * v.x, lt * v.y);
  });
}

// The packed weights from W, W2 and an 1/a that is there already, of every slice.
__global__ void __launch_bounds__(256) k_ilu_pack(int n, const SliceState* __restrict__ st,
                                                  const float* __restrict__ wtv, const float* __restrict__ wtv2,
                                                  const float* __restrict__ ia, float4* __restrict__ wa,
                                                  float2* __restrict__ w2s) {
  const int s = blockIdx.z;
  const float lam = st[s].lam_tv;
  const size_t nat = (size_t)s * n * n, out = (size_t)s * wv_bands(n) * wv_steps(n) * 32;
  skew_pairs(n, [&](int row, int c, int at) {
    const size_t i = nat + (size_t)row * n + 2 * c;
    const float2 w = *reinterpret_cast<const float2*>(wtv + i), a = *reinterpret_cast<const float2*>(ia + i);
    wa[out + at] = make_float4(lam * w.x, a.x, lam * w.y, a.y);
    if (wtv2) {
      const float2 v = *reinterpret_cast<const float2*>(wtv2 + i);
      w2s[out + at] = make_float2(lam * v.x, lam * v.y);
    }
  });
}

// A complex array from the natural to the skewed layout, and back.
__global__ void __launch_bounds__(256) k_to_skewed(int n, const float4* __restrict__ src, float4* __restrict__ dst) {
  const size_t nat = (size_t)blockIdx.z * n * (n / 2), out = (size_t)blockIdx.z * wv_bands(n) * wv_steps(n) * 32;
  skew_pairs(n, [&](int row, int c, int at) { dst[out + at] = src[nat + (size_t)row * (n / 2) + c]; });
}
__global__ void k_from_skewed(int n, const float4* __restrict__ src, float4* __restrict__ dst) {
  const int H = n / 2, K = wv_steps(n), s = blockIdx.y;
  const size_t nat = (size_t)s * n * H, sk = (size_t)s * wv_bands(n) * K * 32;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n * H; i += gridDim.x * blockDim.x) {
    const int row = i / H, c = i % H, L = row & 31;
    dst[nat + i] = src[sk + (size_t)((row >> 5) * K + c + L) * 32 + L];
  }
}

namespace {

typedef void (*IluKernel)(int, int, SliceState*, double*, float4*, const float4*, float4*, float4*, const float4*,
                          const float2*, int, PcgSched, int, int);
// Chunks of 8 steps where the CTA has the registers of an SM to itself (up to
// 256 rows); of 4 with two CTAs of 256^2 per SM; of 5 and 4 above 256 rows,
// where the CTA has more warps.  l1 TV holds W2 in the chunks too: of 3 steps where a
// thread has 128 registers (4 spilled: 304 slices of 256^2 337 -> 275 us, 304 of
// 128^2 132 -> 96, 40 of 512^2 486 -> 385; the row scans before took 297, 95 and 557).
template <bool ANISO>
IluKernel ilu_kernel(int n, bool deep, bool far) {
  constexpr int CS = ANISO ? 3 : 4;
  if (wv_bands(n) > 12) return k_ilu<CS, 512, 1, 0, ANISO>;
  if (wv_bands(n) > 8) return k_ilu<5, 384, 1, 0, ANISO>;
  if (deep) return far ? k_ilu<8, 256, 1, 4, ANISO> : k_ilu<8, 256, 1, 0, ANISO>;
  return far ? k_ilu<CS, 256, 2, 4, ANISO> : k_ilu<CS, 256, 2, 0, ANISO>;
}

}  // namespace

bool ilu_prepare() {
  const cudaFuncAttribute A = cudaFuncAttributeMaxDynamicSharedMemorySize;
  bool ok = true;
  for (int n : {256, 384, 512})
    for (int i = 0; i < 4; ++i) {
      ok = cudaFuncSetAttribute(ilu_kernel<false>(n, i & 1, i & 2), A, wv_rows_bytes(512)) == cudaSuccess && ok;
      ok = cudaFuncSetAttribute(ilu_kernel<true>(n, i & 1, i & 2), A, wv_rows_bytes(512)) == cudaSuccess && ok;
    }
  return ok;
}

// Shapes are numbered 10 * G + S: G = 4 takes long chunks (8 warps per SM), G = 2
// short ones (16); S has no effect.  All shapes give the same results bit for bit.
// A full wave of short chunks serves twice the slices in about 1.9 times the time of a
// wave of long ones (128^2: 608 slices 140 us, 304 74), so the default takes the long
// ones where they need fewer than 1.9 times the waves.  Long and short, us: 128^2 152
// slices 57 and 69, 304 73 and 94, 400 122 and 107, 800 197 and 224; 64^2 300 slices
// 32 and 39, 900 75 and 67, 1500 115 and 129; 256^2 152 slices 132 and 175, 160 217 and
// 197, 304 260 and 254.  (By the batch alone, 152 slices at every size, 304 slices of 128^2
// were no faster than with the row scans before.)  Below 32 rows half the lanes idle and a
// sweep is short against the long chunks' start: 1500 slices of 16^2 37 and 23.
int ilu_default_shape(int n, int batch) {
  const int bands = wv_bands(n), sms = 152;
  if (bands > 8) return 22;  // one form there
  if (n < 32) return batch <= sms ? 42 : 22;
  auto waves = [&](int warps) { return (batch + sms * (warps / bands) - 1) / (sms * (warps / bands)); };
  return 10 * waves(8) < 19 * waves(16) ? 42 : 22;
}

// The shapes that set_tuning takes for a size: those of tuning files and callers from
// when S counted the stages of a shared-memory ring, by the bytes it took.  The sweeps
// need no such room; the set stays what it was.
bool ilu_shape_fits(int n, int shape, bool aniso) {
  const int G = shape / 10, S = shape % 10;
  if ((G != 2 && G != 4) || S < 2 || S > 8 || n % G) return false;
  const long stage = ((long)(aniso ? 44 : 40) * n * G + 16L * 32 * wv_bands(n) * G + 127) / 128 * 128;
  return S * stage <= 200 * 1024;
}

void ilu_step(int batch, int n, cudaStream_t s, SliceState* st, double* part, int mode, float2* r, const float2* q,
              float2* y, float2* z, const float4* wa, const float2* w2s, int shape, int fuse_scalars, PcgSched ps,
              int wait_test, int alpha_np, bool chained) {
  if (shape <= 0) shape = ilu_default_shape(n, batch);
  const bool deep = shape / 10 == 4;
  // r, q, y, z and the weights: 40 bytes a pixel against an L2 of 129 MB.  304
  // slices of 256^2: 247 us with the fetches into L2, 257 without; 16: 96
  // against 94.
  const bool far = 40.0 * n * n * batch > 100e6;
  const IluKernel k = w2s ? ilu_kernel<true>(n, deep, far) : ilu_kernel<false>(n, deep, far);
  auto f4 = [](float2* p) { return reinterpret_cast<float4*>(p); };
  launch_chained(chained, k, dim3(batch), dim3(32 * wv_bands(n)), wv_rows_bytes(n), s, n, mode, st, part, f4(r),
                 reinterpret_cast<const float4*>(q), f4(y), f4(z), wa, w2s, fuse_scalars, ps, wait_test, alpha_np);
}

void penta_pack(int batch, int n, cudaStream_t s, const SliceState* st, const float* wtv, const float* wtv2,
                const float* wdiag, float* ia, float4* wa, float2* w2s) {
  if (wtv2) k_penta_pack<true><<<skew_grid(n, batch), 256, 0, s>>>(n, st, wtv, wtv2, wdiag, ia, wa, w2s);
  else k_penta_pack<false><<<skew_grid(n, batch), 256, 0, s>>>(n, st, wtv, wtv2, wdiag, ia, wa, w2s);
}

void ilu_pack(int batch, int n, cudaStream_t s, const SliceState* st, const float* wtv, const float* wtv2,
              const float* ia, float4* wa, float2* w2s) {
  k_ilu_pack<<<skew_grid(n, batch), 256, 0, s>>>(n, st, wtv, wtv2, ia, wa, w2s);
}

void ilu0_pivots(int batch, int n, cudaStream_t s, SliceState* st, const SliceState* view, float4* wa,
                 const float2* w2s, float* ia) {
  const size_t bytes = (size_t)wv_bands(n) * (n / 2) * 8;
  if (w2s) k_ilu0_pivots<true><<<batch, 32 * wv_bands(n), bytes, s>>>(n, st, view, wa, w2s, ia);
  else k_ilu0_pivots<false><<<batch, 32 * wv_bands(n), bytes, s>>>(n, st, view, wa, w2s, ia);
}

void ilu_skew(int batch, int n, cudaStream_t s, bool to_skewed, const float2* src, float2* dst) {
  const float4* from = reinterpret_cast<const float4*>(src);
  float4* to = reinterpret_cast<float4*>(dst);
  if (to_skewed) k_to_skewed<<<skew_grid(n, batch), 256, 0, s>>>(n, from, to);
  else k_from_skewed<<<dim3(std::min((n * n / 2 + 255) / 256, 64), batch), 256, 0, s>>>(n, from, to);
}

}  // namespace firls
