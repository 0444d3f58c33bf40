// The lifting wavelets and the one-launch form of Phi^T (s o Phi x) on a
// thread-block cluster, instantiated per size and kind in k_wav_haar.cu and
// k_wav_db4.cu.
#pragma once

#include "launch.h"

namespace firls {

// ============================================================ wavelets =====
// Lifting factorisation (Daubechies & Sweldens) arranged to reproduce the
// periodic filter bank a_k = sum_t h_t x_{2k+t}, d_k = sum_t g_t x_{2k+t},
// g_t = (-1)^t h_{3-t}, h the Daubechies-4 taps.  For output pair k, with
// s1_l = x_{2l} + sqrt3 x_{2l+1}:
//   D_k  = x_{2k+3} - (sqrt3/4) s1_{k+1} - ((sqrt3-2)/4) s1_k
//   a_k  = cs (s1_k - D_k),   d_k = -cd D_k,
// cs = (sqrt3-1)/sqrt2, cd = (sqrt3+1)/sqrt2.  The inverse solves these for
// x_{2l}, x_{2l+1} from pairs l-1 and l.  Haar: a = (x0+x1)/sqrt2,
// d = (x0-x1)/sqrt2.
namespace lift {
constexpr float S3 = 1.7320508075688772f;
constexpr float K1 = 0.43301270189221932f;   // sqrt3 / 4
constexpr float K2 = -0.066987298107780677f; // (sqrt3 - 2) / 4
constexpr float CS = 0.51763809020504152f;   // (sqrt3 - 1) / sqrt2
constexpr float CD = 1.9318516525781366f;    // (sqrt3 + 1) / sqrt2
constexpr float ICS = 1.9318516525781366f;   // 1 / CS
constexpr float ICD = 0.51763809020504152f;  // 1 / CD
constexpr float RS2 = 0.70710678118654752f;  // 1 / sqrt2

FI void fwd_db4(float2 x0, float2 x1, float2 x2, float2 x3, float2& a, float2& d) {
  const float2 s1k = cfma(S3, x1, x0);
  const float2 s1n = cfma(S3, x3, x2);
  const float2 D = make_float2(x3.x - K1 * s1n.x - K2 * s1k.x, x3.y - K1 * s1n.y - K2 * s1k.y);
  a = cscale(csub(s1k, D), CS);
  d = cscale(D, -CD);
}
FI void fwd_haar(float2 x0, float2 x1, float2& a, float2& d) {
  a = cscale(cadd(x0, x1), RS2);
  d = cscale(csub(x0, x1), RS2);
}
// from (a_{l-1}, d_{l-1}) and (a_l, d_l) to (x_{2l}, x_{2l+1})
FI void inv_db4(float2 am, float2 dm, float2 al, float2 dl, float2& x0, float2& x1) {
  const float2 Dm = cscale(dm, -ICD);
  const float2 s1m = cfma(ICS, am, Dm);
  const float2 Dl = cscale(dl, -ICD);
  const float2 s1l = cfma(ICS, al, Dl);
  x1 = make_float2(Dm.x + K1 * s1l.x + K2 * s1m.x, Dm.y + K1 * s1l.y + K2 * s1m.y);
  x0 = cfma(-S3, x1, s1l);
}
FI void inv_haar(float2 a, float2 d, float2& x0, float2& x1) {
  x0 = cscale(cadd(a, d), RS2);
  x1 = cscale(csub(a, d), RS2);
}
}  // namespace lift

// ---- every level of one slice on a thread-block cluster ----
// u = Phi^T (s o Phi x) in one launch: the C CTAs of a cluster own R = n/C
// consecutive rows of the slice each, so the whole slice lives in their
// shared memory and only x, the weights and u cross HBM.  All levels run in
// place.  Level l (side m = n >> (l-1), R_l = R >> (l-1) rows per CTA) keeps
// its row r at local row r << (l-1); the row step stores each row as
// [lowpass | highpass], the column step stores output pair k as rows 2k
// (lowpass) and 2k+1 (highpass), so the next level's block is the even rows'
// left halves, and every local position ends holding exactly one
// coefficient.  The column step scales each coefficient by its weight as
// soon as it is final, so no separate pass touches them.
// The Daubechies-4 column step of the last pair needs the next CTA's first
// two rows, the inverse column step of the first pair the previous CTA's last
// pair.  Each exchange e (forward level l: e = l - 1; inverse level l:
// e = 2L - l) has its own halo buffer and mbarrier in the receiving CTA: the
// sender writes the rows there with st.async, which counts the bytes on that
// mbarrier, and the receiver waits for them (bounded).  No buffer is written
// twice in a launch, so one cluster barrier at the start (every mbarrier
// armed before any remote write) is the only cluster-wide synchronisation;
// only the thread range whose pair reads a halo waits for it, just before
// that pair, so the exchange overlaps the rest of the column step.
constexpr int WCL_NMAX = 256;
constexpr int WCL_LMAX = 5;
constexpr int WCL_RMAX = 32;  // rows per CTA: two CTAs per SM fit with the weights mirrored
constexpr int WCL_WIDE_R = 32;  // rows per CTA of the sizes above WCL_NMAX (clusters of 10, 12, 16)

FI unsigned wcl_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
FI unsigned wcl_smem(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
// 16 bytes to the same shared-memory offset in CTA `rank`, counted on that
// CTA's mbarrier at the offset of `bar`
FI void wcl_st_async16(const void* dst, const uint64_t* bar, unsigned rank, float4 v) {
  unsigned ra, rb;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(wcl_smem(dst)), "r"(rank));
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(wcl_smem(bar)), "r"(rank));
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                   ra),
               "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(rb)
               : "memory");
}
// bounded wait (about a second) for the first phase of `bar`, with
// cluster-scope acquire of the remote writes it counted
FI bool wcl_wait(const uint64_t* bar) {
  for (int it = 0; it < 20000; ++it) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0, %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(wcl_smem(bar)), "r"(50000u)
        : "memory");
    if (ok) return true;
  }
  return false;
}
FI void wcl_cp16(void* sdst, const void* gsrc) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(wcl_smem(sdst)), "l"(gsrc) : "memory");
}

// level of exchange e, and the offset (float2) of its halo buffer
__host__ __device__ inline int wcl_ex_level(int L, int e) { return e < L ? e + 1 : 2 * L - e; }
__host__ __device__ inline int wcl_halo_off(int n, int L, int e) {
  int off = 0;
  for (int q = 0; q < e; ++q) off += 2 * (n >> (wcl_ex_level(L, q) - 1));
  return off;
}

// Mallat row (in the n x n coefficient array) of the coefficient held at
// local row rho, column j of CTA `rank` after all L analysis levels.
FI int wcl_coef_row(int rho, int j, int n, int L, int R, int rank) {
  for (int l = 1; l <= L; ++l) {
    const int m = n >> (l - 1), r = rho >> (l - 1);
    const int k = rank * ((R >> (l - 1)) / 2) + (r >> 1);  // global pair index at level l
    if (r & 1) return m / 2 + k;                            // highpass row
    if (j >= m / 2 || l == L) return k;                     // lowpass row, final
  }
  return 0;  // not reached for L >= 1
}

struct WclScale {  // per-coefficient factor: w (MUL_W) or 1/(abar + lam w)
  const float* Wm;  // mirrored weights, or null: read from ws
  const float* ws;
  int n, L, R, rank, mode;
  float lam, abar;
  FI float2 apply(float2 v, int rho, int j) const {
    const float wv = Wm ? Wm[rho * n + j] : __ldg(ws + (size_t)wcl_coef_row(rho, j, n, L, R, rank) * n + j);
    return cscale(v, mode == WAV_MUL_W ? wv : 1.0f / (abar + lam * wv));
  }
};

// one level-l row step over the R_l rows (a warp per row); the inverse of
// level 1 (out != null) writes the samples straight to `out` (row stride n)
// with the optional real projection and partial Re<r, out>
template <int PAIRS>  // pairs per lane of a row
FI float wcl_rows(float2* D, int n, int sr, int Rl, int m, int kind, bool inverse, int nth, float2* out = nullptr,
                  const float2* rr_ = nullptr, int real = 0) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, half = m / 2;
  float acc = 0.f;
  for (int rr = wid; rr < Rl; rr += nth / 32) {
    float2* L = D + rr * sr * n;
    float2 o0[PAIRS], o1[PAIRS];
#pragma unroll
    for (int u = 0; u < PAIRS; ++u) {
      const int k = lane + 32 * u;
      if (k >= half) continue;
      if (!inverse) {
        const float4 p0 = reinterpret_cast<const float4*>(L)[k];
        if (kind == 2) {
          const float4 p1 = reinterpret_cast<const float4*>(L)[k + 1 < half ? k + 1 : 0];
          lift::fwd_db4(make_float2(p0.x, p0.y), make_float2(p0.z, p0.w), make_float2(p1.x, p1.y),
                        make_float2(p1.z, p1.w), o0[u], o1[u]);
        } else {
          lift::fwd_haar(make_float2(p0.x, p0.y), make_float2(p0.z, p0.w), o0[u], o1[u]);
        }
      } else if (kind == 2) {
        const int km = k ? k - 1 : half - 1;
        lift::inv_db4(L[km], L[half + km], L[k], L[half + k], o0[u], o1[u]);
      } else {
        lift::inv_haar(L[k], L[half + k], o0[u], o1[u]);
      }
    }
    if (out) {
#pragma unroll
      for (int u = 0; u < PAIRS; ++u) {
        const int k = lane + 32 * u;
        if (k >= half) continue;
        float4 v = make_float4(o0[u].x, o0[u].y, o1[u].x, o1[u].y);
        if (real) v.y = v.w = 0.f;
        reinterpret_cast<float4*>(out + (size_t)rr * n)[k] = v;
        if (rr_) {
          const float4 q = reinterpret_cast<const float4*>(rr_ + (size_t)rr * n)[k];
          acc += q.x * v.x + q.y * v.y + q.z * v.z + q.w * v.w;
        }
      }
      continue;
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < PAIRS; ++u) {
      const int k = lane + 32 * u;
      if (k >= half) continue;
      if (!inverse) {
        L[k] = o0[u];
        L[half + k] = o1[u];
      } else {
        reinterpret_cast<float4*>(L)[k] = make_float4(o0[u].x, o0[u].y, o1[u].x, o1[u].y);
      }
    }
    __syncwarp();
  }
  return acc;
}

// Pairs [k0, k1) of one column of a level-l column step, streaming down the
// column in place, two pairs per step with every load before the first
// store.  Forward: rows 2 k1 and 2 k1 + 1 (the next part's first rows, or the
// halo) are (e0, e1); the step scales the coefficients that are final after
// this level (highpass rows; lowpass rows right of m/2 or at the last
// level).  Inverse: (e0, e1) is pair k0 - 1 as it was before its update.
FI void wcl_col_pairs(float2* Dc, int rs, int sr, int j, int k0, int k1, float2 e0, float2 e1, int kind,
                      bool inverse, bool lo_final, const WclScale& sc) {
  if (kind != 2) {
    for (int kk = k0; kk < k1; ++kk) {
      float2 o0, o1;
      if (!inverse) {
        lift::fwd_haar(Dc[2 * kk * rs], Dc[(2 * kk + 1) * rs], o0, o1);
        if (lo_final) o0 = sc.apply(o0, 2 * kk * sr, j);
        o1 = sc.apply(o1, (2 * kk + 1) * sr, j);
      } else {
        lift::inv_haar(Dc[2 * kk * rs], Dc[(2 * kk + 1) * rs], o0, o1);
      }
      Dc[2 * kk * rs] = o0;
      Dc[(2 * kk + 1) * rs] = o1;
    }
  } else if (!inverse) {
    float2 r0 = Dc[2 * k0 * rs], r1 = Dc[(2 * k0 + 1) * rs];
    int kk = k0;
    for (; kk + 1 < k1; kk += 2) {
      const bool last = kk + 2 >= k1;
      const float2 r2 = Dc[(2 * kk + 2) * rs], r3 = Dc[(2 * kk + 3) * rs];
      const float2 r4 = last ? e0 : Dc[(2 * kk + 4) * rs];
      const float2 r5 = last ? e1 : Dc[(2 * kk + 5) * rs];
      float2 a0, d0, a1, d1;
      lift::fwd_db4(r0, r1, r2, r3, a0, d0);
      lift::fwd_db4(r2, r3, r4, r5, a1, d1);
      if (lo_final) {
        a0 = sc.apply(a0, 2 * kk * sr, j);
        a1 = sc.apply(a1, (2 * kk + 2) * sr, j);
      }
      Dc[2 * kk * rs] = a0;
      Dc[(2 * kk + 1) * rs] = sc.apply(d0, (2 * kk + 1) * sr, j);
      Dc[(2 * kk + 2) * rs] = a1;
      Dc[(2 * kk + 3) * rs] = sc.apply(d1, (2 * kk + 3) * sr, j);
      r0 = r4;
      r1 = r5;
    }
    if (kk < k1) {  // the last pair alone: its rows 2k+2, 2k+3 are (e0, e1)
      float2 a, d;
      lift::fwd_db4(r0, r1, e0, e1, a, d);
      if (lo_final) a = sc.apply(a, 2 * kk * sr, j);
      Dc[2 * kk * rs] = a;
      Dc[(2 * kk + 1) * rs] = sc.apply(d, (2 * kk + 1) * sr, j);
    }
  } else {
    float2 am = e0, dm = e1;
    int kk = k0;
    for (; kk + 1 < k1; kk += 2) {
      const float2 al = Dc[2 * kk * rs], dl = Dc[(2 * kk + 1) * rs];
      const float2 bl = Dc[(2 * kk + 2) * rs], el = Dc[(2 * kk + 3) * rs];
      float2 x0, x1, y0, y1;
      lift::inv_db4(am, dm, al, dl, x0, x1);
      lift::inv_db4(al, dl, bl, el, y0, y1);
      Dc[2 * kk * rs] = x0;
      Dc[(2 * kk + 1) * rs] = x1;
      Dc[(2 * kk + 2) * rs] = y0;
      Dc[(2 * kk + 3) * rs] = y1;
      am = bl;
      dm = el;
    }
    if (kk < k1) {
      const float2 al = Dc[2 * kk * rs], dl = Dc[(2 * kk + 1) * rs];
      float2 x0, x1;
      lift::inv_db4(am, dm, al, dl, x0, x1);
      Dc[2 * kk * rs] = x0;
      Dc[(2 * kk + 1) * rs] = x1;
    }
  }
}

// Pairs [k0, k1) of one column when the range touches the halo (forward:
// its last pair reads the next CTA's rows 0, 1; inverse: its first pair reads
// the previous CTA's last pair).  Every other pair is done first; the halo is
// waited for only before the pair that reads it, so the exchange overlaps the
// column work.  The inverse order is in-place safe: pairs k0+1.. need pair
// k0 as it was, and pair k0 is updated last.
FI void wcl_col_edge(float2* Dc, const float2* H, const uint64_t* bar, bool& ok, int rs, int sr, int j, int m,
                     int k0, int k1, int kind, bool inverse, bool lo_final, const WclScale& sc) {
  if (!inverse) {
    if (k1 - k0 >= 2)
      wcl_col_pairs(Dc, rs, sr, j, k0, k1 - 1, Dc[2 * (k1 - 1) * rs], Dc[(2 * (k1 - 1) + 1) * rs], kind, false,
                    lo_final, sc);
    ok = wcl_wait(bar) && ok;
    wcl_col_pairs(Dc, rs, sr, j, k1 - 1, k1, H[j], H[m + j], kind, false, lo_final, sc);
  } else {
    if (k1 - k0 >= 2)
      wcl_col_pairs(Dc, rs, sr, j, k0 + 1, k1, Dc[2 * k0 * rs], Dc[(2 * k0 + 1) * rs], kind, true, lo_final, sc);
    ok = wcl_wait(bar) && ok;
    wcl_col_pairs(Dc, rs, sr, j, k0, k0 + 1, H[j], H[m + j], kind, true, lo_final, sc);
  }
}

// One level-l column step over the m columns and R_l rows; H holds the halo
// rows (forward: the next CTA's rows 0, 1; inverse: the previous CTA's last
// pair), counted on `bar` (Daubechies-4 only; null for Haar).  With at least
// 2m threads the pairs of a column are split into `parts` ranges, one thread
// each: every part first reads the rows its neighbouring part will overwrite
// (forward: the next part's first two rows; inverse: the previous part's
// last pair), the CTA synchronises, then all parts stream in place.  Whole
// columns (parts 1) synchronise before the first store too: wcl_push's threads
// read the boundary rows, and another thread than the one that reads a column's
// element there updates it.
FI void wcl_cols(float2* D, const float2* H, const uint64_t* bar, bool& ok, int n, int sr, int Rl, int m, int kind,
                 bool inverse, bool last_level, const WclScale& sc, int nth) {
  const int rs = sr * n, npair = Rl / 2;
  const bool halo = kind == 2;
  int parts = 1;
  while (parts * 2 * m <= nth && npair % (parts * 2) == 0) parts *= 2;  // equal ranges only
  if (parts == 1) {
    if (halo) __syncthreads();  // wcl_push reads the boundary rows that this step overwrites
    for (int j = threadIdx.x; j < m; j += nth) {
      const bool lo_final = last_level || j >= m / 2;
      if (halo)
        wcl_col_edge(D + j, H, bar, ok, rs, sr, j, m, 0, npair, kind, inverse, lo_final, sc);
      else
        wcl_col_pairs(D + j, rs, sr, j, 0, npair, H[j], H[m + j], kind, inverse, lo_final, sc);
    }
    return;
  }
  const int per = npair / parts, tid = threadIdx.x, j = tid % m, p = tid / m, k0 = p * per;
  const bool act = tid < m * parts;
  const bool edge = halo && (inverse ? p == 0 : p + 1 == parts);
  float2* Dc = D + j;
  float2 e0 = make_float2(0.f, 0.f), e1 = e0;
  if (act && !edge) {
    if (!inverse) {
      const bool last = p + 1 == parts;  // Haar: no row beyond the range is read
      e0 = last ? e0 : Dc[2 * (k0 + per) * rs];
      e1 = last ? e1 : Dc[(2 * (k0 + per) + 1) * rs];
    } else if (p > 0) {
      e0 = Dc[(2 * k0 - 2) * rs];
      e1 = Dc[(2 * k0 - 1) * rs];
    }
  }
  __syncthreads();
  if (!act) return;
  const bool lo_final = last_level || j >= m / 2;
  if (edge)
    wcl_col_edge(Dc, H, bar, ok, rs, sr, j, m, k0, k0 + per, kind, inverse, lo_final, sc);
  else
    wcl_col_pairs(Dc, rs, sr, j, k0, k0 + per, e0, e1, kind, inverse, lo_final, sc);
}

// rows row0, row1 (local) of width m to halo buffer Hb of CTA `to`
// (buffer rows of width m), counted on its mbarrier `bar`
FI void wcl_push(const float2* D, const float2* Hb, const uint64_t* bar, int n, int row0, int row1, int m,
                 unsigned to, int nth) {
  const int q4 = m / 2;  // float4 per row
  for (int q = threadIdx.x; q < 2 * q4; q += nth) {
    const int h = q / q4, jj = 2 * (q % q4);
    const float4 v = *reinterpret_cast<const float4*>(D + (h ? row1 : row0) * n + jj);
    wcl_st_async16(Hb + h * m + jj, bar, to, v);
  }
}

// NT, RT, KT: side, rows per CTA and wavelet kind fixed at compile time, so that
// the loop bounds, strides and offsets of every level are constants; LT: the
// levels too (0: from the argument).  One instantiation that took them all from
// its arguments served every size but 256^2 before: 228 us at 304 slices of
// 128^2, against 144 us for four times the pixels at 256^2.
//
// UPD (z = P^{-1} r of a PCG step): the load is the residual update as well:
// r -= alpha q, or r = A^H b - q for a slice at the start of its outer step, and
// the partial ||r||^2 (NaN beyond the FP32 range: k_pcg_scalars then sums r itself).  A launch and a pass over r less than an update of its own
// (solves of 60 slices of 256^2 4231 -> 4125 us, of one of 64^2 1588 -> 1502).  Up
// to WCL_NMAX: above, the clusters leave SMs idle that an update of its own uses
// (8 slices of 512^2: 7697 us apart, 8108 in one).
template <int NT, int RT, int LT, int KT, int TH, bool UPD>
__global__ void __launch_bounds__(TH, NT <= 256 ? 2 : 1)
k_wav_cluster(const float2* x, float2* u, const float* __restrict__ w, int L_arg, int mode, int mirror,
              const float2* r, double* __restrict__ part, int real, SliceState* __restrict__ st, float2* rw,
              const float2* __restrict__ q_in, const float2* __restrict__ atb, int axpy_mode) {
  chained_start();
  const int s = blockIdx.y;
  // the same slice for every CTA of the cluster: all of them leave or none
  if (st != nullptr && !slice_running(st, s)) return;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[32];
  __shared__ Sum3 rr_part[UPD ? TH / 32 : 1];
  constexpr int n = NT, R = RT, kind = KT;
  constexpr unsigned C = NT / RT;
  const int L = LT ? LT : L_arg, tid = threadIdx.x;
  const unsigned rank = wcl_rank();
  float2* D = reinterpret_cast<float2*>(smem);        // [R][n]
  float2* H = D + R * n;                              // halo buffers of the 2L exchanges
  uint64_t* mb = reinterpret_cast<uint64_t*>(H + wcl_halo_off(n, L, 2 * L));  // their mbarriers
  float* Wm = reinterpret_cast<float*>(mb + 2 * L);   // [R][n] weights (mirror)
  const size_t nn = (size_t)n * n;
  const float* ws = w + (size_t)s * nn;
  {
    const float2* xs = x + (size_t)s * nn + (size_t)rank * R * n;
    if (!UPD)
      for (int q = tid; q < R * n / 2; q += TH) wcl_cp16(D + 2 * q, xs + 2 * q);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    if (mirror) {  // the weight of the coefficient each position will hold
      for (int q = tid; q < R * n / 4; q += TH) {
        const int rho = 4 * q / n, j = 4 * q % n;
        wcl_cp16(Wm + 4 * q, ws + (size_t)wcl_coef_row(rho, j, n, L, R, rank) * n + j);
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  }
  if (kind == 2 && tid == 0) {  // arm every exchange: two halo rows of its level
    for (int e = 0; e < 2 * L; ++e) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(wcl_smem(mb + e)) : "memory");
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    for (int e = 0; e < 2 * L; ++e) {
      const unsigned bytes = 2u * (unsigned)(n >> (wcl_ex_level(L, e) - 1)) * 8u;
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(wcl_smem(mb + e)), "r"(bytes)
                   : "memory");
    }
  }
  bool updated = false;
  if (UPD) {
    const int ph = st[s].phase;
    updated = axpy_mode != AXPY_PER_SLICE || slice_working(ph);
    const bool first = axpy_mode == AXPY_INIT || (axpy_mode == AXPY_PER_SLICE && ph == PH_START);
    const float alpha = (float)st[s].alpha;
    const size_t off = ((size_t)s * nn + (size_t)rank * R * n) / 2;
    float4* r4 = reinterpret_cast<float4*>(rw) + off;
    const float4* src = updated && first ? reinterpret_cast<const float4*>(atb) + off : r4;
    const float4* q4 = reinterpret_cast<const float4*>(q_in) + off;
    Sum3 rr{0.f, 0.f, 0.f};
    constexpr int UN = 4;  // 16-byte loads of r and of q in flight per thread
    for (int i0 = tid; i0 < R * n / 2; i0 += UN * TH) {
      float4 rv[UN], qv[UN];
#pragma unroll
      for (int e = 0; e < UN; ++e) {
        const int i = i0 + e * TH;
        if (i < R * n / 2) {
          rv[e] = src[i];
          if (updated) qv[e] = q4[i];
        }
      }
      float acc = 0.f;
#pragma unroll
      for (int e = 0; e < UN; ++e) {
        const int i = i0 + e * TH;
        if (i >= R * n / 2) continue;
        float2 a = make_float2(rv[e].x, rv[e].y), b = make_float2(rv[e].z, rv[e].w);
        if (updated) {
          const float2 qa = make_float2(qv[e].x, qv[e].y), qb = make_float2(qv[e].z, qv[e].w);
          a = first ? csub(a, qa) : cfma(-alpha, qa, a);
          b = first ? csub(b, qb) : cfma(-alpha, qb, b);
          acc += cabs2(a) + cabs2(b);
          r4[i] = make_float4(a.x, a.y, b.x, b.y);
        }
        reinterpret_cast<float4*>(D)[i] = make_float4(a.x, a.y, b.x, b.y);
      }
      rr.add(acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rr.add(rr.from_lane(o));
    if ((tid & 31) == 0) rr_part[tid >> 5] = rr;
  }
  asm volatile("cp.async.wait_group 1;\n" ::: "memory");
  __syncthreads();
  if (UPD && updated && tid < 32) {
    Sum3 rr{0.f, 0.f, 0.f};
    if (tid < TH / 32) rr = rr_part[tid];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rr.add(rr.from_lane(o));
    if (tid == 0) part[((size_t)s * NSLOT + SLOT_RR) * MAXPART + rank] = rr.value();
  }
  if (kind == 2)  // every CTA's mbarriers armed before any remote write
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
  WclScale sc;
  sc.Wm = mirror ? Wm : nullptr;
  sc.ws = ws;
  sc.n = n;
  sc.L = L;
  sc.R = R;
  sc.rank = (int)rank;
  sc.mode = mode;
  sc.lam = st ? st[s].lam : 0.f;
  sc.abar = st ? st[s].abar : 0.f;
  bool ok = true;
#pragma unroll
  for (int l = 1; l <= (LT ? LT : WCL_LMAX); ++l) {
    if (l > L) break;
    const int m = n >> (l - 1), Rl = R >> (l - 1), sr = 1 << (l - 1), e = l - 1;
    wcl_rows<(NT + 63) / 64>(D, n, sr, Rl, m, kind, false, TH);
    __syncthreads();
    const float2* He = H + wcl_halo_off(n, L, e);
    if (kind == 2) {
      wcl_push(D, He, mb + e, n, 0, sr, m, (rank + C - 1) % C, TH);
    }
    if (l == 1) {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
      __syncthreads();
    }
    wcl_cols(D, He, mb + e, ok, n, sr, Rl, m, kind, false, l == L, sc, TH);
    __syncthreads();
  }
  float acc = 0.f;
#pragma unroll
  for (int lr = 0; lr < (LT ? LT : WCL_LMAX); ++lr) {
    const int l = L - lr;
    if (l < 1) break;
    const int m = n >> (l - 1), Rl = R >> (l - 1), sr = 1 << (l - 1), e = 2 * L - l;
    const float2* He = H + wcl_halo_off(n, L, e);
    if (kind == 2) {
      wcl_push(D, He, mb + e, n, (Rl - 2) * sr, (Rl - 1) * sr, m, (rank + 1) % C, TH);
      // the last remote write of this CTA is issued: arrive on the cluster
      // barrier that every CTA waits on before it exits
      if (l == 1) asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
    }
    wcl_cols(D, He, mb + e, ok, n, sr, Rl, m, kind, true, false, sc, TH);
    __syncthreads();
    if (l > 1) {
      wcl_rows<(NT + 63) / 64>(D, n, sr, Rl, m, kind, true, TH);
      __syncthreads();
    } else {  // the last row step writes u
      const size_t off = (size_t)s * nn + (size_t)rank * R * n;
      acc = wcl_rows<(NT + 63) / 64>(D, n, 1, R, n, kind, true, TH, u + off, r ? r + off : nullptr, real);
    }
  }
  if (!ok && st) st[s].fault = 1;  // a halo never arrived: results invalid
  if (part) {
    const double tot = block_sum((double)acc, red);
    if (tid == 0) part[((size_t)s * NSLOT + SLOT_RZ) * MAXPART + rank] = tot;
  }
  // no CTA leaves (releasing its shared memory) while a peer of the cluster
  // may still issue a write into it, even after a halo wait ran out; every
  // CTA reaches this point, so the wait ends
  if (kind == 2) asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}


inline int wcl_smem_bytes(int n, int R, int L, bool mirror) {
  return R * n * 8 + wcl_halo_off(n, L, 2 * L) * 8 + 2 * L * 8 + (mirror ? R * n * 4 : 0);
}

// A launch of the one-launch form: n / R CTAs per cluster and slice.
struct WclArgs {
  const float2* x;
  float2* u;
  const float* w;
  int levels, mode, mirror;
  const float2* r;
  double* part;
  int real;
  SliceState* st;
  int batch;
  cudaStream_t stream;
  bool chained;
  float2* rw;  // residual to update on the way in (x = r = rw), or null
  const float2 *q, *atb;
  int axpy_mode;
};

template <int N, int R, int TH>
inline void wcl_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, int levels, bool mirror, int batch,
                       cudaStream_t stream) {
  cfg = {};
  cfg.gridDim = dim3(N / R, batch);
  cfg.blockDim = dim3(TH);
  cfg.dynamicSmemBytes = wcl_smem_bytes(N, R, levels, mirror);
  cfg.stream = stream;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = N / R;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
}

template <int N, int R, int L, int KT, int TH> bool wcl_launch_as(const WclArgs& a) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[2];
  wcl_config<N, R, TH>(cfg, at, a.levels, a.mirror, a.batch, a.stream);
  if (a.chained) {
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
  }
  auto k = k_wav_cluster<N, R, L, KT, TH, false>;
  if constexpr (N <= WCL_NMAX) {
    if (a.rw) k = k_wav_cluster<N, R, L, KT, TH, true>;
  }
  return cudaLaunchKernelEx(&cfg, k, a.x, a.u, a.w, a.levels, a.mode, a.mirror, a.r,
                            a.part, a.real, a.st, a.rw, a.q, a.atb, a.axpy_mode) == cudaSuccess;
}
template <int N, int R, int L, int KT, int TH> bool wcl_attr_as() {
  const int bytes = wcl_smem_bytes(N, R, L ? L : WCL_LMAX, true);
  const cudaFuncAttribute A = cudaFuncAttributeMaxDynamicSharedMemorySize;
  bool ok = cudaFuncSetAttribute(k_wav_cluster<N, R, L, KT, TH, false>, A, bytes) == cudaSuccess;
  if constexpr (N <= WCL_NMAX)
    ok = cudaFuncSetAttribute(k_wav_cluster<N, R, L, KT, TH, true>, A, bytes) == cudaSuccess && ok;
  return ok;
}
// A cluster above the portable 8 CTAs: how many the device holds at once, 0
// where it cannot be launched.
template <int N, int R, int KT, int TH> int wcl_wide_resident() {
  auto k = k_wav_cluster<N, R, 0, KT, TH, false>;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  wcl_config<N, R, TH>(cfg, at, WCL_LMAX, true, 1, nullptr);
  int clusters = 0;
  if (!wcl_attr_as<N, R, 0, KT, TH>() ||
      cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&clusters, k, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return clusters;
}

// Every (size, rows per CTA) that wcl_rows_per_cta gives, with the threads per
// CTA: enough for two per column of the first level, so that a column's pairs
// are split.
#define WCL_SHAPES(X)                                                                                              \
  X(16, 2, 128) X(16, 4, 128) X(32, 4, 128) X(32, 8, 128) X(48, 6, 128) X(48, 8, 128) X(64, 8, 128) X(64, 16, 128) \
  X(80, 10, 256) X(80, 16, 256) X(96, 12, 256) X(96, 16, 256) X(128, 16, 256) X(128, 32, 256) X(160, 20, 512)      \
  X(160, 32, 512) X(192, 24, 512) X(192, 32, 512) X(256, 32, 512)

// The sizes above WCL_NMAX: one CTA per SM, more CTAs than a portable cluster.
// 512 threads at 512^2: 1024 leave 64 registers and spill (8 slices of 20 PCG
// steps 5.05 against 4.58 ms).
#define WCL_WIDE_SHAPES(X) X(320, 640) X(384, 768) X(512, 512)

template <int KT> bool wcl_launch_kind(int n, int R, const WclArgs& a) {
  if (n == 256 && a.levels == 4) return wcl_launch_as<256, 32, 4, KT, 512>(a);
#define WCL_CASE(N_, R_, T_) \
  if (n == N_ && R == R_) return wcl_launch_as<N_, R_, 0, KT, T_>(a);
  WCL_SHAPES(WCL_CASE)
#undef WCL_CASE
#define WCL_CASE(N_, T_) \
  if (n == N_ && R == WCL_WIDE_R) return wcl_launch_as<N_, WCL_WIDE_R, 0, KT, T_>(a);
  WCL_WIDE_SHAPES(WCL_CASE)
#undef WCL_CASE
  return false;
}
template <int KT> int wcl_wide_kind(int n) {
#define WCL_CASE(N_, T_) \
  if (n == N_) return wcl_wide_resident<N_, WCL_WIDE_R, KT, T_>();
  WCL_WIDE_SHAPES(WCL_CASE)
#undef WCL_CASE
  return 0;
}
template <int KT> bool wcl_attrs_kind() {
  bool ok = wcl_attr_as<256, 32, 4, KT, 512>();
#define WCL_CASE(N_, R_, T_) ok = wcl_attr_as<N_, R_, 0, KT, T_>() && ok;
  WCL_SHAPES(WCL_CASE)
#undef WCL_CASE
  return ok;
}
bool wcl_launch_haar(int n, int R, const WclArgs& a);
bool wcl_launch_db4(int n, int R, const WclArgs& a);
int wcl_wide_haar(int n);
int wcl_wide_db4(int n);
bool wcl_prepare_haar();
bool wcl_prepare_db4();

}  // namespace firls
