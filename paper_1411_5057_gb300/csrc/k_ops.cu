// Non-FFT kernels of the FIRLS hot path: lifting wavelets (Phi, Phi^T),
// weights (Eq. gw, Eq. Wog, Eq. wi), preconditioner set-up and application
// (Eq. pog, Eq. ptv with the L U factors of Sec. 4.2), PCG vector updates
// and the FP64 PCG scalars.
#include "wavelet.cuh"
#include "per_device.h"

namespace firls {

constexpr int WAV_THREADS = 256;
constexpr int WAV_RB = 8;            // output row pairs per CTA of a tiled level
constexpr int COARSE_MAX = 64;       // default largest block kept whole in shared memory
constexpr int COARSE_LIMIT = 64;     // the in-shared-memory transform handles up to 64^2 (2 pairs per lane)
constexpr int COARSE_THREADS = 256;

static int wav_rb(int m, int want = 0) {
  const int rb = want > 0 ? want : WAV_RB;
  return m / 2 < rb ? m / 2 : rb;
}

// One tiled analysis level on the m x m block `in` (row stride ld_in).  The
// horizontal step reads the input rows straight from global memory (16-byte
// pairs), the vertical step works from shared memory.
__global__ void __launch_bounds__(WAV_THREADS)
k_wav_fwd(const float2* __restrict__ in, size_t in_ss, int ld_in, float2* __restrict__ llo, size_t ll_ss,
          int ld_ll, float2* __restrict__ c, float* __restrict__ w, int n, int m, int rb, int kind,
          int mode, int last, const SliceState* __restrict__ st) {
  const int s = blockIdx.y;
  if (st != nullptr && !slice_running(st, s)) return;
  extern __shared__ __align__(16) unsigned char smem[];
  const int half = m / 2;
  const int k0 = blockIdx.x * rb;
  const int nrow = 2 * rb + (kind == 2 ? 2 : 0);
  float2* rt = reinterpret_cast<float2*>(smem);  // [nrow][m] row-transformed
  const float2* src = in + (size_t)s * in_ss;
  for (int idx = threadIdx.x; idx < nrow * half; idx += blockDim.x) {
    const int i = idx / half, k = idx % half;
    const float4* xr = reinterpret_cast<const float4*>(src + (size_t)((2 * k0 + i) % m) * ld_in);
    const float4 p0 = xr[k];
    float2 a, d;
    if (kind == 2) {
      const float4 p1 = xr[k + 1 < half ? k + 1 : 0];
      lift::fwd_db4(make_float2(p0.x, p0.y), make_float2(p0.z, p0.w), make_float2(p1.x, p1.y),
                    make_float2(p1.z, p1.w), a, d);
    } else {
      lift::fwd_haar(make_float2(p0.x, p0.y), make_float2(p0.z, p0.w), a, d);
    }
    rt[i * m + k] = a;
    rt[i * m + half + k] = d;
  }
  __syncthreads();
  const float lam = st ? st[s].lam : 0.f, abar = st ? st[s].abar : 0.f, eps = st ? st[s].eps : 1e-10f;
  float2* cs = c + (size_t)s * n * n;
  float* ws = w ? w + (size_t)s * n * n : nullptr;
  float2* lls = llo + (size_t)s * ll_ss;
  const int nout = min(rb, half - k0);
  for (int idx = threadIdx.x; idx < nout * m; idx += blockDim.x) {
    const int kk = idx / m, j = idx % m;
    float2 a, d;
    if (kind == 2) {
      lift::fwd_db4(rt[(2 * kk) * m + j], rt[(2 * kk + 1) * m + j], rt[(2 * kk + 2) * m + j],
                    rt[(2 * kk + 3) * m + j], a, d);
    } else {
      lift::fwd_haar(rt[(2 * kk) * m + j], rt[(2 * kk + 1) * m + j], a, d);
    }
    const int row = k0 + kk;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int orow = h ? half + row : row;
      const float2 v = h ? d : a;
      if (!h && j < half && !last) {  // LL of a non-final level: raw, to the ping-pong buffer
        lls[(size_t)row * ld_ll + j] = v;
        continue;
      }
      const size_t p = (size_t)orow * n + j;
      if (mode == WAV_RAW) {
        cs[p] = v;
      } else if (mode == WAV_MUL_W) {
        cs[p] = cscale(v, ws[p]);
      } else if (mode == WAV_MUL_PINV) {
        cs[p] = cscale(v, 1.0f / (abar + lam * ws[p]));
      } else {
        ws[p] = rsqrtf(cabs2(v) + eps);
      }
    }
  }
}

// One tiled synthesis level: LL from `lli` (row stride ld_ll), details from c
// (stride n) to the m x m output block.  Vertical step from global memory,
// horizontal step from shared memory; optional partial Re<r, out>.
__global__ void __launch_bounds__(WAV_THREADS)
k_wav_inv(const float2* __restrict__ lli, size_t ll_ss, int ld_ll, const float2* __restrict__ c,
          float2* __restrict__ out, size_t out_ss, int ld_out, int n, int m, int rb, int kind,
          const float2* __restrict__ r, double* __restrict__ part, int real,
          const SliceState* __restrict__ st) {
  const int s = blockIdx.y;
  if (st != nullptr && !slice_running(st, s)) return;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[32];
  const int half = m / 2;
  const int k0 = blockIdx.x * rb;
  const int nout = min(rb, half - k0);
  float2* vs = reinterpret_cast<float2*>(smem);  // [2 rb][m]
  const float2* cs = c + (size_t)s * n * n;
  const float2* ls = lli + (size_t)s * ll_ss;
  for (int idx = threadIdx.x; idx < nout * m; idx += blockDim.x) {
    const int kk = idx / m, j = idx % m;
    const int k = k0 + kk;
    const float2 al = j < half ? ls[(size_t)k * ld_ll + j] : cs[(size_t)k * n + j];
    const float2 dl = cs[(size_t)(half + k) * n + j];
    float2 x0, x1;
    if (kind == 2) {
      const int km = (k - 1 + half) % half;
      const float2 am = j < half ? ls[(size_t)km * ld_ll + j] : cs[(size_t)km * n + j];
      const float2 dm = cs[(size_t)(half + km) * n + j];
      lift::inv_db4(am, dm, al, dl, x0, x1);
    } else {
      lift::inv_haar(al, dl, x0, x1);
    }
    vs[(2 * kk) * m + j] = x0;
    vs[(2 * kk + 1) * m + j] = x1;
  }
  __syncthreads();
  float2* os = out + (size_t)s * out_ss;
  const float2* rs = r ? r + (size_t)s * n * n : nullptr;
  float acc = 0.f;
  for (int idx = threadIdx.x; idx < 2 * nout * half; idx += blockDim.x) {
    const int i = idx / half, l = idx % half;
    const float2* vr = vs + i * m;
    float2 x0, x1;
    if (kind == 2) {
      const int lm = (l - 1 + half) % half;
      lift::inv_db4(vr[lm], vr[half + lm], vr[l], vr[half + l], x0, x1);
    } else {
      lift::inv_haar(vr[l], vr[half + l], x0, x1);
    }
    if (real) {
      x0.y = 0.f;
      x1.y = 0.f;
    }
    const int orow = 2 * k0 + i;
    reinterpret_cast<float4*>(os + (size_t)orow * ld_out)[l] = make_float4(x0.x, x0.y, x1.x, x1.y);
    if (rs) {
      const float4 rv = reinterpret_cast<const float4*>(rs + (size_t)orow * n)[l];
      acc += rdot2(make_float2(rv.x, rv.y), x0) + rdot2(make_float2(rv.z, rv.w), x1);
    }
  }
  if (part) {
    const double tot = block_sum((double)acc, red);
    if (threadIdx.x == 0) part[((size_t)s * NSLOT + SLOT_RZ) * MAXPART + blockIdx.x] = tot;
  }
}

// ---- coarse levels of one slice in shared memory ----
// In-place one-level analysis of the top-left m x m block of S (row stride
// ls): every lane reads the inputs of its pairs, the warp syncs, then writes
// [lo | hi].  m <= COARSE_MAX, so a lane holds at most two pairs.
FI void smem_fwd_level(float2* S, int ls, int m, int kind) {
  const int half = m / 2, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int pass = 0; pass < 2; ++pass) {  // 0: rows, 1: columns
    const int es = pass ? ls : 1;         // element stride along the line
    for (int line = wid; line < m; line += nw) {
      float2* L = pass ? S + line : S + (size_t)line * ls;
      float2 a[2], d[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int k = lane + 32 * u;
        if (k < half) {
          if (kind == 2) {
            lift::fwd_db4(L[(2 * k) * es], L[(2 * k + 1) * es], L[((2 * k + 2) % m) * es],
                          L[((2 * k + 3) % m) * es], a[u], d[u]);
          } else {
            lift::fwd_haar(L[(2 * k) * es], L[(2 * k + 1) * es], a[u], d[u]);
          }
        }
      }
      __syncwarp();
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int k = lane + 32 * u;
        if (k < half) {
          L[k * es] = a[u];
          L[(half + k) * es] = d[u];
        }
      }
      __syncwarp();
    }
    __syncthreads();
  }
}

// In-place inverse of smem_fwd_level (columns first, then rows).
FI void smem_inv_level(float2* S, int ls, int m, int kind) {
  const int half = m / 2, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int pass = 0; pass < 2; ++pass) {  // 0: columns, 1: rows
    const int es = pass ? 1 : ls;
    for (int line = wid; line < m; line += nw) {
      float2* L = pass ? S + (size_t)line * ls : S + line;
      float2 x0[2], x1[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int l = lane + 32 * u;
        if (l < half) {
          if (kind == 2) {
            const int lm = (l - 1 + half) % half;
            lift::inv_db4(L[lm * es], L[(half + lm) * es], L[l * es], L[(half + l) * es], x0[u], x1[u]);
          } else {
            lift::inv_haar(L[l * es], L[(half + l) * es], x0[u], x1[u]);
          }
        }
      }
      __syncwarp();
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int l = lane + 32 * u;
        if (l < half) {
          L[(2 * l) * es] = x0[u];
          L[(2 * l + 1) * es] = x1[u];
        }
      }
      __syncwarp();
    }
    __syncthreads();
  }
}

enum { COARSE_FWD = 1, COARSE_INV = 2 };

// Levels l0..L of one slice on the m0 x m0 block (m0 <= COARSE_MAX) held in
// shared memory.  FWD: analysis of `src`; without INV the coefficients are
// stored per `mode` at their Mallat positions (top-left block of c / w).
// FWD|INV: analysis, per-coefficient scaling (MUL_W or MUL_PINV), synthesis;
// the coarse coefficients never leave shared memory.  INV alone: synthesis
// of the coefficients read from c.  The synthesised block goes to `dst`.
__global__ void __launch_bounds__(COARSE_THREADS)
k_wav_coarse(const float2* __restrict__ src, size_t src_ss, int src_ld, float2* __restrict__ dst, size_t dst_ss,
             int dst_ld, float2* __restrict__ c, float* __restrict__ w, int n, int m0, int nlev, int kind,
             int mode, int flags, const float2* __restrict__ r, double* __restrict__ part, int real,
             const SliceState* __restrict__ st) {
  const int s = blockIdx.x;
  if (st != nullptr && !slice_running(st, s)) return;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[32];
  float2* S = reinterpret_cast<float2*>(smem);
  const int ls = m0 + 1;
  const size_t nn = (size_t)n * n;
  float2* cs = c + (size_t)s * nn;
  float* ws = w ? w + (size_t)s * nn : nullptr;
  const int cnt = m0 * m0;
  // the block goes to shared memory with asynchronous 8-byte copies, all in
  // flight at once (rows keep the odd stride ls that spreads column accesses)
  {
    const float2* sp = (flags & COARSE_FWD) ? src + (size_t)s * src_ss : cs;
    const size_t sld = (flags & COARSE_FWD) ? (size_t)src_ld : (size_t)n;
    for (int idx = threadIdx.x; idx < cnt; idx += blockDim.x) {
      const int rr = idx / m0, cc = idx % m0;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(
                       (unsigned)__cvta_generic_to_shared(S + rr * ls + cc)),
                   "l"(sp + rr * sld + cc)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;\n cp.async.wait_all;\n" ::: "memory");
  }
  __syncthreads();
  if (flags & COARSE_FWD) {
    // the coefficient weights this thread scales, fetched before the levels run
    constexpr int WMAX = COARSE_LIMIT * COARSE_LIMIT / COARSE_THREADS;
    float wv[WMAX];
    if ((flags & COARSE_INV) && ws) {
#pragma unroll
      for (int k = 0; k < WMAX; ++k) {
        const int idx = threadIdx.x + COARSE_THREADS * k;
        wv[k] = idx < cnt ? ws[(size_t)(idx / m0) * n + idx % m0] : 0.f;
      }
    }
    for (int lev = 0; lev < nlev; ++lev) smem_fwd_level(S, ls, m0 >> lev, kind);
    const float lam = st ? st[s].lam : 0.f, abar = st ? st[s].abar : 0.f, eps = st ? st[s].eps : 1e-10f;
    if (flags & COARSE_INV) {
#pragma unroll
      for (int k = 0; k < WMAX; ++k) {
        const int idx = threadIdx.x + COARSE_THREADS * k;
        if (idx < cnt) {
          float2& v = S[(idx / m0) * ls + idx % m0];
          v = cscale(v, mode == WAV_MUL_W ? wv[k] : 1.0f / (abar + lam * wv[k]));
        }
      }
    }
    for (int idx = threadIdx.x; idx < cnt && !(flags & COARSE_INV); idx += blockDim.x) {
      const int rr = idx / m0, cc = idx % m0;
      const size_t p = (size_t)rr * n + cc;
      float2& v = S[rr * ls + cc];
      if (mode == WAV_RAW) {
        cs[p] = v;
      } else if (mode == WAV_MUL_W) {
        cs[p] = cscale(v, ws[p]);
      } else if (mode == WAV_MUL_PINV) {
        cs[p] = cscale(v, 1.0f / (abar + lam * ws[p]));
      } else {
        ws[p] = rsqrtf(cabs2(v) + eps);
      }
    }
    __syncthreads();
  }
  if (!(flags & COARSE_INV)) return;
  for (int lev = nlev - 1; lev >= 0; --lev) smem_inv_level(S, ls, m0 >> lev, kind);
  float2* dp = dst + (size_t)s * dst_ss;
  const float2* rs = r ? r + (size_t)s * nn : nullptr;
  float acc = 0.f;
  for (int idx = threadIdx.x; idx < cnt; idx += blockDim.x) {
    const int rr = idx / m0, cc = idx % m0;
    float2 v = S[rr * ls + cc];
    if (real) v.y = 0.f;
    dp[(size_t)rr * dst_ld + cc] = v;
    if (rs) acc += rdot2(rs[(size_t)rr * n + cc], v);
  }
  if (part) {
    const double tot = block_sum((double)acc, red);
    if (threadIdx.x == 0) part[((size_t)s * NSLOT + SLOT_RZ) * MAXPART] = tot;
  }
}

// Clusters of the one-launch form above WCL_NMAX that the current device
// holds at once (0: it cannot launch them), asked once per device.
static int wide_resident(int n, int kind) {
  static PerDeviceOnce once;
  static int held[64][2][3];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev >= 64) return 0;
  once.run([dev] {
    for (int i = 0; i < 3; ++i) {
      constexpr int side[3] = {320, 384, 512};
      held[dev][0][i] = wcl_wide_haar(side[i]);
      held[dev][1][i] = wcl_wide_db4(side[i]);
    }
    return true;
  });
  const int i = n == 320 ? 0 : n == 384 ? 1 : n == 512 ? 2 : -1;
  return i < 0 ? 0 : held[dev][kind - 1][i];
}

// Rows per CTA of the one-launch form (0 when it does not apply): the
// fewest rows (most CTAs, at most 8 per cluster) for which every level has an
// even number of rows per CTA.  choice: 0 default, 1 weights mirrored in
// shared memory, 2 read from HBM; *mirror receives which.  Above 256^2 only the
// default takes it, with clusters of n / 32 CTAs where the device launches
// them.  Solves of 20 PCG steps, 5 levels, against the tiled levels with 8 rows
// a CTA: 512^2 D4 1 slice 4.8 -> 2.5 ms, 8 slices 6.5 -> 4.6 (two waves of
// clusters, 7 fit at once), 64 slices 25.2 -> 21.4; 320^2 5 slices 3.8 -> 2.1,
// 120 slices 17.3 -> 16.2; 384^2 8 slices 5.0 -> 2.7, 80 slices 19.0 -> 18.6;
// Haar gains more.  No batch is left for which the tiled levels are faster.
static int wcl_rows_per_cta(int n, int L, int kind, int choice, bool* mirror) {
  if (kind != 1 && kind != 2) return 0;
  if (choice != 0 && choice != 1 && choice != 2) return 0;
  if (choice == 0 && n > WCL_NMAX) {
    if (L < 1 || L > WCL_LMAX || (n >> L) % 4 || !wide_resident(n, kind)) return 0;
    if (mirror) *mirror = true;
    return WCL_WIDE_R;
  }
  if (n % 8 || n > WCL_NMAX || L < 1 || L > WCL_LMAX || (n >> L) % 4) return 0;
  for (int C = 8; C >= 1; --C) {
    if (n % (C << L) || n / C > WCL_RMAX) continue;
    if (mirror) *mirror = choice != 2;
    return n / C;
  }
  return 0;
}

static void wcl_launch(const WavArgs& a, int R, bool mirror, const float2* x, const float* w, int mode, float2* u,
                       const float2* r, int real) {
  const WclArgs c{x,    u,    w,       a.levels,
                  mode, mirror ? 1 : 0, r, r ? a.part : nullptr,
                  real, const_cast<SliceState*>(a.st), a.batch, a.stream, a.chained,
                  a.upd_q ? const_cast<float2*>(r) : nullptr, a.upd_q, a.upd_atb, a.upd_mode};
  if (a.kind == 2) wcl_launch_db4(a.n, R, c);
  else wcl_launch_haar(a.n, R, c);
}

static int coarse_smem(int m0) { return m0 * (m0 + 1) * 8; }

// Dynamic shared-memory limits of the wavelet kernels,
// set once per device.
static void set_wav_attrs() {
  static PerDeviceOnce once;
  once.run([] {
    const cudaFuncAttribute A = cudaFuncAttributeMaxDynamicSharedMemorySize;
    bool ok = cudaFuncSetAttribute(k_wav_fwd, A, (2 * 16 + 2) * 512 * 8) == cudaSuccess;
    ok = cudaFuncSetAttribute(k_wav_inv, A, 2 * 16 * 512 * 8) == cudaSuccess && ok;
    ok = cudaFuncSetAttribute(k_wav_coarse, A, coarse_smem(COARSE_LIMIT)) == cudaSuccess && ok;
    ok = wcl_prepare_haar() && ok;
    ok = wcl_prepare_db4() && ok;
    return ok;
  });
}

void wav_prepare() { set_wav_attrs(); }

// First level handled by the coarse kernel: its input side m <= cmax.
static int coarse_first_level(int n, int levels, int cmax = 0) {
  const int lim = cmax > 0 ? (cmax < COARSE_LIMIT ? cmax : COARSE_LIMIT) : COARSE_MAX;
  int l0 = 1;
  while (l0 <= levels && (n >> (l0 - 1)) > lim) ++l0;
  return l0;  // levels + 1 when no level fits
}

// Tiled analysis of levels 1 .. lend; returns the buffer holding LL_lend.
static const float2* tiled_forward(const WavArgs& a, const float2* x, float2* c, float* w, int mode, int lend,
                                   bool ll_final_to_c, size_t* ss, int* ld) {
  const int n = a.n;
  const size_t hh = (size_t)(n / 2) * (n / 2);
  const float2* src = x;
  size_t src_ss = (size_t)n * n;
  int src_ld = n;
  for (int l = 1; l <= lend; ++l) {
    const int m = n >> (l - 1), half = m / 2;
    const bool to_c = ll_final_to_c && l == lend;
    float2* dst = to_c ? c : ((l & 1) ? a.tmpA : a.tmpB);
    const size_t dst_ss = to_c ? (size_t)n * n : hh;
    const int dst_ld = to_c ? n : half;
    const int rb = wav_rb(m, a.rb);
    const int smem = (2 * rb + (a.kind == 2 ? 2 : 0)) * m * 8;
    k_wav_fwd<<<dim3((half + rb - 1) / rb, a.batch), WAV_THREADS, smem, a.stream>>>(
        src, src_ss, src_ld, dst, dst_ss, dst_ld, c, w, n, m, rb, a.kind, mode, to_c ? 1 : 0, a.st);
    src = dst;
    src_ss = dst_ss;
    src_ld = dst_ld;
  }
  *ss = src_ss;
  *ld = src_ld;
  return src;
}

// Tiled synthesis of levels lstart .. 1 with LL_lstart in (lli, ll_ss, ll_ld).
static void tiled_inverse(const WavArgs& a, const float2* lli, size_t ll_ss, int ll_ld, const float2* c,
                          float2* x, int lstart, const float2* r, int real) {
  const int n = a.n;
  const size_t hh = (size_t)(n / 2) * (n / 2);
  for (int l = lstart; l >= 1; --l) {
    const int m = n >> (l - 1), half = m / 2;
    const bool final_level = (l == 1);
    // write into the ping-pong buffer the input does not occupy
    float2* out = final_level ? x : (lli == a.tmpA ? a.tmpB : a.tmpA);
    const size_t out_ss = final_level ? (size_t)n * n : hh;
    const int out_ld = final_level ? n : m;
    const int rb = wav_rb(m, a.rb);
    k_wav_inv<<<dim3((half + rb - 1) / rb, a.batch), WAV_THREADS, 2 * rb * m * 8, a.stream>>>(
        lli, ll_ss, ll_ld, c, out, out_ss, out_ld, n, m, rb, a.kind, final_level ? r : nullptr,
        final_level && r ? a.part : nullptr, real, a.st);
    lli = out;
    ll_ss = out_ss;
    ll_ld = out_ld;
  }
}

void wavelet_forward(const WavArgs& a, const float2* x, float2* c, float* w, int mode) {
  set_wav_attrs();
  const int n = a.n, L = a.levels;
  const int l0 = coarse_first_level(n, L, a.coarse_max);
  size_t ss;
  int ld;
  const float2* ll = tiled_forward(a, x, c, w, mode, l0 - 1, l0 > L, &ss, &ld);
  if (l0 <= L) {
    const int m0 = n >> (l0 - 1);
    k_wav_coarse<<<a.batch, COARSE_THREADS, coarse_smem(m0), a.stream>>>(
        ll, ss, ld, nullptr, 0, 0, c, w, n, m0, L - l0 + 1, a.kind, mode, COARSE_FWD, nullptr, nullptr, 0, a.st);
  }
}

void wavelet_inverse(const WavArgs& a, const float2* c, float2* x, const float2* r, int real) {
  set_wav_attrs();
  const int n = a.n, L = a.levels;
  const int l0 = coarse_first_level(n, L, a.coarse_max);
  if (l0 <= L) {
    const int m0 = n >> (l0 - 1);
    const bool final_coarse = (l0 == 1);
    float2* dst = final_coarse ? x : ((l0 - 1) & 1 ? a.tmpA : a.tmpB);
    const size_t dss = final_coarse ? (size_t)n * n : (size_t)(n / 2) * (n / 2);
    const int dld = final_coarse ? n : m0;
    k_wav_coarse<<<a.batch, COARSE_THREADS, coarse_smem(m0), a.stream>>>(
        nullptr, 0, 0, dst, dss, dld, const_cast<float2*>(c), nullptr, n, m0, L - l0 + 1, a.kind, WAV_RAW,
        COARSE_INV, final_coarse ? r : nullptr, final_coarse && r ? a.part : nullptr, real, a.st);
    if (!final_coarse) tiled_inverse(a, dst, dss, dld, c, x, l0 - 1, r, real);
  } else {
    tiled_inverse(a, c, (size_t)n * n, n, c, x, L, r, real);
  }
}

// u = Phi^T (s o Phi x) with s = w (MUL_W) or 1/(abar + lam w) (MUL_PINV).
void wavelet_apply(const WavArgs& a, const float2* x, float2* c, float* w, int mode, float2* u,
                   const float2* r, int real) {
  set_wav_attrs();
  const int n = a.n, L = a.levels;
  bool mirror = false;
  const int R = wcl_rows_per_cta(n, L, a.kind, a.rb, &mirror);
  if (R > 0) {  // every level on chip, c untouched
    wcl_launch(a, R, mirror, x, w, mode, u, r, real);
    return;
  }
  const int l0 = coarse_first_level(n, L, a.coarse_max);
  if (l0 > L) {
    wavelet_forward(a, x, c, w, mode);
    wavelet_inverse(a, c, u, r, real);
    return;
  }
  size_t ss;
  int ld;
  const float2* ll = tiled_forward(a, x, c, w, mode, l0 - 1, false, &ss, &ld);
  const int m0 = n >> (l0 - 1);
  const bool final_coarse = (l0 == 1);
  float2* dst = final_coarse ? u : const_cast<float2*>(ll);  // LL' overwrites LL in place
  const size_t dss = final_coarse ? (size_t)n * n : ss;
  const int dld = final_coarse ? n : ld;
  k_wav_coarse<<<a.batch, COARSE_THREADS, coarse_smem(m0), a.stream>>>(
      ll, ss, ld, dst, dss, dld, c, w, n, m0, L - l0 + 1, a.kind, mode, COARSE_FWD | COARSE_INV,
      final_coarse ? r : nullptr, final_coarse && r ? a.part : nullptr, real, a.st);
  if (!final_coarse) tiled_inverse(a, dst, dss, dld, c, u, l0 - 1, r, real);
}

// CTAs per slice of the one-launch cluster form of wavelet_apply (0: tiled).
int wavelet_cluster_ctas(int n, int levels, int kind, int rb) {
  const int R = wcl_rows_per_cta(n, levels, kind, rb, nullptr);
  return R ? n / R : 0;
}

// Whether wavelet_apply takes the residual update in (WavArgs::upd_q).
bool wavelet_updates(int n, int levels, int kind, int rb) {
  return n <= WCL_NMAX && wcl_rows_per_cta(n, levels, kind, rb, nullptr) > 0;
}

// Partial-sum count of the wavelet_apply stage that computes Re<r, Phi^T ...>.
int wavelet_apply_ctas(int n, int levels, int kind, int rb, int cmax) {
  const int C = wavelet_cluster_ctas(n, levels, kind, rb);
  if (C > 0) return C;
  if (coarse_first_level(n, levels, cmax) == 1) return 1;
  return (n / 2 + wav_rb(n, rb) - 1) / wav_rb(n, rb);
}

// Launches per wavelet_apply call (for the launch count).
int wavelet_apply_launches(int n, int levels, int kind, int rb, int cmax) {
  if (wavelet_cluster_ctas(n, levels, kind, rb) > 0) return 1;
  const int l0 = coarse_first_level(n, levels, cmax);
  if (l0 > levels) return 2 * levels;
  return 2 * (l0 - 1) + 1;
}

// ================================================================== TV =====

// Isotropic TV (wtv2 null): W_i = (|grad_1 x_i|^2 + |grad_2 x_i|^2 + eps)^(-1/2)
// (Eq. wi).  l1 TV (Eq. l1): W1_i = (|grad_1 x_i|^2 + eps)^(-1/2) into wtv and
// W2_i = (|grad_2 x_i|^2 + eps)^(-1/2) into wtv2.  Zero extension.  Joint TV
// (Sec. 5.6, C > 1 contrasts in consecutive slices, isotropic only): the
// squared gradients of all contrasts of the image are summed under the root,
// and every contrast gets the same W.
__global__ void k_tv_weights(int n, int C, const SliceState* __restrict__ st, const float2* __restrict__ x,
                             float* __restrict__ wtv, float* __restrict__ wtv2) {
  const int s = blockIdx.y;
  if (!slice_running(st, s)) return;
  const float eps = st[s].eps;
  const size_t base = (size_t)s * n * n;
  const size_t img = (size_t)(s - s % C) * n * n;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n * n; i += gridDim.x * blockDim.x) {
    const int r = i / n, c = i % n;
    if (C > 1) {
      float g = 0.f;
      for (int t = 0; t < C; ++t) {
        const size_t bt = img + (size_t)t * n * n;
        const float2 xc = x[bt + i];
        const float2 g1 = c > 0 ? csub(xc, x[bt + i - 1]) : xc;
        const float2 g2 = r > 0 ? csub(xc, x[bt + i - n]) : xc;
        g += cabs2(g1) + cabs2(g2);
      }
      wtv[base + i] = rsqrtf(g + eps);
      continue;
    }
    const float2 xc = x[base + i];
    const float2 g1 = c > 0 ? csub(xc, x[base + i - 1]) : xc;
    const float2 g2 = r > 0 ? csub(xc, x[base + i - n]) : xc;
    if (wtv2) {
      wtv[base + i] = rsqrtf(cabs2(g1) + eps);
      wtv2[base + i] = rsqrtf(cabs2(g2) + eps);
    } else {
      wtv[base + i] = rsqrtf(cabs2(g1) + cabs2(g2) + eps);
    }
  }
}

void tv_weights(int batch, int n, cudaStream_t s, const SliceState* st, const float2* x, float* wtv, float* wtv2,
                int channels) {
  const int N = n * n;
  const int blocks = (N + 255) / 256 < 64 ? (N + 255) / 256 : 64;
  k_tv_weights<<<dim3(blocks, batch), 256, 0, s>>>(n, channels, st, x, wtv, wtv2);
}

// Joint wavelet sparsity (Sec. 5.6, FIRLS_MT): coefficient j of the C
// contrasts of an image forms one non-overlapping group, W_j = (sum_t
// |(Phi x_t)_j|^2 + eps)^(-1/2) (Eq. gw), written to every contrast.  cw holds
// the raw coefficients of all slices.
__global__ void k_joint_wavelet_weights(int N, int C, const SliceState* __restrict__ st,
                                        const float2* __restrict__ cw, float* __restrict__ ww) {
  const int s = blockIdx.y;
  if (!slice_running(st, s)) return;
  const float eps = st[s].eps;
  const size_t img = (size_t)(s - s % C) * N;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x) {
    float g = 0.f;
    for (int t = 0; t < C; ++t) g += cabs2(cw[img + (size_t)t * N + j]);
    ww[(size_t)s * N + j] = rsqrtf(g + eps);
  }
}

void joint_wavelet_weights(int batch, int n, int channels, cudaStream_t s, const SliceState* st, const float2* cw,
                           float* ww) {
  const int N = n * n;
  const int blocks = (N + 255) / 256 < 64 ? (N + 255) / 256 : 64;
  k_joint_wavelet_weights<<<dim3(blocks, batch), 256, 0, s>>>(N, channels, st, cw, ww);
}

// Exact diag(Phi^T diag(w) Phi).  Each 2-D basis function of level l is an
// outer product of 1-D level-l functions f_{l,type}(i - 2^l p) (type 0 low,
// 1 high) whose squares are tabulated (sqtab[(l-1)*2 + type][0 .. sqlen)),
// so the diagonal is a separable sum over levels and subbands:
//   diag(r, c) = sum_l sum_br sum_pr F_{l,br}(r - 2^l pr) T_{l,br}(pr, c),
//   T_{l,br}(pr, c) = sum_{bands (br, bc)} sum_pc F_{l,bc}(c - 2^l pc) w_band(pr, pc),
// indices periodic.  Bands at level l (h = n >> l, Mallat layout):
// (0,1) rows [0,h) cols [h,2h); (1,0) rows [h,2h) cols [0,h); (1,1) rows and
// cols [h,2h); at the last level also (0,0), rows and cols [0,h).
//
// A filter has at most TAPS 2^l taps, so an output meets TAPS coarse rows and a
// T value TAPS coefficients per band: T_{l,br}(p, c) for p = r >> l, .. - (TAPS -
// 1).  A thread owns WD_RB output rows of one column; per level it walks down
// the coarse rows with the last TAPS T values of both types in registers, and
// each fine row adds its filtered sum.  The groups of fine rows that share
// r >> l are fixed at compile time (r0 is a multiple of 16), so only the row
// filter's taps come from shared memory, as one float4 per type.  Bound by the
// load/store pipe (14 weights and 8 tap vectors a pixel at four levels).  T rows
// shared by a CTA, with taps and row indices found per term, took 690 us at 304
// slices of 256^2; this takes 200 (weights stage as a whole: 1028 -> 536 us there,
// 506 -> 166 at 304 x 128^2, 98 -> 45 for one slice).
constexpr int WD_RB = 16, WD_LMAX = 9;  // n <= 512
constexpr int WD_COLS = 64;             // threads: enough CTAs for one slice

template <int TAPS, int LG>  // 2^LG fine rows of the 16 share a coarse row
FI void wd_level(float (&acc)[WD_RB], int n, int l, bool last, int r0, int c, const float* __restrict__ ws,
                 const float* __restrict__ F0, const float* __restrict__ F1, int len0, int len1,
                 const float4 (*fr)[WD_RB]) {
  constexpr int G = 1 << LG, NP = WD_RB >> LG;
  const int h = n >> l, p0 = r0 >> l, cq = c >> l, phase = c & ((1 << l) - 1);
  float f0[TAPS], f1[TAPS];
  int q[TAPS];
#pragma unroll
  for (int i = 0; i < TAPS; ++i) {
    const int sc = phase + (i << l);
    f0[i] = sc < len0 ? F0[sc] : 0.f;
    f1[i] = sc < len1 ? F1[sc] : 0.f;
    q[i] = ((cq - i) % h + h) % h;
  }
  float t0[TAPS] = {}, t1[TAPS] = {};  // [i]: T of coarse row p - i, types 0 and 1
#pragma unroll
  for (int pp = 1 - TAPS; pp < NP; ++pp) {
#pragma unroll
    for (int i = TAPS - 1; i > 0; --i) {
      t0[i] = t0[i - 1];
      t1[i] = t1[i - 1];
    }
    const float* wl = ws + (size_t)(((p0 + pp) % h + h) % h) * n;  // row of type 0
    const float* wh = wl + (size_t)h * n;
    float a = 0.f, b = 0.f;
    if (last) {
#pragma unroll
      for (int i = 0; i < TAPS; ++i) a = fmaf(f0[i], wl[q[i]], a);
    }
#pragma unroll
    for (int i = 0; i < TAPS; ++i) a = fmaf(f1[i], wl[h + q[i]], a);
#pragma unroll
    for (int i = 0; i < TAPS; ++i) b = fmaf(f0[i], wh[q[i]], b);
#pragma unroll
    for (int i = 0; i < TAPS; ++i) b = fmaf(f1[i], wh[h + q[i]], b);
    t0[0] = a;
    t1[0] = b;
    if (pp < 0) continue;
#pragma unroll
    for (int k = 0; k < G; ++k) {
      const float4 u = fr[0][k], v = fr[1][k];
      const float uu[3] = {u.x, u.y, u.z}, vv[3] = {v.x, v.y, v.z};
      float o = acc[pp * G + k];
#pragma unroll
      for (int i = 0; i < TAPS; ++i) o = fmaf(uu[i], t0[i], o);
#pragma unroll
      for (int i = 0; i < TAPS; ++i) o = fmaf(vv[i], t1[i], o);
      acc[pp * G + k] = o;
    }
  }
}

template <int TAPS>
__global__ void __launch_bounds__(WD_COLS, 10) k_wavelet_diag(int n, int levels, const SliceState* __restrict__ st,
                                                          const float* __restrict__ w, float* __restrict__ out,
                                                          const float* __restrict__ sqtab,
                                                          const int* __restrict__ sqlen) {
  const int s = blockIdx.z;
  if (!slice_running(st, s)) return;
  const int r0 = blockIdx.y * WD_RB;
  // fr[l - 1][type][k]: the taps that meet fine row r0 + k (those of its phase)
  __shared__ float4 fr[WD_LMAX][2][WD_RB];
  for (int i = threadIdx.x; i < levels * 2 * WD_RB; i += WD_COLS) {
    const int k = i % WD_RB, type = i / WD_RB % 2, l = i / (2 * WD_RB) + 1;
    const int phase = (r0 + k) & ((1 << l) - 1), len = sqlen[(l - 1) * 2 + type];
    const float* F = sqtab + (size_t)((l - 1) * 2 + type) * n;
    float f[3];
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const int sr = phase + (t << l);
      f[t] = sr < len ? F[sr] : 0.f;
    }
    fr[l - 1][type][k] = make_float4(f[0], f[1], f[2], 0.f);
  }
  __syncthreads();
  const int c = blockIdx.x * WD_COLS + threadIdx.x;
  if (c >= n) return;
  const size_t base = (size_t)s * n * n;
  float acc[WD_RB];
#pragma unroll
  for (int k = 0; k < WD_RB; ++k) acc[k] = 0.f;
  for (int l = 1; l <= levels; ++l) {
    const float* F0 = sqtab + (size_t)(l - 1) * 2 * n;
    const int len0 = sqlen[(l - 1) * 2], len1 = sqlen[(l - 1) * 2 + 1];
    const bool last = l == levels;
    if (l == 1) wd_level<TAPS, 1>(acc, n, l, last, r0, c, w + base, F0, F0 + n, len0, len1, fr[l - 1]);
    else if (l == 2) wd_level<TAPS, 2>(acc, n, l, last, r0, c, w + base, F0, F0 + n, len0, len1, fr[l - 1]);
    else if (l == 3) wd_level<TAPS, 3>(acc, n, l, last, r0, c, w + base, F0, F0 + n, len0, len1, fr[l - 1]);
    else wd_level<TAPS, 4>(acc, n, l, last, r0, c, w + base, F0, F0 + n, len0, len1, fr[l - 1]);
  }
#pragma unroll
  for (int k = 0; k < WD_RB; ++k) out[base + (size_t)(r0 + k) * n + c] = acc[k];
}

void wavelet_diag(int batch, int n, int levels, int kind, cudaStream_t s, const SliceState* st, const float* w,
                  float* out, const float* sqtab, const int* sqlen) {
  const dim3 grid((n + WD_COLS - 1) / WD_COLS, n / WD_RB, batch);  // n % 16 = 0 for every size
  if (kind == 2) k_wavelet_diag<3><<<grid, WD_COLS, 0, s>>>(n, levels, st, w, out, sqtab, sqlen);
  else k_wavelet_diag<1><<<grid, WD_COLS, 0, s>>>(n, levels, st, w, out, sqtab, sqlen);
}

// P = abar I + lam_tv (D1^T W1 D1 + D2^T W2 D2) [+ lam diag(Phi^T W Phi)]
// (Eq. ptv; W1 = W2 = W for isotropic TV, wtv2 null): ia = 1 / a_i, the
// inverse diagonal, a_i = abar + lam_tv (W1_i + W1_{i+1} + W2_i + W2_{i+n}).
// For the Jacobi scale; the sweeps' set-up is k_penta_pack (k_ilu.cu).
__global__ void k_penta(int n, const SliceState* __restrict__ st, const float* __restrict__ wtv,
                        const float* __restrict__ wtv2, const float* __restrict__ wdiag, float* __restrict__ ia) {
  const int s = blockIdx.y;
  if (!slice_running(st, s)) return;
  const float abar = st[s].abar, lt = st[s].lam_tv, lw = st[s].lam;
  const size_t base = (size_t)s * n * n;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n * n; i += gridDim.x * blockDim.x) {
    const int r = i / n, c = i % n;
    const float wc = wtv[base + i];
    const float wr = c < n - 1 ? wtv[base + i + 1] : 0.f;
    float a;
    if (wtv2) {
      const float wd = r < n - 1 ? wtv2[base + i + n] : 0.f;
      a = penta_diag<true>(abar, lt, wc, wr, wtv2[base + i], wd);
    } else {
      const float wd = r < n - 1 ? wtv[base + i + n] : 0.f;
      a = penta_diag<false>(abar, lt, wc, wr, wc, wd);
    }
    if (wdiag) a = fmaf(lw, wdiag[base + i], a);
    ia[base + i] = 1.0f / a;
  }
}

void penta_setup(int batch, int n, cudaStream_t s, const SliceState* st, const float* wtv, const float* wtv2,
                 const float* wdiag, float* ia) {
  const int N = n * n;
  const int blocks = (N + 255) / 256 < 64 ? (N + 255) / 256 : 64;
  k_penta<<<dim3(blocks, batch), 256, 0, s>>>(n, st, wtv, wtv2, wdiag, ia);
}

// =========================================================== PCG vectors ==

int axpy_ctas(int n) {
  const int N = n * n;
  int c = N / 2048;
  if (c < 1) c = 1;
  if (c > MAXPART) c = MAXPART;
  return c;
}

__global__ void k_axpy(int N, int mode_arg, const SliceState* __restrict__ st, double* __restrict__ part,
                       float2* r, const float2* __restrict__ q, const float2* atb) {
  chained_start();
  const int s = blockIdx.y;
  if (!slice_running(st, s)) return;
  const int ph = st[s].phase;
  if (mode_arg == AXPY_PER_SLICE && !slice_working(ph)) return;
  const int mode = mode_arg != AXPY_PER_SLICE ? mode_arg : (ph == PH_START ? AXPY_INIT : AXPY_STEP);
  __shared__ double red[32];
  const float alpha = (float)st[s].alpha;
  const size_t base = (size_t)s * N;
  const int chunk = (N + gridDim.x - 1) / gridDim.x;
  const int lo = blockIdx.x * chunk, hi = min(N, lo + chunk);
  const float2* src = mode == AXPY_INIT ? atb : r;
  constexpr int UN = 4;  // elements in flight per thread
  float acc = 0.f;
  for (int i = lo + threadIdx.x; i < hi; i += UN * blockDim.x) {
    float2 rv[UN], qv[UN];
#pragma unroll
    for (int e = 0; e < UN; ++e) {
      const int j = i + e * blockDim.x;
      if (j < hi) {
        rv[e] = src[base + j];
        qv[e] = q[base + j];
      }
    }
#pragma unroll
    for (int e = 0; e < UN; ++e) {
      const int j = i + e * blockDim.x;
      if (j < hi) {
        rv[e] = mode == AXPY_INIT ? csub(rv[e], qv[e]) : cfma(-alpha, qv[e], rv[e]);
        r[base + j] = rv[e];
        acc += cabs2(rv[e]);
      }
    }
  }
  const double tot = block_sum((double)acc, red);
  if (threadIdx.x == 0) part[((size_t)s * NSLOT + SLOT_RR) * MAXPART + blockIdx.x] = tot;
}

void axpy_step(int batch, int n, cudaStream_t s, const SliceState* st, double* part, int mode, float2* r,
               const float2* q, const float2* atb, bool chained) {
  launch_chained(chained, k_axpy, dim3(axpy_ctas(n), batch), dim3(256), 0, s, n * n, mode, st, part, r, q, atb);
}

// Residual update with a diagonal preconditioner (Jacobi PCG, sdiag = 1 /
// diag(S)) or none (standard CG, sdiag null), for the comparison of Sec. 5.2.
__global__ void k_axpy_diag(int N, int mode_arg, const SliceState* __restrict__ st, double* __restrict__ part,
                            float2* __restrict__ r, const float2* __restrict__ q, const float2* __restrict__ atb,
                            const float* __restrict__ sdiag, float2* __restrict__ z) {
  chained_start();
  const int s = blockIdx.y;
  if (!slice_running(st, s)) return;
  const int ph = st[s].phase;
  if (mode_arg == AXPY_PER_SLICE && !slice_working(ph)) return;
  const int mode = mode_arg != AXPY_PER_SLICE ? mode_arg : (ph == PH_START ? AXPY_INIT : AXPY_STEP);
  __shared__ double red[32];
  const float alpha = (float)st[s].alpha;
  const size_t base = (size_t)s * N;
  const int chunk = (N + gridDim.x - 1) / gridDim.x;
  const int lo = blockIdx.x * chunk, hi = min(N, lo + chunk);
  float rz = 0.f, rr = 0.f;
  for (int i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    const size_t g = base + i;
    const float2 rv = mode == AXPY_INIT ? csub(atb[g], q[g]) : cfma(-alpha, q[g], r[g]);
    r[g] = rv;
    const float sc = sdiag ? sdiag[g] : 1.f;
    z[g] = cscale(rv, sc);
    const float r2 = cabs2(rv);
    rr += r2;
    rz = fmaf(sc, r2, rz);
  }
  const double trz = block_sum((double)rz, red);
  __syncthreads();
  const double trr = block_sum((double)rr, red);
  if (threadIdx.x == 0) {
    part[((size_t)s * NSLOT + SLOT_RZ) * MAXPART + blockIdx.x] = trz;
    part[((size_t)s * NSLOT + SLOT_RR) * MAXPART + blockIdx.x] = trr;
  }
}

void axpy_diag_step(int batch, int n, cudaStream_t s, const SliceState* st, double* part, int mode, float2* r,
                    const float2* q, const float2* atb, const float* sdiag, float2* z, bool chained) {
  launch_chained(chained, k_axpy_diag, dim3(axpy_ctas(n), batch), dim3(256), 0, s, n * n, mode, st, part, r, q, atb, sdiag, z);
}

__global__ void k_jacobi_wavelet(int N, const SliceState* __restrict__ st, const float* __restrict__ wdiag,
                                 float* __restrict__ ia) {
  const int s = blockIdx.y;
  if (!slice_running(st, s)) return;
  const float abar = st[s].abar, lw = st[s].lam;
  const size_t base = (size_t)s * N;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x)
    ia[base + i] = 1.0f / fmaf(lw, wdiag[base + i], abar);
}

void jacobi_wavelet_setup(int batch, int n, cudaStream_t s, const SliceState* st, const float* wdiag, float* ia) {
  const int N = n * n;
  const int blocks = (N + 255) / 256 < 64 ? (N + 255) / 256 : 64;
  k_jacobi_wavelet<<<dim3(blocks, batch), 256, 0, s>>>(N, st, wdiag, ia);
}

// End of a slice's outer step (PH_END): x^{k+1} = x^k + dx, where
// dx = sum_j alpha_j d_j was accumulated from zero by the row FFTs of the PCG
// steps (so its rounding is relative to the step, not to x), up to the last
// step's alpha d, which is added here, and dx is cleared for the next outer
// step; partial ||dx||^2 (SLOT_DX) and ||x^k||^2 (SLOT_XX) for the
// relative change.  Slices stopped by a breakdown are done and keep x^k.
__global__ void k_outer_apply(int N, const SliceState* __restrict__ st, float2* __restrict__ x,
                              float2* __restrict__ dx, const float2* __restrict__ d,
                              double* __restrict__ part) {
  const int s = blockIdx.y;
  if (!slice_running(st, s) || st[s].phase != PH_END) return;
  __shared__ double red[32];
  const size_t base = (size_t)s * N;
  const int chunk = (N + gridDim.x - 1) / gridDim.x;
  const int lo = blockIdx.x * chunk, hi = min(N, lo + chunk);
  const float alpha = (float)st[s].alpha;
  float a = 0.f, b = 0.f;
  for (int i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    const float2 xv = x[base + i], dv = cfma(alpha, d[base + i], dx[base + i]);
    a += cabs2(dv);
    b += cabs2(xv);
    x[base + i] = cadd(xv, dv);
    dx[base + i] = make_float2(0.f, 0.f);
  }
  const double ta = block_sum((double)a, red);
  __syncthreads();
  const double tb = block_sum((double)b, red);
  if (threadIdx.x == 0) {
    part[((size_t)s * NSLOT + SLOT_DX) * MAXPART + blockIdx.x] = ta;
    part[((size_t)s * NSLOT + SLOT_XX) * MAXPART + blockIdx.x] = tb;
  }
}

void outer_apply(int batch, int n, cudaStream_t s, const SliceState* st, float2* x, float2* dx, const float2* d,
                 double* part) {
  k_outer_apply<<<dim3(axpy_ctas(n), batch), 256, 0, s>>>(n * n, st, x, dx, d, part);
}

// ================================================================ groups ===

// W_g = (sum_{j in g} |c_j|^2 + eps)^(-1/2)   (Eq. gw)
__global__ void k_group_norms(int n, int G, const SliceState* __restrict__ st, const int* __restrict__ gidx,
                              const int* __restrict__ goff, int gsize, const float2* __restrict__ c,
                              float* __restrict__ wg) {
  const int s = blockIdx.y;
  if (!slice_running(st, s)) return;
  const float eps = st[s].eps;
  const float2* cs = c + (size_t)s * n * n;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x) {
    const int b = goff ? goff[g] : g * gsize;
    const int e = goff ? goff[g + 1] : b + gsize;
    float acc = 0.f;
    for (int k = b; k < e; ++k) acc += cabs2(cs[gidx[k]]);
    wg[(size_t)s * G + g] = rsqrtf(acc + eps);
  }
}

void group_norms(int batch, int n, int G, cudaStream_t s, const SliceState* st, const int* gidx,
                 const int* goff, int gsize, const float2* c, float* wg, float) {
  const int blocks = (G + 255) / 256 < 256 ? (G + 255) / 256 : 256;
  k_group_norms<<<dim3(blocks, batch), 256, 0, s>>>(n, G, st, gidx, goff, gsize, c, wg);
}

// w_j = sum_{g containing j} W_g = diag(G^T W G)_j  (Eq. Wog), ascending g
__global__ void k_group_gather(int n, int G, const SliceState* __restrict__ st, const int* __restrict__ ioff,
                               const int* __restrict__ iids, const float* __restrict__ wg,
                               float* __restrict__ w) {
  const int s = blockIdx.y;
  if (!slice_running(st, s)) return;
  const float* wgs = wg + (size_t)s * G;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n * n; j += gridDim.x * blockDim.x) {
    float acc = 0.f;
    for (int k = ioff[j]; k < ioff[j + 1]; ++k) acc += wgs[iids[k]];
    w[(size_t)s * n * n + j] = acc;
  }
}

void group_gather(int batch, int n, int G, cudaStream_t s, const SliceState* st, const int* inv_off,
                  const int* inv_ids, const float* wg, float* w) {
  const int N = n * n;
  const int blocks = (N + 255) / 256 < 256 ? (N + 255) / 256 : 256;
  k_group_gather<<<dim3(blocks, batch), 256, 0, s>>>(n, G, st, inv_off, inv_ids, wg, w);
}

__global__ void k_gm_count(int N, int G, int gsize, const int* __restrict__ gidx, const int* __restrict__ goff,
                           int* __restrict__ counts, int* __restrict__ err) {
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x) {
    const int b = goff ? goff[g] : g * gsize;
    const int e = goff ? goff[g + 1] : b + gsize;
    if (e < b) {
      atomicExch(err, 1);
      continue;
    }
    for (int k = b; k < e; ++k) {
      const int j = gidx[k];
      if (j < 0 || j >= N) {
        atomicExch(err, 1);
      } else {
        atomicAdd(&counts[j], 1);
      }
    }
  }
}

// Exclusive scan of counts[0..N) into off[0..N], one block.
__global__ void k_scan_counts(int N, const int* __restrict__ counts, int* __restrict__ off) {
  __shared__ int sums[1024];
  const int t = threadIdx.x, nt = blockDim.x;
  const int chunk = (N + nt - 1) / nt;
  const int lo = min(N, t * chunk), hi = min(N, lo + chunk);
  int acc = 0;
  for (int i = lo; i < hi; ++i) acc += counts[i];
  sums[t] = acc;
  __syncthreads();
  for (int o = 1; o < nt; o <<= 1) {
    const int v = t >= o ? sums[t - o] : 0;
    __syncthreads();
    sums[t] += v;
    __syncthreads();
  }
  int run = t > 0 ? sums[t - 1] : 0;
  for (int i = lo; i < hi; ++i) {
    off[i] = run;
    run += counts[i];
  }
  if (t == nt - 1) off[N] = sums[nt - 1];
}

__global__ void k_gm_fill(int N, int G, int gsize, const int* __restrict__ gidx, const int* __restrict__ goff,
                          const int* __restrict__ ioff, int* __restrict__ cursor, int* __restrict__ iids,
                          const int* __restrict__ err) {
  if (*err) return;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x) {
    const int b = goff ? goff[g] : g * gsize;
    const int e = goff ? goff[g + 1] : b + gsize;
    for (int k = b; k < e; ++k) {
      const int j = gidx[k];
      const int pos = atomicAdd(&cursor[j], 1);
      iids[ioff[j] + pos] = g;
    }
  }
}

__global__ void k_gm_sort(int N, const int* __restrict__ ioff, int* __restrict__ iids, const int* __restrict__ err) {
  if (*err) return;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x) {
    const int b = ioff[j], e = ioff[j + 1];
    for (int a = b + 1; a < e; ++a) {
      const int v = iids[a];
      int k = a - 1;
      while (k >= b && iids[k] > v) {
        iids[k + 1] = iids[k];
        --k;
      }
      iids[k + 1] = v;
    }
  }
}

void group_inverse_build(int n, int G, int gsize, cudaStream_t s, const int* gidx, const int* goff,
                         int* counts, int* inv_off, int* inv_ids, int* cursor, int* err) {
  const int N = n * n;
  const int gb = (G + 255) / 256 < 1024 ? (G + 255) / 256 : 1024;
  const int nb = (N + 255) / 256 < 1024 ? (N + 255) / 256 : 1024;
  k_gm_count<<<gb, 256, 0, s>>>(N, G, gsize, gidx, goff, counts, err);
  k_scan_counts<<<1, 1024, 0, s>>>(N, counts, inv_off);
  k_gm_fill<<<gb, 256, 0, s>>>(N, G, gsize, gidx, goff, inv_off, cursor, inv_ids, err);
  k_gm_sort<<<nb, 256, 0, s>>>(N, inv_off, inv_ids, err);
}

__global__ void k_popcount(int N, const uint8_t* __restrict__ mask, int* __restrict__ counts) {
  const int s = blockIdx.y;
  __shared__ int red[32];
  int acc = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x)
    acc += mask[(size_t)s * N + i] ? 1 : 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += red[i];
    atomicAdd(&counts[s], t);
  }
}

void mask_popcount(int batch, int n, cudaStream_t s, const uint8_t* mask, int* counts) {
  const int N = n * n;
  const int blocks = (N + 255) / 256 < 64 ? (N + 255) / 256 : 64;
  k_popcount<<<dim3(blocks, batch), 256, 0, s>>>(N, mask, counts);
}

// ======================================================== objective sums ===

// C > 1 (joint sparsity, no group map): the first slice of each image sums
// sqrt(sum_t |c_tj|^2 + eps) over its C contrasts, the others contribute 0.
__global__ void k_l21_sum(int n, int C, const float2* __restrict__ c, const int* __restrict__ gidx,
                          const int* __restrict__ goff, int G, int gsize, float eps, double* __restrict__ part,
                          int slot) {
  const int s = blockIdx.y;
  __shared__ double red[32];
  const size_t N = (size_t)n * n;
  const float2* cs = c + (size_t)s * N;
  const int count = gidx ? G : n * n;
  const int chunk = (count + gridDim.x - 1) / gridDim.x;
  const int lo = blockIdx.x * chunk, hi = min(count, lo + chunk);
  const int cc = s % C == 0 ? C : 0;
  float acc = 0.f;
  for (int g = lo + threadIdx.x; g < hi; g += blockDim.x) {
    float ss;
    if (C > 1) {
      if (!cc) break;
      ss = 0.f;
      for (int t = 0; t < cc; ++t) ss += cabs2(cs[(size_t)t * N + g]);
    } else if (!gidx) {
      ss = cabs2(cs[g]);
    } else {
      const int b = goff ? goff[g] : g * gsize;
      const int e = goff ? goff[g + 1] : b + gsize;
      ss = 0.f;
      for (int k = b; k < e; ++k) ss += cabs2(cs[gidx[k]]);
    }
    acc += sqrtf(ss + eps);
  }
  const double tot = block_sum((double)acc, red);
  if (threadIdx.x == 0) part[((size_t)s * NSLOT + slot) * MAXPART + blockIdx.x] = tot;
}

void l21_sum(int batch, int n, cudaStream_t s, const float2* c, const int* gidx, const int* goff, int G, int gsize,
             float eps, double* part, int slot, int channels) {
  k_l21_sum<<<dim3(axpy_ctas(n), batch), 256, 0, s>>>(n, channels, c, gidx, goff, G, gsize, eps, part, slot);
}

// C > 1 (joint TV): the first slice of each image sums sqrt(sum_t |grad
// x_t,i|^2 + eps) over its C contrasts, the others contribute 0.
__global__ void k_tv_sum(int n, int C, const float2* __restrict__ x, float eps, double* __restrict__ part, int slot,
                         int aniso) {
  const int s = blockIdx.y;
  __shared__ double red[32];
  const size_t base = (size_t)s * n * n;
  const int N = n * n;
  const int chunk = (N + gridDim.x - 1) / gridDim.x;
  const int lo = blockIdx.x * chunk, hi = min(N, lo + chunk);
  const int cc = (C == 1 || s % C == 0) ? C : 0;
  float acc = 0.f;
  for (int i = lo + threadIdx.x; i < hi && cc; i += blockDim.x) {
    const int r = i / n, col = i % n;
    float g = 0.f, ga = 0.f;
    for (int t = 0; t < cc; ++t) {
      const size_t bt = base + (size_t)t * N;
      const float2 xc = x[bt + i];
      const float2 g1 = col > 0 ? csub(xc, x[bt + i - 1]) : xc;
      const float2 g2 = r > 0 ? csub(xc, x[bt + i - n]) : xc;
      g += cabs2(g1) + cabs2(g2);
      if (aniso) ga = sqrtf(cabs2(g1) + eps) + sqrtf(cabs2(g2) + eps);
    }
    acc += aniso ? ga : sqrtf(g + eps);
  }
  const double tot = block_sum((double)acc, red);
  if (threadIdx.x == 0) part[((size_t)s * NSLOT + slot) * MAXPART + blockIdx.x] = tot;
}

void tv_sum(int batch, int n, cudaStream_t s, const float2* x, float eps, double* part, int slot, int aniso,
            int channels) {
  k_tv_sum<<<dim3(axpy_ctas(n), batch), 256, 0, s>>>(n, channels, x, eps, part, slot, aniso);
}

// ========================================================== PCG scalars ===

// The scalar kernels give a warp to each slice: its lanes fetch the partial sums
// at once and lane 0 adds them in order, as one thread did (which took 15 us at
// 60 slices of three contrasts, one load after the other).
constexpr int SC_WARPS = 4;  // slices per CTA
FI int sc_slice() { return blockIdx.x * SC_WARPS + (threadIdx.x >> 5); }
static int sc_ctas(int batch) { return (batch + SC_WARPS - 1) / SC_WARPS; }

// sum of slice s's np partial sums, valid in lane 0; called by a whole warp
FI double sum_parts(const double* part, int s, int slot, int np) {
  __shared__ double buf[SC_WARPS][MAXPART];
  double* b = buf[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const double* p = part + ((size_t)s * NSLOT + slot) * MAXPART;
  __syncwarp();
  for (int i = lane; i < np; i += 32) b[i] = p[i];
  __syncwarp();
  double a = 0.0;
  if (lane == 0)
    for (int i = 0; i < np; ++i) a += b[i];
  return a;
}

// The sum over the C contrasts (consecutive slices) of the image that slice s
// belongs to: multi-contrast PCG runs on the stacked unknown (Sec. 5.6), so
// its inner products, and the relative change of the outer step, are sums
// over the contrasts.  Every slice of the image sums in the same order and
// takes the same scalars and the same phase transitions.
FI double image_parts(const double* part, int s, int slot, int np, int C) {
  if (C == 1) return sum_parts(part, s, slot, np);
  const int s0 = s - s % C;
  double a = 0.0;
  for (int t = s0; t < s0 + C; ++t) a += sum_parts(part, t, slot, np);
  return a;
}

// F_eps of every slice from the partial sums of its terms (SLOT_DQ: |M F x - b|^2,
// SLOT_RZ: wavelet, SLOT_RR: TV); of the whole image for each of its C contrasts.
// On the device so that a caller reads 8 bytes a slice, not 6 KB of partials.
__global__ void k_objective(int B, int C, const double* part, int nd, int nr, int wavelet, int tv,
                            const float* __restrict__ lam, const float* __restrict__ lam_tv, double* __restrict__ f) {
  const int s = sc_slice();
  if (s >= B) return;
  const int s0 = s - s % C;
  double sum = 0.0;
  for (int t = s0; t < s0 + C; ++t) {
    double v = 0.5 * sum_parts(part, t, SLOT_DQ, nd);
    if (wavelet) v += (double)lam[t] * sum_parts(part, t, SLOT_RZ, nr);
    if (tv) v += (double)lam_tv[t] * sum_parts(part, t, SLOT_RR, nr);
    sum = t == s0 ? v : sum + v;
  }
  if ((threadIdx.x & 31) == 0) f[s] = sum;
}

void objective_sum(int batch, cudaStream_t s, const double* part, int nd, int nr, bool wavelet, bool tv,
                   const float* lam, const float* lam_tv, double* f, int channels) {
  k_objective<<<sc_ctas(batch), 32 * SC_WARPS, 0, s>>>(batch, channels, part, nd, nr, wavelet, tv, lam, lam_tv, f);
}

// The warm start of each slice: x1 where its objective is finite and no larger
// than that of A^H b, else A^H b.  One launch for the batch (a copy per slice
// took 2 us each: 64 slices of 256^2 130 -> 11 us).
__global__ void k_guard_pick(int N4, const double* __restrict__ f1, const double* __restrict__ f0, const float4* x1,
                             const float4* __restrict__ atb, float4* x0) {
  const int s = blockIdx.y;
  const float4* src = (guard_keeps(f1[s], f0[s]) ? x1 : atb) + (size_t)s * N4;
  float4* dst = x0 + (size_t)s * N4;
#pragma unroll 4
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N4; i += gridDim.x * blockDim.x) dst[i] = src[i];
}

void guard_pick(int batch, int n, cudaStream_t s, const double* f1, const double* f0, const void* x1,
                const float2* atb, void* x0) {
  const int N4 = n * n / 2;
  const int ctas = std::max(1, std::min(32, N4 / 1024));
  k_guard_pick<<<dim3(ctas, batch), 256, 0, s>>>(N4, f1, f0, static_cast<const float4*>(x1),
                                                 reinterpret_cast<const float4*>(atb), static_cast<float4*>(x0));
}

__global__ void k_state_init(int B, SliceState* st, const double* part, int np, const int* counts, int N,
                             const float* lam, const float* lam_tv, float eps, int outer_max, int phase, int C) {
  const int s = sc_slice();
  if (s >= B) return;
  const double rhs2 = image_parts(part, s, SLOT_RHS, np, C);
  if (threadIdx.x & 31) return;
  SliceState v;
  v.rho = 0.0;
  v.alpha = 0.0;
  v.beta = 0.0;
  v.rhs2 = rhs2;
  v.rr = v.rhs2;
  v.rr0 = v.rhs2;
  v.relchg = 0.0;
  v.stall = 0;
  v.phase = phase;
  v.pcg_j = 0;
  v.outer_max = outer_max;
  for (int i = 0; i < MU_WINDOW; ++i) v.hist[i] = 0.f;
  // non-finite k-space on the mask makes A^H b non-finite: the slice is not
  // iterated and counts as a breakdown (its x keeps the start)
  const bool bad = !isfinite(v.rhs2);
  v.active = bad ? 0 : 1;
  v.done = bad ? 1 : 0;
  v.breakdown = bad ? 1 : 0;
  v.pcg_steps = 0;
  v.outer_done = 0;
  v.fault = 0;
  v.lam = lam[s];
  v.lam_tv = lam_tv[s];
  v.abar = (float)((double)counts[s] / (double)N);
  v.eps = eps;
  st[s] = v;
}

void state_init(int batch, cudaStream_t s, SliceState* st, const double* part, int np, const int* counts,
                int n, const float* lam, const float* lam_tv, float eps, int outer_max, int phase, int channels) {
  k_state_init<<<sc_ctas(batch), 32 * SC_WARPS, 0, s>>>(batch, st, part, np, counts, n * n, lam, lam_tv, eps,
                                                   outer_max, phase, channels);
}

// The slices whose outer step is due (PH_BOUNDARY), as a copy of the state in
// which every other slice reads as done: the weight and preconditioner
// set-up kernels, which skip done slices and never write the state, then
// work on exactly those slices.  The slices themselves move to PH_START (this
// macro step's S apply and PCG update form their first residual, after the
// set-up kernels have run).
__global__ void k_boundary_view(int B, SliceState* __restrict__ st, SliceState* __restrict__ view) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= B) return;
  SliceState v = st[s];
  if (v.phase != PH_BOUNDARY) {
    v.done = 1;
  } else if (v.active && !v.done) {
    st[s].phase = PH_START;
  }
  view[s] = v;
}

void boundary_view(int batch, cudaStream_t s, SliceState* st, SliceState* view) {
  k_boundary_view<<<(batch + 127) / 128, 128, 0, s>>>(batch, st, view);
}

__global__ void k_alpha(int B, SliceState* st, const double* part, int np, int C) {
  chained_start();
  const int s = sc_slice();
  if (s >= B || !slice_in_pcg(st, s)) return;
  const double dq = image_parts(part, s, SLOT_DQ, np, C);
  if ((threadIdx.x & 31) == 0) pcg_alpha_from(st + s, dq);
}

void pcg_alpha(int batch, cudaStream_t s, SliceState* st, const double* part, int np, int channels, bool chained) {
  launch_chained(chained, k_alpha, dim3(sc_ctas(batch)), dim3(32 * SC_WARPS), 0, s, batch, st, part, np, channels);
}

// The sum of squares of n4 float4 in FP64, in every lane of the warp that calls it.
FI double wide_norm2(const float4* v, int n4) {
  double a = 0.0;
#pragma unroll 4
  for (int i = threadIdx.x & 31; i < n4; i += 32) {
    const float4 x = v[i];
    a += (double)x.x * x.x + (double)x.y * x.y + (double)x.z * x.z + (double)x.w * x.w;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  return a;
}

// After z = P^{-1} r: rho (first residual, slices at the start of an outer
// step) or beta and the PCG stop (slices in PCG); mode INIT / STEP forces one
// of them for every running slice.
// r (may be null): the residuals [B][N4], for ||r||^2 where the partial sums are not
// finite.  Those of the update inside the wavelet transform are carried in three floats,
// which end at 3.4e38 a CTA; a test there cost up to 0.7 % of a small solve.
__global__ void k_pcg_scalars(int B, SliceState* st, const double* part, int np_rz, int np_rr, int mode,
                              PcgSched ps, int C, const float4* __restrict__ r, int N4) {
  chained_start();
  const int s = sc_slice();
  if (s >= B || !slice_running(st, s) || st[s].fault) return;
  const int ph = st[s].phase;
  const bool init = mode == SCALARS_INIT || (mode == SCALARS_PER_SLICE && ph == PH_START);
  const bool step = mode == SCALARS_STEP || (mode == SCALARS_PER_SLICE && ph == PH_PCG);
  const double rz = image_parts(part, s, SLOT_RZ, np_rz, C);
  double rr = image_parts(part, s, SLOT_RR, np_rr, C);
  const int lane = threadIdx.x & 31;
  if (r != nullptr && __shfl_sync(0xffffffffu, !isfinite(rr), 0)) rr = wide_norm2(r + (size_t)(s - s % C) * N4, C * N4);
  if (lane) return;
  if (init)
    pcg_rho_init_from(st + s, rz, rr);
  else if (step)
    pcg_beta_from(st + s, rz, rr, ps);
}

void pcg_scalars(int batch, cudaStream_t s, SliceState* st, const double* part, int np_rz, int np_rr, int mode,
                 const PcgSched& ps, int channels, bool chained, const float2* r, int n) {
  launch_chained(chained, k_pcg_scalars, dim3(sc_ctas(batch)), dim3(32 * SC_WARPS), 0, s, batch, st, part, np_rz, np_rr, mode, ps,
                 channels, reinterpret_cast<const float4*>(r), n * n / 2);
}

// Outer-loop stop.  kind 0: relative change <= tol.  kind 1: estimated
// distance to the limit <= tol.  Under linear convergence x^k -> x* with
// contraction mu, ||x^k - x*|| ~ relchg_k mu / (1 - mu) (the sum of the
// remaining steps) relative to ||x^k||; mu is the geometric mean contraction
// over the last MU_WINDOW steps, (relchg_k / relchg_{k-W})^(1/W), capped at
// 0.999 (a long window: the rate drifts early on and FP32 rounding jitters
// single steps).  Either kind also stops a slice whose relative change has
// stayed at or below stall_tol for STALL_STEPS consecutive steps: the FP32
// rounding floor of the outer iteration, below which it cannot move.  Kind 1
// stops a slice on a plateau too: from outer step plateau_after on (a whole
// window in the phase of nearly exact inner solves, where the outer
// iteration contracts by far more than 20 % over the window), a relative
// change at or below tol that has not fallen by 20 % over the window is that
// slice's FP32 floor, whatever its level.
__global__ void k_outer_end(int B, SliceState* st, const double* part, int np, float tol, int kind,
                            float stall_tol, int plateau_after, int C) {
  const int s = sc_slice();
  if (s >= B || !slice_running(st, s) || st[s].phase != PH_END) return;
  SliceState* v = st + s;
  const double dx = image_parts(part, s, SLOT_DX, np, C);
  const double xx = image_parts(part, s, SLOT_XX, np, C);
  if (threadIdx.x & 31) return;
  const double rel = xx > 0.0 ? sqrt(dx / xx) : INFINITY;
  const int k = v->outer_done;  // this step's index
  const float old = v->hist[k % MU_WINDOW];  // relchg of step k - MU_WINDOW
  v->hist[k % MU_WINDOW] = (float)rel;
  v->relchg = rel;
  v->outer_done = k + 1;
  v->stall = (stall_tol > 0.f && rel <= (double)stall_tol) ? v->stall + 1 : 0;
  if (v->stall >= STALL_STEPS) {
    v->done = 1;
    return;
  }
  if (tol > 0.f) {
    if (kind == 0) {
      if (rel <= (double)tol) v->done = 1;
    } else if (k >= MU_WINDOW && old > 0.f) {
      const double mu = fmin(pow(rel / (double)old, 1.0 / MU_WINDOW), 0.999);
      if (rel * mu / (1.0 - mu) <= (double)tol && rel <= (double)tol) v->done = 1;
      if (k >= plateau_after && rel <= (double)tol && rel >= 0.8 * (double)old) v->done = 1;
    }
  }
  if (v->outer_done >= v->outer_max) v->done = 1;
  if (!v->done) v->phase = PH_BOUNDARY;  // the next outer step starts
}

void outer_end(int batch, cudaStream_t s, SliceState* st, const double* part, int np, float tol, int kind,
               float stall_tol, int plateau_after, int channels) {
  k_outer_end<<<sc_ctas(batch), 32 * SC_WARPS, 0, s>>>(batch, st, part, np, tol, kind, stall_tol, plateau_after,
                                                  channels);
}

}  // namespace firls
