// Batched dense kernels: partial Cholesky engine, GEMV, triangular solves.
//
// The engine is a right-looking blocked Cholesky restricted to the first e
// columns of each matrix, followed by one long-K symmetric rank-e update of
// the trailing block.  With K = [[K_II, K_IG], [K_GI, K_GG]] and e = n_I this
// yields L_II, L_GI and the local Schur complement S_Gamma = K_GG - L_GI L_GI^T
// (static condensation, Section 4.1).  With the augmented matrix
// [[S_DD, S_DP, I], [S_PD, S_PP, 0], [I, 0, 0]] and e = n_D it yields, in the
// trailing block, S_PP - S_PD S_DD^-1 S_DP (the local coarse matrix of
// Section 4.4), -S_DD^-1 S_DP and -S_DD^-1 (the local constrained solve).
#include <algorithm>
#include <atomic>
#include <type_traits>
#include <vector>

#include "digit_ws.h"
#include "kernels.cuh"

namespace bd {


// 16-byte vectors of T (row starts of the batched matrices are 32-byte aligned).
template <typename T> struct Vec16;
template <> struct Vec16<float> {
  using V = float4;
  static constexpr int N = 4;
  __device__ static float get(const float4 &v, int q) { return q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w; }
  __device__ static void set(float4 &v, int q, float a) {
    if (q == 0) v.x = a; else if (q == 1) v.y = a; else if (q == 2) v.z = a; else v.w = a;
  }
  __device__ static float dot(const float4 a, const float4 b) { return a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w; }
  __device__ static void axpy(float *acc, const float4 a, float s) {
    acc[0] += a.x * s; acc[1] += a.y * s; acc[2] += a.z * s; acc[3] += a.w * s;
  }
};
template <> struct Vec16<double> {
  using V = double2;
  static constexpr int N = 2;
  __device__ static double get(const double2 &v, int q) { return q == 0 ? v.x : v.y; }
  __device__ static void set(double2 &v, int q, double a) {
    if (q == 0) v.x = a; else v.y = a;
  }
  __device__ static double dot(const double2 a, const double2 b) { return a.x * b.x + a.y * b.y; }
  __device__ static void axpy(double *acc, const double2 a, double s) { acc[0] += a.x * s; acc[1] += a.y * s; }
};

// ---- rows below a 128-column panel: L_21 = A_21 L_11^-T (FP32) ----------------------
// The diagonal block is factored already and its 32 x 32 diagonal blocks inverted (k_diag128).  RB rows
// per CTA, staged in shared memory; 32 columns at a time: multiplied by that inverse (4 x 4 tiles),
// then a rank-32 update of the remaining columns (4 x 4 tiles over transposed copies of the solved
// columns and of L_11's, the next 32 columns of L_11 on their way meanwhile).  Rows: those the band lets
// the panel reach.  A chain of latencies: one thread per row substituted here before (22 us for
// the 2,490 rows of a coarse panel on 20 CTAs; 11 us on 78 CTAs of 32 rows now).
constexpr int kPW = kEnginePanel;  // panel width
constexpr int kLDP = kPW + 4;      // row stride of the staged panel (16-byte aligned rows)
constexpr int kLDY = 36;
template <int RB>
constexpr size_t panel_smem() { return sizeof(float) * ((size_t)RB * kLDP + 32 * (kPW + RB) + 32 * kLDY); }

template <int RB>
__global__ void __launch_bounds__(256, 2) k_panel_rows(const MatDesc *__restrict__ desc, float *__restrict__ base,
                                                       int K0, const float *__restrict__ pinv) {
  constexpr int NR = kPW + RB, VPP = kPW / 4;  // VPP: vectors per staged row
  const MatDesc d = desc[blockIdx.y];
  if (K0 >= d.e) return;
  const int w = min(kPW, d.e - K0);
  const BandRows br = band_rows(d, K0 + w, K0 + w);
  const int v0 = blockIdx.x * RB;
  if (v0 >= br.nv) return;
  const int nrows = min(RB, br.nv - v0);
  float *A = base + d.off;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float *P = reinterpret_cast<float *>(smem_raw);  // [RB][kLDP] own rows
  float *PT = P + RB * kLDP;                       // [32][NR]: 32 columns, transposed (L_11 rows, then own)
  float *Yt = PT + 32 * NR;                        // [32][kLDY]: Yt[k][c] = (L_bb^-1)[c][k]
  const int tid = threadIdx.x;
  // L_11 below the sub-block (columns [c0, c0 + 32) of rows [c0 + 32, w): three vectors a thread) and
  // the sub-block's inverse (one)
  float4 lv[3], yv;
  auto fetch = [&](int bq) {
    const int c0 = 32 * bq;
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      const int idx = tid + 256 * u, p = c0 + 32 + idx / 8;
      lv[u] = p < w ? *reinterpret_cast<const float4 *>(A + (long long)(K0 + p) * d.ld + K0 + c0 + (idx % 8) * 4) : float4{};
    }
    yv = *reinterpret_cast<const float4 *>(pinv + ((long long)blockIdx.y * 4 + bq) * 1024 + tid * 4);
  };
  fetch(0);
  // stage: kBatch vector loads in flight per thread and batch
  constexpr int kVec = RB * VPP, kBatch = kVec / 256 < 8 ? kVec / 256 : 8;
  for (int base_i = 0; base_i < kVec; base_i += 256 * kBatch) {
    float4 buf[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int idx = base_i + tid + 256 * u, sr = idx / VPP, cv = idx % VPP;
      const bool ok = cv * 4 < w && sr < nrows;
      buf[u] = ok ? *reinterpret_cast<const float4 *>(A + (long long)br.row(v0 + sr) * d.ld + K0 + cv * 4) : float4{};
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int idx = base_i + tid + 256 * u, sr = idx / VPP, cv = idx % VPP;
      float4 o = buf[u];
      if (cv * 4 + 1 >= w) o.y = 0.f;
      if (cv * 4 + 2 >= w) o.z = 0.f;
      if (cv * 4 + 3 >= w) o.w = 0.f;
      *reinterpret_cast<float4 *>(P + sr * kLDP + cv * 4) = o;
    }
  }
  const int nbk = ceil_div(w, 32), nr4 = (nrows + 3) / 4;
  for (int bq = 0; bq < nbk; ++bq) {
    const int c0 = 32 * bq;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      const int idx = tid + 256 * u, p = c0 + 32 + idx / 8, cv = (idx % 8) * 4;
      if (p < kPW) {
#pragma unroll
        for (int q = 0; q < 4; ++q) PT[(cv + q) * NR + p] = Vec16<float>::get(lv[u], q);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) Yt[((tid & 7) * 4 + q) * kLDY + (tid >> 3)] = Vec16<float>::get(yv, q);
    if (bq + 1 < nbk) fetch(bq + 1);
    __syncthreads();
    // x = a Y^T: four rows RB / 4 apart (consecutive threads read consecutive rows) by four columns a thread
    constexpr int RS = RB / 4;
    const int r0 = tid % RS, j0 = 4 * (tid / RS);
    const bool mine = j0 < 32;
    float x[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) x[i][j] = 0.f;
    if (mine) {
#pragma unroll
      for (int k = 0; k < 32; k += 4) {
        float4 av[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) av[i] = *reinterpret_cast<const float4 *>(P + (r0 + RS * i) * kLDP + c0 + k);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 y = *reinterpret_cast<const float4 *>(Yt + (k + q) * kLDY + j0);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float e = Vec16<float>::get(av[i], q);
            x[i][0] += e * y.x;
            x[i][1] += e * y.y;
            x[i][2] += e * y.z;
            x[i][3] += e * y.w;
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) PT[(j0 + j) * NR + kPW + r0 + RS * i] = x[i][j];
    }
    __syncthreads();
    if (mine) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        *reinterpret_cast<float4 *>(P + (r0 + RS * i) * kLDP + c0 + j0) = make_float4(x[i][0], x[i][1], x[i][2], x[i][3]);
    }
    // rank-32 update of the panel columns [c0 + 32, w), 4 x 4 tiles
    const int jb = c0 + 32, ncol = w - jb;
    if (ncol > 0) {
      const int nc4 = (ncol + 3) / 4;
      for (int mt = tid; mt < nr4 * nc4; mt += 256) {
        const int r0 = 4 * (mt / nc4), j0 = jb + 4 * (mt % nc4);
        float acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
#pragma unroll 8
        for (int k = 0; k < 32; ++k) {
          const float4 x = *reinterpret_cast<const float4 *>(&PT[k * NR + kPW + r0]);
          const float4 y = *reinterpret_cast<const float4 *>(&PT[k * NR + j0]);
          const float av[4] = {x.x, x.y, x.z, x.w}, bv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] += av[i] * bv[j];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (r0 + i >= nrows) continue;
          float *row = P + (r0 + i) * kLDP;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j0 + j < w) row[j0 + j] -= acc[i][j];
        }
      }
    }
  }
  __syncthreads();
  for (int idx = tid; idx < nrows * VPP; idx += 256) {
    const int q = idx / VPP, cv = idx % VPP;
    if (cv * 4 >= w) continue;
    const float *src = P + q * kLDP + cv * 4;
    float *dst = A + (long long)br.row(v0 + q) * d.ld + K0 + cv * 4;
    if (cv * 4 + 4 <= w) {
      *reinterpret_cast<float4 *>(dst) = *reinterpret_cast<const float4 *>(src);
    } else {
      for (int u = 0; cv * 4 + u < w; ++u) dst[u] = src[u];
    }
  }
}

std::atomic<long long> g_launches{0};
void count_launch(int n) { g_launches += n; }
long long launch_count() { return g_launches.load(); }

// ---- FP32 rank-k update of lower tiles: 128x128 CTA tiles, 8x8 outputs per thread ----------
// C[r][c] -= sum_k A[r][k] A[c][k] with
// mode 0 (in-block): rows [k0+w, m), cols [k0+w, min(K1, e)), K = [k0, k0+w), w = one panel
// mode 2 (outer):    rows [K1, m),   cols [K1, e),            K = [K0, K1)
// mode 1 (final):    rows [e, m),    cols [e, m),             K = [0, e)
// K is consumed in chunks of 16 with the next chunk prefetched into registers while the
// current one is used.  (The FP64 updates run on the tensor cores, digits.cu.)
constexpr int kTB2 = 128, kKC2 = 16;

__global__ void __launch_bounds__(256) k_rankk128(const MatDesc *__restrict__ desc, float *__restrict__ base,
                                                  int mode, int k0, int K0, int K1, int nct) {
  const MatDesc d = desc[blockIdx.y];
  int row0, colend, kb, ke;
  if (mode == 0) {
    if (k0 >= d.e) return;
    const int w = min(kEnginePanel, d.e - k0);
    row0 = k0 + w; colend = min(K1, d.e); kb = k0; ke = k0 + w;
  } else if (mode == 2) {
    if (K1 >= d.e) return;
    row0 = K1; colend = d.e; kb = K0; ke = K1;
  } else {
    row0 = d.e; colend = d.m; kb = 0; ke = d.e;
  }
  const BandRows br = band_rows(d, row0, ke);  // rows past the band hold zeros in K = [kb, ke)
  if (mode != 1) colend = min(colend, band_limit(d, ke));
  const int ti = blockIdx.x / nct, tj = blockIdx.x % nct;
  if (tj > ti) return;
  const int v0 = ti * kTB2, c0 = row0 + tj * kTB2;
  if (mode == 1 && d.ifirst && v0 < br.nv) kb = max(kb, d.ifirst[v0] & ~3);  // rows' L starts there
  if (v0 >= br.nv || c0 >= colend || ke <= kb) return;
  float *A = base + d.off;
  __shared__ __align__(16) float As[2][kKC2][kTB2 + 4];
  __shared__ __align__(16) float Bs[2][kKC2][kTB2 + 4];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  // loader: thread -> (row lr, k offset lk): 128 rows x 16 k = 2 x 4 floats per thread per operand
  const int lr = tid >> 1, lk = (tid & 1) * 8;
  const bool va = v0 + lr < br.nv;
  const int ra = va ? br.row(v0 + lr) : 0, rb = c0 + lr;
  const bool vb = rb < colend;
  const float *pa = A + (long long)ra * d.ld, *pb = A + (long long)rb * d.ld;
  float la[8], lb[8];
  auto load = [&](int kk) {
#pragma unroll
    for (int q = 0; q < 8; q += 4) {
      const int k = kk + lk + q;
      if (k + 3 < ke) {
        const float4 x = va ? *reinterpret_cast<const float4 *>(pa + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 y = vb ? *reinterpret_cast<const float4 *>(pb + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        la[q] = x.x; la[q + 1] = x.y; la[q + 2] = x.z; la[q + 3] = x.w;
        lb[q] = y.x; lb[q + 1] = y.y; lb[q + 2] = y.z; lb[q + 3] = y.w;
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          la[q + u] = (va && k + u < ke) ? pa[k + u] : 0.f;
          lb[q + u] = (vb && k + u < ke) ? pb[k + u] : 0.f;
        }
      }
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      As[buf][lk + q][lr] = la[q];
      Bs[buf][lk + q][lr] = lb[q];
    }
  };
  float acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
  load(kb);
  store(0);
  __syncthreads();
  int buf = 0;
  for (int kk = kb; kk < ke; kk += kKC2) {
    const bool more = kk + kKC2 < ke;
    if (more) load(kk + kKC2);
#pragma unroll
    for (int k = 0; k < kKC2; ++k) {
      const float4 a0 = *reinterpret_cast<const float4 *>(&As[buf][k][ty * 4]);
      const float4 a1 = *reinterpret_cast<const float4 *>(&As[buf][k][64 + ty * 4]);
      const float4 b0 = *reinterpret_cast<const float4 *>(&Bs[buf][k][tx * 4]);
      const float4 b1 = *reinterpret_cast<const float4 *>(&Bs[buf][k][64 + tx * 4]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] += av[i] * bv[j];
    }
    if (more) {
      store(buf ^ 1);
      __syncthreads();
      buf ^= 1;
    }
  }
  // thread owns rows {ty*4 + i, 64 + ty*4 + i} and columns {tx*4 + j, 64 + tx*4 + j}
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int v = v0 + (i < 4 ? ty * 4 + i : 64 + ty * 4 + (i - 4));
    if (v >= br.nv) continue;
    float *crow = A + (long long)br.row(v) * d.ld;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = c0 + (j < 4 ? tx * 4 + j : 64 + tx * 4 + (j - 4));
      if (c < colend) crow[c] -= acc[i][j];
    }
  }
}

// 128 rows per CTA share one copy of L_11; with fewer than two such CTAs an SM, 32 rows.  The shell's Jacobians
// (a batch of 502 and a coarse matrix) take 68.9 ms so, 72.2 with 128 rows everywhere and 72.0 with 32;
// the 128x128x32 slab's (1,024 matrices) 41.4, 41.5 and 45.3.
static void launch_panel_rows(const MatDesc *d_desc, float *base, int K0, int max_below, int count, const float *pinv,
                              cudaStream_t s) {
  if (max_below <= 0) return;
  if (ceil_div(max_below, 128) * (long long)count >= 2 * kUpdCtas)
    k_panel_rows<128><<<dim3(ceil_div(max_below, 128), count), 256, panel_smem<128>(), s>>>(d_desc, base, K0, pinv);
  else
    k_panel_rows<32><<<dim3(ceil_div(max_below, 32), count), 256, panel_smem<32>(), s>>>(d_desc, base, K0, pinv);
  count_launch();
}

static void launch_rankk(const MatDesc *d_desc, float *base, int mode, int k0, int K0, int K1, int max_rows,
                         int max_cols, int count, cudaStream_t s) {
  const int nrt = ceil_div(max_rows, kTB2), nct = ceil_div(max_cols, kTB2);
  if (nrt == 0 || nct == 0) return;
  k_rankk128<<<dim3(nrt * nct, count), 256, 0, s>>>(d_desc, base, mode, k0, K0, K1, nct);
  count_launch();
}

// Lower-triangle entries that a band-limited update of rows band_rows(hd, t0, ke) x columns
// [t0, cend) touches: the interior rows up to the band (a trapezoid), then every column of
// the rows from e on (for a dense matrix: rows [t0, m) x columns [t0, cend), c <= r).
static double band_entries(const MatDesc &hd, int t0, int ke, int cend) {
  const long long k = cend - t0;
  if (k <= 0) return 0.0;
  const BandRows br = band_rows(hd, t0, ke);
  const long long iend = t0 + br.ni;
  const long long a = std::max(0LL, std::min(iend, (long long)cend) - t0);
  const long long b = std::max(0LL, iend - cend);
  return (double)(a * (a + 1) / 2 + b * k + (long long)(br.nv - br.ni) * k);
}

// Few matrices (kAheadCount at most) leave the chip idle in the chain of a block's panels (a diagonal
// block is one CTA for 32 us, its rows a few CTAs for 11).  There the trailing update is cut in two:
// first the columns of the next outer block, then, beside that block's panels on a second stream, the
// columns right of it, on kAheadSms fewer CTAs so that the panels find free SMs.  The two sides share
// no column, and the digit planes of the panels' own updates take half of the workspace.  A Jacobian
// of the masked shell (coarse matrix of 2,618 unknowns) takes 3 % less, of the 128x128x32 slab too.  Both
// constants come from these coarse matrices (40 SMs: the same); batches of 9 to about 100 matrices, whose
// panels leave as many SMs idle, were not tried.
constexpr int kAheadCount = 8, kAheadSms = 24;

template <typename T>
void engine_partial_cholesky(const EngineShape &sh, const MatDesc *d_desc, T *base, int *d_err, cudaStream_t s,
                             T *store, ProfHook *prof, int tc, const SliceWs &ws, const LookAhead *ahead) {
  if (sh.count == 0) return;
  constexpr bool f64 = std::is_same<T, double>::value;
  const bool narrow = f64 || tc == 2;  // 64-column panels solved on the tensor cores
  const int PW = narrow ? kPanel64 : kPW;
  T *pinv = static_cast<T *>(ws.pinv);
  const int ob = std::max(kPW, (sh.ob / kPW) * kPW);  // outer block: columns per long-K trailing update
  SliceWs half[2] = {ws, ws};                         // planes of the trailing updates, of the panels ahead
  half[0].bytes = half[1].bytes = (ws.bytes / 2) & ~(size_t)4095;
  half[1].mem = ws.mem + half[0].bytes;
  const bool look = ahead && (f64 || tc) && sh.count <= kAheadCount && sh.max_e > ob &&
                    slice_fits<T>(sh.count, sh.max_m, std::max(ob, PW), half[0]);
  // host copies of the descriptors' sizes and bands: the grids cover the rows and columns
  // the band lets an update reach (the kernels apply the same limits per matrix)
  std::vector<MatDesc> hd(sh.count);
  for (int b = 0; b < sh.count; ++b) {
    hd[b].m = sh.m[b];
    hd[b].e = sh.e[b];
    if (!sh.band.empty()) hd[b].band = sh.band[b];
    if (!sh.id0.empty()) hd[b].id0 = sh.id0[b];
    if (!sh.ifirst.empty()) hd[b].ifirst = sh.ifirst[b];
  }
  // the panels of the outer block from K0 on
  auto block = [&](int K0, cudaStream_t q, const SliceWs &w_s) {
    const int K1 = K0 + ob;
    for (int k0 = K0; k0 < std::min(K1, sh.max_e); k0 += PW) {
      int max_below = 0, max_cols = 0;
      double fl_panel = 0.0, fl_in = 0.0;
      for (int b = 0; b < sh.count; ++b) {
        if (k0 >= sh.e[b]) continue;
        const int w = std::min(PW, sh.e[b] - k0);
        const int below = band_rows(hd[b], k0 + w, k0 + w).nv;
        const int cend = std::min({K1, sh.e[b], band_limit(hd[b], k0 + w)});
        max_below = std::max(max_below, below);
        max_cols = std::max(max_cols, cend - k0 - w);
        fl_panel += (double)w * w * w / 3.0 + (double)below * w * w;
        fl_in += 2.0 * w * band_entries(hd[b], k0 + w, k0 + w, cend);
      }
      if (prof) prof->begin(PROF_PANEL, q);
      if (narrow) {
        launch_diag<T>(d_desc, base, k0, sh.count, d_err, store, w_s, q);
        launch_update<T>(d_desc, base, Upd64{3, k0, 0, PW, 0, 0}, max_below, PW, sh.count, w_s, d_err, q);
      } else if constexpr (!f64) {
        launch_diag128(d_desc, base, k0, sh.count, d_err, store, pinv, q);
        launch_panel_rows(d_desc, base, k0, max_below, sh.count, pinv, q);
      }
      if (prof) prof->end(PROF_PANEL, q, fl_panel, 0.0);
      // the rest of the outer block: rows [k0 + w, m), columns [k0 + w, min(K1, e)); timed
      // with the panels (the long-K class holds only the trailing updates)
      if (max_below > 0 && max_cols > 0) {
        if (prof) prof->begin(PROF_PANEL, q);
        if constexpr (f64) {
          launch_update<T>(d_desc, base, Upd64{0, k0, K1, PW, 0, 0}, max_below, max_cols, sh.count, w_s, d_err, q);
        } else {
          if (tc) launch_update<T>(d_desc, base, Upd64{0, k0, K1, PW, 0, 0}, max_below, max_cols, sh.count, w_s, d_err, q);
          else launch_rankk(d_desc, base, 0, k0, K0, K1, max_below, max_cols, sh.count, q);
        }
        if (prof) prof->end(PROF_PANEL, q, fl_in, 0.0);
      }
    }
  };
  block(0, s, ws);
  for (int K0 = 0; K0 < sh.max_e; K0 += ob) {
    const int K1 = K0 + ob;
    // outer update of the trailing columns [K1, e) with the finished outer panel
    int max_rows = 0, max_cols = 0;
    double fl = 0.0, by = 0.0;
    for (int b = 0; b < sh.count; ++b) {
      if (K1 >= sh.e[b]) continue;
      const int rows = band_rows(hd[b], K1, K1).nv, cend = band_limit(hd[b], K1);
      max_rows = std::max(max_rows, rows);
      max_cols = std::max(max_cols, cend - K1);
      const double ent = band_entries(hd[b], K1, K1, cend);
      fl += 2.0 * ob * ent;
      by += sizeof(T) * (2.0 * ent + (double)ob * rows);
    }
    const bool update = max_rows > 0 && max_cols > 0;
    const Upd64 u{2, K0, K1, PW, K0, K1};
    if (update && look) {
      if (prof) prof->begin(PROF_RANKK, s);
      launch_update<T>(d_desc, base, u, max_rows, max_cols, sh.count, half[0], d_err, s,
                       UpdPart{0, ob / kUpdN, false, 0});
      cudaEventRecord(ahead->cols, s);
      cudaStreamWaitEvent(ahead->s, ahead->cols, 0);
      launch_update<T>(d_desc, base, u, max_rows, max_cols, sh.count, half[0], d_err, s,
                       UpdPart{ob / kUpdN, -1, true, kUpdCtas - kAheadSms});
      if (prof) prof->end(PROF_RANKK, s, fl, by);
      block(K1, ahead->s, half[1]);
      cudaEventRecord(ahead->panels, ahead->s);
      cudaStreamWaitEvent(s, ahead->panels, 0);
      continue;
    }
    if (update) {
      if (prof) prof->begin(PROF_RANKK, s);
      if constexpr (f64) {
        launch_update<T>(d_desc, base, u, max_rows, max_cols, sh.count, ws, d_err, s);
      } else {
        if (tc) launch_update<T>(d_desc, base, u, max_rows, max_cols, sh.count, ws, d_err, s);
        else launch_rankk(d_desc, base, 2, 0, K0, K1, max_rows, max_cols, sh.count, s);
      }
      if (prof) prof->end(PROF_RANKK, s, fl, by);
    }
    if (K1 < sh.max_e) block(K1, s, ws);
  }
  int max_t = 0;
  double fl = 0.0, by = 0.0;
  for (int b = 0; b < sh.count; ++b) {
    const int rows = band_rows(hd[b], sh.e[b], sh.e[b]).nv;  // rows whose L row is not zero
    max_t = std::max(max_t, rows);
    const double n2 = sh.m[b] - sh.e[b];
    if (hd[b].ifirst) {  // row g of the trailing block needs K from ifirst[g] on
      for (int g = 0; g < rows; ++g) {
        const double k = sh.e[b] - (hd[b].ifirst[g] & ~3);
        fl += 2.0 * k * (g + 1);
        by += sizeof(T) * (2.0 * (g + 1) + k);
      }
    } else {
      const double ent = n2 * (n2 + 1) / 2.0;
      fl += 2.0 * sh.e[b] * ent;
      by += sizeof(T) * (2.0 * ent + n2 * sh.e[b]);
    }
  }
  if (max_t > 0) {
    if (prof) prof->begin(PROF_RANKK, s);
    if constexpr (f64) {
      launch_update<T>(d_desc, base, Upd64{1, 0, 0, PW, 0, sh.max_e}, max_t, max_t, sh.count, ws, d_err, s);
    } else {
      if (tc) launch_update<T>(d_desc, base, Upd64{1, 0, 0, PW, 0, sh.max_e}, max_t, max_t, sh.count, ws, d_err, s);
      else launch_rankk(d_desc, base, 1, 0, 0, 0, max_t, max_t, sh.count, s);
    }
    if (prof) prof->end(PROF_RANKK, s, fl, by);
  }
}

// ---- batched GEMV ------------------------------------------------------------
// One CTA (8 warps) per (task, block of kGemvRows rows): each warp owns two rows
// with independent accumulators; x is staged in shared memory.  prof (interface rows of the local
// factors only): row g of matrix b is zero left of prof[b].ifirst[g], non-decreasing, and not read there
// (the 128x128x32 slab's 1,024 matrices: 382 -> 271 us).
constexpr int kGemvRows = 16;

template <typename T>
__global__ void __launch_bounds__(256) k_gemv(const GemvDesc *__restrict__ tasks, const T *__restrict__ A,
                                              const double *__restrict__ x, const int *__restrict__ xidx,
                                              double *__restrict__ y, double alpha, const int *__restrict__ done,
                                              const MatDesc *__restrict__ prof) {
  pdl_wait();
  if (done && *done) return;
  const GemvDesc t = tasks[blockIdx.y];
  const int rbeg = blockIdx.x * kGemvRows;
  if (rbeg >= t.rows) return;
  const int first = prof && prof[blockIdx.y].ifirst ? prof[blockIdx.y].ifirst[rbeg] & ~63 : 0;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *xs = reinterpret_cast<T *>(smem_raw);
  for (int c = first + threadIdx.x; c < t.cols; c += blockDim.x)
    xs[c] = (T)((t.flags & 1) ? x[xidx[t.x_off + c]] : x[t.x_off + c]);
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int r0 = rbeg + wid, r1 = rbeg + wid + 8;
  const bool v0 = r0 < t.rows, v1 = r1 < t.rows;
  const T *row0 = A + t.a_off + (long long)(v0 ? r0 : rbeg) * t.ld;
  const T *row1 = A + t.a_off + (long long)(v1 ? r1 : rbeg) * t.ld;
  T a0 = T(0), a1 = T(0), b0 = T(0), b1 = T(0);
  int c = first + lane;
  for (; c + 32 < t.cols; c += 64) {
    const T x0 = xs[c], x1 = xs[c + 32];
    a0 += row0[c] * x0;
    a1 += row0[c + 32] * x1;
    b0 += row1[c] * x0;
    b1 += row1[c + 32] * x1;
  }
  if (c < t.cols) {
    a0 += row0[c] * xs[c];
    b0 += row1[c] * xs[c];
  }
  const T s0 = warp_sum(a0 + a1), s1 = warp_sum(b0 + b1);
  if (lane == 0) {
    if (v0) {
      const double v = alpha * (double)s0;
      y[t.y_off + r0] = (t.flags & 2) ? y[t.y_off + r0] + v : v;
    }
    if (v1) {
      const double v = alpha * (double)s1;
      y[t.y_off + r1] = (t.flags & 2) ? y[t.y_off + r1] + v : v;
    }
  }
}

// ---- batched symmetric GEMV (FP32): S = nparts CTAs (8 warps each) per matrix -------
// The matrix is read as 32 x 32 tiles of its lower block triangle, each once: tile (I, J),
// J < I, serves both y_I += A_IJ x_J and y_J += A_IJ^T x_I; a diagonal tile serves
// y_I += A_II x_I.  CTA s of a matrix takes the s-th of S contiguous runs of the row-major
// tile order and splits it over its warps the same way.  A lane holds 4 columns of every fourth row of
// its tile (eight 16-byte loads, the next tile's in flight meanwhile) and multiplies from
// registers: its eight row sums stay in registers along a block row and are reduced over the eight
// lanes of a row at its end; its four column sums are reduced over the four lanes of a column per tile.
// Both end in the warp's own partial vector, so no two warps write the same word.  The CTA
// adds its warps' vectors in warp order; with S > 1 it stores the sum in `scratch` and the last CTA
// of the matrix to finish (counter per matrix, reset by that CTA) adds the S sums in order
// s = 0 .. S-1.  Deterministic; half the bytes of a full GEMV.  Bound by HBM: with the tiles copied
// to shared memory and read there twice it was bound by those reads (160 a tile against 190 clocks of
// HBM time; 206 us for the 1,024 matrices of order 772; now 168 us, 7.3 TB/s).
// Plain rows of B go to the CTAs round-robin.
__global__ void __launch_bounds__(256, 2) k_symv_batched(const SymvTask *__restrict__ tasks, const float *__restrict__ A,
                                                         const double *__restrict__ x, const int *__restrict__ xidx,
                                                         double *__restrict__ y, double alpha,
                                                         const int *__restrict__ done, float *__restrict__ scratch,
                                                         int *__restrict__ counter, int ld_scr) {
  pdl_wait();
  if (done && *done) return;
  const SymvTask t = tasks[blockIdx.x];
  const int S = t.nparts, sidx = t.part;
  const int n = t.n, nb = (n + 31) >> 5, np = nb * 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float *xs = reinterpret_cast<float *>(smem_raw);  // [np]
  float *part = xs + np;                             // [8][np]
  __shared__ int last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int c = tid; c < np; c += 256)
    xs[c] = c < n ? (float)((t.flags & 1) ? x[xidx[t.x_off + c]] : x[t.x_off + c]) : 0.f;
  for (int c = tid; c < 8 * np; c += 256) part[c] = 0.f;
  __syncthreads();
  const float *a = A + t.a_off;
  float *mine = part + warp * np;
  const long long ntiles = (long long)nb * (nb + 1) / 2;
  const long long c0 = ntiles * sidx / S, c1 = ntiles * (sidx + 1) / S;  // this CTA's run
  const int s0 = (int)(c0 + (c1 - c0) * warp / 8), s1 = (int)(c0 + (c1 - c0) * (warp + 1) / 8);
  // tile index s = I (I + 1) / 2 + J  ->  (I, J)
  int I = 0;
  while ((I + 1) * (I + 2) / 2 <= s0) ++I;
  int J = s0 - I * (I + 1) / 2;
  const int lr = lane >> 3, lc = (lane & 7) * 4;  // this lane's first row and column in a tile
  float4 v[8], nx[8];
  auto load = [&](float4 (&b)[8], int ti, int tj) {
    const float *p = a + (long long)(32 * ti + lr) * t.ld + 32 * tj + lc;
    if (32 * ti + 32 <= n) {  // tj <= ti: every entry inside
#pragma unroll
      for (int i = 0; i < 8; ++i) b[i] = *reinterpret_cast<const float4 *>(p + (long long)(4 * i) * t.ld);
    } else {
      const int c = 32 * tj + lc;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
        if (32 * ti + lr + 4 * i < n && c < n) {
          q = *reinterpret_cast<const float4 *>(p + (long long)(4 * i) * t.ld);
          if (c + 1 >= n) q.y = 0.f;
          if (c + 2 >= n) q.z = 0.f;
          if (c + 3 >= n) q.w = 0.f;
        }
        b[i] = q;
      }
    }
  };
  float rs[8], xr[8];  // sums of this lane's rows along the block row; x at those rows
  auto rows = [&](int ti) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      rs[i] = 0.f;
      xr[i] = xs[32 * ti + 4 * i + lr];
    }
  };
  auto flush = [&](int ti) {  // lane -> row 4 i + lr, i the low three bits of the lane
    const bool b2 = lane & 4, b1 = lane & 2, b0 = lane & 1;
    float p4[4], p2[2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      p4[i] = (b2 ? rs[4 + i] : rs[i]) + __shfl_xor_sync(0xffffffffu, b2 ? rs[i] : rs[4 + i], 4);
#pragma unroll
    for (int i = 0; i < 2; ++i)
      p2[i] = (b1 ? p4[2 + i] : p4[i]) + __shfl_xor_sync(0xffffffffu, b1 ? p4[i] : p4[2 + i], 2);
    const float r = (b0 ? p2[1] : p2[0]) + __shfl_xor_sync(0xffffffffu, b0 ? p2[0] : p2[1], 1);
    mine[32 * ti + 4 * (lane & 7) + lr] += r;
    __syncwarp();
  };
  if (s0 < s1) {
    load(v, I, J);
    rows(I);
  }
  for (int s = s0; s < s1; ++s) {
    const int ci = I, cj = J;
    if (++J > I) { ++I; J = 0; }
    if (s + 1 < s1) load(nx, I, J);  // in flight while this tile is multiplied
    const float4 xc = *reinterpret_cast<const float4 *>(xs + 32 * cj + lc);
#pragma unroll
    for (int i = 0; i < 8; ++i) rs[i] += (v[i].x * xc.x + v[i].y * xc.y) + (v[i].z * xc.z + v[i].w * xc.w);
    if (cj < ci) {
      float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        c.x += v[i].x * xr[i];
        c.y += v[i].y * xr[i];
        c.z += v[i].z * xr[i];
        c.w += v[i].w * xr[i];
      }
      const bool b4 = lane & 16, b3 = lane & 8;  // lane -> column lc + 2 b4 + b3
      const float e0 = (b4 ? c.z : c.x) + __shfl_xor_sync(0xffffffffu, b4 ? c.x : c.z, 16);
      const float e1 = (b4 ? c.w : c.y) + __shfl_xor_sync(0xffffffffu, b4 ? c.y : c.w, 16);
      const float e = (b3 ? e1 : e0) + __shfl_xor_sync(0xffffffffu, b3 ? e0 : e1, 8);
      mine[32 * cj + lc + (b4 ? 2 : 0) + (b3 ? 1 : 0)] += e;
      __syncwarp();
    }
    if (I != ci || s + 1 == s1) {
      flush(ci);
      if (s + 1 < s1) rows(I);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = nx[i];
  }
  // plain rows of B: one warp per row, rows dealt to the CTAs round-robin
  for (int r = sidx + S * warp; r < t.nb; r += 8 * S) {
    const float *brow = A + t.b_off + (long long)r * t.ld;
    float acc = 0.f;
    for (int c = lane; c < n; c += 32) acc += brow[c] * xs[c];
    acc = warp_sum(acc);
    if (lane == 0) {
      const double o = alpha * (double)acc;
      y[t.yb_off + r] = (t.flags & 2) ? y[t.yb_off + r] + o : o;
    }
  }
  __syncthreads();
  auto column = [&](int r) {
    float s = part[r];
#pragma unroll
    for (int w = 1; w < 8; ++w) s += part[w * np + r];
    return s;
  };
  if (S == 1) {
    for (int r = tid; r < n; r += 256) {
      const double o = alpha * (double)column(r);
      y[t.y_off + r] = (t.flags & 2) ? y[t.y_off + r] + o : o;
    }
    return;
  }
  float *mysum = scratch + ((long long)t.scr + sidx) * ld_scr;
  for (int r = tid; r < n; r += 256) mysum[r] = column(r);
  __threadfence();
  __syncthreads();
  if (tid == 0) last = (atomicAdd(&counter[t.ctr], 1) == S - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();
  const float *sums = scratch + (long long)t.scr * ld_scr;
  for (int r = tid; r < n; r += 256) {
    float s = __ldcg(sums + r);
    for (int q = 1; q < S; ++q) s += __ldcg(sums + (long long)q * ld_scr + r);
    const double o = alpha * (double)s;
    y[t.y_off + r] = (t.flags & 2) ? y[t.y_off + r] + o : o;
  }
  if (tid == 0) counter[t.ctr] = 0;  // ready for the next launch
}

static size_t symv_fix_smem(int max_n) {
  const size_t nb = (max_n + 31) / 32;
  return nb * 32 * (8 * sizeof(double) + sizeof(int2)) + ((nb + 3) & ~(size_t)3) * sizeof(int) + 8 * 32 * 33 * sizeof(int2);
}
template <typename T>
size_t symv_smem(int max_n) {
  const size_t np = (size_t)((max_n + 31) / 32) * 32;
  return std::is_same<T, double>::value ? symv_fix_smem(max_n) : sizeof(T) * 9 * np;
}

// The CTAs of a launch: whole matrices while they fill the resident slots (a split costs a
// partial-sum round trip and shorter prefetch runs), largest first, and the ones that would make up
// a last, part-empty wave split over several CTAs.  Which ones and into how many parts is decided by
// scheduling the CTAs on the slots with a cost of their tiles plus a fixed part (staging, reduction),
// for every candidate.  1,024 matrices of order 772 on 304 slots (two CTAs an SM): 112 of them in halves,
// three waves of whole matrices and one of halves instead of four.  The fixed parts were fitted when
// three CTAs shared an SM and not again.
std::vector<SymvTask> symv_plan(const std::vector<SymvTask> &tasks, int slots, int *scratch_rows, int *counters) {
  constexpr double kFix = 24.0, kSplitFix = 20.0;  // in tiles of 32 x 32
  const int n = (int)tasks.size();
  auto tiles = [](const SymvTask &t) { const double b = (t.n + 31) / 32; return b * (b + 1) / 2; };
  std::vector<int> order(n);
  for (int i = 0; i < n; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return tasks[a].n > tasks[b].n; });
  double total = 0.0;
  for (const SymvTask &t : tasks) total += tiles(t);
  slots = std::max(1, slots);
  auto parts_of = [&](int i, int tail, int p) {  // parts of the i-th matrix of the order
    const double w = tiles(tasks[order[i]]);
    const int most = (int)std::max(1.0, std::min(16.0, w / 8.0));  // one tile per warp at least
    int q = i >= n - tail ? p : 1;
    if (w > total / slots) q = std::max(q, (int)std::ceil(w * slots / total));
    return std::min(q, most);
  };
  auto makespan = [&](int tail, int p) {
    std::vector<double> load(slots, 0.0);  // a heap of the slots' finishing times
    auto later = [](double a, double b) { return a > b; };
    for (int i = 0; i < n; ++i) {
      const int q = parts_of(i, tail, p);
      const double c = tiles(tasks[order[i]]) / q + kFix + (q > 1 ? kSplitFix : 0.0);
      for (int k = 0; k < q; ++k) {
        std::pop_heap(load.begin(), load.end(), later);
        load.back() += c;
        std::push_heap(load.begin(), load.end(), later);
      }
    }
    return *std::max_element(load.begin(), load.end());
  };
  int best_tail = 0, best_p = 1;
  double best = makespan(0, 1);
  for (int tail : {n % slots, n % slots + slots, n / 2, n})
    for (int p : {2, 3, 4, 5, 6, 8, 12, 16}) {
      if (tail <= 0 || tail > n) continue;
      const double m = makespan(tail, p);
      if (m < 0.98 * best) { best = m; best_tail = tail; best_p = p; }
    }
  std::vector<SymvTask> out;
  int rows = 0, ctrs = 0;
  for (int i = 0; i < n; ++i) {
    SymvTask t = tasks[order[i]];
    t.nparts = parts_of(i, best_tail, best_p);
    if (t.nparts > 1) {
      t.scr = rows;
      t.ctr = ctrs++;
      rows += t.nparts;
    }
    for (t.part = 0; t.part < t.nparts; ++t.part) out.push_back(t);
  }
  *scratch_rows = rows;
  *counters = ctrs;
  return out;
}


void launch_symv_batched(int ntasks, int max_n, const SymvTask *d_tasks, const float *A, const double *x,
                         const int *xidx, double *y, double alpha, const int *done, float *scratch, int *counter,
                         int ld_scr, cudaStream_t s) {
  if (ntasks == 0 || max_n == 0) return;
  launch_pdl(k_symv_batched, ntasks, 256, symv_smem<float>(max_n), s, d_tasks, A, x, xidx, y, alpha, done, scratch,
                                                                    counter, ld_scr);
  count_launch();
}

// ---- FP64 symmetric products in integer arithmetic --------------------------------
// The FP64 pipe (2 multiply-adds per SM and clock) cannot keep up with HBM: a symmetric product needs
// 5.4 of them per SM and clock at the copy rate.  So the operators' lower block triangles are kept a
// second time as 32 x 32 tiles of fixed-point numbers: A = D A' D with D the powers of two of the
// diagonal's square roots, so that the positive definite A' has |A'_rc| <= 1 whatever the units or the
// contrast of the two media; every tile of A' is rounded once to 55 bits below its power of two 2^e,
// X = 2^28 h + l with |h|, |l| <= 2^27 (8 bytes, as the FP64 entry; error at most 2^(e - 56)); D x
// likewise by segments of 32.  A tile's product with a segment is then four 32 x 32 -> 64-bit integer
// multiply-adds per entry, exact, and two FP64 instructions per row and tile.  Packed tiles in the order
// of k_symv_batched; the same parts, partial vectors and fixed orders.
__device__ __forceinline__ double pow2(int e) {  // 2^e, e clamped to the normal range
  return __hiloint2double((max(min(e, 1023), -1022) + 1023) << 20, 0);
}
// v 2^e, by two factors where 2^e is no normal number
__device__ __forceinline__ double scale2(double v, int e) {
  if (e < -1022 || e > 1023) return v * pow2(e / 2) * pow2(e - e / 2);
  return v * pow2(e);
}
__device__ __forceinline__ int2 fix_split(double x, int e) {  // |x| < 2^e
  const long long X = __double2ll_rn(scale2(x, 55 - e));
  const int lo = (int)(X & ((1 << 28) - 1)), l = lo - ((lo >> 27) << 28);
  return make_int2((int)((X - l) >> 28), l);
}
// exponent of a tile or segment that holds an infinity or a NaN; such a segment of x keeps the FP64
// numbers themselves, and its products are those of fix_special
constexpr int kFixNan = 1 << 20;
constexpr int kFixZero = -(1 << 20);
// the exponent e of a number times 2^se, |v| 2^se < 2^e
__device__ __forceinline__ int fix_exp(double v, int se) {
  const int mag = __double2hiint(v) & 0x7fffffff;
  return (mag | __double2loint(v)) == 0 ? kFixZero : mag >= 0x7ff00000 ? kFixNan : (mag >> 20) - 1022 + se;
}
// D's exponent from a diagonal entry: half of its own, rounded up
__device__ __forceinline__ int fix_half(double v) {
  const int e = fix_exp(v, 0);
  return e == kFixZero || e == kFixNan ? 0 : (e + 1) >> 1;
}

// One tile per CTA, grid-stride over a matrix's tiles: task.a_off -> packed tile task.f_off + s.
__global__ void __launch_bounds__(256) k_fix_tiles(const FixTask *__restrict__ tasks, const double *__restrict__ A,
                                                   int2 *__restrict__ tiles, int *__restrict__ ex) {
  const FixTask t = tasks[blockIdx.y];
  const int nb = (t.n + 31) >> 5, ntiles = nb * (nb + 1) / 2;
  __shared__ int smax[8], half[64];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int s = blockIdx.x; s < ntiles; s += gridDim.x) {
    int I = (int)((sqrtf(8.f * s + 1.f) - 1.f) * 0.5f);
    while ((I + 1) * (I + 2) / 2 <= s) ++I;
    while (I * (I + 1) / 2 > s) --I;
    const int J = s - I * (I + 1) / 2;
    if (tid < 64) {  // D of the tile's rows, then of its columns; a diagonal tile stores it
      const int r = 32 * (tid < 32 ? I : J) + lane;
      half[tid] = r < t.n ? fix_half(A[t.a_off + (long long)r * (t.ld + 1)]) : 0;
      if (I == J && tid < 32) ex[t.d_off + r] = half[tid];
    }
    double v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = 32 * I + warp + 8 * q, c = 32 * J + lane;
      v[q] = r < t.n && c < t.n ? A[t.a_off + (long long)r * t.ld + c] : 0.0;
    }
    __syncthreads();
    int e = kFixZero, se[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      se[q] = half[warp + 8 * q] + half[32 + lane];
      e = max(e, fix_exp(v[q], -se[q]));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) smax[warp] = e;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 8; ++q) e = max(e, smax[q]);
    __syncthreads();
    if (e == kFixZero) e = 0;
    if (tid == 0) ex[t.f_off + s] = e;
    int2 *out = tiles + (t.f_off + s) * 1024;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      out[(warp + 8 * q) * 32 + lane] = e == kFixNan ? make_int2(0, 0) : fix_split(v[q], e + se[q]);
  }
}

__device__ __forceinline__ void mad_wide(long long &acc, int a, int b) { acc += (long long)a * b; }

// 32 products of a tile (exponent ea) with a segment (eb) where 2^(ea + eb - 82) is no normal number or one
// of the two is marked; v: their fixed-point sum.  A marked segment holds FP64 numbers: a plain sum, in
// which infinities keep their signs.
__device__ __forceinline__ double fix_special(const int2 *a, int stride, const int2 *x, int ea, int eb, double v) {
  if (ea == kFixNan) return __hiloint2double(0x7ff80000, 0);
  if (eb != kFixNan) return scale2(v, ea + eb - 82);
  double s = 0.0;
#pragma unroll 1
  for (int c = 0; c < 32; ++c) {
    const int2 t = a[c * stride];
    s += scale2(fma((double)t.x, 268435456.0, (double)t.y), ea - 55) * __hiloint2double(x[c].y, x[c].x);
  }
  return s;
}

__global__ void __launch_bounds__(256) k_symv_fix(const SymvTask *__restrict__ tasks, const int2 *__restrict__ tiles,
                                                  const int *__restrict__ ex, const double *__restrict__ x,
                                                  const int *__restrict__ xidx, double *__restrict__ y, double alpha,
                                                  const int *__restrict__ done, double *__restrict__ scratch,
                                                  int *__restrict__ counter, int ld_scr) {
  pdl_wait();
  if (done && *done) return;
  const SymvTask t = tasks[blockIdx.x];
  const int S = t.nparts, sidx = t.part;
  const int n = t.n, nb = (n + 31) >> 5, np = nb * 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double *part = reinterpret_cast<double *>(smem_raw);       // [8][np]
  int2 *xs = reinterpret_cast<int2 *>(part + 8 * np);        // [np] the segments of x, split
  int *xe = reinterpret_cast<int *>(xs + np);                // [nb] their exponents
  int2 *stage = reinterpret_cast<int2 *>(xe + ((nb + 3) & ~3));  // [8][32][33]
  __shared__ int last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int *dx = ex + t.d_off;  // exponents of D
  for (int b = warp; b < nb; b += 8) {
    const int c = 32 * b + lane;
    const double v = c < n ? ((t.flags & 1) ? x[xidx[t.x_off + c]] : x[t.x_off + c]) : 0.0;
    const int se = dx[c];
    int e = __reduce_max_sync(0xffffffffu, fix_exp(v, se));
    if (e == kFixZero) e = 0;
    if (e == kFixNan) {
      const double w = v * pow2(se);
      xs[c] = make_int2(__double2loint(w), __double2hiint(w));
    } else {
      xs[c] = fix_split(v, e - se);
    }
    if (lane == 0) xe[b] = e;
  }
  for (int c = tid; c < 8 * np; c += 256) part[c] = 0.0;
  __syncthreads();
  const long long ntiles = (long long)nb * (nb + 1) / 2;
  const long long c0 = ntiles * sidx / S, c1 = ntiles * (sidx + 1) / S;  // this CTA's run
  const int s0 = (int)(c0 + (c1 - c0) * warp / 8), s1 = (int)(c0 + (c1 - c0) * (warp + 1) / 8);
  int2 *tile = stage + warp * 32 * 33;
  double *mine = part + warp * np;
  int I = 0;
  while ((I + 1) * (I + 2) / 2 <= s0) ++I;
  int J = s0 - I * (I + 1) / 2;
  const int4 *src = reinterpret_cast<const int4 *>(tiles + t.f_off * 1024) + lane;
  const int *et = ex + t.f_off;
  int4 buf[16];
  int e1 = 0;
  auto load = [&](int s) {
#pragma unroll
    for (int i = 0; i < 16; ++i) buf[i] = src[(long long)s * 512 + 32 * i];
    e1 = et[s];
  };
  // sum of 32 products as FP64: (h h) 2^56 + (h l + l h) 2^28 + l l, the low part rounded to 2^28
  auto value = [&](long long hh, long long m, long long ll, int ea, const int2 *a, int stride, int seg) {
    const int eb = xe[seg], s = ea + eb - 82;
    m += (ll + (1 << 27)) >> 28;
    const double v = fma(__ll2double_rn(hh), 268435456.0, __ll2double_rn(m));
    // one test for all that is rare, shared by the warp
    if ((unsigned)(s + 1022) > 2045u) return fix_special(a, stride, xs + 32 * seg, ea, eb, v);
    return v * __hiloint2double((s + 1023) << 20, 0);
  };
  if (s0 < s1) load(s0);
  double racc = 0.0;  // row sums of the current block row
  for (int s = s0; s < s1; ++s) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {  // entries 64 i + 2 lane, + 1 of the tile
      int2 *p = tile + (2 * i + (lane >> 4)) * 33 + 2 * (lane & 15);
      p[0] = make_int2(buf[i].x, buf[i].y);
      p[1] = make_int2(buf[i].z, buf[i].w);
    }
    __syncwarp();
    const int ci = I, cj = J, e = e1;
    if (++J > I) { ++I; J = 0; }
    if (s + 1 < s1) load(s + 1);  // in flight while this tile is multiplied
    long long hh = 0, m = 0, ll = 0;
#pragma unroll 8
    for (int c = 0; c < 32; ++c) {
      const int2 a = tile[lane * 33 + c], b = xs[32 * cj + c];
      mad_wide(hh, a.x, b.x);
      mad_wide(m, a.x, b.y);
      mad_wide(m, a.y, b.x);
      mad_wide(ll, a.y, b.y);
    }
    racc += value(hh, m, ll, e, tile + lane * 33, 1, cj);
    if (cj < ci) {
      hh = m = ll = 0;
#pragma unroll 8
      for (int r = 0; r < 32; ++r) {
        const int2 a = tile[r * 33 + lane], b = xs[32 * ci + r];
        mad_wide(hh, a.x, b.x);
        mad_wide(m, a.x, b.y);
        mad_wide(m, a.y, b.x);
        mad_wide(ll, a.y, b.y);
      }
      mine[32 * cj + lane] += value(hh, m, ll, e, tile + lane, 33, ci);
    }
    if (I != ci || s + 1 == s1) {
      mine[32 * ci + lane] += racc;
      racc = 0.0;
    }
    __syncwarp();
  }
  __syncthreads();
  auto column = [&](int r) {
    double v = part[r];
#pragma unroll
    for (int w = 1; w < 8; ++w) v += part[w * np + r];
    return v;
  };
  if (S == 1) {
    for (int r = tid; r < n; r += 256) {
      const double o = alpha * (column(r) * pow2(dx[r]));
      y[t.y_off + r] = (t.flags & 2) ? y[t.y_off + r] + o : o;
    }
    return;
  }
  double *mysum = scratch + ((long long)t.scr + sidx) * ld_scr;
  for (int r = tid; r < n; r += 256) mysum[r] = column(r);
  __threadfence();
  __syncthreads();
  if (tid == 0) last = (atomicAdd(&counter[t.ctr], 1) == S - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();
  const double *sums = scratch + (long long)t.scr * ld_scr;
  for (int r = tid; r < n; r += 256) {
    double v = __ldcg(sums + r);
    for (int q = 1; q < S; ++q) v += __ldcg(sums + (long long)q * ld_scr + r);
    const double o = alpha * (v * pow2(dx[r]));
    y[t.y_off + r] = (t.flags & 2) ? y[t.y_off + r] + o : o;
  }
  if (tid == 0) counter[t.ctr] = 0;  // ready for the next launch
}

template <typename T>
int symv_occupancy(int max_n) {
  int occ = 0;
  const cudaError_t e =
      std::is_same<T, double>::value
          ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_symv_fix, 256, symv_smem<T>(max_n))
          : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_symv_batched, 256, symv_smem<T>(max_n));
  if (e != cudaSuccess) return 0;
  return occ;
}

void launch_fix_tiles(int n, int max_n, const FixTask *d_tasks, const double *A, int2 *tiles, int *ex, cudaStream_t s) {
  if (n == 0 || max_n == 0) return;
  const int nb = ceil_div(max_n, 32);
  k_fix_tiles<<<dim3(std::min(nb * (nb + 1) / 2, 64), n), 256, 0, s>>>(d_tasks, A, tiles, ex);
  count_launch();
}
void launch_symv_fix(int ntasks, int max_n, const SymvTask *d_tasks, const int2 *tiles, const int *ex, const double *x,
                     const int *xidx, double *y, double alpha, const int *done, double *scratch, int *counter,
                     int ld_scr, cudaStream_t s) {
  if (ntasks == 0 || max_n == 0) return;
  launch_pdl(k_symv_fix, ntasks, 256, symv_fix_smem(max_n), s, d_tasks, tiles, ex, x, xidx, y, alpha, done, scratch, counter,
                                                       ld_scr);
  count_launch();
}

// y[a] = (acc ? y[a] : 0) + alpha sum_p A[p][a] x[p]: one CTA per (task, 64 columns);
// x may instead be a sparse product evaluated while staging (csr.ptr set).  A lane takes two
// columns (coalesced rows), the 8 warps split the rows with 8 loads in flight each and add up their
// partial sums in shared memory in a fixed order.  prof as in k_gemv: the rows that reach the CTA's
// columns come first, and only they are read.  Bound by HBM: 780 us for the interface rows of the
// 128x128x32 slab's 1,024 matrices before (all rows, four loads in flight, x staged per 32 columns), 364 us now.
constexpr int kGemvTCols = 64;
template <typename T>
__global__ void __launch_bounds__(256) k_gemv_t(const GemvDesc *__restrict__ tasks, const T *__restrict__ A,
                                                const double *__restrict__ x, const int *__restrict__ xidx,
                                                double *__restrict__ y, double alpha, const int *__restrict__ done,
                                                const CsrIn csr, const MatDesc *__restrict__ prof) {
  if (done && *done) return;
  const GemvDesc t = tasks[blockIdx.y];
  const int c0 = blockIdx.x * kGemvTCols;
  if (c0 >= t.cols) return;
  const int rows = prof ? min(t.rows, profile_rows(prof[blockIdx.y], c0 + kGemvTCols)) : t.rows;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *xs = reinterpret_cast<T *>(smem_raw);
  __shared__ T part[8][kGemvTCols];
  for (int p = threadIdx.x; p < rows; p += blockDim.x)
    xs[p] = (T)(csr.ptr ? csr_row(csr, t.x_off + p) : (t.flags & 1) ? x[xidx[t.x_off + p]] : x[t.x_off + p]);
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const T *col0 = A + t.a_off + min(c0 + lane, t.cols - 1), *col1 = A + t.a_off + min(c0 + 32 + lane, t.cols - 1);
  const long long ld = t.ld;
  T a0 = T(0), a1 = T(0), b0 = T(0), b1 = T(0);
  for (int p = wid; p < rows; p += 32) {
    T u[4], v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = min(p + 8 * q, rows - 1);
      u[q] = col0[r * ld];
      v[q] = col1[r * ld];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (p + 8 * q < rows) {
        const T xv = xs[p + 8 * q];
        if (q & 1) {
          a1 += u[q] * xv;
          b1 += v[q] * xv;
        } else {
          a0 += u[q] * xv;
          b0 += v[q] * xv;
        }
      }
    }
  }
  part[wid][lane] = a0 + a1;
  part[wid][32 + lane] = b0 + b1;
  __syncthreads();
  const int a = c0 + threadIdx.x;
  if (threadIdx.x < kGemvTCols && a < t.cols) {
    T sum = T(0);
#pragma unroll
    for (int k = 0; k < 8; ++k) sum += part[k][threadIdx.x];
    const double v = alpha * (double)sum;
    y[t.y_off + a] = (t.flags & 2) ? y[t.y_off + a] + v : v;
  }
}

// Batched GEMVs of many small matrices (deluxe blocks, Psi): one CTA per task covering all of
// its rows / columns, so the staging of x and the task descriptor are paid once per matrix.
// y = alpha A x (+ y): 8 warps over the rows, two rows at a time per warp, lanes over the
// columns (coalesced rows).  Bound by the latency of its loads: two in flight per lane before,
// eight now (the Krylov part of an FP64 Newton solve on the 32x32x16 slab 3.80 -> 3.59 ms with the transposed product's).
template <typename T>
__global__ void __launch_bounds__(256) k_gemv_task(const GemvDesc *__restrict__ tasks, const T *__restrict__ A,
                                                   const double *__restrict__ x, const int *__restrict__ xidx,
                                                   double *__restrict__ y, double alpha,
                                                   const int *__restrict__ done) {
  pdl_wait();
  if (done && *done) return;
  const GemvDesc t = tasks[blockIdx.x];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *xs = reinterpret_cast<T *>(smem_raw);
  for (int c = threadIdx.x; c < t.cols; c += blockDim.x)
    xs[c] = (T)((t.flags & 1) ? x[xidx[t.x_off + c]] : x[t.x_off + c]);
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int r0 = 2 * wid; r0 < t.rows; r0 += 16) {
    const int r1 = r0 + 1;
    const bool v1 = r1 < t.rows;
    const T *row0 = A + t.a_off + (long long)r0 * t.ld;
    const T *row1 = A + t.a_off + (long long)(v1 ? r1 : r0) * t.ld;
    T a0 = T(0), b0 = T(0);
    for (int c = lane; c < t.cols; c += 128) {  // eight loads in flight
      T u[4], v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int cc = c + 32 * q < t.cols ? c + 32 * q : c;
        u[q] = row0[cc];
        v[q] = row1[cc];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const T xv = c + 32 * q < t.cols ? xs[c + 32 * q] : T(0);
        a0 += u[q] * xv;
        b0 += v[q] * xv;
      }
    }
    const T s0 = warp_sum(a0), s1 = warp_sum(b0);
    if (lane == 0) {
      const double v = alpha * (double)s0;
      y[t.y_off + r0] = (t.flags & 2) ? y[t.y_off + r0] + v : v;
      if (v1) {
        const double w = alpha * (double)s1;
        y[t.y_off + r1] = (t.flags & 2) ? y[t.y_off + r1] + w : w;
      }
    }
  }
}

// y[a] = (acc ? y[a] : 0) + alpha sum_p A[p][a] x[p]: one CTA per task, one thread per column
// (coalesced rows), x staged (gathered, or a sparse product when csr.ptr is set).
template <typename T>
__global__ void __launch_bounds__(256) k_gemv_t_task(const GemvDesc *__restrict__ tasks, const T *__restrict__ A,
                                                     const double *__restrict__ x, const int *__restrict__ xidx,
                                                     double *__restrict__ y, double alpha,
                                                     const int *__restrict__ done, const CsrIn csr) {
  pdl_wait();
  if (done && *done) return;
  const GemvDesc t = tasks[blockIdx.x];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *xs = reinterpret_cast<T *>(smem_raw);
  for (int p = threadIdx.x; p < t.rows; p += blockDim.x)
    xs[p] = (T)(csr.ptr ? csr_row(csr, t.x_off + p) : (t.flags & 1) ? x[xidx[t.x_off + p]] : x[t.x_off + p]);
  __syncthreads();
  const T *base = A + t.a_off;
  const long long ld = t.ld;
  for (int a = threadIdx.x; a < t.cols; a += blockDim.x) {
    T a0 = T(0), a1 = T(0);
    int p = 0;
    for (; p + 7 < t.rows; p += 8) {  // eight loads in flight
      T u[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) u[q] = base[(p + q) * ld + a];
#pragma unroll
      for (int q = 0; q < 8; q += 2) {
        a0 += u[q] * xs[p + q];
        a1 += u[q + 1] * xs[p + q + 1];
      }
    }
    for (; p < t.rows; ++p) a0 += base[p * ld + a] * xs[p];
    const double v = alpha * (double)(a0 + a1);
    y[t.y_off + a] = (t.flags & 2) ? y[t.y_off + a] + v : v;
  }
}

template <typename T>
void launch_gemv_task(int ntasks, int max_rows, int max_cols, const GemvDesc *d_tasks, const T *A, const double *x,
                      const int *xidx, double *y, double alpha, const int *done, cudaStream_t s) {
  if (ntasks == 0 || max_rows == 0) return;
  launch_pdl(k_gemv_task<T>, ntasks, 256, sizeof(T) * (size_t)std::max(1, max_cols), s, d_tasks, A, x, xidx, y, alpha, done);
  count_launch();
}

template <typename T>
void launch_gemv_t_task(int ntasks, int max_rows, int max_cols, const GemvDesc *d_tasks, const T *A,
                        const double *x, const int *xidx, double *y, double alpha, const int *done, cudaStream_t s,
                        const CsrIn *csr) {
  if (ntasks == 0 || max_cols == 0) return;
  const int threads = max_cols <= 128 ? 128 : 256;
  const size_t sm = sizeof(T) * (size_t)std::max(1, max_rows);
  const CsrIn c = csr ? *csr : CsrIn{};
  // without csr this follows the join with the coarse solve's stream: an ordinary launch
  launch_maybe_pdl(csr != nullptr, k_gemv_t_task<T>, ntasks, threads, sm, s, d_tasks, A, x, xidx, y, alpha, done, c);
  count_launch();
}

// y (+)= A x for one large symmetric matrix stored in full (n x n, row-major, ld a multiple
// of 8, zero padding columns), reading only its lower block triangle.  The CTA of rows
// [I0, I0 + 8) takes
//   the row strip     A[I0 .. I0+8)[0 .. I0+8)   (diagonal 8 x 8 block included; one warp
//                     per row, 16-byte loads, four in flight per lane), and
//   the column strip  A[I0+8 .. n)[I0 .. I0+8)   (the symmetric images of the same rows'
//                     entries right of the diagonal block; 16-byte loads, 32 / (8 / VN) rows
//                     per warp instruction, four instructions in flight),
// so every CTA reads n x 8 values and the kernel touches half the matrix: the repeated
// products of an iterative refinement find it in L2.  x staged in shared memory in T,
// accumulation in T, partial sums added in a fixed order.  The coarse solve of large
// coarse problems.
template <typename T>
__global__ void __launch_bounds__(256) k_symv_rows(int n, const T *__restrict__ A, int ld,
                                                   const double *__restrict__ x, double *__restrict__ y,
                                                   int accumulate, const int *__restrict__ done) {
  pdl_wait();
  if (done && *done) return;
  using VT = typename Vec16<T>::V;
  constexpr int VN = Vec16<T>::N;
  constexpr int LPR = 8 / VN;    // lanes per 8-wide row segment of the column strip
  constexpr int RPI = 32 / LPR;  // column-strip rows per warp instruction
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *xs = reinterpret_cast<T *>(smem_raw);
  __shared__ T part[8][8];  // [warp][column of the block]: column-strip sums
  const int npad = (n + 7) & ~7;
  for (int c = threadIdx.x; c < npad; c += blockDim.x) xs[c] = c < n ? (T)x[c] : T(0);
  __syncthreads();
  const int I0 = blockIdx.x * 8, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = I0 + warp;
  // row strip: columns [0, I0 + 8) (I0 + 8 <= npad; padding columns are zero)
  T rs = T(0);
  if (row < n) {
    const VT *a = reinterpret_cast<const VT *>(A + (long long)row * ld);
    const VT *xv = reinterpret_cast<const VT *>(xs);
    const int nv = (I0 + 8) / VN;
    T acc0 = T(0), acc1 = T(0), acc2 = T(0), acc3 = T(0);
    int v = lane;
    for (; v + 96 < nv; v += 128) {
      const VT a0 = a[v], a1 = a[v + 32], a2 = a[v + 64], a3 = a[v + 96];
      acc0 += Vec16<T>::dot(a0, xv[v]);
      acc1 += Vec16<T>::dot(a1, xv[v + 32]);
      acc2 += Vec16<T>::dot(a2, xv[v + 64]);
      acc3 += Vec16<T>::dot(a3, xv[v + 96]);
    }
    for (; v < nv; v += 32) acc0 += Vec16<T>::dot(a[v], xv[v]);
    rs = warp_sum((acc0 + acc1) + (acc2 + acc3));
  }
  // column strip: rows [I0 + 8, n), columns [I0, I0 + 8); lane -> (row in the group, vector)
  T cs[VN];
#pragma unroll
  for (int q = 0; q < VN; ++q) cs[q] = T(0);
  {
    const int sub = lane / LPR, seg = lane % LPR;
    const T *col = A + I0 + seg * VN;
    constexpr int kStride = 8 * RPI;  // rows between a warp's consecutive instructions
    for (int j = I0 + 8 + warp * RPI + sub; j < n; j += 4 * kStride) {
      VT v[4];
      T xj[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int jj = j + u * kStride;
        v[u] = jj < n ? *reinterpret_cast<const VT *>(col + (long long)jj * ld) : VT{};
        xj[u] = jj < n ? xs[jj] : T(0);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) Vec16<T>::axpy(cs, v[u], xj[u]);
    }
#pragma unroll
    for (int q = 0; q < VN; ++q)
#pragma unroll
      for (int off = LPR; off < 32; off <<= 1) cs[q] += __shfl_xor_sync(0xffffffffu, cs[q], off);
    if (sub == 0) {
#pragma unroll
      for (int q = 0; q < VN; ++q) part[warp][seg * VN + q] = cs[q];
    }
  }
  __syncthreads();
  if (lane == 0 && row < n) {
    T t = rs;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += part[w][warp];
    y[row] = accumulate ? y[row] + (double)t : (double)t;
  }
}

template <typename T>
void launch_symv_rows(int n, const T *A, int ld, const double *x, double *y, int accumulate, const int *done,
                      cudaStream_t s) {
  if (n == 0) return;
  launch_pdl(k_symv_rows<T>, ceil_div(n, 8), 256, sizeof(T) * (size_t)((n + 7) & ~7), s, n, A, ld, x, y, accumulate, done);
  count_launch();
}

template <typename T>
void launch_gemv(int ntasks, int max_rows, int max_cols, const GemvDesc *d_tasks, const T *A, const double *x,
                 const int *xidx, double *y, double alpha, const int *done, cudaStream_t s, const MatDesc *prof) {
  if (ntasks == 0 || max_rows == 0) return;
  dim3 g(ceil_div(max_rows, kGemvRows), ntasks);
  const size_t sm = sizeof(T) * (size_t)std::max(1, max_cols);
  launch_pdl(k_gemv<T>, g, 256, sm, s, d_tasks, A, x, xidx, y, alpha, done, prof);
  count_launch();
}

template <typename T>
void launch_gemv_t(int ntasks, int max_rows, int max_cols, const GemvDesc *d_tasks, const T *A, const double *x,
                   const int *xidx, double *y, double alpha, const int *done, cudaStream_t s, const CsrIn *csr,
                   const MatDesc *prof) {
  if (ntasks == 0 || max_cols == 0) return;
  dim3 g(ceil_div(max_cols, kGemvTCols), ntasks);
  const size_t sm = sizeof(T) * (size_t)std::max(1, max_rows);
  k_gemv_t<T><<<g, 256, sm, s>>>(d_tasks, A, x, xidx, y, alpha, done, csr ? *csr : CsrIn{}, prof);
  count_launch();
}

// ---- batched triangular solves (one CTA of 32 warps per matrix) ---------------
// y = L^-1 b (lower, blocks in increasing order) or y = L^-T b (upper, decreasing),
// 32-row blocks, one barrier per block.  While warp 0 finishes block k (adds the
// contributions gathered for it, then substitutes with the factored diagonal block
// from the engine's store), warps 1..31 gather everything the next block needs
// that is already final: its diagonal block, the sums over the solved blocks before
// k (16-byte vector loads, several in flight per lane) and the 32 x 32 tile that
// couples it to block k.  Buffers alternate between blocks; the vector lives in
// shared memory.
template <typename T>
__global__ void __launch_bounds__(1024) k_trsv(const MatDesc *__restrict__ desc, const int *__restrict__ vec_off,
                                               const T *__restrict__ base, const T *__restrict__ store,
                                               const double *__restrict__ b, double *__restrict__ y, int transpose) {
  using VT = typename Vec16<T>::V;
  constexpr int VN = Vec16<T>::N, VPR = kNB / VN, RPW = 32 / VPR;
  const MatDesc d = desc[blockIdx.x];
  const int n = d.e;
  const T *L = base + d.off;
  // dynamic shared memory: six 32 x 33 tiles, then the vector
  typedef T Tile[32][33];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Tile *Lb = reinterpret_cast<Tile *>(smem_raw);  // [2] diagonal block
  Tile *Lt = Lb + 2;    // [2] coupling tile: lower Lt[j][c] = L[r0n + j][r0 + c]; upper Lt[c][j] = L[r0 + c][r0n + j]
  Tile *part = Lb + 4;  // [2] lower: part[0][j] = prefix sums; upper: part[w][j] per warp
  T *v = reinterpret_cast<T *>(Lb + 6);
  const int off = vec_off[blockIdx.x];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nblk = ceil_div(n, 32);
  for (int i = threadIdx.x; i < n; i += blockDim.x) v[i] = (T)b[off + i];
  if (nblk > 0) {
    const int b0 = transpose ? nblk - 1 : 0;
    Lb[0][wid][lane] = store[((long long)d.dblk + b0) * kNB * kNB + wid * kNB + lane];
  }
  __syncthreads();
  for (int q = 0; q < nblk; ++q) {
    const int buf = q & 1, nb = buf ^ 1;
    const int bk = transpose ? nblk - 1 - q : q;
    const int r0 = bk * 32, r1 = min(n, r0 + 32);
    if (wid == 0) {
      const int r = r0 + lane;
      T vr = (r < r1) ? v[r] : T(0);
      if (q > 0) {
        if (!transpose) {  // previous block [r0 - 32, r0)
          T s = part[buf][0][lane];
#pragma unroll 8
          for (int c = 0; c < 32; ++c) s += Lt[buf][lane][c] * v[r0 - 32 + c];
          vr -= s;
        } else {  // previous block [r1, min(n, r1 + 32))
          T s = T(0);
#pragma unroll 8
          for (int k = 1; k < 32; ++k) s += part[buf][k][lane];
          const int cnt = min(32, n - r1);
          for (int c = 0; c < cnt; ++c) s += Lt[buf][c][lane] * v[r1 + c];
          vr -= s;
        }
      }
      const T rdl = T(1) / Lb[buf][lane][lane];
      if (!transpose) {
        for (int c = 0; c < r1 - r0; ++c) {
          const T xc = __shfl_sync(0xffffffffu, vr * rdl, c);
          if (lane == c) vr = xc;
          else if (lane > c) vr -= Lb[buf][lane][c] * xc;
        }
      } else {
        for (int c = r1 - r0 - 1; c >= 0; --c) {
          const T xc = __shfl_sync(0xffffffffu, vr * rdl, c);
          if (lane == c) vr = xc;
          else if (lane < c) vr -= Lb[buf][c][lane] * xc;
        }
      }
      if (r < r1) v[r] = vr;
    } else {
      const int bn = transpose ? bk - 1 : bk + 1;  // next block
      if (bn >= 0 && bn < nblk) {
        const int r0n = bn * 32;
        for (int j = wid - 1; j < 32; j += 31)
          Lb[nb][j][lane] = store[((long long)d.dblk + bn) * kNB * kNB + j * kNB + lane];
        if (!transpose) {
          // rows r0n + j: prefix over the columns [0, r0) and the tile against [r0, r1)
          for (int j = wid - 1; j < 32; j += 31) {
            const int rn = r0n + j;
            T s = T(0), tv = T(0);
            if (rn < n) {
              const T *Lr = L + (long long)rn * d.ld;
              tv = Lr[r0 + lane];  // r1 - r0 = 32 here: block k is not the last one
              const VT *Lv = reinterpret_cast<const VT *>(Lr);
              const VT *vv = reinterpret_cast<const VT *>(v);
              const int nv = r0 / VN;
              // columns left of rn - band hold zeros (banded factor): start at the band
              const int i0 = d.band >= n ? 0 : max(0, rn - d.band) / VN;
              T a0 = T(0), a1 = T(0), a2 = T(0), a3 = T(0);
              int i = i0 + lane;
              for (; i + 96 < nv; i += 128) {
                const VT l0 = Lv[i], l1 = Lv[i + 32], l2 = Lv[i + 64], l3 = Lv[i + 96];
                a0 += Vec16<T>::dot(l0, vv[i]);
                a1 += Vec16<T>::dot(l1, vv[i + 32]);
                a2 += Vec16<T>::dot(l2, vv[i + 64]);
                a3 += Vec16<T>::dot(l3, vv[i + 96]);
              }
              for (; i < nv; i += 32) a0 += Vec16<T>::dot(Lv[i], vv[i]);
              s = warp_sum((a0 + a1) + (a2 + a3));
            }
            Lt[nb][j][lane] = tv;
            if (lane == 0) part[nb][0][j] = s;
          }
        } else {
          // columns r0n + j (the next block): sums over the rows [r1, n), tile against the rows [r0, r1)
          const int cq = lane % VPR, rq = lane / VPR;
          T acc[VN];
#pragma unroll
          for (int u = 0; u < VN; ++u) acc[u] = T(0);
          const T *Lc = L + r0n + VN * cq;
          constexpr int kStep = 31 * RPW;
          // rows past the band of the block's last column hold zeros there (banded factor)
          const int cend = d.band >= n ? n : min(n, r0n + 32 + d.band);
          int c = r1 + RPW * (wid - 1) + rq;
          for (; c + 3 * kStep < cend; c += 4 * kStep) {
            const VT l0 = *reinterpret_cast<const VT *>(Lc + (long long)c * d.ld);
            const VT l1 = *reinterpret_cast<const VT *>(Lc + (long long)(c + kStep) * d.ld);
            const VT l2 = *reinterpret_cast<const VT *>(Lc + (long long)(c + 2 * kStep) * d.ld);
            const VT l3 = *reinterpret_cast<const VT *>(Lc + (long long)(c + 3 * kStep) * d.ld);
            Vec16<T>::axpy(acc, l0, v[c]);
            Vec16<T>::axpy(acc, l1, v[c + kStep]);
            Vec16<T>::axpy(acc, l2, v[c + 2 * kStep]);
            Vec16<T>::axpy(acc, l3, v[c + 3 * kStep]);
          }
          for (; c < cend; c += kStep)
            Vec16<T>::axpy(acc, *reinterpret_cast<const VT *>(Lc + (long long)c * d.ld), v[c]);
#pragma unroll
          for (int u = 0; u < VN; ++u)
#pragma unroll
            for (int o = VPR; o < 32; o <<= 1) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], o);
          if (rq == 0)
#pragma unroll
            for (int u = 0; u < VN; ++u) part[nb][wid][VN * cq + u] = acc[u];
          for (int j = wid - 1; j < 32; j += 31)
            Lt[nb][j][lane] = (r0 + j < r1) ? L[(long long)(r0 + j) * d.ld + r0n + lane] : T(0);
        }
      }
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < n; i += blockDim.x) y[off + i] = (double)v[i];
}

template <typename T>
void launch_trsv(int count, int max_n, const MatDesc *d_desc, const int *vec_off, const T *base, const T *store,
                 const double *b, double *y, bool transpose, cudaStream_t s) {
  if (count == 0) return;
  const size_t sm = sizeof(T) * (6 * 32 * 33 + (size_t)std::max(4, max_n + 4));
  k_trsv<T><<<count, 1024, sm, s>>>(d_desc, vec_off, base, store, b, y, transpose ? 1 : 0);
  count_launch();
}

// Large local problems stage vectors of up to ~25k entries in shared memory.
size_t dense_smem_limit() { return 200 * 1024; }
bool dense_configure() {
  const int lim = (int)dense_smem_limit();
  bool ok = true;
  ok &= cudaFuncSetAttribute(k_panel_rows<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)panel_smem<128>()) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_panel_rows<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)panel_smem<32>()) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_trsv<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_trsv<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_gemv<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_gemv<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_gemv_t<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_gemv_t<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_symv_rows<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_symv_batched, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_symv_fix, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_symv_rows<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_gemv_task<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_gemv_task<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_gemv_t_task<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) == cudaSuccess;
  ok &= cudaFuncSetAttribute(k_gemv_t_task<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) == cudaSuccess;
  return ok;
}

#define BD_INST(T)                                                                                              \
  template void engine_partial_cholesky<T>(const EngineShape &, const MatDesc *, T *, int *, cudaStream_t,    \
                                           T *, ProfHook *, int, const SliceWs &, const LookAhead *);                                              \
  template void launch_gemv<T>(int, int, int, const GemvDesc *, const T *, const double *, const int *,        \
                               double *, double, const int *, cudaStream_t, const MatDesc *);                  \
  template void launch_symv_rows<T>(int, const T *, int, const double *, double *, int, const int *,           \
                                    cudaStream_t);                                                             \
  template size_t symv_smem<T>(int);                                                                           \
  template int symv_occupancy<T>(int);                                                                         \
  template void launch_gemv_task<T>(int, int, int, const GemvDesc *, const T *, const double *, const int *,   \
                                    double *, double, const int *, cudaStream_t);                              \
  template void launch_gemv_t_task<T>(int, int, int, const GemvDesc *, const T *, const double *, const int *, \
                                      double *, double, const int *, cudaStream_t, const CsrIn *);             \
  template void launch_gemv_t<T>(int, int, int, const GemvDesc *, const T *, const double *, const int *,      \
                                 double *, double, const int *, cudaStream_t, const CsrIn *, const MatDesc *);                  \
  template void launch_trsv<T>(int, int, const MatDesc *, const int *, const T *, const T *, const double *,   \
                               double *, bool, cudaStream_t);
BD_INST(float)
BD_INST(double)

}  // namespace bd
