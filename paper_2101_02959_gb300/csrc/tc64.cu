// FP64 rank-k updates of the partial Cholesky on the tensor cores.
//
// GB300 runs FP64 arithmetic at 2 fused multiply-adds per SM and clock, so the long products
// C[r][c] -= sum_k A[r][k] A[c][k] of the factorisation are formed from exact integer products
// instead (the splitting of Ozaki, Ogita, Oishi and Rump, Numerical Algorithms 59, 2012, with
// fixed-point digits).  Over a group of 128 columns k every row is scaled by a power of two and
// rounded once to a 55-bit integer X = sum_{s=1..7} d_s 256^{7-s}, digits d_s in [-128, 128],
// which bfloat16 holds exactly.  A product of two rows is sum_w 256^{14-w} P_w with
// P_w = sum_{s+t=w} sum_k d_s e_t; each P_w is an integer below 7 * 128 * 2^14 < 2^24, so the
// FP32 accumulators of tcgen05.mma hold it exactly.  The terms w = 2 .. 9 are formed (34 of the 49
// digit products); what is left out is below 2^-57 of the largest product, and the operands'
// rounding below 2^-56 of the row's largest entry.  The P_w are combined as 64-bit integers,
// rounded once to FP64, scaled back and added in FP64, so a group of 128 columns costs one FP64
// rounding per entry where the SIMT loop has 128.
//
// Two kernels: k_slice64 writes the digit planes of the rows an update reads, in the order the
// MMA kernel's shared-memory operands have, so that every operand tile is one contiguous bulk copy;
// k_update64 multiplies them.  The workspace is bounded: batches that need more are
// processed in runs of matrices, and K in runs of kSliceK columns.
//
// Measured (one Jacobian's factorisations, FP64): 64 subdomains of H/h = 12 592 ms with the SIMT
// updates and panels, 69 ms here; 32 subdomains of H/h = 8 34 ms and 7.0 ms.  The rounding error of
// the formed Schur complements (S times the constant vector, which it annihilates, relative to S)
// is 1.83e-16 and 1.72e-16 at H/h = 12, 1.46e-16 and 1.40e-16 at H/h = 8.
#include <algorithm>

#include "kernels.cuh"
#include "tc_ptx.cuh"

namespace bd {

namespace {

constexpr int kDig = 7;            // digit planes per operand
constexpr int kWts = 8;            // weights w = 2 .. 9, one accumulator each
constexpr int kUM = 128, kUN = 64; // output tile
constexpr int kUK = 32;            // K elements per pipeline stage (one 64-byte row of bf16)
constexpr int kGrp = 128;          // K elements per scaling group
constexpr int kBlkBytes = 64 * kUK * 2;  // one digit plane of 64 rows x 32 columns
constexpr int kABytes = kDig * 2 * kBlkBytes, kBBytes = kDig * kBlkBytes;
constexpr int kStageBytes = kABytes + kBBytes;
constexpr int kStages = 2;
constexpr int kU64Smem = kStages * kStageBytes + 1024;
constexpr int kUThreads = 320;     // warps 0-7 drain the accumulators, 8 loads, 9 issues the MMAs
constexpr int kExNan = 1 << 20;    // exponent mark of a row that holds an infinity or a NaN
constexpr int kExMin = 60 - 1022;  // smallest row exponent (keeps the scale factor finite)

// Rows, columns and K range of an update.
struct Range {
  int row0, colend, kb, ke, w;
};
// mode 0: an outer block by its finished panel [K0, K0 + pw): rows [K0 + w, m), columns up to K1;
// mode 1: rows and columns [e, m), K = [K0, min(K1, e)); mode 2: rows [K1, m), columns [K1, e),
// K = [ka, kz) inside the outer block [K0, K1); mode 3: the panel solve, rows [K0 + w, m),
// K = [K0, K0 + w), columns of the panel (B from the inverse of its diagonal block).
__device__ inline bool upd_range(const MatDesc &d, const Upd64 &u, Range &r) {
  if (u.mode == 1) {
    r.row0 = d.e; r.colend = d.m; r.kb = u.ka; r.ke = min(u.kz, d.e); r.w = 0;
    return r.kb < r.ke;
  }
  if (u.mode == 2) {
    r.row0 = u.K1; r.colend = d.e; r.kb = u.ka; r.ke = min(u.kz, u.K1); r.w = 0;
    return u.K1 < d.e && r.kb < r.ke;
  }
  if (u.K0 >= d.e) return false;
  r.w = min(u.pw, d.e - u.K0);
  r.row0 = u.K0 + r.w; r.kb = u.K0; r.ke = u.K0 + r.w;
  r.colend = u.mode == 0 ? min(u.K1, d.e) : r.w;
  return true;
}

// Columns of the update as a count of leading virtual rows (row(v) = column of the update).
__device__ inline int virt_cols(const MatDesc &d, const Upd64 &u, const Range &r, const BandRows &br) {
  if (u.mode == 3) return r.w;
  if (u.mode == 1) return br.nv;
  return max(0, min(r.colend, band_limit(d, r.ke)) - r.row0);
}

}  // namespace

// One 16-thread team per row and group of 128 columns, 8 columns a thread: the row's scale from the
// largest magnitude of the group, then the seven digits of every entry.  Bound by the FP64 pipe (one
// multiply and one conversion per entry) and by its writes; small beside the products.
__global__ void __launch_bounds__(256) k_slice64(const MatDesc *__restrict__ desc, const double *__restrict__ base,
                                                 Upd64 u, const double *__restrict__ pinv, unsigned char *__restrict__ sl,
                                                 int *__restrict__ ex, int nrb, int nkc, int ng) {
  const int b = blockIdx.z, g = blockIdx.y;
  const MatDesc d = desc[b];
  Range r;
  if (!upd_range(d, u, r)) return;
  const int k0 = r.kb + g * kGrp;
  if (k0 >= r.ke) return;
  const int t = threadIdx.x & 15, v = blockIdx.x * 16 + (threadIdx.x >> 4);
  const double *src;
  bool valid;
  int kend = r.ke;
  if (pinv) {  // rows of the panel's block inverse, K relative to the panel
    if (blockIdx.x * 16 >= ((r.w + 63) & ~63)) return;
    valid = v < r.w;
    src = pinv + ((long long)b * u.pw + (valid ? v : 0)) * u.pw - r.kb;
  } else {
    const BandRows br = band_rows(d, r.row0, r.ke);
    if (blockIdx.x * 16 >= ((br.nv + kUM - 1) / kUM) * kUM) return;
    valid = v < br.nv;
    src = base + d.off + (long long)(valid ? br.row(v) : 0) * d.ld;
  }
  const int k = k0 + 8 * t;
  double x[8];
  if (valid && k + 8 <= kend) {
#pragma unroll
    for (int q = 0; q < 8; q += 2) {
      const double2 p = *reinterpret_cast<const double2 *>(src + k + q);  // k even, rows 16-byte aligned
      x[q] = p.x;
      x[q + 1] = p.y;
    }
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = (valid && k + q < kend) ? src[k + q] : 0.0;
  }
  int mag = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) mag = max(mag, __double2hiint(x[q]) & 0x7fffffff);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) mag = max(mag, __shfl_xor_sync(0xffffffffu, mag, o));
  const bool bad = mag >= 0x7ff00000;
  const int e = max((mag >> 20) - 1022, kExMin);  // every |x| < 2^e
  if (t == 0) ex[((long long)b * ng + g) * (nrb * 64) + v] = bad ? kExNan : e;
  const int kc = g * (kGrp / kUK) + (t >> 2);
  if (k0 + (t >> 2) * kUK >= kend) return;
  const double scale = __hiloint2double((1023 + 55 - e) << 20, 0);
  uint32_t pk[kDig][4];
#pragma unroll
  for (int q = 0; q < 8; q += 2) {
    long long X = bad ? 0 : __double2ll_rn(x[q] * scale), Y = bad ? 0 : __double2ll_rn(x[q + 1] * scale);
#pragma unroll
    for (int s = kDig - 1; s >= 0; --s) {
      const int dx = s ? (int)(signed char)(X & 255) : (int)X, dy = s ? (int)(signed char)(Y & 255) : (int)Y;
      X = (X - dx) >> 8;
      Y = (Y - dy) >> 8;
      pk[s][q >> 1] = __byte_perm(__float_as_uint((float)dx), __float_as_uint((float)dy), 0x7632);
    }
  }
  unsigned char *dst = sl + ((((long long)b * nkc + kc) * kDig) * nrb + (v >> 6)) * kBlkBytes + (v & 63) * 64 +
                       (((t & 3) ^ ((v >> 1) & 3)) * 16);
#pragma unroll
  for (int s = 0; s < kDig; ++s)
    *reinterpret_cast<uint4 *>(dst + (long long)s * nrb * kBlkBytes) = make_uint4(pk[s][0], pk[s][1], pk[s][2], pk[s][3]);
}

// One 128 x 64 tile per CTA.  Warp 8 streams the digit planes (two stages of 32 columns), warp 9
// issues the 34 x 2 MMAs of a stage into the eight accumulators (8 x 64 tensor-memory columns), and
// after each group of 128 columns warps 0-7 combine them (warp q: lanes 32 (q & 3) .., columns
// 32 (q >> 2) ..) while the MMAs of the next group already refill the accumulators that
// were read first.  N = 64 and not 128 because eight accumulators of 128 columns exceed tensor memory;
// the MMAs are then bound by reading A from shared memory (48 of their 32 tensor clocks).
__global__ void __launch_bounds__(kUThreads, 1) k_update64(const MatDesc *__restrict__ desc, double *__restrict__ base,
                                                           Upd64 u, const unsigned char *__restrict__ sl,
                                                           const int *__restrict__ ex, int nrb, int nkc, int ng,
                                                           const unsigned char *__restrict__ slb,
                                                           const int *__restrict__ exb, int nct, int *__restrict__ err) {
  const int b = blockIdx.y;
  const MatDesc d = desc[b];
  Range r;
  if (!upd_range(d, u, r)) return;
  const BandRows br = band_rows(d, r.row0, r.ke);
  const int ncv = virt_cols(d, u, r, br);
  const int ti = blockIdx.x / nct, tj = blockIdx.x % nct;
  const int v0 = ti * kUM, c0 = tj * kUN;
  if (v0 >= br.nv || c0 >= ncv || (u.mode != 3 && c0 > v0 + kUM - 1)) return;
  // first column of K that a row of the tile reaches (rows of each kind start in order)
  int ks = r.kb;
  if (v0 >= br.ni) {
    const int idb = d.id0 < d.m ? d.id0 : d.m;
    const int first = br.row(v0);
    if (first < idb) {
      if (d.ifirst && r.row0 <= d.e) {
        ks = max(ks, d.ifirst[first - d.e]);
        if (v0 + kUM > br.ni + br.nmid && br.nv > br.ni + br.nmid) ks = r.kb;
      }
    } else {
      ks = max(ks, first - idb);
    }
  }
  if (ks >= r.ke) return;
  const int ch0 = (ks - r.kb) / kUK, ch1 = (r.ke - r.kb + kUK - 1) / kUK;
  const int g0 = ch0 / (kGrp / kUK), g1 = (ch1 + kGrp / kUK - 1) / (kGrp / kUK);

  extern __shared__ unsigned char smem_raw[];
  __shared__ uint64_t bars[2 * kStages + 1 + kWts];
  __shared__ uint32_t tmem_slot;
  __shared__ int failed;
  __shared__ int ecol[2][kUN];
  const uint32_t raw0 = tcp::smem_addr(smem_raw);
  const uint32_t tiles = (raw0 + 1023u) & ~1023u;
  unsigned char *tp = smem_raw + (tiles - raw0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t bfull = tcp::smem_addr(&bars[0]), bempty = tcp::smem_addr(&bars[kStages]),
                 bacc = tcp::smem_addr(&bars[2 * kStages]), bfree = tcp::smem_addr(&bars[2 * kStages + 1]);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     tcp::smem_addr(&tmem_slot)),
                 "r"((uint32_t)(kWts * kUN)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      tcp::mbar_init(bfull + 8 * s, 1);
      tcp::mbar_init(bempty + 8 * s, 1);
    }
    tcp::mbar_init(bacc, 1);
    for (int w = 0; w < kWts; ++w) tcp::mbar_init(bfree + 8 * w, 8);
    asm volatile("fence.mbarrier_init.release.cluster;");
    failed = 0;
  }
  tcp::fence_before();
  __syncthreads();
  tcp::fence_after();
  const uint32_t tmem = tmem_slot;
  double acc[32];
#pragma unroll
  for (int q = 0; q < 32; ++q) acc[q] = 0.0;

  if (warp == 8) {
    if (lane == 0) {
      bool ok = true;
      const int rbA = v0 >> 6, rbB = c0 >> 6;
      const int nrbB = u.mode == 3 ? (u.pw + 63) / 64 : nrb;
      int n = 0;
      for (int c = ch0; c < ch1; ++c, ++n) {
        const int s = n % kStages;
        if (n >= kStages && !tcp::mbar_wait(bempty + 8 * s, ((n / kStages) - 1) & 1)) { ok = false; break; }
        const uint32_t bar = bfull + 8 * s, dst = tiles + s * kStageBytes;
        tcp::mbar_expect(bar, kStageBytes);
        const unsigned char *pa = sl + (((long long)b * nkc + c) * kDig * nrb + rbA) * kBlkBytes;
        const unsigned char *pb = u.mode == 3
                                      ? slb + (((long long)b * (u.pw / kUK) + c) * kDig * nrbB + rbB) * kBlkBytes
                                      : sl + (((long long)b * nkc + c) * kDig * nrb + rbB) * kBlkBytes;
#pragma unroll
        for (int q = 0; q < kDig; ++q) {
          tcp::bulk_load(dst + q * 2 * kBlkBytes, pa + (long long)q * nrb * kBlkBytes, 2 * kBlkBytes, bar);
          tcp::bulk_load(dst + kABytes + q * kBlkBytes, pb + (long long)q * nrbB * kBlkBytes, kBlkBytes, bar);
        }
      }
      // the copies in flight must land before the CTA releases its shared memory
      for (int m = max(0, n - kStages); m < n; ++m) ok &= tcp::mbar_wait(bfull + 8 * (m % kStages), (m / kStages) & 1);
      if (!ok) failed = 1;
    }
  } else if (warp == 9) {
    if (lane == 0) {
      bool ok = true;
      const uint32_t idesc = tcp::idesc_bf16(kUM, kUN);
      int n = 0;
      for (int g = g0; g < g1 && ok; ++g) {
        const int ca = max(ch0, g * (kGrp / kUK)), cz = min(ch1, (g + 1) * (kGrp / kUK));
        for (int c = ca; c < cz && ok; ++c, ++n) {
          const int s = n % kStages;
          if (!tcp::mbar_wait(bfull + 8 * s, (n / kStages) & 1)) { ok = false; break; }
          tcp::fence_after();
          const uint32_t A = tiles + s * kStageBytes, B = A + kABytes;
#pragma unroll
          for (int w = 0; w < kWts; ++w) {
            if (c == ca && g > g0) {  // the accumulator's last group must have been read
              if (!tcp::mbar_wait(bfree + 8 * w, (g - g0 - 1) & 1)) { ok = false; break; }
              tcp::fence_after();
            }
#pragma unroll
            for (int i = 0; i < kDig; ++i) {
              const int j = w - i;  // digit indices from 0: weight w + 2
              if (j < 0 || j >= kDig) continue;
              const bool fresh = c == ca && i == (w < kDig ? 0 : w - kDig + 1);
#pragma unroll
              for (int t = 0; t < kUK / 16; ++t)
                tcp::mma_f16(tmem + w * kUN, tcp::sw64_desc(A + i * 2 * kBlkBytes + 32 * t),
                             tcp::sw64_desc(B + j * kBlkBytes + 32 * t), idesc, fresh && t == 0 ? 0u : 1u);
            }
          }
          tcp::mma_commit(bempty + 8 * s);
        }
        tcp::mma_commit(bacc);
      }
      if (!ok) failed = 1;
    }
  } else {
    const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * 32);
    const int v = v0 + (warp & 3) * 32 + lane, cq = (warp >> 2) * 32;
    bool ok = true;
    for (int g = g0; g < g1; ++g) {
      const int par = (g - g0) & 1;
      if (warp < 2) {  // the columns' exponents of this group
        const int c = c0 + tid;
        ecol[par][tid] = u.mode == 3 ? exb[((long long)b * ((u.pw + kGrp - 1) / kGrp) + g) * (((u.pw + 63) / 64) * 64) + c]
                                     : ex[((long long)b * ng + g) * (nrb * 64) + c];
      }
      const int er = ex[((long long)b * ng + g) * (nrb * 64) + v];
      ok = ok && tcp::mbar_wait(bacc, par);  // after a missed wait the loop only keeps the barriers in step
      asm volatile("bar.sync 1, 256;" ::: "memory");
      tcp::fence_after();
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {  // 16 columns at a time (registers)
        long long I[16];
        uint32_t t[16];
        int x8[16];
#pragma unroll
        for (int w = 0; w < kWts; ++w) {
          tcp::tmem_ld16(taddr + w * kUN + 16 * hf, t);
          tcp::tmem_wait_ld();
          if (hf == 1) {
            tcp::fence_before();
            __syncwarp();
            if (lane == 0) tcp::mbar_arrive(bfree + 8 * w);
          }
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const int x = __float2int_rn(__uint_as_float(t[q]));
            if (w == 0) I[q] = x;
            else if (w < 6) I[q] = (I[q] << 8) + x;
            else if (w == 6) x8[q] = x;
            else I[q] += (x8[q] + ((x + 128) >> 8) + 128) >> 8;  // weights 8 and 9, rounded
          }
        }
        // unit of I: 2^(er + ec - 110) 256^7 = 2^(er + ec - 54)
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          const int ec = ecol[par][cq + 16 * hf + q];
          const int s = er + ec - 54;
          const double sc = (er == kExNan || ec == kExNan)
                                ? __hiloint2double(0x7ff80000, 0)
                                : __hiloint2double(max(min(s, 1023) + 1023, 0) << 20, 0);
          acc[16 * hf + q] = fma(__ll2double_rn(I[q]), sc, acc[16 * hf + q]);
        }
      }
    }
    if (!ok) failed = 1;
  }
  __syncwarp();
  tcp::fence_before();
  __syncthreads();
  tcp::fence_after();
  if (failed) {
    if (tid == 0) atomicOr(err, DEV_ERR_TIMEOUT);
  } else {
    // accumulators through shared memory (the operand stages are done), then C row by row
    double *stage = reinterpret_cast<double *>(tp);  // [128][65]
    if (warp < 8) {
      const int row = (warp & 3) * 32 + lane, cq = (warp >> 2) * 32;
#pragma unroll
      for (int q = 0; q < 32; ++q) stage[row * (kUN + 1) + cq + q] = acc[q];
    }
    __syncthreads();
    double *C = base + d.off;
    const int vc0 = c0 + lane, vc1 = c0 + 32 + lane;
    const int col0 = u.mode == 3 ? u.K0 + vc0 : (vc0 < ncv ? br.row(vc0) : 0);
    const int col1 = u.mode == 3 ? u.K0 + vc1 : (vc1 < ncv ? br.row(vc1) : 0);
    for (int row = warp; row < kUM; row += kUThreads / 32) {
      const int v = v0 + row;
      if (v >= br.nv) break;
      double *crow = C + (long long)br.row(v) * d.ld;
      const double a0 = stage[row * (kUN + 1) + lane], a1 = stage[row * (kUN + 1) + 32 + lane];
      if (u.mode == 3) {
        if (vc0 < ncv) crow[col0] = a0;
        if (vc1 < ncv) crow[col1] = a1;
      } else {
        if (vc0 < ncv && vc0 <= v) crow[col0] -= a0;
        if (vc1 < ncv && vc1 <= v) crow[col1] -= a1;
      }
    }
  }
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)(kWts * kUN)));
}

// ---- factored diagonal block of a panel and its inverse ---------------------------
// One CTA per matrix: the w x w block (w <= 64) at K0 in two 32-column halves.  Writes L_11 in
// place, its 32 x 32 diagonal blocks to the block store and the inverse Y = L_11^-1 to pinv, so
// the rows below become one product on the tensor cores.
//
// A warp issues one FP64 instruction in 64 clocks (measured, dependent or not) and the SM four of
// them at a time, so the work is spread over the four schedulers: in ldl_inv32 warps 0-3 hold
// every fourth column of the block and of its inverse (lane = row) and eliminate one column a step,
// root-free: the step's chain is one reciprocal, one scaling, one update (about 560 clocks), and the
// other updates fit beside it; the square roots of the 32 pivots are taken together at the end.
// Between the halves 32 x 32 x 32 products over all warps (L_21 = A_21 Y_11^T,
// A_22 -= L_21 L_21^T, Y_21 = -Y_22 (L_21 Y_11)), column groups paired so that the schedulers get
// equal triangles.  Panels of 64 columns and not 128: the count of FP64 instructions grows with the
// cube of the width.
constexpr int kDP = kPanel64, kDLD = kDP + 1;
constexpr size_t kDiagSmem = sizeof(double) * (2 * (size_t)kDP * kDLD + 32 * 33);

// Lower Cholesky factor of the 32 x 32 block of P at (o, o) and its inverse into Y; warps 0-3.
// Columns at and after the block's width hold the identity.
__device__ __forceinline__ void ldl_inv32(double *P, double *Y, int o, int s, int lane, double (*Lc)[2][32],
                                          double *piv, bool &bad) {
  double a[8], y[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int t = 4 * q + s;
    a[q] = t <= lane ? P[(o + lane) * kDLD + o + t] : 0.0;
    y[q] = t == lane ? 1.0 : 0.0;
  }
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    const int q0 = c >> 2, buf = c & 1;
    if (s == (c & 3)) {
      double p = __shfl_sync(0xffffffffu, a[q0], c);
      if (!(p > 0.0)) { bad = true; p = 1.0; }
      const double inv = 1.0 / p;
      Lc[buf][0][lane] = a[q0];                           // the column before scaling
      Lc[buf][1][lane] = lane > c ? a[q0] * inv : 0.0;   // unit-lower column
      if (lane == c) piv[c] = p;
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");
    const double l = Lc[buf][1][lane];
#pragma unroll
    for (int d = 0; d < 4; ++d) {  // the next column's owner updates it first
      const int q = q0 + (d == 3 ? 1 : 0);
      if (d == 0 || d == 3) {
        if (q < 8 && 4 * q + s > c) a[q] -= l * Lc[buf][0][4 * q + s];
      }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (q > q0 + 1 && 4 * q + s > c) a[q] -= l * Lc[buf][0][4 * q + s];
      if (q <= q0 && 4 * q + s <= c) {
        const double yc = __shfl_sync(0xffffffffu, y[q], c);
        y[q] -= l * yc;
      }
    }
  }
  asm volatile("bar.sync 1, 128;" ::: "memory");
  const double pl = piv[lane], rs = rsqrt(pl);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int t = 4 * q + s;
    const double rt = __shfl_sync(0xffffffffu, rs, t);
    P[(o + lane) * kDLD + o + t] = lane < t ? 0.0 : (lane == t ? pl * rs : a[q] * rt);
    Y[(o + lane) * kDLD + o + t] = t <= lane ? y[q] * rs : 0.0;
  }
}

__global__ void __launch_bounds__(256) k_diag64(const MatDesc *__restrict__ desc, double *__restrict__ base, int K0,
                                                int *__restrict__ err, double *__restrict__ store,
                                                double *__restrict__ pinv) {
  const MatDesc d = desc[blockIdx.x];
  if (K0 >= d.e) return;
  const int w = min(kDP, d.e - K0);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double *P = reinterpret_cast<double *>(smem_raw);  // [64][65] the block, lower, identity past w
  double *Y = P + kDP * kDLD;                        // [64][65] its inverse
  double *T = Y + kDP * kDLD;                        // [32][33]
  __shared__ double Lc[2][2][32], piv[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double *A = base + d.off + (long long)K0 * d.ld + K0;
  {
    const int i = tid >> 2, j0 = (tid & 3) * 16;
    double v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = (i < w && j0 + q <= i) ? A[(long long)i * d.ld + j0 + q] : (i == j0 + q ? 1.0 : 0.0);
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      P[i * kDLD + j0 + q] = v[q];
      Y[i * kDLD + j0 + q] = 0.0;
    }
  }
  bool bad = false;
  const int nbk = ceil_div(w, 32);
  const int grp = 4 * (warp < 4 ? warp : 11 - warp);  // this warp's four columns (rows) of a triangle
  for (int h = 0; h < nbk; ++h) {
    const int o = 32 * h;
    __syncthreads();
    if (warp < 4) ldl_inv32(P, Y, o, warp, lane, Lc, piv, bad);
    __syncthreads();
    double *sb = store + ((long long)d.dblk + K0 / kNB + h) * kNB * kNB;
    for (int q = tid; q < 1024; q += 256) sb[q] = P[(o + (q >> 5)) * kDLD + o + (q & 31)];
    if (h == 0 && nbk > 1) {
      double x[4] = {0.0, 0.0, 0.0, 0.0};  // L_21 = A_21 Y_11^T (Y_11 lower: k <= column)
#pragma unroll 4
      for (int k = 0; k < grp + 4; ++k) {
        const double l = P[(32 + lane) * kDLD + k];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] += l * Y[(grp + u) * kDLD + k];
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 4; ++u) P[(32 + lane) * kDLD + grp + u] = x[u];
      __syncthreads();
      // A_22 -= L_21 L_21^T, the ten 8 x 8 blocks of its lower part
      for (int q = warp; q < 10; q += 8) {
        const int bi = q < 1 ? 0 : q < 3 ? 1 : q < 6 ? 2 : 3, bj = q - bi * (bi + 1) / 2;
        const int r = 32 + 8 * bi + (lane >> 2), c = 32 + 8 * bj + (lane & 3) * 2;
        double x0 = 0.0, x1 = 0.0;
#pragma unroll 8
        for (int k = 0; k < 32; ++k) {
          const double l = P[r * kDLD + k];
          x0 += l * P[c * kDLD + k];
          x1 += l * P[(c + 1) * kDLD + k];
        }
        if (r < w && c <= r) P[r * kDLD + c] -= x0;
        if (r < w && c + 1 <= r) P[r * kDLD + c + 1] -= x1;
      }
    }
  }
  if (nbk > 1) {  // Y_21 = -Y_22 (L_21 Y_11)
    double x[4] = {0.0, 0.0, 0.0, 0.0};
    const int g2 = 28 - grp;  // columns g2 .. g2 + 3: k >= column
#pragma unroll 4
    for (int k = g2; k < 32; ++k) {
      const double l = P[(32 + lane) * kDLD + k];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] += l * Y[k * kDLD + g2 + u];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) T[lane * 33 + g2 + u] = x[u];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = 0.0;
#pragma unroll 4
    for (int k = 0; k < grp + 4; ++k) {  // lane = column, rows grp .. grp + 3: k <= row
      const double t = T[k * 33 + lane];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] += Y[(32 + grp + u) * kDLD + 32 + k] * t;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) Y[(32 + grp + u) * kDLD + lane] = -x[u];
  }
  __syncthreads();
  if (bad && lane == 0) atomicOr(err, DEV_ERR_NOT_SPD);
  double *out = pinv + (long long)blockIdx.x * kDP * kDP;
#pragma unroll 4
  for (int q = tid; q < kDP * kDP; q += 256) {
    const int i = q / kDP, j = q % kDP;
    out[q] = (i < w && j <= i) ? Y[i * kDLD + j] : 0.0;
    if (i < w && j <= i) A[(long long)i * d.ld + j] = P[i * kDLD + j];
  }
}

void launch_diag64(const MatDesc *d_desc, double *base, int K0, int count, int *err, double *store, double *pinv,
                   cudaStream_t s) {
  k_diag64<<<count, 256, kDiagSmem, s>>>(d_desc, base, K0, err, store, pinv);
  count_launch();
}

bool tc64_configure() {
  return cudaFuncSetAttribute(k_update64, cudaFuncAttributeMaxDynamicSharedMemorySize, kU64Smem) == cudaSuccess &&
         cudaFuncSetAttribute(k_diag64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDiagSmem) == cudaSuccess;
}

// Workspace of the digit planes of one matrix (rows x cols) and of a panel inverse.
static size_t planes_bytes(int rows, int cols) {
  return (size_t)ceil_div(cols, kUK) * kDig * 2 * ceil_div(rows, kUM) * kBlkBytes;
}
static size_t rows_bytes(int rows, int cols) {
  return planes_bytes(rows, cols) + (size_t)ceil_div(cols, kGrp) * 2 * ceil_div(rows, kUM) * 64 * sizeof(int);
}
static size_t inv_bytes() { return planes_bytes(1, kPanel64) / 2 + 64 * sizeof(int); }
static_assert(kPanel64 == 64, "the inverse's digit planes are one block of 64 rows");

size_t slice64_bytes(int count, int max_rows, int max_e) {
  return (size_t)std::max(1, count) * (rows_bytes(std::max(max_rows, 1), std::min(std::max(max_e, 1), kSliceK)) + inv_bytes());
}

// Runs of matrices whose planes fit the workspace; the final update (mode 1) also in runs of
// kSliceK columns (each run rounds C once more, so they are long).
void launch_update64(const MatDesc *d_desc, double *base, Upd64 u, int max_rows, int max_cols, int count,
                     const Slice64 &ws, int *err, cudaStream_t s, const double *pinv) {
  if (max_rows <= 0 || max_cols <= 0 || count <= 0) return;
  const int za = u.mode == 1 || u.mode == 2 ? u.ka : u.K0, zz = u.mode == 1 || u.mode == 2 ? u.kz : u.K0 + u.pw;
  const int kmax = std::min(zz - za, kSliceK), nrb = 2 * ceil_div(max_rows, kUM);
  const int run = (int)std::max<size_t>(1, std::min<size_t>((size_t)count, ws.bytes / (rows_bytes(max_rows, kmax) + inv_bytes())));
  const int nrt = ceil_div(max_rows, kUM), nct = ceil_div(max_cols, kUN);
  unsigned char *sl = ws.mem, *slb = sl + (size_t)run * planes_bytes(max_rows, kmax);
  int *ex = reinterpret_cast<int *>(slb + (size_t)run * (planes_bytes(1, kPanel64) / 2));
  int *exb = ex + (size_t)run * ceil_div(kmax, kGrp) * nrb * 64;
  for (int b0 = 0; b0 < count; b0 += run) {
    const int nb = std::min(run, count - b0);
    for (int ka = za; ka < zz; ka += kSliceK) {
      Upd64 q = u;
      q.ka = ka;
      q.kz = std::min(zz, ka + kSliceK);
      const int kw = q.kz - ka, nkc = ceil_div(kw, kUK), ng = ceil_div(kw, kGrp);
      k_slice64<<<dim3(nrb * 4, ng, nb), 256, 0, s>>>(d_desc + b0, base, q, nullptr, sl, ex, nrb, nkc, ng);
      count_launch();
      if (u.mode == 3) {
        const double *pv = pinv + (size_t)b0 * u.pw * u.pw;
        k_slice64<<<dim3(4, 1, nb), 256, 0, s>>>(d_desc + b0, base, q, pv, slb, exb, 1, kPanel64 / kUK, 1);
        count_launch();
      }
      k_update64<<<dim3(nrt * nct, nb), kUThreads, kU64Smem, s>>>(d_desc + b0, base, q, sl, ex, nrb, nkc, ng, slb, exb,
                                                                 nct, err);
      count_launch();
    }
  }
}

}  // namespace bd
