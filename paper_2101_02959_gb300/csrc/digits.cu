// Rank-k updates of the partial Cholesky on the tensor cores by exact digit products.
//
// GB300 runs FP64 arithmetic at 2 fused multiply-adds per SM and clock, and its tensor cores sum
// FP32 products with truncation, so the long products C[r][c] -= sum_k A[r][k] A[c][k] are formed from
// exact integer products instead (the splitting of Ozaki, Ogita, Oishi and Rump, Numerical
// Algorithms 59, 2012, with fixed-point digits).  Over a group of columns k every row is scaled
// by a power of two and rounded once to an integer X = sum_s d_s B^{D-s} of D digits, which bfloat16
// holds exactly.  A product of two rows is sum_w B^{2D-w} P_w with P_w = sum_{s+t=w} sum_k d_s e_t; each
// P_w is an integer below 2^24, so the FP32 accumulators of tcgen05.mma hold it exactly.
//   FP64: B = 256, D = 7 (55 bits), groups of 128 columns (7 * 128 * 2^14 < 2^24), w = 2 .. 9, 34 of
//   the 49 digit products.  With rows below 2^er and 2^ec over a group: an operand's rounding is at most
//   2^(er - 56) (2^-55 of the row's largest entry), the digit products left out 2^-61 2^(er + ec) a column.
//   The P_w are combined as 64-bit integers in units of weight 7, into which weights 8 and 9 are
//   rounded (2^-55 2^(er + ec) a group), converted to FP64 with one rounding, scaled back and added.
//   FP32: B = 512, D = 3 (26 bits), groups of 64 columns (3 * 64 * 2^16 < 2^24), w = 2 .. 4, 6 of the 9
//   digit products: 2^(er - 27) for an operand, 2^-26 2^(er + ec) a column left out, combined and added
//   in FP32: one rounding per group where a chain of FP32 multiply-adds has one per column and an FP32
//   accumulator of the tensor cores loses the low bits at every step.
// These are bounds below the rows' largest entries.  A Cholesky factor's rows are bounded by their
// diagonals, so there they are those of any backward-stable sum; the products of two different matrices
// scale the columns first (ColScale).  FP64 rows' products below 2^-968 are lost (matrices of entries
// below 1e-290); FP32 keeps its whole range.
//
// Two kernels: k_slice writes the digit planes of the rows an update reads, in the order the
// MMA kernel's shared-memory operands have, so that every operand tile is one contiguous bulk copy;
// k_update multiplies them.  The workspace is bounded: batches that need more are
// processed in runs of matrices, and the final update in runs of kSliceK columns.
//
// Measured (one Jacobian's factorisations, FP64): 64 subdomains of H/h = 12 592 ms with the SIMT
// updates and panels, 69 ms here; 32 subdomains of H/h = 8 34 ms and 7.0 ms.  The rounding error of
// the formed Schur complements (S times the constant vector, which it annihilates, relative to S)
// is 1.83e-16 and 1.72e-16 at H/h = 12, 1.46e-16 and 1.40e-16 at H/h = 8.  FP32, 1,024 subdomains of
// H/h = 8: 19.6 ms of updates per Jacobian against 16.7 with a TF32 hi + lo split that lost the
// accumulators' low bits; a time step solved until the FP64 residual stops falling takes 10 Newton
// iterations instead of 32 (13 with SIMT FP32).
#include <algorithm>
#include <stdexcept>
#include <string>

#include "digit_ws.h"
#include "kernels.cuh"
#include "tc_ptx.cuh"

namespace bd {

namespace {

template <typename T> struct Dig;
template <> struct Dig<double> {
  // digits, weights, K group, tile columns, pipeline stages, columns of an epilogue pass
  static constexpr int D = DigitDims<double>::D, W = 8, Grp = DigitDims<double>::Grp, N = kUpdN, Stages = 2, Epi = 8;
  static constexpr int ExLow = 60 - 1022;  // below it a row is lifted first (keeps the scale factor finite)
};
template <> struct Dig<float> {
  static constexpr int D = DigitDims<float>::D, W = 3, Grp = DigitDims<float>::Grp, N = kUpdN, Stages = 4, Epi = 16;
  static constexpr int ExLow = 30 - 126;
};
constexpr int kUM = kUpdM;         // tile rows
constexpr int kUK = kUpdK;         // K elements per pipeline stage
constexpr int kBlkBytes = kDigitBlk;
template <typename T> constexpr int a_bytes() { return Dig<T>::D * 2 * kBlkBytes; }
template <typename T> constexpr int stage_bytes() { return a_bytes<T>() + Dig<T>::D * (Dig<T>::N / 64) * kBlkBytes; }
// warps 0-15 drain the accumulators and write C, 16 loads, 17 issues the MMAs, 18 lists the tiles
constexpr int kDrain = 16, kUThreads = 32 * (kDrain + 3);
// a drain warp's share of a tile, staged Epi columns at a time
template <typename T> constexpr int epi_bytes() { return 32 * (Dig<T>::Epi + 1) * (int)sizeof(T); }
template <typename T> constexpr int update_smem() {
  return Dig<T>::Stages * stage_bytes<T>() + kDrain * epi_bytes<T>() + 1024;
}
constexpr uint32_t kTmemCols = 512;
constexpr int kSms = kUpdCtas;
constexpr int kExNan = 1 << 20;    // exponent mark of a row that holds an infinity or a NaN

// Rows, columns and K range of an update.
struct Range {
  int row0, colend, kb, ke, w;
};
// mode 0: an outer block by its finished panel [K0, K0 + pw): rows [K0 + w, m), columns up to K1;
// mode 1: rows and columns [e, m), K = [K0, min(K1, e)); mode 2: rows [K1, m), columns [K1, e),
// K = [ka, kz) inside the outer block [K0, K1); mode 3: the panel solve, rows [K0 + w, m),
// K = [K0, K0 + w), columns of the panel (B from the inverse of its diagonal block); mode 4: the plain
// product C = A B^T of n x n matrices (desc.e = desc.m = n).
__device__ inline bool upd_range(const MatDesc &d, const Upd64 &u, Range &r) {
  if (u.mode == 1) {
    r.row0 = d.e; r.colend = d.m; r.kb = u.ka; r.ke = min(u.kz, d.e); r.w = 0;
    return r.kb < r.ke;
  }
  if (u.mode == 2) {
    r.row0 = u.K1; r.colend = d.e; r.kb = u.ka; r.ke = min(u.kz, u.K1); r.w = 0;
    return u.K1 < d.e && r.kb < r.ke;
  }
  if (u.mode == 4) {
    r.row0 = 0; r.colend = d.m; r.kb = u.ka; r.ke = min(u.kz, d.m); r.w = 0;
    return r.kb < r.ke;
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
  if (u.mode == 1 || u.mode == 4) return br.nv;
  return max(0, min(r.colend, band_limit(d, r.ke)) - r.row0);
}

}  // namespace

// The digits of one entry, most significant first (x scaled so that |x| < 2^e becomes |X| <= B^D / 2).
__device__ __forceinline__ void digits(double x, double scale, int (&dg)[7]) {
  long long X = __double2ll_rn(x * scale);
#pragma unroll
  for (int s = 6; s > 0; --s) {
    dg[s] = (int)(signed char)(X & 255);
    X = (X - dg[s]) >> 8;
  }
  dg[0] = (int)X;
}
__device__ __forceinline__ void digits(float x, float scale, int (&dg)[3]) {
  int X = __float2int_rn(x * scale);
#pragma unroll
  for (int s = 2; s > 0; --s) {
    dg[s] = ((X & 511) ^ 256) - 256;  // signed low nine bits
    X = (X - dg[s]) >> 9;
  }
  dg[0] = X;
}
// top word of a value's magnitude and the exponent e with magnitude < 2^e; the factor 2^(bits - e)
__device__ __forceinline__ int mag_bits(double x) { return __double2hiint(x) & 0x7fffffff; }
__device__ __forceinline__ int mag_bits(float x) { return __float_as_int(x) & 0x7fffffff; }
__device__ __forceinline__ int mag_exp(double, int m) { return (m >> 20) - 1022; }
__device__ __forceinline__ int mag_exp(float, int m) { return (m >> 23) - 126; }
__device__ __forceinline__ bool mag_bad(double, int m) { return m >= 0x7ff00000; }
__device__ __forceinline__ bool mag_bad(float, int m) { return m >= 0x7f800000; }
__device__ __forceinline__ double fix_scale(double, int e) { return __hiloint2double((1023 + 55 - e) << 20, 0); }
__device__ __forceinline__ float fix_scale(float, int e) { return __int_as_float((127 + 26 - e) << 23); }

// Scaling of the columns of K in products of two different matrices: C = (A D) (B D^-1)^T with D powers of
// two, so that entries of columns of different size (the two media) keep their bits below the row's
// largest.  Panel solve: D^-1 from the square roots of the block's diagonal before its factorisation, which
// bound the entries of its columns (the pivots do not: where one is small because the block is nearly
// singular, scaling by it takes the bits of all other columns), as k_diag leaves it: kPanelExp ints per
// matrix, the exponents, and 0 behind them where they differ by three or less and nothing is scaled (FP64
// multiplies on every entry cost the H/h = 12 cube 2 of 78 ms).  Plain product: the square roots of B's
// diagonal.
template <typename T>
struct ColScale {
  const int *pexp = nullptr;      // panel solve
  const T *B = nullptr;           // plain product, with B's descriptors
  const MatDesc *desc = nullptr;
  int sign = 1;                   // +1 for A, -1 for B
};
__device__ __forceinline__ double exp2i(double, int e) { return __hiloint2double((e + 1023) << 20, 0); }
__device__ __forceinline__ float exp2i(float, int e) { return __int_as_float((e + 127) << 23); }
template <typename T>
__device__ __forceinline__ T col_factor(const ColScale<T> &c, int b, int k) {
  int e = 0;
  if (c.pexp) {
    e = c.pexp[b * kPanelExp + k];
  } else {
    const T v = c.B[c.desc[b].off + (long long)k * (c.desc[b].ld + 1)];
    const int m = mag_bits(v);
    if (m > 0 && !mag_bad(v, m)) e = (mag_exp(v, m) + 1) >> 1;
  }
  constexpr int most = sizeof(T) == 8 ? 1000 : 120;
  return exp2i(T(0), c.sign * max(-most, min(e, most)));
}

// One team of Grp / 8 threads per row and group of columns, 8 columns a thread: the row's scale from
// the largest magnitude of the group, then the digits of every entry.  The long-K launch of 32 matrices
// of H/h = 8 moves 323 MB in 94 us (3.4 TB/s, most of it planes of 14 bytes per entry; the FP64 pipe is
// 68 % busy with a multiply and a conversion per entry), in FP32 120 MB in 49 us.
template <typename T>
__global__ void __launch_bounds__(256) k_slice(const MatDesc *__restrict__ desc, const T *__restrict__ base,
                                               Upd64 u, const T *__restrict__ pinv, unsigned char *__restrict__ sl,
                                               int *__restrict__ ex, int nrb, int nkc, int ng, ColScale<T> cs) {
  using C = Dig<T>;
  constexpr int TM = C::Grp / 8, RPC = 256 / TM;  // threads of a team, rows per CTA
  const int b = blockIdx.z, g = blockIdx.y;
  const MatDesc d = desc[b];
  Range r;
  if (!upd_range(d, u, r)) return;
  const int k0 = r.kb + g * C::Grp;
  if (k0 >= r.ke) return;
  const int t = threadIdx.x % TM, v = blockIdx.x * RPC + threadIdx.x / TM;
  const T *src;
  bool valid;
  if (pinv) {  // rows of the panel's block inverse, K relative to the panel
    if (blockIdx.x * RPC >= 64 * (C::N / 64)) return;
    valid = v < r.w;
    src = pinv + ((long long)b * u.pw + (valid ? v : 0)) * u.pw - r.kb;
  } else {
    const BandRows br = band_rows(d, r.row0, r.ke);
    if (blockIdx.x * RPC >= ((br.nv + kUM - 1) / kUM) * kUM) return;
    valid = v < br.nv;
    src = base + d.off + (long long)(valid ? br.row(v) : 0) * d.ld;
  }
  const int k = k0 + 8 * t;
  T x[8];
  if (valid && k + 8 <= r.ke && (reinterpret_cast<uintptr_t>(src + k) & 15) == 0) {
    constexpr int VN = 16 / (int)sizeof(T);
#pragma unroll
    for (int q = 0; q < 8; q += VN) *reinterpret_cast<int4 *>(&x[q]) = *reinterpret_cast<const int4 *>(src + k + q);
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = (valid && k + q < r.ke) ? src[k + q] : T(0);
  }
  if (cs.pexp ? cs.pexp[b * kPanelExp + kPanel64] != 0 : cs.B != nullptr) {
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (k + q < r.ke) x[q] *= col_factor(cs, b, k + q - r.kb);
  }
  int mag = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) mag = max(mag, mag_bits(x[q]));
#pragma unroll
  for (int o = TM / 2; o > 0; o >>= 1) mag = max(mag, __shfl_xor_sync(0xffffffffu, mag, o));
  const bool bad = mag_bad(T(0), mag);
  const int e = mag > 0 ? mag_exp(T(0), mag) : 0;  // every |x| < 2^e
  if (t == 0) ex[((long long)b * ng + g) * (nrb * 64) + v] = bad ? kExNan : e;
  const int kc = g * (C::Grp / kUK) + (t >> 2);
  if (k0 + (t >> 2) * kUK >= r.ke) return;
  int up = 0;
  if (e < C::ExLow) {  // a row of very small entries, exact times 2^60
    up = 60;
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] *= T(1ll << 60);
  }
  const T scale = fix_scale(T(0), max(e + up, C::ExLow));
  uint32_t pk[C::D][4];
#pragma unroll
  for (int q = 0; q < 8; q += 2) {
    int dx[C::D], dy[C::D];
    digits(bad ? T(0) : x[q], scale, dx);
    digits(bad ? T(0) : x[q + 1], scale, dy);
#pragma unroll
    for (int s = 0; s < C::D; ++s)  // bf16: the upper halves of the exact FP32 values
      pk[s][q >> 1] = __byte_perm(__float_as_uint((float)dx[s]), __float_as_uint((float)dy[s]), 0x7632);
  }
  unsigned char *dst = sl + ((((long long)b * nkc + kc) * C::D) * nrb + (v >> 6)) * kBlkBytes + (v & 63) * 64 +
                       (((t & 3) ^ ((v >> 1) & 3)) * 16);
#pragma unroll
  for (int s = 0; s < C::D; ++s)
    *reinterpret_cast<uint4 *>(dst + (long long)s * nrb * kBlkBytes) = make_uint4(pk[s][0], pk[s][1], pk[s][2], pk[s][3]);
}

// A tile of an update, as the scheduling warp hands it to the others.
struct Tile {
  long long off;
  int ld, b, v0, c0, ch0, ch1, ncv;  // descriptor, first virtual row and column, K chunks, columns
  BandRows br;
};

// Tile (ti, tj) of matrix b; false when it holds no entry of the update.
__device__ inline bool make_tile(const MatDesc *__restrict__ desc, const MatDesc *__restrict__ out, const Upd64 &u,
                                 int b, int ti, int tj, int n, Tile &t) {
  const MatDesc d = desc[b];
  Range r;
  if (!upd_range(d, u, r)) return false;
  t.v0 = ti * kUM;
  t.c0 = tj * n;
  if (u.mode < 3 && t.c0 > t.v0 + kUM - 1) return false;
  t.br = band_rows(d, r.row0, r.ke);
  t.ncv = virt_cols(d, u, r, t.br);
  if (t.v0 >= t.br.nv || t.c0 >= t.ncv) return false;
  // first column of K that a row of the tile reaches (rows of each kind start in order)
  int ks = r.kb;
  if (t.v0 >= t.br.ni) {
    const int idb = d.id0 < d.m ? d.id0 : d.m;
    const int first = t.br.row(t.v0);
    if (first < idb) {
      if (d.ifirst && r.row0 <= d.e) {
        ks = max(ks, d.ifirst[first - d.e]);
        if (t.v0 + kUM > t.br.ni + t.br.nmid && t.br.nv > t.br.ni + t.br.nmid) ks = r.kb;
      }
    } else {
      ks = max(ks, first - idb);
    }
  }
  if (ks >= r.ke) return false;
  t.off = out[b].off;
  t.ld = out[b].ld;
  t.b = b;
  t.ch0 = (ks - r.kb) / kUK;
  t.ch1 = (r.ke - r.kb + kUK - 1) / kUK;
  return true;
}

// Digit planes and row exponents of one operand: blocks of 64 rows, chunks and groups of columns.
struct Planes {
  const unsigned char *sl;
  const int *ex;
  int nrb, nkc, ng;
};

// Reads one group's accumulators (CPW columns from taddr) and adds sum_w B^(2D-w) P_w 2^(er + ec) to
// acc; the accumulator of weight w is released on bfree + 8 w once read.
__device__ __forceinline__ void drain(uint32_t taddr, uint32_t bfree, int lane, int er, const int *ecol, bool,
                                      double (&acc)[16]) {
  long long I[16];
  // the 64-bit sum in steps of three weights, 256 (256 P_w + P_(w+1)) + P_(w+2)
#pragma unroll
  for (int w = 0; w < 6; w += 3) {
    uint32_t t0[16], t1[16], t2[16];
    tcp::tmem_ld16(taddr + w * 64, t0);
    tcp::tmem_ld16(taddr + (w + 1) * 64, t1);
    tcp::tmem_ld16(taddr + (w + 2) * 64, t2);
    tcp::tmem_wait_ld();
    tcp::fence_before();
    __syncwarp();
    if (lane < 3) tcp::mbar_arrive(bfree + 8 * (w + lane));
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int x0 = __float2int_rn(__uint_as_float(t0[q])), x1 = __float2int_rn(__uint_as_float(t1[q])),
                x2 = __float2int_rn(__uint_as_float(t2[q]));
      const long long h = (long long)x0 * 65536 + ((long long)x1 * 256 + x2);
      I[q] = w == 0 ? h << 24 : I[q] + h;
    }
  }
  {
    uint32_t t0[16], t1[16];
    tcp::tmem_ld16(taddr + 6 * 64, t0);
    tcp::tmem_ld16(taddr + 7 * 64, t1);
    tcp::tmem_wait_ld();
    tcp::fence_before();
    __syncwarp();
    if (lane < 2) tcp::mbar_arrive(bfree + 8 * (6 + lane));
#pragma unroll
    for (int q = 0; q < 16; ++q) {  // weights 8 and 9, rounded
      const int x0 = __float2int_rn(__uint_as_float(t0[q])), x1 = __float2int_rn(__uint_as_float(t1[q]));
      I[q] += (x0 + ((x1 + 128) >> 8) + 128) >> 8;
    }
  }
  // unit of I: 2^(er + ec - 110) 256^7 = 2^(er + ec - 54)
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const int ec = ecol[q];
    const int s = er + ec - 54;
    const double sc = (er == kExNan || ec == kExNan) ? __hiloint2double(0x7ff80000, 0)
                                                     : __hiloint2double(max(min(s, 1023) + 1023, 0) << 20, 0);
    acc[q] = fma(__ll2double_rn(I[q]), sc, acc[q]);
  }
}
__device__ __forceinline__ float half_scale(int e) {  // 2^(e - 17), subnormal below e = -109; NaN for a marked row
  return e == kExNan ? __int_as_float(0x7fc00000) : __int_as_float(e >= -109 ? (e - 17 + 127) << 23 : 1 << (e + 132));
}
// low: a row or column of the warp lies below 2^-46, where the factor 2^(er + ec - 34) of all products may
// be no normal number
__device__ __forceinline__ void drain(uint32_t taddr, uint32_t bfree, int lane, int er, const int *ecol, bool low,
                                      float (&acc)[Dig<float>::N / 4]) {
  constexpr int N = Dig<float>::N, NH = N / 64;
  const float fr = half_scale(er);
#pragma unroll
  for (int hf = 0; hf < NH; ++hf) {
    uint32_t t2[16], t3[16], t4[16];
    tcp::tmem_ld16(taddr + 16 * hf, t2);
    tcp::tmem_ld16(taddr + N + 16 * hf, t3);
    tcp::tmem_ld16(taddr + 2 * N + 16 * hf, t4);
    tcp::tmem_wait_ld();
    if (hf == NH - 1) {
      tcp::fence_before();
      __syncwarp();
      if (lane < 3) tcp::mbar_arrive(bfree + 8 * lane);
    }
    // unit of weight 4: 2^(er + ec - 52) 512^2 = 2^(er - 17) 2^(ec - 17)
    float p[16];
#pragma unroll
    for (int q = 0; q < 16; ++q)
      p[q] = fmaf(fmaf(__uint_as_float(t2[q]), 512.f, __uint_as_float(t3[q])), 512.f, __uint_as_float(t4[q]));
    float f2 = fr;
    if (low) {
      // a small row's factor on the sum, a large one's on the column's: no partial product leaves the
      // range that the result has
      const bool small = er < 0 || er == kExNan;
      const float f1 = small ? fr : 1.f / 65536.f;
      f2 = small ? 1.f : __int_as_float((er - 1 + 127) << 23);
#pragma unroll
      for (int q = 0; q < 16; ++q) p[q] *= f1;
    }
#pragma unroll
    for (int q = 0; q < 16; ++q)
      acc[16 * hf + q] = fmaf(p[q], f2 * __int_as_float(ecol[16 * hf + q]), acc[16 * hf + q]);
  }
}

// Persistent CTAs, one per SM, over the 128 x 64 tiles of a batch.  Warp 18 lists the tiles (32
// candidates at a time, one per lane), warp 16 streams their digit planes (stages of 32 columns of K),
// warp 17 issues the MMAs of a stage into one accumulator per weight, and warps 0-15 combine the
// accumulators after each group of columns and at a tile's end subtract the sums from C, while
// loads and MMAs run on into the next group and tile; an accumulator is refilled as soon as it has
// been read.  64 columns: eight FP64 accumulators fill tensor memory, and a wider FP32 tile measured
// slower where the matrices are small (26 ms of updates against 35 on the masked shell).  Counters (32
// matrices of H/h = 8): the long-K update takes 517 us in FP64 with the tensor pipe 18 % active, the FP64
// pipe 38 % and DRAM at 13 %, 131 us in FP32 with 13 %, none and 10 %; short ones 4 to 7 % and 5 to 10 %.
// So neither the tensor pipe nor memory bounds it: an MMA reads A again from shared memory, and between
// groups the MMAs wait for the drain, which in FP64 does not fit its 96 registers (628 bytes of spill
// stores a thread); for short K the reading and writing of C is added.
template <typename T>
__global__ void __launch_bounds__(kUThreads, 1) k_update(const MatDesc *__restrict__ desc,
                                                         const MatDesc *__restrict__ out, T *__restrict__ base, Upd64 u,
                                                         Planes pa, Planes pb, int nct, int per, int total,
                                                         int *__restrict__ err) {
  using C = Dig<T>;
  constexpr int N = C::N, S = C::Stages, CPG = C::Grp / kUK;
  constexpr int CPW = N / 4;  // columns of a drain warp
  extern __shared__ unsigned char smem_raw[];
  __shared__ uint64_t bars[2 * S + 1 + C::W + 4];
  __shared__ uint32_t tmem_slot;
  __shared__ int failed;
  __shared__ Tile ring[2][32];
  __shared__ int ring_n[2];
  __shared__ int ecols[kDrain][CPW];
  const uint32_t raw0 = tcp::smem_addr(smem_raw);
  const uint32_t tiles = (raw0 + 1023u) & ~1023u;
  unsigned char *tp = smem_raw + (tiles - raw0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t bfull = tcp::smem_addr(&bars[0]), bempty = bfull + 8 * S, bacc = bempty + 8 * S,
                 bfree = bacc + 8, blist = bfree + 8 * C::W, bused = blist + 16;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     tcp::smem_addr(&tmem_slot)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int s = 0; s < 2 * S + 1; ++s) tcp::mbar_init(bfull + 8 * s, 1);
    for (int w = 0; w < C::W; ++w) tcp::mbar_init(bfree + 8 * w, kDrain);
    for (int k = 0; k < 2; ++k) {
      tcp::mbar_init(blist + 8 * k, 1);
      tcp::mbar_init(bused + 8 * k, kDrain + 2);
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
    failed = 0;
  }
  tcp::fence_before();
  __syncthreads();
  tcp::fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp == kDrain + 2) {
    bool ok = true;
    for (int k = 0; ok; ++k) {
      const int slot = k & 1;
      if (k >= 2) ok = tcp::mbar_wait(bused + 8 * slot, ((k >> 1) - 1) & 1);
      const long long idx = blockIdx.x + (32LL * k + lane) * gridDim.x;
      Tile t;
      const bool valid = idx < total && make_tile(desc, out, u, (int)(idx / per), (int)(idx % per) / nct,
                                                  u.ct0 + (int)(idx % per) % nct, N, t);
      const unsigned m = __ballot_sync(0xffffffffu, valid);
      if (valid) ring[slot][__popc(m & ((1u << lane) - 1u))] = t;
      const bool last = blockIdx.x + 32LL * (k + 1) * gridDim.x >= total;
      if (lane == 0) ring_n[slot] = __popc(m) | (last ? 256 : 0);
      __syncwarp();
      if (lane == 0) tcp::mbar_arrive(blist + 8 * slot);
      if (last) break;
    }
    if (!ok) failed = 1;
  } else if (warp == kDrain) {
    if (lane == 0) {
      bool ok = true;
      int n = 0;
      for (int k = 0; ok; ++k) {
        const int slot = k & 1;
        if (!tcp::mbar_wait(blist + 8 * slot, (k >> 1) & 1)) { ok = false; break; }
        const int cnt = ring_n[slot];
        for (int q = 0; q < (cnt & 255) && ok; ++q) {
          const Tile &t = ring[slot][q];
          const int ch1 = t.ch1;
          const unsigned char *qa = pa.sl + (((long long)t.b * pa.nkc + t.ch0) * C::D * pa.nrb + (t.v0 >> 6)) * kBlkBytes;
          const unsigned char *qb = pb.sl + (((long long)t.b * pb.nkc + t.ch0) * C::D * pb.nrb + (t.c0 >> 6)) * kBlkBytes;
          for (int c = t.ch0; c < ch1; ++c, ++n) {
            const int s = n % S;
            if (n >= S && !tcp::mbar_wait(bempty + 8 * s, ((n / S) - 1) & 1)) { ok = false; break; }
            const uint32_t bar = bfull + 8 * s, dst = tiles + s * stage_bytes<T>();
            tcp::mbar_expect(bar, stage_bytes<T>());
#pragma unroll
            for (int i = 0; i < C::D; ++i) {
              tcp::bulk_load(dst + i * 2 * kBlkBytes, qa + (long long)i * pa.nrb * kBlkBytes, 2 * kBlkBytes, bar);
              tcp::bulk_load(dst + a_bytes<T>() + i * (N / 64) * kBlkBytes, qb + (long long)i * pb.nrb * kBlkBytes,
                             (N / 64) * kBlkBytes, bar);
            }
            qa += (long long)C::D * pa.nrb * kBlkBytes;
            qb += (long long)C::D * pb.nrb * kBlkBytes;
          }
        }
        tcp::mbar_arrive(bused + 8 * slot);
        if (cnt & 256) break;
      }
      // the copies in flight must land before the CTA releases its shared memory
      for (int m = max(0, n - S); m < n; ++m) ok &= tcp::mbar_wait(bfull + 8 * (m % S), (m / S) & 1);
      if (!ok) failed = 1;
    }
  } else if (warp == kDrain + 1) {
    if (lane == 0) {
      bool ok = true;
      const uint32_t idesc = tcp::idesc_bf16(kUM, N);
      const uint64_t dA0 = tcp::sw64_desc(tiles);
      int n = 0, G = 0;
      for (int k = 0; ok; ++k) {
        const int slot = k & 1;
        if (!tcp::mbar_wait(blist + 8 * slot, (k >> 1) & 1)) { ok = false; break; }
        const int cnt = ring_n[slot];
        for (int q = 0; q < (cnt & 255) && ok; ++q) {
          const int ch0 = ring[slot][q].ch0, ch1 = ring[slot][q].ch1;
          for (int ca = ch0; ca < ch1 && ok; ++G) {
            const int cz = min(ch1, (ca / CPG + 1) * CPG);
            for (int c = ca; c < cz; ++c, ++n) {
              const int s = n % S;
              if (!tcp::mbar_wait(bfull + 8 * s, (n / S) & 1)) { ok = false; break; }
              tcp::fence_after();
              // descriptors of the stage; the digit planes and K steps are constant offsets
              const uint64_t dA = dA0 + (uint64_t)(s * (stage_bytes<T>() >> 4)), dB = dA + (a_bytes<T>() >> 4);
              const uint32_t keep = c == ca ? 0u : 1u;
#pragma unroll
              for (int w = 0; w < C::W; ++w) {
                if (c == ca && G > 0) {  // the accumulator's last group must have been read
                  if (!tcp::mbar_wait(bfree + 8 * w, (G - 1) & 1)) { ok = false; break; }
                  tcp::fence_after();
                }
#pragma unroll
                for (int i = 0; i < C::D; ++i) {
                  const int j = w - i;  // digit indices from 0: weight w + 2
                  if (j < 0 || j >= C::D) continue;
                  const bool first = i == (w < C::D ? 0 : w - C::D + 1);
#pragma unroll
                  for (int t = 0; t < kUK / 16; ++t)
                    tcp::mma_f16(tmem + w * N, dA + ((i * 2 * kBlkBytes + 32 * t) >> 4),
                                 dB + ((j * (N / 64) * kBlkBytes + 32 * t) >> 4), idesc, first && t == 0 ? keep : 1u);
                }
              }
              tcp::mma_commit(bempty + 8 * s);
            }
            tcp::mma_commit(bacc);
            ca = cz;
          }
        }
        tcp::mbar_arrive(bused + 8 * slot);
        if (cnt & 256) break;
      }
      if (!ok) failed = 1;
    }
  } else {
    // rows and columns of this warp, its epilogue buffer and its copy of the columns' exponents
    const int cq = (warp >> 2) * CPW, rq = (warp & 3) * 32;
    const uint32_t taddr = tmem + ((uint32_t)rq << 16) + (uint32_t)cq;
    T *stage = reinterpret_cast<T *>(tp + S * stage_bytes<T>() + warp * epi_bytes<T>());  // [32][Epi + 1]
    int *ecol = ecols[warp];
    bool ok = true;
    int G = 0;
    for (int k = 0; ok; ++k) {
      const int slot = k & 1;
      ok = tcp::mbar_wait(blist + 8 * slot, (k >> 1) & 1);
      if (!ok) break;
      const int cnt = ring_n[slot];
      for (int q = 0; q < (cnt & 255) && ok; ++q) {
        const Tile t = ring[slot][q];
        const int g0 = t.ch0 / CPG, g1 = (t.ch1 + CPG - 1) / CPG;
        // the matrix row of this lane's tile row
        const int vrow = t.v0 + rq + lane, myrow = t.br.row(min(vrow, t.br.nv - 1)), nrow = min(32, t.br.nv - t.v0 - rq);
        if (u.mode < 3 && lane < nrow && t.c0 + cq < t.ncv)  // C towards L2 while the products form
          asm volatile("prefetch.global.L2 [%0];" ::"l"(base + t.off + (long long)myrow * t.ld + t.br.row(t.c0 + cq)));
        T acc[CPW];
#pragma unroll
        for (int c = 0; c < CPW; ++c) acc[c] = T(0);
        // the exponents of a group are fetched while the group before it is drained
        const int *exr = pa.ex + (long long)t.b * pa.ng * (pa.nrb * 64) + t.v0 + rq + lane;
        const int *exc = pb.ex + (long long)t.b * pb.ng * (pb.nrb * 64) + t.c0 + cq + lane % CPW;
        const int rstep = pa.nrb * 64, cstep = pb.nrb * 64;
        int er1 = exr[(long long)g0 * rstep], ec1 = exc[(long long)g0 * cstep];
        for (int g = g0; g < g1; ++g, ++G) {
          const int er = er1;
          const bool low = sizeof(T) == 4 && __any_sync(0xffffffffu, er < -46 || ec1 < -46);
          ecol[lane % CPW] = sizeof(T) == 8 ? ec1 : __float_as_int(half_scale(ec1));
          __syncwarp();
          if (g + 1 < g1) {
            er1 = exr[(long long)(g + 1) * rstep];
            ec1 = exc[(long long)(g + 1) * cstep];
          }
          ok = ok && tcp::mbar_wait(bacc, G & 1);
          tcp::fence_after();
          drain(taddr, bfree, lane, er, ecol, low, acc);
          __syncwarp();
        }
        if (!ok) break;
        // through shared memory: row segments of C, all of a pass's loads in flight
        constexpr int EC = C::Epi, RPI = 32 / EC, NI = 32 / RPI;  // columns, rows per access, accesses
        const int r0 = lane / EC, lc = lane % EC;
#pragma unroll
        for (int c1 = 0; c1 < CPW; c1 += EC) {
#pragma unroll
          for (int c = 0; c < EC; ++c) stage[lane * (EC + 1) + c] = acc[c1 + c];
          __syncwarp();
          const int vc = t.c0 + cq + c1 + lc;
          T *Cc = base + t.off + (u.mode == 3 ? u.K0 + vc : t.br.row(vc < t.ncv ? vc : 0));
          // rows of this lane: r0 + RPI i below nrow, on or below the diagonal
          const int rmin = u.mode >= 3 ? 0 : vc - t.v0 - rq, rend = vc < t.ncv ? nrow : 0;
          T cv[NI];
          if (u.mode < 3) {
#pragma unroll
            for (int i = 0; i < NI; ++i) {
              const int r = r0 + RPI * i, row = __shfl_sync(0xffffffffu, myrow, r);
              cv[i] = Cc[(long long)row * t.ld];  // rows and columns past the tile's repeat valid ones
            }
          }
#pragma unroll
          for (int i = 0; i < NI; ++i) {
            const int r = r0 + RPI * i, row = __shfl_sync(0xffffffffu, myrow, r);
            const T a = stage[r * (EC + 1) + lc];
            if (r >= rmin && r < rend) Cc[(long long)row * t.ld] = u.mode >= 3 ? a : cv[i] - a;
          }
          __syncwarp();
        }
      }
      if (lane == 0) tcp::mbar_arrive(bused + 8 * slot);
      if (cnt & 256) break;
    }
    if (!ok) failed = 1;
  }
  __syncwarp();
  tcp::fence_before();
  __syncthreads();
  tcp::fence_after();
  if (failed && tid == 0) atomicOr(err, DEV_ERR_TIMEOUT);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

// ---- factored diagonal block of a panel and its inverse ---------------------------
// One CTA per matrix: the w x w block (w <= 64) at K0 in two 32-column halves.  Writes L_11 in
// place, its 32 x 32 diagonal blocks to the block store and the inverse Y = L_11^-1 to pinv, so
// the rows below become one product on the tensor cores.
//
// A warp's FP64 instruction takes 64 clocks of its scheduler (2 multiply-adds a clock and SM), four warps
// of an SM at a time (70 to 74 us a launch, the FP64 pipe 59 % busy on the SMs that have a matrix), so the work is spread over the four schedulers: in ldl_inv32 warps 0-3 hold
// every fourth column of the block and of its inverse (lane = row) and eliminate one column a step,
// root-free: the step's chain is one update, one reciprocal, one scaling, and the other updates run
// beside it; the square roots of the 32 pivots are taken together at the end.
// Between the halves 32 x 32 x 32 products over all warps (L_21 = A_21 Y_11^T,
// A_22 -= L_21 L_21^T, Y_21 = -Y_22 (L_21 Y_11)), column groups paired so that the schedulers get
// equal triangles.  Panels of 64 columns and not 128: the count of FP64 instructions grows with the
// cube of the width.
constexpr int kDP = kPanel64, kDLD = kDP + 1;
template <typename T>
constexpr size_t diag_smem() {
  return sizeof(T) * (2 * (size_t)kDP * kDLD + 32 * 33);
}

// 1 / p: one step of Householder's third-order iteration y (1 + e + e^2), e = 1 - p y, from the FP32
// reciprocal (relative error 2^-23, so 2^-66 after the step); far outside the FP32 range, the division.
__device__ __forceinline__ double recip(double p) {
  if (!(p > 1e-30 && p < 1e30)) return 1.0 / p;
  const double y = (double)__fdividef(1.f, (float)p), e = fma(-p, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
// the hardware estimate, within a unit in the last place (the level of FP32 rounding in the factors) over the
// whole range; __fdividef(1, p) is zero from p = 2^126 on, and 1 / p makes the pivot chain longer (a step
// of the masked shell takes 106.6 ms with the division above 8e37, 105.1 with either estimate)
__device__ __forceinline__ float recip(float p) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(p));
  return r;
}

// Lower Cholesky factor of the 32 x 32 block P (row stride LP) and its inverse into Y (LY); warps 0-3.
// Columns at and after the block's width hold the identity.  The owner of column c + 1 updates it
// first, publishes it and arrives at the column's barrier before it makes the rest of step c's
// updates, so that the others never wait for those; four column buffers and two barriers in turn keep
// the steps apart.
template <int LP, int LY, typename T>
__device__ __forceinline__ void ldl_inv32(T *P, T *Y, int s, int lane, T (*Lc)[2][32], T *piv, bool &bad) {
  T a[8], y[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int t = 4 * q + s;
    a[q] = t <= lane ? P[lane * LP + t] : T(0);
    y[q] = t == lane ? T(1) : T(0);
  }
  auto publish = [&](int c, T col) {  // column c, held by this warp
    T p = __shfl_sync(0xffffffffu, col, c);
    if (!(p > T(0))) { bad = true; p = T(1); }
    const T inv = recip(p);
    Lc[c & 3][0][lane] = col;                            // the column before scaling
    Lc[c & 3][1][lane] = lane > c ? col * inv : T(0);   // unit-lower column
    if (lane == c) piv[c] = p;
    __threadfence_block();
  };
  if (s == 0) publish(0, a[0]);
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    const int q0 = c >> 2, buf = c & 3;
    // column c is published: its owner has arrived already (at c = 0 everyone waits)
    if (c > 0 && s == (c & 3)) __syncwarp();
    else if (c & 1) asm volatile("bar.sync 2, 128;" ::: "memory");
    else asm volatile("bar.sync 1, 128;" ::: "memory");
    const T l = Lc[buf][1][lane];
    const int qn = (c + 1) >> 2;  // the next column's index in its owner
    const bool next = c < 31 && s == ((c + 1) & 3);
    if (next) {
      a[qn < 8 ? qn : 0] -= l * Lc[buf][0][c + 1 < 32 ? c + 1 : 0];
      publish(c + 1, a[qn < 8 ? qn : 0]);
      if ((c + 1) & 1) asm volatile("bar.arrive 2, 128;" ::: "memory");
      else asm volatile("bar.arrive 1, 128;" ::: "memory");
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (q >= q0 && 4 * q + s > c && !(next && q == qn)) a[q] -= l * Lc[buf][0][4 * q + s];
      if (q <= q0 && 4 * q + s <= c) {
        const T yc = __shfl_sync(0xffffffffu, y[q], c);
        y[q] -= l * yc;
      }
    }
  }
  asm volatile("bar.sync 1, 128;" ::: "memory");
  const T pl = piv[lane], rs = T(1) / sqrt(pl);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int t = 4 * q + s;
    const T rt = __shfl_sync(0xffffffffu, rs, t);
    P[lane * LP + t] = lane < t ? T(0) : (lane == t ? pl * rs : a[q] * rt);
    Y[lane * LY + t] = t <= lane ? y[q] * rs : T(0);
  }
}

template <typename T>
__global__ void __launch_bounds__(256) k_diag(const MatDesc *__restrict__ desc, T *__restrict__ base, int K0,
                                              int *__restrict__ err, T *__restrict__ store, T *__restrict__ pinv,
                                              int *__restrict__ pexp) {
  const MatDesc d = desc[blockIdx.x];
  if (K0 >= d.e) return;
  const int w = min(kDP, d.e - K0);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *P = reinterpret_cast<T *>(smem_raw);  // [64][65] the block, lower, identity past w
  T *Y = P + kDP * kDLD;                        // [64][65] its inverse
  T *Tm = Y + kDP * kDLD;                       // [32][33]
  __shared__ T Lc[4][2][32], piv[32], dg[kDP];  // dg: the diagonal before the factorisation
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  T *A = base + d.off + (long long)K0 * d.ld + K0;
  {
    const int i = tid >> 2, j0 = (tid & 3) * 16;
    T v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = (i < w && j0 + q <= i) ? A[(long long)i * d.ld + j0 + q] : (i == j0 + q ? T(1) : T(0));
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      P[i * kDLD + j0 + q] = v[q];
      Y[i * kDLD + j0 + q] = T(0);
      if (i == j0 + q) dg[i] = v[q];
    }
  }
  bool bad = false;
  const int nbk = ceil_div(w, 32);
  const int grp = 4 * (warp < 4 ? warp : 11 - warp);  // this warp's four columns (rows) of a triangle
  for (int h = 0; h < nbk; ++h) {
    const int o = 32 * h;
    __syncthreads();
    if (warp < 4) ldl_inv32<kDLD, kDLD>(P + o * kDLD + o, Y + o * kDLD + o, warp, lane, Lc, piv, bad);
    __syncthreads();
    T *sb = store + ((long long)d.dblk + K0 / kNB + h) * kNB * kNB;
    for (int q = tid; q < 1024; q += 256) sb[q] = P[(o + (q >> 5)) * kDLD + o + (q & 31)];
    if (h == 0 && nbk > 1) {
      T x[4] = {T(0), T(0), T(0), T(0)};  // L_21 = A_21 Y_11^T (Y_11 lower: k <= column)
#pragma unroll 4
      for (int k = 0; k < grp + 4; ++k) {
        const T l = P[(32 + lane) * kDLD + k];
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
        T x0 = T(0), x1 = T(0);
#pragma unroll 8
        for (int k = 0; k < 32; ++k) {
          const T l = P[r * kDLD + k];
          x0 += l * P[c * kDLD + k];
          x1 += l * P[(c + 1) * kDLD + k];
        }
        if (r < w && c <= r) P[r * kDLD + c] -= x0;
        if (r < w && c + 1 <= r) P[r * kDLD + c + 1] -= x1;
      }
    }
  }
  if (nbk > 1) {  // Y_21 = -Y_22 (L_21 Y_11)
    T x[4] = {T(0), T(0), T(0), T(0)};
    const int g2 = 28 - grp;  // columns g2 .. g2 + 3: k >= column
#pragma unroll 4
    for (int k = g2; k < 32; ++k) {
      const T l = P[(32 + lane) * kDLD + k];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] += l * Y[k * kDLD + g2 + u];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) Tm[lane * 33 + g2 + u] = x[u];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = T(0);
#pragma unroll 4
    for (int k = 0; k < grp + 4; ++k) {  // lane = column, rows grp .. grp + 3: k <= row
      const T t = Tm[k * 33 + lane];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] += Y[(32 + grp + u) * kDLD + 32 + k] * t;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) Y[(32 + grp + u) * kDLD + lane] = -x[u];
  }
  __syncthreads();
  if (bad && lane == 0) atomicOr(err, DEV_ERR_NOT_SPD);
  T *out = pinv + (long long)blockIdx.x * kDP * kDP;
  if (tid < 32) {  // column scaling of the panel solve
    int e[2], lo = 1 << 20, hi = -(1 << 20);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int i = lane + 32 * c;
      const int m = mag_bits(dg[i]);
      const bool use = i < w && m > 0 && !mag_bad(dg[i], m);
      e[c] = use ? -((mag_exp(dg[i], m) + 1) >> 1) : 0;
      if (use) {
        lo = min(lo, e[c]);
        hi = max(hi, e[c]);
      }
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    int *pe = pexp + blockIdx.x * kPanelExp;
    pe[lane] = e[0];
    pe[lane + 32] = e[1];
    if (lane == 0) pe[kPanel64] = hi - lo > 3;
  }
#pragma unroll 4
  for (int q = tid; q < kDP * kDP; q += 256) {
    const int i = q / kDP, j = q % kDP;
    out[q] = (i < w && j <= i) ? Y[i * kDLD + j] : T(0);
    if (i < w && j <= i) A[(long long)i * d.ld + j] = P[i * kDLD + j];
  }
}

// ---- FP32 diagonal block of a 128-column panel --------------------------------------
// One CTA per matrix, 32 columns at a time: factor and inverse as above, the block's rows below by
// that inverse (warp = four columns, lane = row), rank-32 update of the rest (4 x 4 tiles a thread).
// A latency chain of 128 pivots: 44 us with one warp factoring and one thread per row substituting,
// 33 us here.  The inverses of the four 32 x 32 diagonal blocks go to pinv.  A coarse matrix of 2,600
// unknowns runs 21 of these one after another.
constexpr int kWP = kEnginePanel, kWLD = kWP + 1;
constexpr size_t kDiag128Smem = sizeof(float) * (size_t)kWP * kWLD;

__global__ void __launch_bounds__(256) k_diag128(const MatDesc *__restrict__ desc, float *__restrict__ base, int K0,
                                                 int *__restrict__ err, float *__restrict__ store,
                                                 float *__restrict__ pinv) {
  const MatDesc d = desc[blockIdx.x];
  if (K0 >= d.e) return;
  const int w = min(kWP, d.e - K0);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float *P = reinterpret_cast<float *>(smem_raw);  // [128][129] the block, lower, identity past w
  __shared__ float Y[32 * 33], Lc[4][2][32], piv[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float *A = base + d.off + (long long)K0 * d.ld + K0;
  for (int r0 = warp; r0 < kWP; r0 += 64) {  // eight rows in flight per warp
    float v[8][4];
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int r = r0 + 8 * q, j = 32 * c + lane;
        v[q][c] = (r < w && j <= r) ? A[(long long)r * d.ld + j] : (r == j ? 1.f : 0.f);
      }
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
      for (int c = 0; c < 4; ++c) P[(r0 + 8 * q) * kWLD + 32 * c + lane] = v[q][c];
  }
  bool bad = false;
  const int nbk = ceil_div(w, 32), grp = 4 * (warp < 4 ? warp : 11 - warp);
  for (int h = 0; h < nbk; ++h) {
    const int o = 32 * h;
    __syncthreads();
    if (warp < 4) ldl_inv32<kWLD, 33>(P + o * kWLD + o, Y, warp, lane, Lc, piv, bad);
    __syncthreads();
    float *sb = store + ((long long)d.dblk + K0 / kNB + h) * kNB * kNB;
    float *inv = pinv + ((long long)blockIdx.x * 4 + h) * 1024;  // for the rows below the panel
    for (int q = tid; q < 1024; q += 256) {
      const int i = q >> 5, j = q & 31;
      sb[q] = P[(o + i) * kWLD + o + j];
      inv[q] = j <= i ? Y[i * 33 + j] : 0.f;
    }
    if (h + 1 == nbk) break;
    const int nrb = nbk - h - 1;  // 32-row blocks below
    float x[3][4];
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
      for (int u = 0; u < 4; ++u) x[b][u] = 0.f;
#pragma unroll 4
    for (int k = 0; k < grp + 4; ++k) {  // Y lower: k <= column
      float y[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) y[u] = Y[(grp + u) * 33 + k];
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        if (b < nrb) {
          const float l = P[(o + 32 + 32 * b + lane) * kWLD + o + k];
#pragma unroll
          for (int u = 0; u < 4; ++u) x[b][u] += l * y[u];
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < 3; ++b)
      if (b < nrb)
#pragma unroll
        for (int u = 0; u < 4; ++u) P[(o + 32 + 32 * b + lane) * kWLD + o + grp + u] = x[b][u];
    __syncthreads();
    // rows and columns from o + 32 on, lower 4 x 4 tiles
    const int n4 = 8 * nrb, nt = n4 * (n4 + 1) / 2;
    for (int t = tid; t < nt; t += 256) {
      int ti = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
      while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
      while (ti * (ti + 1) / 2 > t) --ti;
      const int tj = t - ti * (ti + 1) / 2, r = o + 32 + 4 * ti, c = o + 32 + 4 * tj;
      float a[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) a[i][j] = 0.f;
#pragma unroll 8
      for (int k = 0; k < 32; ++k) {
        float p[4], q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          p[i] = P[(r + i) * kWLD + o + k];
          q[i] = P[(c + i) * kWLD + o + k];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) a[i][j] += p[i] * q[j];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (r + i < w && c + j <= r + i) P[(r + i) * kWLD + c + j] -= a[i][j];
    }
  }
  __syncthreads();
  if (bad && lane == 0) atomicOr(err, DEV_ERR_NOT_SPD);
  for (int r = warp; r < w; r += 8)
    for (int j = lane; j <= r; j += 32) A[(long long)r * d.ld + j] = P[r * kWLD + j];
}

void launch_diag128(const MatDesc *d_desc, float *base, int K0, int count, int *err, float *store, float *pinv,
                    cudaStream_t s) {
  k_diag128<<<count, 256, kDiag128Smem, s>>>(d_desc, base, K0, err, store, pinv);
  count_launch();
}

template <typename T>
void launch_diag(const MatDesc *d_desc, T *base, int K0, int count, int *err, T *store, const SliceWs &ws,
                 cudaStream_t s) {
  k_diag<T><<<count, 256, diag_smem<T>(), s>>>(d_desc, base, K0, err, store, static_cast<T *>(ws.pinv), ws.pexp);
  count_launch();
}

template <typename T>
static bool configure() {
  return cudaFuncSetAttribute(k_update<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, update_smem<T>()) == cudaSuccess &&
         cudaFuncSetAttribute(k_diag<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)diag_smem<T>()) == cudaSuccess;
}
bool digits_configure() {
  return configure<float>() && configure<double>() &&
         cudaFuncSetAttribute(k_diag128, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDiag128Smem) == cudaSuccess;
}

// A launch that the workspace cannot hold is refused (an error of the sizes computed at setup).
static int ws_run(size_t ws_bytes, size_t one, int count) {
  const int run = digit_run(ws_bytes, one, count);
  if (run < 1)
    throw std::length_error("digit workspace of " + std::to_string(ws_bytes) + " bytes, " + std::to_string(one) +
                            " needed for one matrix");
  return run;
}

template <typename T>
bool slice_fits(int count, int max_rows, int cols, const SliceWs &ws) {
  return cols <= kSliceK && upd_layout<T>(count, max_rows, cols).bytes <= ws.bytes;
}

// Runs of matrices whose planes fit the workspace; the final update (mode 1) also in runs of
// kSliceK columns (each run rounds C once more, so they are long).
template <typename T>
void launch_update(const MatDesc *d_desc, T *base, Upd64 u, int max_rows, int max_cols, int count,
                   const SliceWs &ws, int *err, cudaStream_t s, const UpdPart &part) {
  if (max_rows <= 0 || max_cols <= 0 || count <= 0) return;
  using C = Dig<T>;
  const bool panel = u.mode == 0 || u.mode == 3;
  const int za = panel ? u.K0 : u.ka, zz = panel ? u.K0 + u.pw : u.kz;
  const int kmax = std::min(zz - za, kSliceK), nrb = digit_rows(max_rows) / 64;
  const int run = ws_run(ws.bytes, upd_layout<T>(1, max_rows, kmax).bytes, count);
  const int nrt = ceil_div(max_rows, kUM), rpc = 256 / (C::Grp / 8), rest = ceil_div(max_cols, C::N) - part.ct0;
  const int nct = part.nct < 0 ? rest : std::min(rest, part.nct), ctas = part.ctas > 0 ? part.ctas : kSms;
  if (nct <= 0) return;
  const UpdLayout lay = upd_layout<T>(run, max_rows, kmax);
  unsigned char *sl = ws.mem, *slb = sl + lay.inv;
  int *ex = reinterpret_cast<int *>(sl + lay.ex), *exb = reinterpret_cast<int *>(sl + lay.ex_inv);
  for (int b0 = 0; b0 < count; b0 += run) {
    const int nb = std::min(run, count - b0);
    for (int ka = za; ka < zz; ka += kSliceK) {
      Upd64 q = u;
      q.ka = ka;
      q.kz = std::min(zz, ka + kSliceK);
      q.ct0 = part.ct0;
      const int kw = q.kz - ka, nkc = ceil_div(kw, kUK), ng = ceil_div(kw, C::Grp);
      const Planes pa{sl, ex, nrb, nkc, ng}, pi{slb, exb, C::N / 64, kPanel64 / kUK, 1};
      if (u.mode == 3) {
        const T *pv = static_cast<const T *>(ws.pinv) + (size_t)b0 * u.pw * u.pw;
        const int *pe = ws.pexp + (size_t)b0 * kPanelExp;
        k_slice<T><<<dim3(nrb * 64 / rpc, ng, nb), 256, 0, s>>>(d_desc + b0, base, q, nullptr, sl, ex, nrb, nkc, ng,
                                                                     ColScale<T>{pe, nullptr, nullptr, 1});
        k_slice<T><<<dim3(C::N / rpc, 1, nb), 256, 0, s>>>(d_desc + b0, base, q, pv, slb, exb, C::N / 64,
                                                               kPanel64 / kUK, 1, ColScale<T>{pe, nullptr, nullptr, -1});
        count_launch(2);
      } else if (!part.sliced) {
        k_slice<T><<<dim3(nrb * 64 / rpc, ng, nb), 256, 0, s>>>(d_desc + b0, base, q, nullptr, sl, ex, nrb, nkc, ng,
                                                                      ColScale<T>{});
        count_launch();
      }
      const int per = nrt * nct, total = per * nb;
      k_update<T><<<std::min(total, ctas), kUThreads, update_smem<T>(), s>>>(d_desc + b0, d_desc + b0, base, q, pa,
                                                                            u.mode == 3 ? pi : pa, nct, per, total, err);
      count_launch();
    }
  }
}

// C = A B^T for `count` pairs of n x n matrices (n = desc.m = desc.e; the same n in all three
// descriptors of a pair), in runs of pairs whose planes fit the workspace.
template <typename T>
void launch_product(const MatDesc *d_a, const T *A, const MatDesc *d_b, const T *B, const MatDesc *d_c, T *Cm, int count,
                    int max_n, const SliceWs &ws, int *err, cudaStream_t s) {
  if (count <= 0 || max_n <= 0) return;
  using C = Dig<T>;
  const int nrb = digit_rows(max_n) / 64, nkc = ceil_div(max_n, kUK), ng = ceil_div(max_n, C::Grp);
  const int run = ws_run(ws.bytes, product_bytes<T>(1, max_n), count);
  const int nrt = ceil_div(max_n, kUM), nct = ceil_div(max_n, C::N), rpc = 256 / (C::Grp / 8);
  const size_t planes = (size_t)run * digit_planes<T>(nrb * 64, max_n);
  unsigned char *sl[2] = {ws.mem, ws.mem + planes};
  int *ex[2] = {reinterpret_cast<int *>(ws.mem + 2 * planes), nullptr};
  ex[1] = ex[0] + (size_t)run * ng * nrb * 64;
  const Upd64 u{4, 0, 0, 0, 0, max_n};
  for (int b0 = 0; b0 < count; b0 += run) {
    const int nb = std::min(run, count - b0), per = nrt * nct, total = per * nb;
    k_slice<T><<<dim3(nrb * 64 / rpc, ng, nb), 256, 0, s>>>(d_a + b0, A, u, nullptr, sl[0], ex[0], nrb, nkc, ng,
                                                           ColScale<T>{nullptr, B, d_b + b0, 1});
    k_slice<T><<<dim3(nrb * 64 / rpc, ng, nb), 256, 0, s>>>(d_b + b0, B, u, nullptr, sl[1], ex[1], nrb, nkc, ng,
                                                           ColScale<T>{nullptr, B, d_b + b0, -1});
    k_update<T><<<std::min(total, kSms), kUThreads, update_smem<T>(), s>>>(
        d_a + b0, d_c + b0, Cm, u, Planes{sl[0], ex[0], nrb, nkc, ng}, Planes{sl[1], ex[1], nrb, nkc, ng}, nct, per, total,
        err);
    count_launch(3);
  }
}

#define BD_DIG_INST(T)                                                                                       \
  template void launch_diag<T>(const MatDesc *, T *, int, int, int *, T *, const SliceWs &, cudaStream_t);   \
  template void launch_update<T>(const MatDesc *, T *, Upd64, int, int, int, const SliceWs &, int *,       \
                                 cudaStream_t, const UpdPart &);                                 \
  template bool slice_fits<T>(int, int, int, const SliceWs &);                                               \
  template void launch_product<T>(const MatDesc *, const T *, const MatDesc *, const T *, const MatDesc *, T *, int, \
                                  int, const SliceWs &, int *, cudaStream_t);
BD_DIG_INST(float)
BD_DIG_INST(double)

}  // namespace bd
