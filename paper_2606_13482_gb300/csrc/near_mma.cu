// Near-field product on the tensor cores, FP64-class accuracy.
//
// y[r][i] = sum over the near blocks of the target box of M[i][n] x[r][n] is a
// dense contraction per (target box, source box) pair.  The double-float form
// spends 48 FP32 instructions on every complex multiply-add and the FP64 form
// four FP64 ones at a 64th of the FP32 rate; here every operand is cut into
// 10-bit digits (an error-free fixed-point splitting, Ozaki et al. 2012) and
// digit products run as FP16 MMAs with FP32 accumulation, which are exact:
//
//   a = 2^(EA + 1) sum_i a_i 2^(-9 - 10 i),  |a_0| <= 256, |a_i| <= 512
//
// (double-float entries: a = 2^EA sum_i a_i 2^(-9 - 10 i), |a_i| <= 512, the first digit too;
// x has the form above in both), with one exponent EA per (block, row) of the matrix (found at setup) and one
// exponent EX per (source box, right-hand side) of x.  NS = 5 digits (50 bits
// below the row's largest entry) stand for the double-float entries of mixed
// handles, NS = 6 (60 bits) for FP64 ones.  The sum over a group of 8 complex
// columns of one digit pair is at most 16 * 512 * 512 = 2^22, so an MMA (or, with FP64
// entries, a chain of the two pairs that hold a top digit, 2^21 each; with double-float ones
// that chain would reach 1.5 * 2^22) started from the accumulator 1.5 * 2^23 returns its exact integer sum in the low bits of the
// FP32 result, and one integer add moves it to a 32-bit running sum.  Pairs of
// equal weight i + j share a running sum: weights 0..3 exactly, weight 4 (and 5)
// in an FP32 accumulator whose rounding lies 2^-58 below the row maximum.  At
// the end of a source box the sums are scaled into an FP64 accumulator.
//
// What bounds it: the FP16 MMAs, 4 (NS (NS + 1) / 2) real multiply-adds per
// complex one at 1,024 per clock and SM (mma.sync, measured 984), i.e. 3.75
// clocks per entry and 64 vectors; up to 8 vectors the matrix stream (16 bytes
// an entry) and its splitting.  tcgen05 would quadruple the MMA rate but wants the
// integer flush of every 8 columns read back from TMEM (320 columns x 128 lanes
// per flush), which costs more than the MMAs it saves.
//
// Work split: a warp owns 16 rows of a target box and 8 NT right-hand sides and
// streams the box's block row on its own -- no barriers.  The MMA fragment of a
// thread is rows g, g + 8 of columns t, t + 4 (k = 2t, 2t + 1 are the real and
// imaginary parts of a column), so a thread splits exactly the four entries that
// it loads, in registers; entries, and the digits of x that k_near_digits has laid
// out in fragment order, arrive by 16-byte asynchronous copies in a ring of the
// warp's own.  Sharing the split entries of a 32-row tile in shared memory
// between 8 warps (one barrier per 16 or 32 columns) measured 5.3 ms instead of
// 3.8 for the 4-wavelength sphere (1.1e8 entries) and 64 vectors, the warps
// waiting on one another half of the time.
//
// Measured there, A and the scalar part together, ms (before: double-float on
// the FP32 pipes, or FP64 arithmetic): 64 vectors 4.1 (33), 16 1.1 (7.3), 8 0.80
// (4.6); FP64 handles, 8 vectors, 1.4 (13.3).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "device_api.cuh"
#include "digits.cuh"

namespace efie {

static_assert(NEAR_MMA_ROWS == 16, "one MMA row tile per warp");
__device__ __forceinline__ uint32_t nm_packf(float d0, float d1) {
  const __half2 h = __floats2half2_rn(d0, d1);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float nm_pow2(int e) { return __int_as_float((e + 127) << 23); }
// digits of a double-float value hi + lo: every step is exact but the last
// rounding.  s9 = 2^(9 - E), s19 = 2^(19 - E), s29 = 2^(29 - E).  The rounding of
// the second digit looks at lo, so that the third one stays within 512.
__device__ __forceinline__ void nm_digits_df(float hi, float lo, float s9, float s19, float s29, float* d) {
  const float M = 12582912.f;
  d[0] = __fsub_rn(__fmaf_rn(hi, s9, M), M);
  float r = __fmaf_rn(hi, s9, -d[0]);
  r = __fmul_rn(r, 1024.f);
  d[1] = __fsub_rn(__fadd_rn(__fmaf_rn(lo, s19, r), M), M);
  r = __fsub_rn(r, d[1]);
  const float h2 = __fsub_rn(__fmaf_rn(r, 1024.f, M), M);
  r = __fmaf_rn(r, 1024.f, -h2);
  r = __fmaf_rn(lo, s29, r);
  const float l2 = __fsub_rn(__fadd_rn(r, M), M);
  d[2] = __fadd_rn(h2, l2);
  r = __fsub_rn(r, l2);
  d[3] = __fsub_rn(__fmaf_rn(r, 1024.f, M), M);
  r = __fmaf_rn(r, 1024.f, -d[3]);
  d[4] = __fsub_rn(__fmaf_rn(r, 1024.f, M), M);
}

// ---------------------------------------------------------------- row exponents (setup)
// rexp[rexp_off[x] + (j - near_ptr[x]) nrow + row]: E with max |entry| < 2^E over
// the row of block j; one CTA per block, a thread per row (column reads coalesce)
template <bool F64>
__global__ void k_near_rexp(const void* __restrict__ M, const int64_t* __restrict__ blk_off,
                            const int64_t* __restrict__ near_ptr, const int32_t* __restrict__ near_src,
                            const int32_t* __restrict__ blk_tgt, const int64_t* __restrict__ box_ptr,
                            const int64_t* __restrict__ rexp_off, int16_t* __restrict__ rexp) {
  const int64_t j = blockIdx.x;
  const int x = blk_tgt[j], y = near_src[j];
  const int nrow = (int)(box_ptr[x + 1] - box_ptr[x]), ncol = (int)(box_ptr[y + 1] - box_ptr[y]);
  int16_t* out = rexp + rexp_off[x] + (j - near_ptr[x]) * nrow;
  for (int row = threadIdx.x; row < nrow; row += blockDim.x) {
    int E;
    if (F64) {
      const double2* Mb = (const double2*)M + blk_off[j] + row;
      int mx = 0;
      for (int c = 0; c < ncol; ++c) {
        const double2 a = Mb[(int64_t)c * nrow];
        mx = max(mx, max(__double2hiint(a.x) & 0x7fffffff, __double2hiint(a.y) & 0x7fffffff));
      }
      E = nm_row_exponent(mx);
    } else {
      const float4* Mb = (const float4*)M + blk_off[j] + row;
      int mx = 0;
      for (int c = 0; c < ncol; ++c) {
        const float4 a = Mb[(int64_t)c * nrow];
        mx = max(mx, max(__float_as_int(a.x) & 0x7fffffff, __float_as_int(a.z) & 0x7fffffff));
      }
      const int f = mx >> 23;
      E = f == 255 ? NM_ENAN : max(f - 126, -90);
    }
    out[row] = (int16_t)E;
  }
}

// ---------------------------------------------------------------- digits of x
// One CTA per (box, 8 right-hand sides), a warp per right-hand side: the
// exponent of the box's values, then their digits in MMA B-fragment order,
// xd[kg][ntile][digit][lane] = (column t, column t + 4), each as half2 (real,
// imaginary), kg a group of 8 columns, lane = 4 (rhs % 8) + t.  Missing columns
// and right-hand sides are zeros.  Reads x once more from L2; a few percent of
// the product.
template <int NS>
__global__ void __launch_bounds__(256) k_near_digits(const double2* __restrict__ x, int64_t ld, int nr, int ntt,
                                                     const int64_t* __restrict__ box_ptr,
                                                     const int64_t* __restrict__ kg_off, uint2* __restrict__ xd,
                                                     int16_t* __restrict__ xexp) {
  const int box = blockIdx.x, nt = blockIdx.y, n = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t c0 = box_ptr[box];
  const int ncol = (int)(box_ptr[box + 1] - c0);
  const int r = nt * 8 + n;
  const double2* xr = x + (int64_t)r * ld + c0;
  int mx = 0;
  if (r < nr)
    for (int c = lane; c < ncol; c += 32) {
      const double2 v = xr[c];
      mx = max(mx, max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff));
    }
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  // a box of subnormal numbers only: its own exponent, the values raised by 2^64
  const bool sub = (mx >> 20) == 0;
  const int E = sub ? 32 - __clz(mx) - 1042 : nm_exponent(mx), Ed = sub ? E + 64 : E;
  if (lane == 0) xexp[((int64_t)box * ntt + nt) * 8 + n] = (int16_t)E;
  const bool zero = r >= nr || E == NM_ENAN;
  const int npair = ((ncol + 7) / 8) * 4;
  for (int cp = lane; cp < npair; cp += 32) {
    const int c = (cp >> 2) * 8 + (cp & 3);
    double2 v0 = make_double2(0, 0), v1 = v0;
    if (!zero && c < ncol) v0 = xr[c];
    if (!zero && c + 4 < ncol) v1 = xr[c + 4];
    if (sub) {
      const double up = 18446744073709551616.0;
      v0 = make_double2(v0.x * up, v0.y * up), v1 = make_double2(v1.x * up, v1.y * up);
    }
    int a0[NS], a1[NS], b0[NS], b1[NS];
    nm_digits<NS>(nm_fixed(v0.x, Ed), a0);
    nm_digits<NS>(nm_fixed(v0.y, Ed), b0);
    nm_digits<NS>(nm_fixed(v1.x, Ed), a1);
    nm_digits<NS>(nm_fixed(v1.y, Ed), b1);
    uint2* o = xd + (((kg_off[box] + (cp >> 2)) * ntt + nt) * NS) * 32 + n * 4 + (cp & 3);
#pragma unroll
    for (int s = 0; s < NS; ++s) o[s * 32] = make_uint2(nm_pack(a0[s], b0[s]), nm_pack(a1[s], b1[s]));
  }
}

// ---------------------------------------------------------------- product
__device__ __forceinline__ void nm_cp16(void* dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(bytes)
               : "memory");
}

// Per warp: a ring of RD column groups (entries, 2 KB, and the digits of x),
// and the FP64 accumulators.  RD - 1 groups are in flight, which covers DRAM's
// latency: a group is 30 NT MMAs long.  Blocks per SM and RD as measured (4-
// wavelength sphere, near A, ms): NT = 1 (8 vectors) 4 blocks, RD 3 0.53, 3
// blocks, RD 4 0.53, 2 blocks, RD 4 0.55; NT = 2 (16) 2 blocks, RD 4 0.74, 3
// blocks, RD 3 0.99 (spills); NT = 4 (64) 2 blocks, RD 2 2.65, 1 block, RD 3 3.49,
// and 2.95 with NT = 2.
template <bool F64, int NT>
struct NmCfg {
  static constexpr int NS = F64 ? 6 : 5;
  static constexpr int RD = NT == 4 ? 2 : NT == 2 ? 4 : 3;
  static constexpr int XW = NT * NS * 16;          // 16-byte words of digits per group
  static constexpr int SLOT = 128 + XW;            // and of a ring slot
  static constexpr int WARP_BYTES = RD * SLOT * 16;
  static constexpr int SMEM = 4 * (WARP_BYTES + 8 * NT * 32 * 8);
};

// a source box of the list: first entry of the block, first column group, box, columns
struct NmBox {
  int64_t m, x;
  int y, nc;
};

// grid: tile groups of both operators, the groups of 8 NT right-hand sides of
// one tile group next to each other (the matrix comes from DRAM once).  A block's four warps take four row tiles, or, with wk = 2 or 4, 4 / wk tiles and
// the source boxes s, s + wk, .. each, summed at the end in a fixed order.
template <bool F64, int NT>
__global__ void __launch_bounds__(128, NT == 1 ? 4 : 2)
k_near_mma(const NearMma pa, const NearMma pb, int nr, int ntt, int wk) {
  using Cfg = NmCfg<F64, NT>;
  constexpr int NS = Cfg::NS, RD = Cfg::RD;
  constexpr int NG = F64 ? 5 : 4;  // digit-pair weights summed exactly
  extern __shared__ __align__(16) unsigned char nm_smem[];
  __shared__ NearMma P;  // this block's operator, out of the registers
  __shared__ NmBox boxes[4][32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint4* ring = reinterpret_cast<uint4*>(nm_smem + warp * Cfg::WARP_BYTES);
  double* acc = reinterpret_cast<double*>(nm_smem + 4 * Cfg::WARP_BYTES);  // [8 NT][128]
  const int tpb = 4 / wk;  // row tiles per block
  const int nba = (pa.ntiles + tpb - 1) / tpb, ngr = ntt / NT;
  const int tg = (int)blockIdx.x / ngr;
  const bool second = tg >= nba;
  if (tid == 0) P = second ? pb : pa;
  __syncthreads();
  const int wks = warp % wk;  // this warp's stream of source boxes
  const int tile = (tg - (second ? nba : 0)) * tpb + warp / wk;
  const int nt0 = ((int)blockIdx.x - tg * ngr) * NT;
  const bool active = tile < P.ntiles;
#pragma unroll
  for (int v = 0; v < 8 * NT; ++v) acc[v * 128 + tid] = 0.0;
  int xb = 0, row0 = 0, nrow = 0;
  const int g = lane >> 2, t = lane & 3;
  if (active) {
    xb = P.tiles[2 * tile], row0 = P.tiles[2 * tile + 1];
    nrow = (int)(P.box_ptr[xb + 1] - P.box_ptr[xb]);
    const int ra = row0 + g, rb = ra + 8;
    const bool oka = ra < nrow, okb = rb < nrow;
    const int64_t j0 = P.near_ptr[xb];
    const int nblk = (int)(P.near_ptr[xb + 1] - j0);
    const int16_t* rexp = P.rexp + P.rexp_off[xb];
    // 1.5 * 2^23 four times over, behind a mov so that they stay in four
    // consecutive registers instead of being copied there before every MMA
    float mg[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) asm volatile("mov.b32 %0, 0x4B400000;" : "=f"(mg[v]));
    constexpr uint32_t MB = 0x4B400000;
    int run[NT][NG][8];
    float fl[NT][8];
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int v = 0; v < 8; ++v) {
#pragma unroll
        for (int w = 0; w < NG; ++w) run[n][w][v] = 0;
        fl[n][v] = 0.f;
      }
    int nk = 0;  // column groups in the running sums: each flush has left MB there once per group

    // source boxes, 32 of the stream at a time, one per lane
    for (int b0 = wks; b0 < nblk; b0 += 32 * wk) {
      const int bj = b0 + lane * wk;
      NmBox bi = {0, 0, 0, 0};
      if (bj < nblk) {
        bi.y = P.near_src[j0 + bj];
        bi.nc = (int)(P.box_ptr[bi.y + 1] - P.box_ptr[bi.y]);
        bi.m = P.blk_off[j0 + bj];
        bi.x = P.kg_off[bi.y] * ntt + nt0;
      }
      __syncwarp();
      boxes[warp][lane] = bi;
      __syncwarp();
      const NmBox* bl = boxes[warp];
      const unsigned have = __ballot_sync(0xffffffffu, bi.nc > 0);
      if (have == 0) continue;
      // loader: column groups in order, box lb (of the lanes in `left`), group lk
      unsigned left = have;
      int lb = __ffs(left) - 1, lk = 0;
      int lnc = bl[lb].nc;
      const uint4* lm = reinterpret_cast<const uint4*>(P.M) + bl[lb].m;
      const uint4* lx = reinterpret_cast<const uint4*>(P.xd) + bl[lb].x * (NS * 16) + lane;
      auto load = [&](int slot) {
        if (left) {
          const int c = lk * 8 + t;
          const bool k0 = c < lnc, k1 = c + 4 < lnc;
          const uint4* m0 = lm + (int64_t)(k0 ? c : 0) * nrow;
          const uint4* m1 = lm + (int64_t)(k1 ? c + 4 : 0) * nrow;
          uint4* d = ring + slot * Cfg::SLOT + lane;
          nm_cp16(d, m0 + (oka ? ra : 0), oka && k0 ? 16 : 0);
          nm_cp16(d + 32, m0 + (okb ? rb : 0), okb && k0 ? 16 : 0);
          nm_cp16(d + 64, m1 + (oka ? ra : 0), oka && k1 ? 16 : 0);
          nm_cp16(d + 96, m1 + (okb ? rb : 0), okb && k1 ? 16 : 0);
#pragma unroll
          for (int i = 0; i < Cfg::XW / 32 + (Cfg::XW % 32 != 0); ++i)
            if (Cfg::XW % 32 == 0 || i < Cfg::XW / 32 || lane < Cfg::XW % 32)
              asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(
                               (uint32_t)__cvta_generic_to_shared(d + 128 + 32 * i)),
                           "l"(lx + 32 * i)
                           : "memory");
          lx += ntt * (NS * 16);
          if (++lk * 8 >= lnc) {
            left &= left - 1;
            lk = 0;
            if (left) {
              lb = __ffs(left) - 1;
              lnc = bl[lb].nc;
              lm = reinterpret_cast<const uint4*>(P.M) + bl[lb].m;
              lx = reinterpret_cast<const uint4*>(P.xd) + bl[lb].x * (NS * 16) + lane;
            }
          }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
      };
#pragma unroll
      for (int q = 0; q < RD - 1; ++q) load(q);
      int slot = 0;
      unsigned todo = have;
      // row exponents of the first box; of the following ones, a box ahead
      int cb = __ffs(todo) - 1;
      int jn = b0 + cb * wk;
      int nea = oka ? rexp[jn * nrow + ra] : 0, neb = okb ? rexp[jn * nrow + rb] : 0;
      while (todo) {
        const int nc = bl[cb].nc, y = bl[cb].y;
        const int ea = nea, eb = neb;
        todo &= todo - 1;
        if (todo) {
          cb = __ffs(todo) - 1;
          jn = b0 + cb * wk;
          nea = oka ? rexp[jn * nrow + ra] : 0, neb = okb ? rexp[jn * nrow + rb] : 0;
        }
        const bool bada = ea == NM_ENAN, badb = eb == NM_ENAN;
        const float sa9 = F64 || bada ? 0.f : nm_pow2(9 - ea), sb9 = F64 || badb ? 0.f : nm_pow2(9 - eb);
        const int nkg = (nc + 7) / 8;
#pragma unroll 1
        for (int kg = 0; kg < nkg; ++kg) {
          load(slot == 0 ? RD - 1 : slot - 1);  // the slot that the last group has left
          asm volatile("cp.async.wait_group %0;\n" ::"n"(RD - 1) : "memory");
          __syncwarp();
          const uint4* cur = ring + slot * Cfg::SLOT;
          // split: a[s] = rows g, g + 8 of column t, then of column t + 4
          uint32_t a[NS][4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint4 w = cur[q * 32 + lane];
            if constexpr (F64) {
              const int E = (q & 1) ? eb : ea;
              const bool bad = (q & 1) ? badb : bada;
              int dr[NS], di[NS];
              nm_digits<NS>(bad ? 0 : nm_fixed(__hiloint2double(w.y, w.x), E), dr);
              nm_digits<NS>(bad ? 0 : nm_fixed(__hiloint2double(w.w, w.z), E), di);
#pragma unroll
              for (int s = 0; s < NS; ++s) a[s][q] = nm_pack(dr[s], di[s]);
            } else {
              const float s9 = (q & 1) ? sb9 : sa9, s19 = s9 * 1024.f, s29 = s19 * 1024.f;
              float dr[NS], di[NS];
              nm_digits_df(__uint_as_float(w.x), __uint_as_float(w.y), s9, s19, s29, dr);
              nm_digits_df(__uint_as_float(w.z), __uint_as_float(w.w), s9, s19, s29, di);
#pragma unroll
              for (int s = 0; s < NS; ++s) a[s][q] = nm_packf(dr[s], di[s]);
            }
          }
          slot = slot == RD - 1 ? 0 : slot + 1;
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            const uint2* xq = reinterpret_cast<const uint2*>(cur + 128) + n * (NS * 32) + lane;
            uint2 x[NS];
#pragma unroll
            for (int s = 0; s < NS; ++s) x[s] = xq[s * 32];
#pragma unroll
            for (int part = 0; part < 2; ++part) {
              // real: ar xr - ai xi; imaginary: ar xi + ai xr
              uint32_t c0[NS], c1[NS];
#pragma unroll
              for (int s = 0; s < NS; ++s) {
                c0[s] = part ? __byte_perm(x[s].x, 0, 0x1032) : x[s].x ^ 0x80000000u;
                c1[s] = part ? __byte_perm(x[s].y, 0, 0x1032) : x[s].y ^ 0x80000000u;
              }
#pragma unroll
              for (int w = 0; w < NG; ++w)
#pragma unroll
                for (int i = 0; i <= w; ++i) {
                  if (F64 && w > 0 && i == w) continue;  // chained to (0, w) below
                  float d[4];
                  nm_mma(d, a[i], c0[w - i], c1[w - i], mg);
                  if (F64 && w > 0 && i == 0) nm_mma(d, a[w], c0[0], c1[0], d);
#pragma unroll
                  for (int v = 0; v < 4; ++v) run[n][w][part * 4 + v] += __float_as_int(d[v]);
                }
              float* f = &fl[n][part * 4];
#pragma unroll
              for (int i = 0; i <= NG; ++i) nm_mma(f, a[i], c0[NG - i], c1[NG - i], f);
            }
          }
          __syncwarp();  // every lane has read this slot before the next load refills it
          ++nk;
          if (kg + 1 < nkg && (kg + 1) % (NM_PIECE / 8) != 0) continue;
          // end of the box (or of NM_PIECE of its columns): running sums into the
          // FP64 accumulators, T = 2^30 g0 + 2^20 g1 + 2^10 g2 + g3 in units of 2^-48 and
          // the next weight(s) below it
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            const int xe = __ldg(reinterpret_cast<const int*>(P.xexp + ((int64_t)y * ntt + nt0 + n) * 8) + t);
            const NmCol x0 = nm_col((int16_t)(xe & 0xffff)), x1 = nm_col(xe >> 16);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              const NmCol xc = (v & 1) ? x1 : x0;
              const double sc = nm_scale(v < 2 ? ea : eb, xc, F64 ? 46 : 51);
#pragma unroll
              for (int part = 0; part < 2; ++part) {
                const int q = part * 4 + v;
                // wrapping arithmetic: the sums themselves fit in 32 bits
                int r_[NG];
#pragma unroll
                for (int w = 0; w < NG; ++w) {
                  r_[w] = (int)((uint32_t)run[n][w][q] - MB * (uint32_t)(nk * (F64 && w > 0 ? w : w + 1)));
                  run[n][w][q] = 0;
                }
                long long T = ((long long)r_[0] << 30) + ((long long)r_[1] << 20) + ((long long)r_[2] << 10) + r_[3];
                double* ap = acc + (n * 8 + q) * 128 + tid;
                if constexpr (F64) {
                  const int low = r_[4] + __float2int_rn(fl[n][q] * 0.0009765625f);
                  *ap = fma(nm_raise((double)T, xc), sc, fma(nm_raise((double)low, xc), sc * 0.0009765625, *ap));
                } else {
                  T = T * 16 + __float2int_rn(fl[n][q] * 0.015625f);
                  *ap = fma(nm_raise((double)T, xc), sc, *ap);
                }
                fl[n][q] = 0.f;
              }
            }
          }
          nk = 0;
        }
      }
      asm volatile("cp.async.wait_all;\n" ::: "memory");
    }
  }
  if (wk > 1) __syncthreads();
  if (!active || wks != 0) return;
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int row = row0 + g + (v < 2 ? 0 : 8);
      const int r = (nt0 + n) * 8 + 2 * t + (v & 1);
      if (row >= nrow || r >= nr) continue;
      double re = 0.0, im = 0.0;
      for (int k = 0; k < wk; ++k) {  // the streams' sums, in a fixed order
        re += acc[(n * 8 + v) * 128 + tid + 32 * k];
        im += acc[(n * 8 + 4 + v) * 128 + tid + 32 * k];
      }
      P.y[(int64_t)r * P.ld + P.box_ptr[xb] + row] = make_double2(re, im);
    }
}

// ---------------------------------------------------------------- launchers
int near_mma_ntiles8(int nr) { return nr <= 8 ? 1 : nr <= 16 ? 2 : nr <= 32 ? 4 : 8; }
int near_mma_max_nr(bool f64) { return f64 ? 8 : 64; }
int near_mma_digits(bool f64) { return f64 ? 6 : 5; }

void launch_near_rexp(const void* M, bool f64, const int64_t* blk_off, const int64_t* near_ptr,
                      const int32_t* near_src, const int32_t* blk_tgt, int64_t n_blocks, const int64_t* box_ptr,
                      const int64_t* rexp_off, int16_t* rexp, cudaStream_t s) {
  if (n_blocks <= 0) return;
  if (f64)
    k_near_rexp<true><<<(unsigned)n_blocks, 128, 0, s>>>(M, blk_off, near_ptr, near_src, blk_tgt, box_ptr, rexp_off,
                                                         rexp);
  else
    k_near_rexp<false><<<(unsigned)n_blocks, 128, 0, s>>>(M, blk_off, near_ptr, near_src, blk_tgt, box_ptr, rexp_off,
                                                          rexp);
}

void launch_near_digits(const double2* x, int64_t ld, int nr, bool f64, const int64_t* box_ptr, int64_t n_boxes,
                        const int64_t* kg_off, uint2* xd, int16_t* xexp, cudaStream_t s) {
  if (n_boxes <= 0 || nr <= 0) return;
  const int ntt = near_mma_ntiles8(nr);
  const dim3 grid((unsigned)n_boxes, (unsigned)ntt);
  if (f64) k_near_digits<6><<<grid, 256, 0, s>>>(x, ld, nr, ntt, box_ptr, kg_off, xd, xexp);
  else k_near_digits<5><<<grid, 256, 0, s>>>(x, ld, nr, ntt, box_ptr, kg_off, xd, xexp);
}

template <bool F64, int NT>
static void run_near_mma(const NearMma& a, const NearMma& b, int nr, int ntt, cudaStream_t s) {
  static SmemAttr attr;
  using Cfg = NmCfg<F64, NT>;
  smem_attr_once(k_near_mma<F64, NT>, Cfg::SMEM, attr.v);
  // source boxes over 2 or 4 warps of a block while the row tiles alone leave
  // the chip's warp slots (8 to 16 per SM) less than half full
  const int groups = ntt / NT, slots = 152 * (NT == 1 ? 16 : 8);
  const int64_t warps = (int64_t)(a.ntiles + b.ntiles) * groups;
  const int wk = warps * 4 <= slots ? 4 : warps * 2 <= slots ? 2 : 1;
  const int tpb = 4 / wk;
  const int64_t blocks = ((a.ntiles + tpb - 1) / tpb + (b.ntiles + tpb - 1) / tpb) * (int64_t)groups;
  k_near_mma<F64, NT><<<(unsigned)blocks, 128, Cfg::SMEM, s>>>(a, b, nr, ntt, wk);
}

// both near operators (a second one with ntiles = 0 is absent) on nr right-hand
// sides, at most near_mma_max_nr; every row of every box is written
void launch_near_mma(const NearMma& a, const NearMma& b, int nr, bool f64, cudaStream_t s) {
  if (nr <= 0 || a.ntiles + b.ntiles <= 0) return;
  const int ntt = near_mma_ntiles8(nr);
  if (f64) run_near_mma<true, 1>(a, b, nr, ntt, s);
  else if (ntt == 1) run_near_mma<false, 1>(a, b, nr, ntt, s);
  else if (ntt == 2) run_near_mma<false, 2>(a, b, nr, ntt, s);
  else run_near_mma<false, 4>(a, b, nr, ntt, s);
}

}  // namespace efie
