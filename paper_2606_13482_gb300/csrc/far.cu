// Far-field kernels of the fast matvec (charges through interpolation) and small vector kernels.
//
//  k_anterp : leaf anterpolation q_{d,b} = sum_{n in b} j_n m_{d,n} and the
//             charge component q_{4,b} = sum_{c in b} rho_c m^phi_c
//             (Eq. TAfactor, Sec. VI-A); one CTA per leaf box, one thread
//             per grid point gathering over the moments that cover it.
//  k_mode   : tensor mode products with the knot-insertion transfers
//             C^L / C^R and their transposes (Eq. interleveltransfer, Sec. IV-B).
//  k_dft    : stabilize + zero-pad + DFT fused into one n x s' complex
//             matrix per axis (F P, P = B_stab^{-1} S), inverse likewise
//             (P^T F^{-1}); Sec. III-C, Sec. V-B.
//  k_mac    : frequency-domain translation R_x = sum_{y in IL(x)} K_{x-y} Q_y
//             (Eq. TAfactorBspline, Toeplitz structure), spectra stored
//             frequency-major so one frequency of all boxes is contiguous.
//  k_interp : interpolation (the transpose of anterpolation), one warp per
//             basis function, lanes over channels.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "device_api.cuh"
#include "plan.hpp"
#include "../../include/efie.h"

namespace efie {

// ---------------------------------------------------------------- mode product
template <typename R, bool CM>
__global__ void k_mode(const cpx_t<R>* __restrict__ in, View vin, cpx_t<R>* __restrict__ out,
                       View vout, int64_t B, int C, int ax, int nin, int e0, int e1, int e2,
                       const void* __restrict__ M0, const void* __restrict__ M1,
                       const int8_t* __restrict__ sel, const int64_t* __restrict__ srcmap,
                       bool accumulate) {
  using T = cpx_t<R>;
  const int64_t total = B * e0 * e1 * e2 * (int64_t)C;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t t = idx;
    int c = (int)(t % C);
    t /= C;
    int j2 = (int)(t % e2);
    t /= e2;
    int j1 = (int)(t % e1);
    t /= e1;
    int j0 = (int)(t % e0);
    int64_t b = t / e0;
    int64_t bs = srcmap ? srcmap[b] : b;
    int jo = ax == 0 ? j0 : (ax == 1 ? j1 : j2);
    int64_t step = ax == 0 ? vin.s0 : (ax == 1 ? vin.s1 : vin.s2);
    int64_t base = bs * vin.sb + (int64_t)(ax == 0 ? 0 : j0) * vin.s0 +
                   (int64_t)(ax == 1 ? 0 : j1) * vin.s1 + (int64_t)(ax == 2 ? 0 : j2) * vin.s2 + c;
    const void* Mv = (sel && sel[3 * b + ax]) ? M1 : M0;
    T acc = mk<R>(0, 0);
    if (CM) {
      const T* M = (const T*)Mv + (int64_t)jo * nin;
      for (int i = 0; i < nin; ++i) cfma(acc, M[i], in[base + i * step]);
    } else {
      const R* M = (const R*)Mv + (int64_t)jo * nin;
      for (int i = 0; i < nin; ++i) {
        T v = in[base + i * step];
        acc.x = fma(M[i], v.x, acc.x);
        acc.y = fma(M[i], v.y, acc.y);
      }
    }
    int64_t o = b * vout.sb + (int64_t)j0 * vout.s0 + (int64_t)j1 * vout.s1 + (int64_t)j2 * vout.s2 + c;
    if (accumulate) acc = cadd(acc, out[o]);
    out[o] = acc;
  }
}

// Line form: one thread owns LPT lines (box, the two other indices, LPT
// consecutive channels), loads their nin inputs into registers once and writes
// all nout outputs; the one or two matrices of the pass sit in shared memory,
// so each matrix value read feeds LPT complex MACs.
template <typename R, bool CM, int NMAX, int LPT>
__global__ void k_mode_line(const cpx_t<R>* __restrict__ in, View vin, cpx_t<R>* __restrict__ out,
                            View vout, int64_t B, int C, int ax, int nin, int e0, int e1, int e2,
                            const void* __restrict__ M0, const void* __restrict__ M1,
                            const int8_t* __restrict__ sel, const int64_t* __restrict__ srcmap,
                            bool accumulate) {
  using T = cpx_t<R>;
  extern __shared__ unsigned char smem_raw[];
  const int nout = ax == 0 ? e0 : (ax == 1 ? e1 : e2);
  const int msz = nout * nin;
  const int esz = CM ? (int)sizeof(T) : (int)sizeof(R);
  const int nmat = M1 && M1 != M0 ? 2 : 1;
  for (int i = threadIdx.x; i < msz * esz / 4; i += blockDim.x) {
    ((int*)smem_raw)[i] = ((const int*)M0)[i];
    if (nmat == 2) ((int*)smem_raw)[msz * esz / 4 + i] = ((const int*)M1)[i];
  }
  __syncthreads();
  const int ea = ax == 0 ? e1 : e0, eb = ax == 2 ? e1 : e2;
  const int64_t sa_in = ax == 0 ? vin.s1 : vin.s0, sb_in = ax == 2 ? vin.s1 : vin.s2;
  const int64_t sa_out = ax == 0 ? vout.s1 : vout.s0, sb_out = ax == 2 ? vout.s1 : vout.s2;
  const int64_t step_in = ax == 0 ? vin.s0 : (ax == 1 ? vin.s1 : vin.s2);
  const int64_t step_out = ax == 0 ? vout.s0 : (ax == 1 ? vout.s1 : vout.s2);
  const int CL = C / LPT;  // channel groups
  const int64_t lines = B * ea * eb * (int64_t)CL;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < lines;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t t = idx;
    const int c = (int)(t % CL) * LPT;
    t /= CL;
    const int ib = (int)(t % eb);
    t /= eb;
    const int ia = (int)(t % ea);
    const int64_t b = t / ea;
    const int64_t bs = srcmap ? srcmap[b] : b;
    const T* ip = in + bs * vin.sb + ia * sa_in + ib * sb_in + c;
    T v[NMAX][LPT];
#pragma unroll
    for (int i = 0; i < NMAX; ++i)
      if (i < nin)
#pragma unroll
        for (int l = 0; l < LPT; ++l) v[i][l] = ip[i * step_in + l];
    const unsigned char* Ms = smem_raw + ((nmat == 2 && sel && sel[3 * b + ax]) ? (size_t)msz * esz : 0);
    T* op = out + b * vout.sb + ia * sa_out + ib * sb_out + c;
    for (int j = 0; j < nout; ++j) {
      T acc[LPT];
#pragma unroll
      for (int l = 0; l < LPT; ++l) acc[l] = mk<R>(0, 0);
      if (CM) {
        const T* M = (const T*)Ms + j * nin;
#pragma unroll
        for (int i = 0; i < NMAX; ++i)
          if (i < nin) {
            const T m = M[i];
#pragma unroll
            for (int l = 0; l < LPT; ++l) cfma(acc[l], m, v[i][l]);
          }
      } else {
        const R* M = (const R*)Ms + j * nin;
#pragma unroll
        for (int i = 0; i < NMAX; ++i)
          if (i < nin) {
            const R m = M[i];
#pragma unroll
            for (int l = 0; l < LPT; ++l) {
              acc[l].x = fma(m, v[i][l].x, acc[l].x);
              acc[l].y = fma(m, v[i][l].y, acc[l].y);
            }
          }
      }
#pragma unroll
      for (int l = 0; l < LPT; ++l) {
        T r = acc[l];
        if (accumulate) r = cadd(r, op[j * step_out + l]);
        op[j * step_out + l] = r;
      }
    }
  }
}

template <typename R, bool CM, int NMAX, int LPT>
static void run_mode_line(const cpx_t<R>* in, View vin, cpx_t<R>* out, View vout, int64_t B, int C, int ax,
                          int nin, int e0, int e1, int e2, const void* M0, const void* M1, const int8_t* sel,
                          const int64_t* srcmap, bool accumulate, size_t smem, cudaStream_t s) {
  static SmemAttr attr;
  smem_attr_once(k_mode_line<R, CM, NMAX, LPT>, 96 * 1024, attr.v);
  const int ea = ax == 0 ? e1 : e0, eb = ax == 2 ? e1 : e2;
  int64_t lines = B * ea * eb * (int64_t)(C / LPT);
  int64_t blocks = ceil_div(lines, 128);
  if (blocks > 152 * 32) blocks = 152 * 32;
  k_mode_line<R, CM, NMAX, LPT><<<(unsigned)blocks, 128, smem, s>>>(in, vin, out, vout, B, C, ax, nin, e0, e1, e2,
                                                                     M0, M1, sel, srcmap, accumulate);
}

template <typename R, bool CM>
static bool dispatch_mode_line(const cpx_t<R>* in, View vin, cpx_t<R>* out, View vout, int64_t B, int C, int ax,
                               int nin, int e0, int e1, int e2, const void* M0, const void* M1,
                               const int8_t* sel, const int64_t* srcmap, bool accumulate, size_t smem,
                               cudaStream_t s) {
  const bool two = (C % 2) == 0 && sizeof(R) == 4;
#define EFIE_ML(NM)                                                                                          \
  if (nin <= NM) {                                                                                           \
    if constexpr (sizeof(R) == 4) {                                                                          \
      if (two) {                                                                                             \
        run_mode_line<R, CM, NM, 2>(in, vin, out, vout, B, C, ax, nin, e0, e1, e2, M0, M1, sel, srcmap,     \
                                    accumulate, smem, s);                                                    \
        return true;                                                                                         \
      }                                                                                                      \
    }                                                                                                        \
    run_mode_line<R, CM, NM, 1>(in, vin, out, vout, B, C, ax, nin, e0, e1, e2, M0, M1, sel, srcmap,         \
                                accumulate, smem, s);                                                        \
    return true;                                                                                             \
  }
  EFIE_ML(9)
  EFIE_ML(13)
  EFIE_ML(21)
#undef EFIE_ML
  return false;
}

// ---------------------------------------------------------------- tiled mode products
// Mode products along long axes (more than 21 splines in, or more than 40
// values): a small GEMM per group of 32 lines-of-16-bytes.  A block holds the
// matrix in shared memory for all of its groups, transposed to [in][out] and cut
// into tiles of 8 outputs; the group's input lines are staged by double-buffered
// 16-byte asynchronous copies; a warp owns JT outputs of all 32 units (a unit
// is two adjacent FP32 channels or one FP64 one), so one staged input value
// feeds JT outputs and one broadcast matrix value two (FP32) lines.
//   MODE 0: real matrix (M1 where sel says so), 1: complex, 2: rows f and n - f of
//   the forward transform from four real sums, 3: two sources, real (sibling-
//   shared upward transfer).
// Every output sums over its inputs in ascending order with the line kernels'
// sequence of multiply-adds, so the results are theirs bit for bit.
//
// What bounds it: the FP32 (or FP64) multiply-adds, 4 per complex product; shared
// memory takes 8 wavefronts for every 64 of them.  It replaces one thread per
// output, which read every input nout times and every matrix value from L1 (k_mode),
// and register-resident lines of up to 40 values, which spilled.  On a nonuniform
// tree with 32 boxes of 41^3 splines (77 frequencies per axis) and 52 of 25^3, 64
// vectors, ms: forward 333 -> 62, inverse 437 -> 63 (with k_mode_tile2 below), upward 181 -> 11, downward
// 27 -> 7.  Up to 21 inputs the register-resident line kernels stay: there the
// passes run near the memory bandwidth.
template <int MODE>
struct TileArgs {
  View vin, vout;
  int64_t items;   // groups over all boxes
  int ngrp;        // groups per box
  int C, ax, nin, nout, ea, eb, n;
  const void *M0, *M1;
  const int8_t* sel;
  const int64_t* srcmap;
  bool accumulate;
  const int64_t *src0, *src1;
  const int8_t *bit0, *bit1;
};

__device__ __forceinline__ void tile_cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

template <typename R, int MODE, int JT>
__global__ void __launch_bounds__(320) k_mode_tile(const cpx_t<R>* __restrict__ in, cpx_t<R>* __restrict__ out,
                                                   const TileArgs<MODE> a) {
  using T = cpx_t<R>;
  constexpr int LPT = 16 / (int)sizeof(T);      // channels per unit
  constexpr bool CM = MODE == 1 || MODE == 2;
  using E = typename std::conditional<CM, T, R>::type;
  constexpr int NSRC = MODE == 3 ? 2 : 1;
  extern __shared__ __align__(16) unsigned char tile_smem[];
  const int nj = MODE == 2 ? a.n / 2 + 1 : a.nout;
  const int njt = (nj + JT - 1) / JT;
  const int nmat = (MODE == 0 && a.M1 && a.M1 != a.M0) || MODE == 3 ? 2 : 1;
  const int msz = a.nin * njt * 8;
  E* Ms = reinterpret_cast<E*>(tile_smem);                                          // [nmat][nin][njt][8]
  uint4* tl = reinterpret_cast<uint4*>(tile_smem + sizeof(E) * (size_t)msz * nmat); // [2][NSRC][nin][32]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
  for (int e = tid; e < msz * nmat; e += blockDim.x) {
    const int m = e / msz, r = e - m * msz, i = r / (njt * 8), q = r - i * (njt * 8), jt = q >> 3, jl = q & 7;
    const int j = jt * JT + jl;
    E v = E();
    if (jl < JT && j < nj) v = reinterpret_cast<const E*>(m ? a.M1 : a.M0)[(int64_t)j * a.nin + i];
    Ms[e] = v;
  }
  const int CL = a.C / LPT;
  const int units = a.ea * a.eb * CL;
  const int64_t sa_in = a.ax == 0 ? a.vin.s1 : a.vin.s0, sb_in = a.ax == 2 ? a.vin.s1 : a.vin.s2;
  const int64_t sa_out = a.ax == 0 ? a.vout.s1 : a.vout.s0, sb_out = a.ax == 2 ? a.vout.s1 : a.vout.s2;
  const int64_t step_in = a.ax == 0 ? a.vin.s0 : (a.ax == 1 ? a.vin.s1 : a.vin.s2);
  const int64_t step_out = a.ax == 0 ? a.vout.s0 : (a.ax == 1 ? a.vout.s1 : a.vout.s2);
  // offset of this lane's unit inside a box
  auto where = [&](int64_t item, int64_t& b, int& c, int& ia, int& ib) {
    b = item / a.ngrp;
    int u = (int)(item - b * a.ngrp) * 32 + lane;
    const bool ok = u < units;
    if (!ok) u = 0;
    c = (u % CL) * LPT;
    const int t = u / CL;
    ib = t % a.eb;
    ia = t / a.eb;
    return ok;
  };
  auto stage = [&](int64_t item, int buf) {
    int64_t b;
    int c, ia, ib;
    const bool ok = where(item, b, c, ia, ib);
    if (ok)
#pragma unroll
      for (int q = 0; q < NSRC; ++q) {
        const int64_t bs = MODE == 3 ? (q ? a.src1[b] : a.src0[b]) : a.srcmap ? a.srcmap[b] : b;
        if (bs < 0) continue;
        const T* ip = in + bs * a.vin.sb + ia * sa_in + ib * sb_in + c;
        uint4* d = tl + ((size_t)(buf * NSRC + q) * a.nin) * 32 + lane;
        for (int i = warp; i < a.nin; i += nw) tile_cp16(d + i * 32, ip + i * step_in);
      }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  int buf = 0;
  int64_t item = blockIdx.x;
  if (item < a.items) stage(item, 0);
  for (; item < a.items; item += gridDim.x, buf ^= 1) {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();  // this group's lines are in (and Ms, the first time); the other buffer is free
    if (item + gridDim.x < a.items) stage(item + gridDim.x, buf ^ 1);
    int64_t b;
    int c, ia, ib;
    const bool ok = where(item, b, c, ia, ib);
    T* op = out + b * a.vout.sb + ia * sa_out + ib * sb_out + c;
    const E* Ma = Ms;
    const E* Mb = Ms;
    bool have0 = true, have1 = false;
    if (MODE == 0 && nmat == 2 && a.sel && a.sel[3 * b + a.ax]) Ma += msz;
    if (MODE == 3) {
      have0 = a.src0[b] >= 0, have1 = a.src1[b] >= 0;
      if (a.bit0[b]) Ma += msz;
      if (have1 && a.bit1[b]) Mb += msz;
    }
    const uint4* t0 = tl + ((size_t)buf * NSRC * a.nin) * 32 + lane;
    const uint4* t1 = t0 + (size_t)a.nin * 32;
    for (int jt = warp; jt < njt; jt += nw) {
      R acc[JT][MODE == 2 ? 4 * LPT : 2 * LPT];
#pragma unroll
      for (int j = 0; j < JT; ++j)
#pragma unroll
        for (int q = 0; q < (MODE == 2 ? 4 * LPT : 2 * LPT); ++q) acc[j][q] = (R)0;
      auto run = [&](const uint4* tp, const E* M) {
        const E* m0 = M + jt * 8;
#pragma unroll 2
        for (int i = 0; i < a.nin; ++i) {
          const uint4 w = tp[i * 32];
          T v[LPT];
          if constexpr (LPT == 2) {
            v[0] = mk<R>((R)__uint_as_float(w.x), (R)__uint_as_float(w.y));
            v[1] = mk<R>((R)__uint_as_float(w.z), (R)__uint_as_float(w.w));
          } else {
            v[0] = mk<R>((R)__hiloint2double(w.y, w.x), (R)__hiloint2double(w.w, w.z));
          }
          E m[8];
          const uint4* mp = reinterpret_cast<const uint4*>(m0 + (size_t)i * njt * 8);
#pragma unroll
          for (int q = 0; q < (int)sizeof(E) * 8 / 16; ++q) reinterpret_cast<uint4*>(m)[q] = mp[q];
#pragma unroll
          for (int j = 0; j < JT; ++j)
#pragma unroll
            for (int l = 0; l < LPT; ++l) {
              if constexpr (MODE == 2) {
                acc[j][4 * l] = fma(m[j].x, v[l].x, acc[j][4 * l]);
                acc[j][4 * l + 1] = fma(m[j].y, v[l].y, acc[j][4 * l + 1]);
                acc[j][4 * l + 2] = fma(m[j].x, v[l].y, acc[j][4 * l + 2]);
                acc[j][4 * l + 3] = fma(m[j].y, v[l].x, acc[j][4 * l + 3]);
              } else if constexpr (MODE == 1) {
                acc[j][2 * l] = fma(m[j].x, v[l].x, acc[j][2 * l]);
                acc[j][2 * l] = fma(-m[j].y, v[l].y, acc[j][2 * l]);
                acc[j][2 * l + 1] = fma(m[j].x, v[l].y, acc[j][2 * l + 1]);
                acc[j][2 * l + 1] = fma(m[j].y, v[l].x, acc[j][2 * l + 1]);
              } else {
                acc[j][2 * l] = fma(m[j], v[l].x, acc[j][2 * l]);
                acc[j][2 * l + 1] = fma(m[j], v[l].y, acc[j][2 * l + 1]);
              }
            }
        }
      };
      if constexpr (MODE == 3) {
        if (have0 && !have1) run(t0, Ma);
        else if (have0) {
          // both sources of an input index before the next index
          const E *ma = Ma + jt * 8, *mb = Mb + jt * 8;
#pragma unroll 2
          for (int i = 0; i < a.nin; ++i) {
            const uint4 w[2] = {t0[i * 32], t1[i * 32]};
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              T v[LPT];
              if constexpr (LPT == 2) {
                v[0] = mk<R>((R)__uint_as_float(w[q].x), (R)__uint_as_float(w[q].y));
                v[1] = mk<R>((R)__uint_as_float(w[q].z), (R)__uint_as_float(w[q].w));
              } else {
                v[0] = mk<R>((R)__hiloint2double(w[q].y, w[q].x), (R)__hiloint2double(w[q].w, w[q].z));
              }
              E m[8];
              const uint4* mp = reinterpret_cast<const uint4*>((q ? mb : ma) + (size_t)i * njt * 8);
#pragma unroll
              for (int r = 0; r < (int)sizeof(E) * 8 / 16; ++r) reinterpret_cast<uint4*>(m)[r] = mp[r];
#pragma unroll
              for (int j = 0; j < JT; ++j)
#pragma unroll
                for (int l = 0; l < LPT; ++l) {
                  acc[j][2 * l] = fma(m[j], v[l].x, acc[j][2 * l]);
                  acc[j][2 * l + 1] = fma(m[j], v[l].y, acc[j][2 * l + 1]);
                }
            }
          }
        }
      } else {
        run(t0, Ma);
      }
      if (ok)
#pragma unroll
        for (int j = 0; j < JT; ++j) {
          const int jo = jt * JT + j;
          if (jo >= nj) break;
#pragma unroll
          for (int l = 0; l < LPT; ++l) {
            if constexpr (MODE == 2) {
              const R s1 = acc[j][4 * l], s2 = acc[j][4 * l + 1], s3 = acc[j][4 * l + 2], s4 = acc[j][4 * l + 3];
              op[jo * step_out + l] = mk<R>(s1 - s2, s3 + s4);
              if (jo != 0 && 2 * jo != a.n) op[(int64_t)(a.n - jo) * step_out + l] = mk<R>(s1 + s2, s3 - s4);
            } else {
              T r = mk<R>(acc[j][2 * l], acc[j][2 * l + 1]);
              if (a.accumulate) r = cadd(r, op[jo * step_out + l]);
              op[jo * step_out + l] = r;
            }
          }
        }
    }
  }
}

// The FP32 complex and paired passes (MODE 1 and 2) with two units (four lines)
// per lane: a broadcast matrix value feeds four lines instead of two, which
// halves the shared-memory returns per multiply-add.  The sums of JT outputs of
// four lines stay in registers (up to 168: twelve warps per SM, whatever the
// block size BT), a warp owns one tile of JT outputs, and the inputs come in
// pieces of 16 through a ring of three, so that three blocks of four warps fit on
// an SM with their matrices.  Same sums in the same order as k_mode_tile.
//
// What bounds it: issue slots (three quarters taken, four fifths of them
// multiply-adds; register-bank conflicts take most of the others).  41 -> 77
// complex outputs, 64 vectors, 32 boxes of 77 x 77 lines: 3.93 -> 3.59 ms; the
// transforms of that tree: forward 68.7 -> 62.1, inverse 69.1 -> 63.4 ms.  Reading
// the next input's values ahead by hand changed nothing.
constexpr int T2_PI = 16, T2_RD = 3;
template <int MODE, int JT, int BT>
__global__ void __launch_bounds__(BT, 384 / BT) k_mode_tile2(const float2* __restrict__ in, float2* __restrict__ out,
                                                             const TileArgs<MODE> a) {
  extern __shared__ __align__(16) unsigned char tile_smem[];
  const int nj = MODE == 2 ? a.n / 2 + 1 : a.nout;
  const int njt = (nj + JT - 1) / JT;
  constexpr int JP = JT + (JT & 1);  // matrix tile, padded to 16 bytes
  const int msz = a.nin * njt * JP;
  float2* Ms = reinterpret_cast<float2*>(tile_smem);               // [nin][njt][JP]
  float4* ring = reinterpret_cast<float4*>(Ms + msz);              // [T2_RD][T2_PI][64]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
  for (int e = tid; e < msz; e += blockDim.x) {
    const int i = e / (njt * JP), q = e - i * (njt * JP), jt = q / JP, jl = q - jt * JP, j = jt * JT + jl;
    Ms[e] = jl < JT && j < nj ? reinterpret_cast<const float2*>(a.M0)[(int64_t)j * a.nin + i] : make_float2(0.f, 0.f);
  }
  const int CL = a.C / 2, units = a.ea * a.eb * CL;
  const int64_t sa_in = a.ax == 0 ? a.vin.s1 : a.vin.s0, sb_in = a.ax == 2 ? a.vin.s1 : a.vin.s2;
  const int64_t sa_out = a.ax == 0 ? a.vout.s1 : a.vout.s0, sb_out = a.ax == 2 ? a.vout.s1 : a.vout.s2;
  const int64_t step_in = a.ax == 0 ? a.vin.s0 : (a.ax == 1 ? a.vin.s1 : a.vin.s2);
  const int64_t step_out = a.ax == 0 ? a.vout.s0 : (a.ax == 1 ? a.vout.s1 : a.vout.s2);
  // offset of unit 32 h + lane of an item in its box (-1: past the last)
  auto offset = [&](int64_t item, int h, bool output) -> int64_t {
    const int64_t b = item / a.ngrp;
    const int u = (int)(item - b * a.ngrp) * 64 + 32 * h + lane;
    if (u >= units) return -1;
    const int c = (u % CL) * 2, t = u / CL, ib = t % a.eb, ia = t / a.eb;
    return output ? b * a.vout.sb + ia * sa_out + ib * sb_out + c : b * a.vin.sb + ia * sa_in + ib * sb_in + c;
  };
  const int npc = (a.nin + T2_PI - 1) / T2_PI;
  // loader: pieces of the block's items in order
  int64_t litem = blockIdx.x, lo0 = -1, lo1 = -1;
  int lpc = 0;
  if (litem < a.items) lo0 = offset(litem, 0, false), lo1 = offset(litem, 1, false);
  auto load = [&](int slot) {
    if (litem < a.items) {
      float4* d = ring + slot * (T2_PI * 64) + lane;
      const int i0 = lpc * T2_PI, i1 = min(a.nin, i0 + T2_PI);
      for (int i = i0 + warp; i < i1; i += nw) {
        if (lo0 >= 0) tile_cp16(d + (i - i0) * 64, in + lo0 + i * step_in);
        if (lo1 >= 0) tile_cp16(d + (i - i0) * 64 + 32, in + lo1 + i * step_in);
      }
      if (++lpc == npc) {
        lpc = 0;
        litem += gridDim.x;
        if (litem < a.items) lo0 = offset(litem, 0, false), lo1 = offset(litem, 1, false);
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
#pragma unroll
  for (int q = 0; q < T2_RD - 1; ++q) load(q);
  int slot = 0;
  constexpr int NA = MODE == 2 ? 4 : 2;  // sums per output and line
  for (int64_t item = blockIdx.x; item < a.items; item += gridDim.x) {
    float acc[JT][4][NA];
#pragma unroll
    for (int j = 0; j < JT; ++j)
#pragma unroll
      for (int l = 0; l < 4; ++l)
#pragma unroll
        for (int q = 0; q < NA; ++q) acc[j][l][q] = 0.f;
    for (int pc = 0; pc < npc; ++pc) {
      asm volatile("cp.async.wait_group %0;\n" ::"n"(T2_RD - 2) : "memory");
      __syncthreads();  // this piece is in for every warp, and every warp has left the one before
      load(slot == 0 ? T2_RD - 1 : slot - 1);
      if (warp < njt) {
        const float4* tp = ring + slot * (T2_PI * 64) + lane;
        const int i0 = pc * T2_PI, cnt = min(T2_PI, a.nin - i0);
        const float4* mp = reinterpret_cast<const float4*>(Ms + ((size_t)i0 * njt + warp) * JP);
#pragma unroll 2
        for (int i = 0; i < cnt; ++i) {
          const float4 w0 = tp[i * 64], w1 = tp[i * 64 + 32];
          const float2 v[4] = {make_float2(w0.x, w0.y), make_float2(w0.z, w0.w), make_float2(w1.x, w1.y),
                               make_float2(w1.z, w1.w)};
          float2 m[JP];
#pragma unroll
          for (int q = 0; q < JP / 2; ++q) {
            const float4 t = mp[(size_t)i * njt * (JP / 2) + q];
            m[2 * q] = make_float2(t.x, t.y);
            m[2 * q + 1] = make_float2(t.z, t.w);
          }
#pragma unroll
          for (int j = 0; j < JT; ++j)
#pragma unroll
            for (int l = 0; l < 4; ++l) {
              if constexpr (MODE == 2) {
                acc[j][l][0] = fmaf(m[j].x, v[l].x, acc[j][l][0]);
                acc[j][l][1] = fmaf(m[j].y, v[l].y, acc[j][l][1]);
                acc[j][l][2] = fmaf(m[j].x, v[l].y, acc[j][l][2]);
                acc[j][l][3] = fmaf(m[j].y, v[l].x, acc[j][l][3]);
              } else {
                acc[j][l][0] = fmaf(m[j].x, v[l].x, acc[j][l][0]);
                acc[j][l][0] = fmaf(-m[j].y, v[l].y, acc[j][l][0]);
                acc[j][l][1] = fmaf(m[j].x, v[l].y, acc[j][l][1]);
                acc[j][l][1] = fmaf(m[j].y, v[l].x, acc[j][l][1]);
              }
            }
        }
      }
      slot = slot == T2_RD - 1 ? 0 : slot + 1;
    }
    if (warp < njt)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int64_t o = offset(item, h, true);
        if (o < 0) continue;
        float2* op = out + o;
#pragma unroll
        for (int j = 0; j < JT; ++j) {
          const int jo = warp * JT + j;
          if (jo >= nj) break;
          const float* p = acc[j][2 * h];
          const float* q = acc[j][2 * h + 1];
          if constexpr (MODE == 2) {
            *reinterpret_cast<float4*>(op + jo * step_out) =
                make_float4(p[0] - p[1], p[2] + p[3], q[0] - q[1], q[2] + q[3]);
            if (jo != 0 && 2 * jo != a.n)
              *reinterpret_cast<float4*>(op + (int64_t)(a.n - jo) * step_out) =
                  make_float4(p[0] + p[1], p[2] - p[3], q[0] + q[1], q[2] - q[3]);
          } else {
            float4 r = make_float4(p[0], p[1], q[0], q[1]);
            if (a.accumulate) {
              const float4 old = *reinterpret_cast<const float4*>(op + jo * step_out);
              r = make_float4(r.x + old.x, r.y + old.y, r.z + old.z, r.w + old.w);
            }
            *reinterpret_cast<float4*>(op + jo * step_out) = r;
          }
        }
      }
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
}

template <int MODE, int JT, int BT>
static void run_mode_tile2_bt(const float2* in, float2* out, const TileArgs<MODE>& a, int warps, size_t smem,
                              cudaStream_t s) {
  const int bps = (int)std::max<size_t>(1, std::min<size_t>(220 * 1024 / (smem + 1024), 384 / BT));
  static SmemAttr attr;
  smem_attr_once(k_mode_tile2<MODE, JT, BT>, (int)smem, attr.v);
  k_mode_tile2<MODE, JT, BT>
      <<<(unsigned)std::min<int64_t>(a.items, (int64_t)152 * bps), 32 * warps, smem, s>>>(in, out, a);
}
template <int MODE, int JT>
static bool run_mode_tile2(const float2* in, float2* out, int64_t B, TileArgs<MODE> a, cudaStream_t s) {
  const int nj = MODE == 2 ? a.n / 2 + 1 : a.nout, njt = (nj + JT - 1) / JT;
  const size_t smem = sizeof(float2) * (size_t)a.nin * njt * (JT + (JT & 1)) + (size_t)T2_RD * T2_PI * 64 * 16;
  const int64_t units = (int64_t)a.ea * a.eb * (a.C / 2);
  if (njt > 12 || smem > 200 * 1024 || units > 0x7fffffff - 64) return false;
  a.ngrp = (int)((units + 63) / 64);
  a.items = B * a.ngrp;
  if (a.items <= 0) return true;
  const int warps = std::max(njt, 4);  // spare warps help to load
  if (warps <= 4) run_mode_tile2_bt<MODE, JT, 128>(in, out, a, warps, smem, s);
  else if (warps <= 6) run_mode_tile2_bt<MODE, JT, 192>(in, out, a, warps, smem, s);
  else run_mode_tile2_bt<MODE, JT, 384>(in, out, a, warps, smem, s);
  return true;
}

// false when the matrix and two input buffers do not fit in shared memory, or
// when a unit's 16 bytes would not be aligned (an odd channel count in FP32)
template <typename R, int MODE>
static bool launch_mode_tile(const cpx_t<R>* in, cpx_t<R>* out, int64_t B, TileArgs<MODE> a, cudaStream_t s) {
  // FP32 complex passes: two units per lane, up to 12 tiles of outputs (84 to 96
  // outputs, 144 paired ones); beyond that k_mode_tile, whose warps take several
  // tiles in turn.  The tile that leaves less of its last one empty.
  if constexpr (sizeof(R) == 4 && (MODE == 1 || MODE == 2)) {
    if (a.C % 2 == 0 && !a.srcmap) {
      const auto pad = [&](int nj, int jt) { return (nj + jt - 1) / jt * jt; };
      if constexpr (MODE == 2) {
        const int nj = a.n / 2 + 1;
        if (pad(nj, 5) < pad(nj, 6) ? run_mode_tile2<MODE, 5>(in, out, B, a, s)
                                    : run_mode_tile2<MODE, 6>(in, out, B, a, s))
          return true;
      } else if (pad(a.nout, 7) < pad(a.nout, 8) ? run_mode_tile2<MODE, 7>(in, out, B, a, s)
                                                 : run_mode_tile2<MODE, 8>(in, out, B, a, s)) {
        return true;
      }
    }
  }
  constexpr int LPT = 16 / (int)sizeof(cpx_t<R>);
  constexpr bool CM = MODE == 1 || MODE == 2;
  if (a.C % LPT != 0) return false;
  const int nj = MODE == 2 ? a.n / 2 + 1 : a.nout;
  const int jt = ((nj + 6) / 7) * 7 < ((nj + 7) / 8) * 8 ? 7 : 8;  // the tile that leaves less of its last one empty
  const int njt = (nj + jt - 1) / jt;
  const int nmat = (MODE == 0 && a.M1 && a.M1 != a.M0) || MODE == 3 ? 2 : 1;
  const size_t smem = (CM ? 2 : 1) * sizeof(R) * (size_t)a.nin * njt * 8 * nmat +
                      (size_t)2 * (MODE == 3 ? 2 : 1) * a.nin * 512;
  if (smem > 200 * 1024) return false;
  const int64_t units = (int64_t)a.ea * a.eb * (a.C / LPT);
  if (units > 0x7fffffff - 32) return false;
  a.ngrp = (int)((units + 31) / 32);
  a.items = B * a.ngrp;
  if (a.items <= 0) return true;
  // warps share the staged lines: one per output tile, at most 10
  const int per = (njt + 9) / 10, warps = (njt + per - 1) / per;
  int bps = (int)std::min<size_t>(220 * 1024 / (smem + 1024), 2048 / (size_t)(32 * warps));
  bps = std::max(1, std::min(bps, 16));
  const int64_t blocks = std::min<int64_t>(a.items, (int64_t)152 * bps);
  if (jt == 7) {
    static SmemAttr attr;
    smem_attr_once(k_mode_tile<R, MODE, 7>, (int)smem, attr.v);
    k_mode_tile<R, MODE, 7><<<(unsigned)blocks, 32 * warps, smem, s>>>(in, out, a);
  } else {
    static SmemAttr attr;
    smem_attr_once(k_mode_tile<R, MODE, 8>, (int)smem, attr.v);
    k_mode_tile<R, MODE, 8><<<(unsigned)blocks, 32 * warps, smem, s>>>(in, out, a);
  }
  return true;
}

// ---------------------------------------------------------------- sibling-shared transfers
// Upward transfer as a tree over the children of each parent: the product
// q_P = sum_c (C_x(c) (x) C_y(c) (x) C_z(c)) q_c is taken one axis at a time,
// summing after each axis the (at most two) partial results that will see the
// same matrices on the remaining axes -- z for children sharing (b_x, b_y),
// then y for groups sharing b_x, then x.  Each output unit g of a pass is
// out[g] = M(bit0[g]) in[src0[g]] + M(bit1[g]) in[src1[g]] (src1 < 0: absent),
// M(0) = C^L, M(1) = C^R, real, applied along axis ax.  The intermediates are
// about a quarter of those of transferring every child separately.
template <typename R, int NMAX, int LPT>
__global__ void k_mode_pair(const cpx_t<R>* __restrict__ in, View vin, cpx_t<R>* __restrict__ out, View vout,
                            int64_t G, int C, int ax, int nin, int e0, int e1, int e2, const R* __restrict__ M0,
                            const R* __restrict__ M1, const int64_t* __restrict__ src0,
                            const int64_t* __restrict__ src1, const int8_t* __restrict__ bit0,
                            const int8_t* __restrict__ bit1) {
  using T = cpx_t<R>;
  extern __shared__ unsigned char smem_raw[];
  const int nout = ax == 0 ? e0 : (ax == 1 ? e1 : e2);
  const int msz = nout * nin;
  R* Ms = reinterpret_cast<R*>(smem_raw);  // [2][nout][nin]
  for (int i = threadIdx.x; i < msz; i += blockDim.x) {
    Ms[i] = M0[i];
    Ms[msz + i] = M1[i];
  }
  __syncthreads();
  const int ea = ax == 0 ? e1 : e0, eb = ax == 2 ? e1 : e2;
  const int64_t sa_in = ax == 0 ? vin.s1 : vin.s0, sb_in = ax == 2 ? vin.s1 : vin.s2;
  const int64_t sa_out = ax == 0 ? vout.s1 : vout.s0, sb_out = ax == 2 ? vout.s1 : vout.s2;
  const int64_t step_in = ax == 0 ? vin.s0 : (ax == 1 ? vin.s1 : vin.s2);
  const int64_t step_out = ax == 0 ? vout.s0 : (ax == 1 ? vout.s1 : vout.s2);
  const int CL = C / LPT;
  const int64_t lines = G * ea * eb * (int64_t)CL;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < lines;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t t = idx;
    const int c = (int)(t % CL) * LPT;
    t /= CL;
    const int ib = (int)(t % eb);
    t /= eb;
    const int ia = (int)(t % ea);
    const int64_t g = t / ea;
    // g0 < 0: an output without inputs (a leaf on the parent level of a
    // nonuniform tree), written as zeros
    const int64_t g0 = src0[g], g1 = src1[g];
    const T* ip0 = in + (g0 >= 0 ? g0 : 0) * vin.sb + ia * sa_in + ib * sb_in + c;
    const T* ip1 = in + (g1 >= 0 ? g1 : (g0 >= 0 ? g0 : 0)) * vin.sb + ia * sa_in + ib * sb_in + c;
    T v0[NMAX][LPT], v1[NMAX][LPT];
#pragma unroll
    for (int i = 0; i < NMAX; ++i)
      if (i < nin)
#pragma unroll
        for (int l = 0; l < LPT; ++l) {
          v0[i][l] = g0 >= 0 ? ip0[i * step_in + l] : mk<R>(0, 0);
          v1[i][l] = g1 >= 0 ? ip1[i * step_in + l] : mk<R>(0, 0);
        }
    const R* Ma = Ms + (bit0[g] ? msz : 0);
    const R* Mb = Ms + (g1 >= 0 && bit1[g] ? msz : 0);
    T* op = out + g * vout.sb + ia * sa_out + ib * sb_out + c;
    for (int j = 0; j < nout; ++j) {
      T acc[LPT];
#pragma unroll
      for (int l = 0; l < LPT; ++l) acc[l] = mk<R>(0, 0);
#pragma unroll
      for (int i = 0; i < NMAX; ++i)
        if (i < nin) {
          const R ma = Ma[j * nin + i], mb = Mb[j * nin + i];
#pragma unroll
          for (int l = 0; l < LPT; ++l) {
            acc[l].x = fma(ma, v0[i][l].x, acc[l].x);
            acc[l].y = fma(ma, v0[i][l].y, acc[l].y);
            acc[l].x = fma(mb, v1[i][l].x, acc[l].x);
            acc[l].y = fma(mb, v1[i][l].y, acc[l].y);
          }
        }
#pragma unroll
      for (int l = 0; l < LPT; ++l) op[j * step_out + l] = acc[l];
    }
  }
}

template <typename R>
void launch_mode_pair(const cpx_t<R>* in, View vin, cpx_t<R>* out, View vout, int64_t G, int C, int ax, int nin,
                      int e0, int e1, int e2, const R* M0, const R* M1, const int64_t* src0, const int64_t* src1,
                      const int8_t* bit0, const int8_t* bit1, cudaStream_t s) {
  const int ea = ax == 0 ? e1 : e0, eb = ax == 2 ? e1 : e2;
  const int nout = ax == 0 ? e0 : (ax == 1 ? e1 : e2);
  if (G <= 0) return;
  const size_t smem = 2 * sizeof(R) * (size_t)nout * nin;
  const bool two = (C % 2) == 0 && sizeof(R) == 4;
  const int lpt = two ? 2 : 1;
  const int64_t lines = G * ea * eb * (int64_t)(C / lpt);
  int64_t blocks = ceil_div(lines, 128);
  if (blocks > 152 * 32) blocks = 152 * 32;
#define EFIE_MP(NM)                                                                                          \
  if (nin <= NM) {                                                                                           \
    if (two && NM <= 9) {                                                                                    \
      auto k = k_mode_pair<R, NM, (sizeof(R) == 4 && NM <= 9) ? 2 : 1>;                                      \
      k<<<(unsigned)blocks, 128, smem, s>>>(in, vin, out, vout, G, C, ax, nin, e0, e1, e2, M0, M1, src0,    \
                                            src1, bit0, bit1);                                               \
    } else {                                                                                                 \
      const int64_t lines1 = G * ea * eb * (int64_t)C;                                                       \
      int64_t blocks1 = ceil_div(lines1, 128);                                                               \
      if (blocks1 > 152 * 32) blocks1 = 152 * 32;                                                            \
      auto k = k_mode_pair<R, NM, 1>;                                                                        \
      k<<<(unsigned)blocks1, 128, smem, s>>>(in, vin, out, vout, G, C, ax, nin, e0, e1, e2, M0, M1, src0,   \
                                             src1, bit0, bit1);                                              \
    }                                                                                                        \
    return;                                                                                                  \
  }
  EFIE_MP(9)
  EFIE_MP(13)
  EFIE_MP(21)
#undef EFIE_MP
  if (nin <= TRANSFER_MAX_SPLINES) {
    TileArgs<3> t{};
    t.vin = vin, t.vout = vout, t.C = C, t.ax = ax, t.nin = nin, t.nout = nout, t.ea = ea, t.eb = eb;
    t.M0 = M0, t.M1 = M1, t.src0 = src0, t.src1 = src1, t.bit0 = bit0, t.bit1 = bit1;
    if (launch_mode_tile<R, 3>(in, out, G, t, s)) return;
    throw EfieError{EFIE_EINVAL, "transfer: the parent level has too many splines per axis"};
  }
  throw EfieError{EFIE_EINVAL, "transfer: more than 40 splines per axis below the top level"};
}

// ---------------------------------------------------------------- fused sparse transfers
// Knot insertion touches few splines: where s doubles, a transfer matrix has
// little more than one nonzero per child spline (12 of 117 for 9 -> 13 splines).
// A thread owns 16 bytes (two FP32 channels or one FP64) of an output point and
// takes the nested sums over the nonzeros of its three matrix rows straight from
// the source grids, so the intermediates of the axis-by-axis passes never exist.
// The sums run in the passes' order (z inside y inside x; both children of an
// index before the next index) and leave out exact zeros only, so the results
// are theirs bit for bit.
//
// What bounds it: the chains of dependent loads, (nonzeros per row)^3 of 16 bytes
// per output -- 6.3 upward and 2.4 downward on average for 9 -> 13 splines, up to 216
// at a parent's centre.  So in FP32 rows of more than 8 loads keep the passes (11 -> 15
// splines, 22 upward: 0.31 ms in passes, 0.76 fused; 7 downward: 0.33 and 0.31); in
// FP64, where the passes multiply every zero on a pipe of two operations per
// clock, up to 40.  Dense constant-s transfers (three nonzeros per child spline)
// keep the passes.  Measured, ms, upward and downward: 10-wavelength sphere, FP32,
// 64 vectors 10.2 -> 8.2 and 10.2 -> 6.3; 4-wavelength sphere, FP64, 8 vectors 1.67 ->
// 0.28 and 1.29 -> 0.23.
template <typename R>
struct U16;
template <>
struct U16<float> {
  using T = float4;
  static __device__ __forceinline__ T zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  static __device__ __forceinline__ void fma1(float c, const T& v, T& a) {
    a.x = fmaf(c, v.x, a.x), a.y = fmaf(c, v.y, a.y), a.z = fmaf(c, v.z, a.z), a.w = fmaf(c, v.w, a.w);
  }
  static __device__ __forceinline__ T add(const T& a, const T& b) {
    return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
  }
};
template <>
struct U16<double> {
  using T = double2;
  static __device__ __forceinline__ T zero() { return make_double2(0.0, 0.0); }
  static __device__ __forceinline__ void fma1(double c, const T& v, T& a) {
    a.x = fma(c, v.x, a.x), a.y = fma(c, v.y, a.y);
  }
  static __device__ __forceinline__ T add(const T& a, const T& b) { return make_double2(a.x + b.x, a.y + b.y); }
};

// ptr [rows + 1], then idx and coef of the entries, into shared memory
template <typename R>
struct SparseRows {
  const int* ptr;
  const int* idx;
  const R* coef;
};
template <typename R>
__device__ __forceinline__ SparseRows<R> stage_rows(const SparseMat<R>& m, unsigned char* smem) {
  R* coef = reinterpret_cast<R*>(smem);
  int* idx = reinterpret_cast<int*>(coef + m.nnz);
  int* ptr = idx + m.nnz;
  for (int i = threadIdx.x; i < m.nnz; i += blockDim.x) coef[i] = m.coef[i], idx[i] = m.idx[i];
  for (int i = threadIdx.x; i <= m.rows; i += blockDim.x) ptr[i] = m.ptr[i];
  __syncthreads();
  return {ptr, idx, coef};
}

// parent grids from their children (child[8 pb + 4 bx + 2 by + bz], -1: none);
// entries of a row: child index * 2 + half, ascending
template <typename R>
__global__ void __launch_bounds__(256) k_up_fused(const typename U16<R>::T* __restrict__ q,
                                                  typename U16<R>::T* __restrict__ out, int ppb, int nb, int U, int sp,
                                                  int spp, const SparseMat<R> m, const int32_t* __restrict__ child) {
  using T = typename U16<R>::T;
  extern __shared__ __align__(16) unsigned char up_smem[];
  const SparseRows<R> rows = stage_rows(m, up_smem);
  const int64_t pb = blockIdx.x / nb;
  const int p0 = (int)(blockIdx.x - pb * nb) * ppb, npt = spp * spp * spp, csz = sp * sp * sp * U;
  int ch[8];
  {
    const int4 c0 = __ldg(reinterpret_cast<const int4*>(child + 8 * pb)),
               c1 = __ldg(reinterpret_cast<const int4*>(child + 8 * pb) + 1);
    ch[0] = c0.x, ch[1] = c0.y, ch[2] = c0.z, ch[3] = c0.w, ch[4] = c1.x, ch[5] = c1.y, ch[6] = c1.z, ch[7] = c1.w;
  }
  for (int e = threadIdx.x; e < ppb * U; e += blockDim.x) {
    const int pt = p0 + e / U, u = e % U;
    if (pt >= npt) break;
    const int Z = pt % spp, Y = (pt / spp) % spp, X = pt / (spp * spp);
    const int z0 = rows.ptr[Z], z1 = rows.ptr[Z + 1];
    T ax = U16<R>::zero();
    for (int ex = rows.ptr[X]; ex < rows.ptr[X + 1]; ++ex) {
      const int i = rows.idx[ex] >> 1;
      const bool bx = rows.idx[ex] & 1;
      const int h0 = bx ? ch[4] : ch[0], h1 = bx ? ch[5] : ch[1], h2 = bx ? ch[6] : ch[2], h3 = bx ? ch[7] : ch[3];
      if ((h0 & h1 & h2 & h3) < 0) continue;  // no child on this side (-1 each)
      T ay = U16<R>::zero();
      for (int ey = rows.ptr[Y]; ey < rows.ptr[Y + 1]; ++ey) {
        const int j = rows.idx[ey] >> 1;
        const bool by = rows.idx[ey] & 1;
        const int g0 = by ? h2 : h0, g1 = by ? h3 : h1;
        if ((g0 & g1) < 0) continue;
        // an absent child's terms are exact zeros: its sibling's values, coefficient 0
        const T* q0 = q + (int64_t)(g0 < 0 ? g1 : g0) * csz + (i * sp + j) * sp * U + u;
        const T* q1 = q + (int64_t)(g1 < 0 ? g0 : g1) * csz + (i * sp + j) * sp * U + u;
        T az = U16<R>::zero();
#pragma unroll 3
        for (int ez = z0; ez < z1; ++ez) {
          const int k = rows.idx[ez] >> 1;
          const bool bz = rows.idx[ez] & 1;
          const R c = (bz ? g1 : g0) < 0 ? (R)0 : rows.coef[ez];
          U16<R>::fma1(c, __ldg((bz ? q1 : q0) + k * U), az);
        }
        U16<R>::fma1(rows.coef[ey], az, ay);
      }
      U16<R>::fma1(rows.coef[ex], ay, ax);
    }
    out[(pb * npt + pt) * U + u] = ax;
  }
}

// child grids += their parents' (rows of m: half * sp + child spline, entries the
// parent splines ascending)
template <typename R>
__global__ void __launch_bounds__(256) k_down_fused(const typename U16<R>::T* __restrict__ r,
                                                    typename U16<R>::T* __restrict__ out, int ppb, int nb, int U,
                                                    int sp, int spp, const SparseMat<R> m,
                                                    const int64_t* __restrict__ parent,
                                                    const int8_t* __restrict__ bits) {
  using T = typename U16<R>::T;
  extern __shared__ __align__(16) unsigned char down_smem[];
  const SparseRows<R> rows = stage_rows(m, down_smem);
  const int64_t b = blockIdx.x / nb;
  const int p0 = (int)(blockIdx.x - b * nb) * ppb, npt = sp * sp * sp;
  const int kz = bits[3 * b + 2] ? sp : 0, ky = bits[3 * b + 1] ? sp : 0, kx = bits[3 * b] ? sp : 0;
  const T* rb = r + parent[b] * ((int64_t)spp * spp * spp * U);
  for (int e = threadIdx.x; e < ppb * U; e += blockDim.x) {
    const int pt = p0 + e / U, u = e % U;
    if (pt >= npt) break;
    const int k = pt % sp + kz, j = (pt / sp) % sp + ky, i = pt / (sp * sp) + kx;
    const int x0 = rows.ptr[i], x1 = rows.ptr[i + 1];
    T* op = out + (b * npt + pt) * U + u;
    const T old = *op;
    T az = U16<R>::zero();
    for (int ez = rows.ptr[k]; ez < rows.ptr[k + 1]; ++ez) {
      const int Z = rows.idx[ez];
      T ay = U16<R>::zero();
      for (int ey = rows.ptr[j]; ey < rows.ptr[j + 1]; ++ey) {
        const T* rp = rb + (rows.idx[ey] * spp + Z) * U + u;
        T ax = U16<R>::zero();
#pragma unroll 3
        for (int ex = x0; ex < x1; ++ex)
          U16<R>::fma1(rows.coef[ex], __ldg(rp + rows.idx[ex] * (spp * spp * U)), ax);
        U16<R>::fma1(rows.coef[ey], ax, ay);
      }
      U16<R>::fma1(rows.coef[ez], ay, az);
    }
    *op = U16<R>::add(az, old);
  }
}

template <typename R>
static size_t rows_smem(const SparseMat<R>& m) {
  return (size_t)m.nnz * (sizeof(R) + sizeof(int)) + sizeof(int) * (size_t)(m.rows + 1);
}
template <typename R>
void launch_up_fused(const cpx_t<R>* q, cpx_t<R>* out, int64_t Bp, int C, int sp, int spp, const SparseMat<R>& m,
                     const int32_t* child, cudaStream_t s) {
  using T = typename U16<R>::T;
  const int U = C * (int)sizeof(cpx_t<R>) / 16;
  if (Bp <= 0) return;
  // blocks of 1,024 units of one parent box (fewer where the boxes alone leave the chip empty)
  const int npt = spp * spp * spp;
  int ppb = std::max(1, 1024 / U);
  while (ppb > 1 && ppb * U > 256 && Bp * ceil_div(npt, ppb) < 152 * 8) ppb /= 2;
  const int nb = (int)ceil_div(npt, ppb);
  k_up_fused<R><<<(unsigned)(Bp * nb), 256, rows_smem(m), s>>>(reinterpret_cast<const T*>(q),
                                                               reinterpret_cast<T*>(out), ppb, nb, U, sp, spp, m,
                                                               child);
}
template <typename R>
void launch_down_fused(const cpx_t<R>* r, cpx_t<R>* out, int64_t B, int C, int sp, int spp, const SparseMat<R>& m,
                       const int64_t* parent, const int8_t* bits, cudaStream_t s) {
  using T = typename U16<R>::T;
  const int U = C * (int)sizeof(cpx_t<R>) / 16;
  if (B <= 0) return;
  const int npt = sp * sp * sp;
  int ppb = std::max(1, 1024 / U);
  while (ppb > 1 && ppb * U > 256 && B * ceil_div(npt, ppb) < 152 * 8) ppb /= 2;
  const int nb = (int)ceil_div(npt, ppb);
  k_down_fused<R><<<(unsigned)(B * nb), 256, rows_smem(m), s>>>(reinterpret_cast<const T*>(r),
                                                                reinterpret_cast<T*>(out), ppb, nb, U, sp, spp, m,
                                                                parent, bits);
}

// ---------------------------------------------------------------- DFT passes
// The transform passes apply M = F P (forward, n x s') or M = P^T F^{-1}
// (inverse, s' x n) along one axis, F the n-point DFT and P real.  Because F's
// rows f and n - f (columns, for F^{-1}) are complex conjugates and P is real,
// M[n-f] = conj(M[f]) (forward) and M[:, n-f] = conj(M[:, f]) (inverse), so a
// pair of outputs (inputs) shares one set of real products:
//   forward: with M[f] = A + iB and four real sums S1 = sum A Re v,
//            S2 = sum B Im v, S3 = sum A Im v, S4 = sum B Re v,
//            y_f = (S1 - S2) + i (S3 + S4), y_{n-f} = (S1 + S2) + i (S3 - S4);
//   inverse: M v_f + conj(M) v_{n-f} = A u + i B w with u = v_f + v_{n-f},
//            w = v_f - v_{n-f}.
// That is half the multiply-adds of the dense product, with only rows
// (columns) 0 .. n/2 of M read.  Same line mapping as k_mode_line.
template <typename R, int NMAX, int LPT>
__global__ void k_dft_fwd_line(const cpx_t<R>* __restrict__ in, View vin, cpx_t<R>* __restrict__ out, View vout,
                               int64_t B, int C, int ax, int nin, int e0, int e1, int e2,
                               const cpx_t<R>* __restrict__ M, int n) {
  using T = cpx_t<R>;
  extern __shared__ unsigned char smem_raw[];
  T* Ms = reinterpret_cast<T*>(smem_raw);  // rows 0 .. n/2 of M
  const int nh = n / 2 + 1;
  for (int i = threadIdx.x; i < nh * nin; i += blockDim.x) Ms[i] = M[i];
  __syncthreads();
  const int ea = ax == 0 ? e1 : e0, eb = ax == 2 ? e1 : e2;
  const int64_t sa_in = ax == 0 ? vin.s1 : vin.s0, sb_in = ax == 2 ? vin.s1 : vin.s2;
  const int64_t sa_out = ax == 0 ? vout.s1 : vout.s0, sb_out = ax == 2 ? vout.s1 : vout.s2;
  const int64_t step_in = ax == 0 ? vin.s0 : (ax == 1 ? vin.s1 : vin.s2);
  const int64_t step_out = ax == 0 ? vout.s0 : (ax == 1 ? vout.s1 : vout.s2);
  const int CL = C / LPT;
  const int64_t lines = B * ea * eb * (int64_t)CL;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < lines;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t t = idx;
    const int c = (int)(t % CL) * LPT;
    t /= CL;
    const int ib = (int)(t % eb);
    t /= eb;
    const int ia = (int)(t % ea);
    const int64_t b = t / ea;
    const T* ip = in + b * vin.sb + ia * sa_in + ib * sb_in + c;
    T v[NMAX][LPT];
#pragma unroll
    for (int i = 0; i < NMAX; ++i)
      if (i < nin)
#pragma unroll
        for (int l = 0; l < LPT; ++l) v[i][l] = ip[i * step_in + l];
    T* op = out + b * vout.sb + ia * sa_out + ib * sb_out + c;
    for (int f = 0; f < nh; ++f) {
      R s1[LPT], s2[LPT], s3[LPT], s4[LPT];
#pragma unroll
      for (int l = 0; l < LPT; ++l) s1[l] = s2[l] = s3[l] = s4[l] = (R)0;
      const T* Mr = Ms + f * nin;
#pragma unroll
      for (int i = 0; i < NMAX; ++i)
        if (i < nin) {
          const T m = Mr[i];
#pragma unroll
          for (int l = 0; l < LPT; ++l) {
            s1[l] = fma(m.x, v[i][l].x, s1[l]);
            s2[l] = fma(m.y, v[i][l].y, s2[l]);
            s3[l] = fma(m.x, v[i][l].y, s3[l]);
            s4[l] = fma(m.y, v[i][l].x, s4[l]);
          }
        }
      const bool pair = f != 0 && 2 * f != n;
#pragma unroll
      for (int l = 0; l < LPT; ++l) {
        op[f * step_out + l] = mk<R>(s1[l] - s2[l], s3[l] + s4[l]);
        if (pair) op[(n - f) * step_out + l] = mk<R>(s1[l] + s2[l], s3[l] - s4[l]);
      }
    }
  }
}

// Inverse passes keep the nout (= s') outputs of a line in registers and
// stream the conjugate input pairs (f, n - f) through them.
template <typename R, int AMAX>
__global__ void k_dft_inv_line(const cpx_t<R>* __restrict__ in, View vin, cpx_t<R>* __restrict__ out, View vout,
                               int64_t B, int C, int ax, int nin_unused, int e0, int e1, int e2,
                               const cpx_t<R>* __restrict__ M, int n) {
  using T = cpx_t<R>;
  extern __shared__ unsigned char smem_raw[];
  T* Ms = reinterpret_cast<T*>(smem_raw);  // [f][a], f = 0 .. n/2
  const int nout = ax == 0 ? e0 : (ax == 1 ? e1 : e2);
  const int nh = n / 2 + 1;
  for (int i = threadIdx.x; i < nout * nh; i += blockDim.x) {
    const int f = i / nout, a = i - f * nout;
    Ms[i] = M[(int64_t)a * n + f];
  }
  __syncthreads();
  const int ea = ax == 0 ? e1 : e0, eb = ax == 2 ? e1 : e2;
  const int64_t sa_in = ax == 0 ? vin.s1 : vin.s0, sb_in = ax == 2 ? vin.s1 : vin.s2;
  const int64_t sa_out = ax == 0 ? vout.s1 : vout.s0, sb_out = ax == 2 ? vout.s1 : vout.s2;
  const int64_t step_in = ax == 0 ? vin.s0 : (ax == 1 ? vin.s1 : vin.s2);
  const int64_t step_out = ax == 0 ? vout.s0 : (ax == 1 ? vout.s1 : vout.s2);
  const int64_t lines = B * ea * eb * (int64_t)C;
  const int np = (n - 1) / 2;     // conjugate pairs (f, n - f), f = 1 .. np
  const bool mid = (n % 2) == 0;  // f = n/2 pairs with itself
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < lines;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t t = idx;
    const int c = (int)(t % C);
    t /= C;
    const int ib = (int)(t % eb);
    t /= eb;
    const int ia = (int)(t % ea);
    const int64_t b = t / ea;
    const T* ip = in + b * vin.sb + ia * sa_in + ib * sb_in + c;
    T acc[AMAX];
    {
      const T v0 = ip[0];
#pragma unroll
      for (int a = 0; a < AMAX; ++a)
        if (a < nout) acc[a] = cmul(Ms[a], v0);
    }
    T z1 = np > 0 ? ip[step_in] : mk<R>(0, 0), z2 = np > 0 ? ip[(int64_t)(n - 1) * step_in] : mk<R>(0, 0);
    for (int f = 1; f <= np; ++f) {
      const T u = mk<R>(z1.x + z2.x, z1.y + z2.y), w = mk<R>(z1.x - z2.x, z1.y - z2.y);
      if (f < np) {  // next pair's loads in flight during this pair's products
        z1 = ip[(int64_t)(f + 1) * step_in];
        z2 = ip[(int64_t)(n - f - 1) * step_in];
      }
      const T* Mr = Ms + f * nout;
#pragma unroll
      for (int a = 0; a < AMAX; ++a)
        if (a < nout) {
          const T m = Mr[a];
          acc[a].x = fma(m.x, u.x, acc[a].x);
          acc[a].x = fma(-m.y, w.y, acc[a].x);
          acc[a].y = fma(m.x, u.y, acc[a].y);
          acc[a].y = fma(m.y, w.x, acc[a].y);
        }
    }
    if (mid) {
      const T* Mr = Ms + (n / 2) * nout;
      const T vm = ip[(int64_t)(n / 2) * step_in];
#pragma unroll
      for (int a = 0; a < AMAX; ++a)
        if (a < nout) cfma(acc[a], Mr[a], vm);
    }
    T* op = out + b * vout.sb + ia * sa_out + ib * sb_out + c;
#pragma unroll
    for (int a = 0; a < AMAX; ++a)
      if (a < nout) op[a * step_out] = acc[a];
  }
}

// FP64 passes with the mirror symmetry as well.  P is symmetric under reversal of
// both its axes, so with the rows of M turned by a phase, H[f] = e^{-i theta_f} M[f],
// e^{2 i theta_f} = w^{f (shat - 1)}, H[f][s' - 1 - j] = conj(H[f][j]): inputs j and s' - 1 - j
// fold into u = v_j + v_j', w = v_j - v_j' and
//   y_f = P1 + i P2, y_{n-f} = P1 - i P2,  P1 = sum Re H u, P2 = sum Im H w,
// half the multiply-adds of the conjugate pairing alone; the outputs of the inverse
// pass fold the same way.  The phases of the forward and the inverse pass
// cancel across the translation, which multiplies frequency by frequency, so
// spectra are simply kept turned.  FP64 is bound by its pipe (two operations per
// clock and SM).  4-wavelength sphere, 8 vectors, ms: forward 6.0 -> 3.6, inverse
// 5.9 -> 3.4.  (FP32 passes are bound by memory and keep their order of sums.)
// Blocks of one warp where larger ones would leave SMs without work.
template <int NH>
__global__ void __launch_bounds__(128) k_dft_fwd_fold(const double2* __restrict__ in, View vin,
                                                      double2* __restrict__ out, View vout, int64_t B, int C, int ax,
                                                      int nin, int e0, int e1, int e2, const double2* __restrict__ M,
                                                      int n) {
  extern __shared__ unsigned char smem_raw[];
  double2* Ms = reinterpret_cast<double2*>(smem_raw);  // [f][h], f = 0 .. n/2, h = columns 0 .. (nin - 1) / 2
  const int nh = n / 2 + 1, hc = (nin + 1) / 2, half = nin / 2;
  for (int i = threadIdx.x; i < nh * hc; i += blockDim.x) Ms[i] = M[(i / hc) * nin + i % hc];
  __syncthreads();
  const int ea = ax == 0 ? e1 : e0, eb = ax == 2 ? e1 : e2;
  const int64_t sa_in = ax == 0 ? vin.s1 : vin.s0, sb_in = ax == 2 ? vin.s1 : vin.s2;
  const int64_t sa_out = ax == 0 ? vout.s1 : vout.s0, sb_out = ax == 2 ? vout.s1 : vout.s2;
  const int64_t step_in = ax == 0 ? vin.s0 : (ax == 1 ? vin.s1 : vin.s2);
  const int64_t step_out = ax == 0 ? vout.s0 : (ax == 1 ? vout.s1 : vout.s2);
  const int64_t lines = B * ea * eb * (int64_t)C;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < lines;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t t = idx;
    const int c = (int)(t % C);
    t /= C;
    const int ib = (int)(t % eb);
    t /= eb;
    const int ia = (int)(t % ea);
    const int64_t b = t / ea;
    const double2* ip = in + b * vin.sb + ia * sa_in + ib * sb_in + c;
    double2 u[NH], w[NH], mid = make_double2(0, 0);
#pragma unroll
    for (int j = 0; j < NH; ++j)
      if (j < half) {
        const double2 p = ip[j * step_in], q = ip[(int64_t)(nin - 1 - j) * step_in];
        u[j] = cadd(p, q);
        w[j] = csub(p, q);
      }
    if (hc > half) mid = ip[half * step_in];
    double2* op = out + b * vout.sb + ia * sa_out + ib * sb_out + c;
    for (int f = 0; f < nh; ++f) {
      const double2* Mr = Ms + f * hc;
      double2 p1 = make_double2(0, 0), p2 = p1;
#pragma unroll
      for (int j = 0; j < NH; ++j)
        if (j < half) {
          const double2 m = Mr[j];
          p1.x = fma(m.x, u[j].x, p1.x);
          p1.y = fma(m.x, u[j].y, p1.y);
          p2.x = fma(m.y, w[j].x, p2.x);
          p2.y = fma(m.y, w[j].y, p2.y);
        }
      if (hc > half) {
        const double m = Mr[half].x;
        p1.x = fma(m, mid.x, p1.x);
        p1.y = fma(m, mid.y, p1.y);
      }
      op[f * step_out] = make_double2(p1.x - p2.y, p1.y + p2.x);
      if (f != 0) op[(int64_t)(n - f) * step_out] = make_double2(p1.x + p2.y, p1.y - p2.x);
    }
  }
}
template <int NH>
__global__ void __launch_bounds__(128) k_dft_inv_fold(const double2* __restrict__ in, View vin,
                                                      double2* __restrict__ out, View vout, int64_t B, int C, int ax,
                                                      int e0, int e1, int e2, const double2* __restrict__ M, int n) {
  extern __shared__ unsigned char smem_raw[];
  double2* Ms = reinterpret_cast<double2*>(smem_raw);  // [f][a], f = 0 .. n/2, a = 0 .. (nout - 1) / 2
  const int nout = ax == 0 ? e0 : (ax == 1 ? e1 : e2);
  const int nh = n / 2 + 1, hc = (nout + 1) / 2, half = nout / 2;
  for (int i = threadIdx.x; i < nh * hc; i += blockDim.x) Ms[i] = M[(int64_t)(i % hc) * n + i / hc];
  __syncthreads();
  const int ea = ax == 0 ? e1 : e0, eb = ax == 2 ? e1 : e2;
  const int64_t sa_in = ax == 0 ? vin.s1 : vin.s0, sb_in = ax == 2 ? vin.s1 : vin.s2;
  const int64_t sa_out = ax == 0 ? vout.s1 : vout.s0, sb_out = ax == 2 ? vout.s1 : vout.s2;
  const int64_t step_in = ax == 0 ? vin.s0 : (ax == 1 ? vin.s1 : vin.s2);
  const int64_t step_out = ax == 0 ? vout.s0 : (ax == 1 ? vout.s1 : vout.s2);
  const int64_t lines = B * ea * eb * (int64_t)C;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < lines;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t t = idx;
    const int c = (int)(t % C);
    t /= C;
    const int ib = (int)(t % eb);
    t /= eb;
    const int ia = (int)(t % ea);
    const int64_t b = t / ea;
    const double2* ip = in + b * vin.sb + ia * sa_in + ib * sb_in + c;
    double2 E[NH], O[NH], mid = make_double2(0, 0);
    const double2 v0 = ip[0];
#pragma unroll
    for (int a = 0; a < NH; ++a)
      if (a < half) {
        E[a] = make_double2(Ms[a].x * v0.x, Ms[a].x * v0.y);
        O[a] = make_double2(0, 0);
      }
    if (hc > half) mid = make_double2(Ms[half].x * v0.x, Ms[half].x * v0.y);
    double2 z1 = nh > 1 ? ip[step_in] : v0, z2 = nh > 1 ? ip[(int64_t)(n - 1) * step_in] : v0;
    for (int f = 1; f < nh; ++f) {
      const double2 u = cadd(z1, z2), w = csub(z1, z2);
      if (f + 1 < nh) {  // next pair's loads in flight during this pair's products
        z1 = ip[(int64_t)(f + 1) * step_in];
        z2 = ip[(int64_t)(n - f - 1) * step_in];
      }
      const double2* Mr = Ms + f * hc;
#pragma unroll
      for (int a = 0; a < NH; ++a)
        if (a < half) {
          const double2 m = Mr[a];
          E[a].x = fma(m.x, u.x, E[a].x);
          E[a].y = fma(m.x, u.y, E[a].y);
          O[a].x = fma(m.y, w.x, O[a].x);
          O[a].y = fma(m.y, w.y, O[a].y);
        }
      if (hc > half) {
        mid.x = fma(Mr[half].x, u.x, mid.x);
        mid.y = fma(Mr[half].x, u.y, mid.y);
      }
    }
    double2* op = out + b * vout.sb + ia * sa_out + ib * sb_out + c;
#pragma unroll
    for (int a = 0; a < NH; ++a)
      if (a < half) {
        op[a * step_out] = make_double2(E[a].x - O[a].y, E[a].y + O[a].x);
        op[(int64_t)(nout - 1 - a) * step_out] = make_double2(E[a].x + O[a].y, E[a].y - O[a].x);
      }
    if (hc > half) op[half * step_out] = mid;
  }
}

// the folded pass, for turned matrices (see above) of odd length n and up to 21
// splines; false where it does not apply
bool launch_dft_fold(const double2* in, View vin, double2* out, View vout, int64_t B, int C, int ax, int nin, int e0,
                     int e1, int e2, const double2* M, int n, bool inverse, cudaStream_t s) {
  const int ea = ax == 0 ? e1 : e0, eb = ax == 2 ? e1 : e2;
  const int ns = inverse ? (ax == 0 ? e0 : (ax == 1 ? e1 : e2)) : nin, half = ns / 2;
  const int64_t lines = B * ea * eb * (int64_t)C;
  if (half > 10 || n % 2 == 0) return false;
  if (lines <= 0) return true;
  const size_t smem = sizeof(double2) * (size_t)(n / 2 + 1) * ((ns + 1) / 2);
  if (smem > 48 * 1024) return false;
  const int th = ceil_div(lines, 128) < 152 * 2 ? 32 : 128;
  const unsigned blocks = (unsigned)std::min<int64_t>(ceil_div(lines, th), (int64_t)152 * 32 * (128 / th));
#define EFIE_FOLD(NH)                                                                                       \
  if (half <= NH) {                                                                                         \
    if (inverse) k_dft_inv_fold<NH><<<blocks, th, smem, s>>>(in, vin, out, vout, B, C, ax, e0, e1, e2, M, n); \
    else k_dft_fwd_fold<NH><<<blocks, th, smem, s>>>(in, vin, out, vout, B, C, ax, nin, e0, e1, e2, M, n);   \
    return true;                                                                                            \
  }
  EFIE_FOLD(4)
  EFIE_FOLD(6)
  EFIE_FOLD(10)
#undef EFIE_FOLD
  return false;
}

// Fused second and third passes (FP32, 32 channels), one block per
// (box, x-frequency) slab.  Forward: the slab t[b][fx][y][z][c] (SP x SP x 32
// values, the output of the x pass) is staged in shared memory; a warp takes
// a pair of y-frequencies (fy, n - fy), lane = channel, forms the two rows
// T[z] of the y pass in registers (the conjugate-row pairing of the line
// kernels) and from each row the n z-frequencies, which it stores straight
// into the spectrum layout Q[fx][fy][fz][b][c] (256 contiguous bytes per
// warp store).  The y-pass intermediate never goes to HBM: per box the pass
// pair reads n SP^2 and writes n^3 values instead of reading and writing
// n SP^2 + n^2 SP.  What bounds it: issue slots (two thirds taken) with HBM at
// 4.5 TB/s.  1,016 boxes of 9^3 splines, 16 vectors: 215 -> 175 us (one matrix read per
// row and a warp of eight idle before).
template <int SP>
__global__ void __launch_bounds__(256, SP == 9 ? 3 : 1)
    k_dft_fwd_yz(const float2* __restrict__ in, float2* __restrict__ out, int64_t B, const float2* __restrict__ M,
                 int n) {
  extern __shared__ float4 fyz_smem[];
  float2* slab = reinterpret_cast<float2*>(fyz_smem);  // [SP][SP][32]
  float2* Ms = slab + SP * SP * 32;                    // rows 0 .. n/2 of M, [f][SP]
  const int nh = n / 2 + 1;
  const int64_t sl = blockIdx.x;
  const int64_t b = sl / n;
  const int fx = (int)(sl - b * n);
  {
    const float4* src = reinterpret_cast<const float4*>(in + sl * (SP * SP * 32));
    float4* dst = reinterpret_cast<float4*>(slab);
    for (int i = threadIdx.x; i < SP * SP * 16; i += blockDim.x) tile_cp16(dst + i, src + i);
    for (int i = threadIdx.x; i < nh * SP; i += blockDim.x) Ms[i] = M[i];
    asm volatile("cp.async.wait_all;\n" ::: "memory");
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int64_t fstride = B * 32;  // between consecutive z-frequencies
  for (int fy = warp; fy < nh; fy += nw) {
    // y pass: a[z] = (S1, S3), c[z] = (S2, S4) over the slab's y lines
    float2 t0[SP], t1[SP];
#pragma unroll
    for (int z = 0; z < SP; ++z) t0[z] = t1[z] = make_float2(0.f, 0.f);
    const float2* Mr = Ms + fy * SP;
#pragma unroll 1
    for (int y = 0; y < SP; ++y) {
      const float2 m = Mr[y];
      const float2* sv = slab + y * SP * 32 + lane;
#pragma unroll
      for (int z = 0; z < SP; ++z) {
        const float2 v = sv[z * 32];
        t0[z].x = fmaf(m.x, v.x, t0[z].x);
        t0[z].y = fmaf(m.x, v.y, t0[z].y);
        t1[z].x = fmaf(m.y, v.y, t1[z].x);
        t1[z].y = fmaf(m.y, v.x, t1[z].y);
      }
    }
    // rows fy and n - fy: (S1 - S2) + i (S3 + S4) and (S1 + S2) + i (S3 - S4)
#pragma unroll
    for (int z = 0; z < SP; ++z) {
      const float2 a = t0[z], c = t1[z];
      t0[z] = make_float2(a.x - c.x, a.y + c.y);
      t1[z] = make_float2(a.x + c.x, a.y - c.y);
    }
    // a matrix value serves both rows
    float2* op = out + (((int64_t)fx * n + fy) * n * B + b) * 32 + lane;
    float2* oq = out + (((int64_t)fx * n + (n - fy)) * n * B + b) * 32 + lane;
    const bool ypair = fy != 0 && 2 * fy != n;
    for (int fz = 0; fz < nh; ++fz) {
      const float2* Mz = Ms + fz * SP;
      const bool zpair = fz != 0 && 2 * fz != n;
      float s1 = 0.f, s2 = 0.f, s3 = 0.f, s4 = 0.f, r1 = 0.f, r2 = 0.f, r3 = 0.f, r4 = 0.f;
#pragma unroll
      for (int z = 0; z < SP; ++z) {
        const float2 m = Mz[z];
        s1 = fmaf(m.x, t0[z].x, s1);
        s2 = fmaf(m.y, t0[z].y, s2);
        s3 = fmaf(m.x, t0[z].y, s3);
        s4 = fmaf(m.y, t0[z].x, s4);
        r1 = fmaf(m.x, t1[z].x, r1);
        r2 = fmaf(m.y, t1[z].y, r2);
        r3 = fmaf(m.x, t1[z].y, r3);
        r4 = fmaf(m.y, t1[z].x, r4);
      }
      op[fz * fstride] = make_float2(s1 - s2, s3 + s4);
      if (zpair) op[(int64_t)(n - fz) * fstride] = make_float2(s1 + s2, s3 - s4);
      if (ypair) {
        oq[fz * fstride] = make_float2(r1 - r2, r3 + r4);
        if (zpair) oq[(int64_t)(n - fz) * fstride] = make_float2(r1 + r2, r3 - r4);
      }
    }
  }
}

// k_dft_inv_line for FP32 and pairs of channels with a thread's whole input line in
// flight: the n values of 16 bytes go to the thread's own column of shared memory
// by asynchronous copies, without registers (four pairs ahead in registers cost
// more in resident warps than they gave: 37.7 -> 43.1 ms for all inverse passes of 300,000
// unknowns, 64 vectors; this form with k_dft_inv_zy below 24.2).  Same sums in the same
// order.
//
// What bounds it: HBM, 5.1 to 5.9 TB/s on the larger passes (4.2 before).  13^3 splines,
// 816 MB: 214 -> 146 us.
template <int AMAX>
__global__ void __launch_bounds__(128) k_dft_inv_stage(const float2* __restrict__ in, View vin,
                                                       float2* __restrict__ out, View vout, int64_t B, int C, int ax,
                                                       int e0, int e1, int e2, const float2* __restrict__ M, int n) {
  extern __shared__ float4 izy_smem[];
  constexpr int AP = AMAX + (AMAX & 1);
  float4* S = izy_smem + threadIdx.x;                        // [n][128], this thread's column
  float2* Ms = reinterpret_cast<float2*>(izy_smem + n * 128);  // [f][a < AP], f = 0 .. n/2
  const int nout = ax == 0 ? e0 : (ax == 1 ? e1 : e2);
  const int nh = n / 2 + 1;
  for (int i = threadIdx.x; i < nh * AP; i += blockDim.x) {
    const int f = i / AP, a = i - f * AP;
    Ms[i] = a < nout ? M[(int64_t)a * n + f] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  const int ea = ax == 0 ? e1 : e0, eb = ax == 2 ? e1 : e2;
  const int64_t sa_in = ax == 0 ? vin.s1 : vin.s0, sb_in = ax == 2 ? vin.s1 : vin.s2;
  const int64_t sa_out = ax == 0 ? vout.s1 : vout.s0, sb_out = ax == 2 ? vout.s1 : vout.s2;
  const int64_t step_in = ax == 0 ? vin.s0 : (ax == 1 ? vin.s1 : vin.s2);
  const int64_t step_out = ax == 0 ? vout.s0 : (ax == 1 ? vout.s1 : vout.s2);
  const int CL = C / 2;
  const int64_t lines = B * ea * eb * (int64_t)CL;
  const int np = (n - 1) / 2;     // conjugate pairs (f, n - f), f = 1 .. np
  const bool mid = (n % 2) == 0;  // f = n/2 pairs with itself
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < lines;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t t = idx;
    const int c = (int)(t % CL) * 2;
    t /= CL;
    const int ib = (int)(t % eb);
    t /= eb;
    const int ia = (int)(t % ea);
    const int64_t b = t / ea;
    const float2* ip = in + b * vin.sb + ia * sa_in + ib * sb_in + c;
    for (int f = 0; f < n; ++f) tile_cp16(S + f * 128, ip + f * step_in);
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    float2 acc[AP][2];
    const float4* Mr = reinterpret_cast<const float4*>(Ms);
    {
      const float4 v = S[0];
      const float2 v0[2] = {make_float2(v.x, v.y), make_float2(v.z, v.w)};
#pragma unroll
      for (int a = 0; a < AP; a += 2) {
        const float4 m = Mr[a / 2];
#pragma unroll
        for (int l = 0; l < 2; ++l) {
          acc[a][l] = cmul(make_float2(m.x, m.y), v0[l]);
          acc[a + 1][l] = cmul(make_float2(m.z, m.w), v0[l]);
        }
      }
    }
#pragma unroll 2
    for (int f = 1; f <= np; ++f) {
      const float4 z1 = S[f * 128], z2 = S[(n - f) * 128];
      const float2 u[2] = {make_float2(z1.x + z2.x, z1.y + z2.y), make_float2(z1.z + z2.z, z1.w + z2.w)};
      const float2 w[2] = {make_float2(z1.x - z2.x, z1.y - z2.y), make_float2(z1.z - z2.z, z1.w - z2.w)};
      Mr += AP / 2;
#pragma unroll
      for (int a = 0; a < AMAX; ++a) {
        const float4 mm = Mr[a / 2];
        const float2 m = a & 1 ? make_float2(mm.z, mm.w) : make_float2(mm.x, mm.y);
#pragma unroll
        for (int l = 0; l < 2; ++l) {
          acc[a][l].x = fmaf(m.x, u[l].x, acc[a][l].x);
          acc[a][l].x = fmaf(-m.y, w[l].y, acc[a][l].x);
          acc[a][l].y = fmaf(m.x, u[l].y, acc[a][l].y);
          acc[a][l].y = fmaf(m.y, w[l].x, acc[a][l].y);
        }
      }
    }
    if (mid) {
      const float4 v = S[(n / 2) * 128];
      const float2 vm[2] = {make_float2(v.x, v.y), make_float2(v.z, v.w)};
      const float2* Mm = Ms + (n / 2) * AP;
#pragma unroll
      for (int a = 0; a < AMAX; ++a)
#pragma unroll
        for (int l = 0; l < 2; ++l) cfma(acc[a][l], Mm[a], vm[l]);
    }
    float2* op = out + b * vout.sb + ia * sa_out + ib * sb_out + c;
#pragma unroll
    for (int a = 0; a < AMAX; ++a)
      if (a < nout)
        *reinterpret_cast<float4*>(op + a * step_out) = make_float4(acc[a][0].x, acc[a][0].y, acc[a][1].x, acc[a][1].y);
  }
}

// Inverse counterpart: the z and y inverse passes of one (box, x-frequency)
// slab, lane = channel.  A warp copies the y-frequency rows fy = warp, warp + SP, ..
// of the slab (n spectrum values of 256 bytes each) to shared memory by 16-byte
// asynchronous copies, all of them in flight at once.  Phase 1: it forms the SP
// outputs of the z pass of each of its rows (conjugate input pairs folded as in
// k_dft_inv_line) and puts them in the place of the row's first SP values.  Phase 2: a
// warp takes one z and folds the y-frequency pairs into t[b][fx][y][z][c], the
// input of the x pass.
//
// What bounds it: issue slots (two thirds taken) with HBM at 4.6 TB/s.  1,016 boxes of
// 9^3 splines, 16 vectors: 326 -> 178 us (rows came pair by pair before, two loads in flight
// per warp, and phase 2 read every pair once per output).
template <int SP>
__global__ void __launch_bounds__(32 * SP) k_dft_inv_zy(const float2* __restrict__ in, float2* __restrict__ out,
                                                        int64_t B, const float2* __restrict__ M, int n) {
  extern __shared__ float4 izy_smem[];
  constexpr int SPP = SP + (SP & 1);
  float2* S = reinterpret_cast<float2*>(izy_smem);  // [fy][fz][32]; after phase 1 [fy][z < SP][32]
  float2* Ms = S + (int64_t)n * n * 32;             // [f][a < SPP] = M[a][f], f = 0 .. n/2
  const int nh = n / 2 + 1;
  const int np = (n - 1) / 2;
  const bool mid = (n % 2) == 0;
  const int64_t sl = blockIdx.x;
  const int64_t b = sl / n;
  const int fx = (int)(sl - b * n);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t fstride = B * 32;
  for (int fy = warp; fy < n; fy += SP) {
    const float2* ip = in + (((int64_t)fx * n + fy) * n * B + b) * 32 + (lane & 15) * 2;
    float2* d = S + (int64_t)fy * n * 32 + (lane & 15) * 2;
    for (int f = lane >> 4; f < n; f += 2) tile_cp16(d + f * 32, ip + f * fstride);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  }
  for (int i = threadIdx.x; i < nh * SPP; i += blockDim.x) {
    const int f = i / SPP, a = i - f * SPP;
    Ms[i] = a < SP ? M[(int64_t)a * n + f] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  for (int fy = warp; fy < n; fy += SP) {
    if (fy + SP < n) asm volatile("cp.async.wait_group 1;\n" ::: "memory");  // n < 2 SP: two rows at most
    else asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncwarp();
    float2* ip = S + (int64_t)fy * n * 32 + lane;
    float2 acc[SPP];
    const float4* Mr = reinterpret_cast<const float4*>(Ms);
    {
      const float2 v0 = ip[0];
#pragma unroll
      for (int a = 0; a < SPP; a += 2) {
        const float4 m = Mr[a / 2];
        acc[a] = make_float2(m.x * v0.x - m.y * v0.y, m.x * v0.y + m.y * v0.x);
        acc[a + 1] = make_float2(m.z * v0.x - m.w * v0.y, m.z * v0.y + m.w * v0.x);
      }
    }
#pragma unroll 2
    for (int f = 1; f <= np; ++f) {
      const float2 z1 = ip[f * 32], z2 = ip[(n - f) * 32];
      const float2 u = make_float2(z1.x + z2.x, z1.y + z2.y), w = make_float2(z1.x - z2.x, z1.y - z2.y);
      Mr += SPP / 2;
#pragma unroll
      for (int a = 0; a < SP; ++a) {
        const float4 mm = Mr[a / 2];
        const float2 m = a & 1 ? make_float2(mm.z, mm.w) : make_float2(mm.x, mm.y);
        acc[a].x = fmaf(m.x, u.x, acc[a].x);
        acc[a].x = fmaf(-m.y, w.y, acc[a].x);
        acc[a].y = fmaf(m.x, u.y, acc[a].y);
        acc[a].y = fmaf(m.y, w.x, acc[a].y);
      }
    }
    if (mid) {
      const float2 vm = ip[(n / 2) * 32];
      const float2* Mm = Ms + (n / 2) * SPP;
#pragma unroll
      for (int a = 0; a < SP; ++a) {
        const float2 m = Mm[a];
        acc[a].x = fmaf(m.x, vm.x, fmaf(-m.y, vm.y, acc[a].x));
        acc[a].y = fmaf(m.x, vm.y, fmaf(m.y, vm.x, acc[a].y));
      }
    }
#pragma unroll
    for (int a = 0; a < SP; ++a) ip[a * 32] = acc[a];  // SP <= n; the lane's own column
  }
  __syncthreads();
  {
    const int z = warp;
    const float2* U = S + z * 32 + lane;
    const int64_t row = (int64_t)n * 32;
    float2 acc[SPP];
    const float4* Mr = reinterpret_cast<const float4*>(Ms);
    {
      const float2 v0 = U[0];
#pragma unroll
      for (int a = 0; a < SPP; a += 2) {
        const float4 m = Mr[a / 2];
        acc[a] = make_float2(m.x * v0.x - m.y * v0.y, m.x * v0.y + m.y * v0.x);
        acc[a + 1] = make_float2(m.z * v0.x - m.w * v0.y, m.z * v0.y + m.w * v0.x);
      }
    }
#pragma unroll 2
    for (int f = 1; f <= np; ++f) {
      const float2 z1 = U[f * row], z2 = U[(n - f) * row];
      const float2 u = make_float2(z1.x + z2.x, z1.y + z2.y), w = make_float2(z1.x - z2.x, z1.y - z2.y);
      Mr += SPP / 2;
#pragma unroll
      for (int a = 0; a < SP; ++a) {
        const float4 mm = Mr[a / 2];
        const float2 m = a & 1 ? make_float2(mm.z, mm.w) : make_float2(mm.x, mm.y);
        acc[a].x = fmaf(m.x, u.x, acc[a].x);
        acc[a].x = fmaf(-m.y, w.y, acc[a].x);
        acc[a].y = fmaf(m.x, u.y, acc[a].y);
        acc[a].y = fmaf(m.y, w.x, acc[a].y);
      }
    }
    if (mid) {
      const float2 vm = U[(n / 2) * row];
      const float2* Mm = Ms + (n / 2) * SPP;
#pragma unroll
      for (int a = 0; a < SP; ++a) {
        const float2 m = Mm[a];
        acc[a].x = fmaf(m.x, vm.x, fmaf(-m.y, vm.y, acc[a].x));
        acc[a].y = fmaf(m.x, vm.y, fmaf(m.y, vm.x, acc[a].y));
      }
    }
    float2* op = out + sl * (SP * SP * 32) + z * 32 + lane;
#pragma unroll
    for (int y = 0; y < SP; ++y) op[y * (SP * 32)] = acc[y];
  }
}

// Whether the fused forward (y, z) / inverse (z, y) passes take a level of
// sp splines per axis and FFT length n (9, 13 or 21 splines; shared memory).
static size_t dft_yz_smem(int sp, int n, bool inverse) {
  const int nh = n / 2 + 1;
  return inverse ? sizeof(float2) * ((size_t)n * n * 32 + (size_t)nh * (sp + (sp & 1)))
                 : sizeof(float2) * ((size_t)sp * sp * 32 + (size_t)nh * sp);
}
bool dft_yz_fits(int sp, int n) { return (sp == 9 || sp == 13 || sp == 21) && dft_yz_smem(sp, n, false) <= 200 * 1024; }
// (at most two rows of a slab per warp, whose sums take the place of the inputs)
bool dft_zy_fits(int sp, int n) {
  return (sp == 9 || sp == 13) && sp <= n && n < 2 * sp && dft_yz_smem(sp, n, true) <= 200 * 1024;
}

// Fused y-z forward (in: t[b][fx][y][z][32] -> out: Q[fx][fy][fz][b][32]) or
// z-y inverse (in: Q layout -> out: t layout).  Returns false when they do not
// apply (splines per axis other than 9, 13 or 21, or shared memory).
bool launch_dft_yz(const float2* in, float2* out, int64_t B, int sp, int n, const float2* M, bool inverse,
                   cudaStream_t s) {
  const int64_t slabs = B * (int64_t)n;
  if (slabs <= 0) return true;
  if (slabs > 0x7FFFFFFFLL) return false;
  const size_t smem = dft_yz_smem(sp, n, inverse);
  if (inverse ? !dft_zy_fits(sp, n) : smem > 200 * 1024) return false;
  // one y-frequency pair per warp and round, the warps even over the rounds
  const int rounds = (n / 2 + 8) / 8, warps = (n / 2 + rounds) / rounds;
#define EFIE_YZ(SPV, KERNEL, WARPS)                                             \
  if (sp == SPV) {                                                              \
    static SmemAttr attr;                                                       \
    smem_attr_once(KERNEL<SPV>, (int)smem, attr.v);                             \
    KERNEL<SPV><<<(unsigned)slabs, 32 * (WARPS), smem, s>>>(in, out, B, M, n);  \
    return true;                                                                \
  }
  if (inverse) {
    EFIE_YZ(9, k_dft_inv_zy, 9)
    EFIE_YZ(13, k_dft_inv_zy, 13)
    return false;
  }
  EFIE_YZ(9, k_dft_fwd_yz, warps)
  EFIE_YZ(13, k_dft_fwd_yz, warps)
  EFIE_YZ(21, k_dft_fwd_yz, warps)
#undef EFIE_YZ
  return false;
}

// forward (inverse = false: M is n x nin, nin inputs -> n outputs along ax) or
// inverse (M is nout x n, n inputs -> nout outputs); returns false when no
// specialisation fits (the caller then uses launch_mode)
template <typename R>
bool launch_dft(const cpx_t<R>* in, View vin, cpx_t<R>* out, View vout, int64_t B, int C, int ax, int nin,
                int e0, int e1, int e2, const cpx_t<R>* M, int n, bool inverse, cudaStream_t s) {
  using T = cpx_t<R>;
  const int ea = ax == 0 ? e1 : e0, eb = ax == 2 ? e1 : e2;
  const int nout = ax == 0 ? e0 : (ax == 1 ? e1 : e2);
  const int nh = n / 2 + 1;
  const bool two = (C % 2) == 0 && sizeof(R) == 4;
  const int lpt = two ? 2 : 1;
  const int64_t lines = B * ea * eb * (int64_t)(C / lpt);
  if (lines <= 0) return true;
  int64_t blocks = ceil_div(lines, 128);
  if (blocks > 152 * 32) blocks = 152 * 32;
  if (!inverse) {
    const size_t smem = sizeof(T) * (size_t)nh * nin;
    if (smem > 96 * 1024) return false;
#define EFIE_DF(NM)                                                                                          \
  if (nin <= NM) {                                                                                           \
    if (two) {                                                                                               \
      auto k = k_dft_fwd_line<R, NM, sizeof(R) == 4 ? 2 : 1>;                                                \
      static SmemAttr attr;                                                                  \
      smem_attr_once(k, 96 * 1024, attr.v);                                                                    \
      k<<<(unsigned)blocks, 128, smem, s>>>(in, vin, out, vout, B, C, ax, nin, e0, e1, e2, M, n);            \
      return true;                                                                                           \
    }                                                                                                        \
    const int64_t lines1 = B * ea * eb * (int64_t)C;                                                         \
    int64_t blocks1 = ceil_div(lines1, 128);                                                                 \
    if (blocks1 > 152 * 32) blocks1 = 152 * 32;                                                              \
    auto k = k_dft_fwd_line<R, NM, 1>;                                                                       \
    static SmemAttr attr1;                                                                   \
    smem_attr_once(k, 96 * 1024, attr1.v);                                                                     \
    k<<<(unsigned)blocks1, 128, smem, s>>>(in, vin, out, vout, B, C, ax, nin, e0, e1, e2, M, n);             \
    return true;                                                                                             \
  }
    EFIE_DF(9)
    EFIE_DF(13)
    EFIE_DF(21)
#undef EFIE_DF
    if (nin <= 40) {
      TileArgs<2> t{};
      t.vin = vin, t.vout = vout, t.C = C, t.ax = ax, t.nin = nin, t.nout = nout, t.ea = ea, t.eb = eb, t.n = n;
      t.M0 = M;
      return launch_mode_tile<R, 2>(in, out, B, t, s);
    }
    return false;
  }
  const size_t smem = sizeof(T) * (size_t)nout * nh;
  if (smem > 96 * 1024) return false;
#define EFIE_DI(AM)                                                                                          \
  if (nout <= AM) {                                                                                          \
    if constexpr (sizeof(R) == 4) {                                                                          \
      const size_t sm = (size_t)n * 2048 + sizeof(T) * (size_t)nh * (AM + (AM & 1));                         \
      if (two && sm <= 100 * 1024) {                                                                         \
        static SmemAttr attr2;                                                                               \
        smem_attr_once(k_dft_inv_stage<AM>, 100 * 1024, attr2.v);                                            \
        k_dft_inv_stage<AM><<<(unsigned)blocks, 128, sm, s>>>(in, vin, out, vout, B, C, ax, e0, e1, e2, M, n); \
        return true;                                                                                         \
      }                                                                                                      \
    }                                                                                                        \
    const int64_t lines1 = B * ea * eb * (int64_t)C;                                                         \
    int64_t blocks1 = ceil_div(lines1, 128);                                                                 \
    if (blocks1 > 152 * 32) blocks1 = 152 * 32;                                                              \
    auto k = k_dft_inv_line<R, AM>;                                                                          \
    static SmemAttr attr1;                                                                                   \
    smem_attr_once(k, 96 * 1024, attr1.v);                                                                   \
    k<<<(unsigned)blocks1, 128, smem, s>>>(in, vin, out, vout, B, C, ax, nin, e0, e1, e2, M, n);             \
    return true;                                                                                             \
  }
  EFIE_DI(9)
  EFIE_DI(13)
  EFIE_DI(21)
#undef EFIE_DI
  return false;
}

template <typename R>
void launch_mode(const cpx_t<R>* in, View vin, cpx_t<R>* out, View vout, int64_t B, int C, int ax,
                 int nin, int e0, int e1, int e2, const void* M0, const void* M1, bool complex_m,
                 const int8_t* sel, const int64_t* srcmap, bool accumulate, cudaStream_t s) {
  int64_t total = B * e0 * e1 * e2 * (int64_t)C;
  if (total <= 0) return;
  const int nout = ax == 0 ? e0 : (ax == 1 ? e1 : e2);
  const size_t esz = complex_m ? sizeof(cpx_t<R>) : sizeof(R);
  const size_t smem = (size_t)nout * nin * esz * ((M1 && M1 != M0) ? 2 : 1);
  if (smem <= 96 * 1024) {
    bool done = complex_m ? dispatch_mode_line<R, true>(in, vin, out, vout, B, C, ax, nin, e0, e1, e2, M0, M1, sel,
                                                        srcmap, accumulate, smem, s)
                          : dispatch_mode_line<R, false>(in, vin, out, vout, B, C, ax, nin, e0, e1, e2, M0, M1,
                                                         sel, srcmap, accumulate, smem, s);
    if (done) return;
  }
  {
    const int ea = ax == 0 ? e1 : e0, eb = ax == 2 ? e1 : e2;
    const auto fill = [&](auto t) {
      t.vin = vin, t.vout = vout, t.C = C, t.ax = ax, t.nin = nin, t.nout = nout, t.ea = ea, t.eb = eb;
      t.M0 = M0, t.M1 = M1, t.sel = sel, t.srcmap = srcmap, t.accumulate = accumulate;
      return t;
    };
    // one complex matrix (sel picks between two real ones only)
    if (complex_m ? (M1 == nullptr || M1 == M0) && launch_mode_tile<R, 1>(in, out, B, fill(TileArgs<1>{}), s)
                  : launch_mode_tile<R, 0>(in, out, B, fill(TileArgs<0>{}), s))
      return;
  }
  int64_t blocks = ceil_div(total, 256);
  if (blocks > 152 * 64) blocks = 152 * 64;
  if (complex_m)
    k_mode<R, true><<<(unsigned)blocks, 256, 0, s>>>(in, vin, out, vout, B, C, ax, nin, e0, e1, e2, M0,
                                                     M1, sel, srcmap, accumulate);
  else
    k_mode<R, false><<<(unsigned)blocks, 256, 0, s>>>(in, vin, out, vout, B, C, ax, nin, e0, e1, e2, M0,
                                                      M1, sel, srcmap, accumulate);
}

// ---------------------------------------------------------------- leaf grids
// Channel order inside a grid point: c = d * nr + r (component d = 0..2 the
// vector part, 3 the charge part; r the right-hand side), so the vector part
// of one point is 3 nr contiguous values and the charge part nr more.

// Gather lists (setup): the moments re-indexed by grid point.  For leaf box b
// and point pt of its sp^3 grid, entries [ptr[pt], ptr[pt+1]) (offsets within
// the box) hold (k, m_0, m_1, m_2) for every RWG k of the box (local index)
// whose moment block covers pt, in increasing k; triangles likewise hold
// (t, m^phi).  A box's entries start where its RWGs' moment data starts
// (mr_off / 3, mt_off), since both orderings hold the same entries.  One CTA
// per box, one thread per point; the covering test reads each basis
// function's base and extents, so the lists are deterministic.
// Points are taken GB_PTS at a time (the per-point counters live in shared
// memory), so leaves of any spline count fit; thread 0 carries the running
// list offsets from one group of points to the next.
constexpr int GB_PTS = 8192;

template <typename R>
__global__ void k_gather_build(const R* __restrict__ mr, const int32_t* __restrict__ mr_base,
                               const int32_t* __restrict__ mr_ext, const int64_t* __restrict__ mr_off,
                               const R* __restrict__ mt, const int32_t* __restrict__ mt_base,
                               const int32_t* __restrict__ mt_ext, const int64_t* __restrict__ mt_off,
                               const int64_t* __restrict__ box_rwg_ptr, const int64_t* __restrict__ box_tri_ptr,
                               int sp, int32_t* __restrict__ gptr_r, int32_t* __restrict__ gptr_t,
                               R* __restrict__ gr, R* __restrict__ gt) {
  extern __shared__ int32_t gcnt[];  // [2][min(npts, GB_PTS)]
  const int b = blockIdx.x, npts = sp * sp * sp;
  const int gp = npts < GB_PTS ? npts : GB_PTS;
  const int64_t k0 = box_rwg_ptr[b], k1 = box_rwg_ptr[b + 1];
  const int64_t t0 = box_tri_ptr[b], t1 = box_tri_ptr[b + 1];
  auto covers = [&](const int32_t* base, const int32_t* ext, int64_t i, int p0, int p1, int p2, int& e) {
    const int a0 = p0 - base[3 * i], a1 = p1 - base[3 * i + 1], a2 = p2 - base[3 * i + 2];
    const int e0 = ext[3 * i], e1 = ext[3 * i + 1], e2 = ext[3 * i + 2];
    if ((unsigned)a0 >= (unsigned)e0 || (unsigned)a1 >= (unsigned)e1 || (unsigned)a2 >= (unsigned)e2) return false;
    e = (a0 * e1 + a1) * e2 + a2;
    return true;
  };
  int32_t* pr = gptr_r + (int64_t)b * (npts + 1);
  int32_t* pt_ = gptr_t + (int64_t)b * (npts + 1);
  R* outr = gr + 4 * (k0 < k1 ? mr_off[k0] / 3 : 0);
  R* outt = gt + 2 * (t0 < t1 ? mt_off[t0] : 0);
  int32_t rr = 0, rt = 0;  // running offsets (thread 0)
  for (int q0 = 0; q0 < npts; q0 += gp) {
    const int q1 = q0 + gp < npts ? q0 + gp : npts;
    for (int pt = q0 + threadIdx.x; pt < q1; pt += blockDim.x) {
      const int p0 = pt / (sp * sp), p1 = (pt / sp) % sp, p2 = pt % sp;
      int cr = 0, ct = 0, e;
      for (int64_t i = k0; i < k1; ++i) cr += covers(mr_base, mr_ext, i, p0, p1, p2, e);
      for (int64_t i = t0; i < t1; ++i) ct += covers(mt_base, mt_ext, i, p0, p1, p2, e);
      gcnt[pt - q0] = cr;
      gcnt[gp + pt - q0] = ct;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int pt = q0; pt < q1; ++pt) {
        const int32_t vr = gcnt[pt - q0], vt = gcnt[gp + pt - q0];
        gcnt[pt - q0] = rr;
        gcnt[gp + pt - q0] = rt;
        pr[pt] = rr;
        pt_[pt] = rt;
        rr += vr;
        rt += vt;
      }
      if (q1 == npts) {
        pr[npts] = rr;
        pt_[npts] = rt;
      }
    }
    __syncthreads();
    for (int pt = q0 + threadIdx.x; pt < q1; pt += blockDim.x) {
      const int p0 = pt / (sp * sp), p1 = (pt / sp) % sp, p2 = pt % sp;
      int64_t pos = gcnt[pt - q0];
      int e;
      for (int64_t i = k0; i < k1; ++i)
        if (covers(mr_base, mr_ext, i, p0, p1, p2, e)) {
          const R* m = mr + mr_off[i] + 3 * e;
          R* o = outr + 4 * pos++;
          o[0] = (R)(i - k0);
          o[1] = m[0];
          o[2] = m[1];
          o[3] = m[2];
        }
      pos = gcnt[gp + pt - q0];
      for (int64_t i = t0; i < t1; ++i)
        if (covers(mt_base, mt_ext, i, p0, p1, p2, e)) {
          R* o = outt + 2 * pos++;
          o[0] = (R)(i - t0);
          o[1] = mt[mt_off[i] + e];
        }
    }
    __syncthreads();  // gcnt is reused by the next group of points
  }
}

// ---------------------------------------------------------------- anterpolation
// q[b][pt][d nr + r] = sum over the gather list of pt: m_d x_r[k] (d < 3) and
// sum of m^phi rho_r[t] (d = 3).  Blocks are (leaf box, part of its grid points);
// the box's currents and charges are staged in shared memory (ak basis
// functions at a time: all of them wherever they fit, else several passes
// over the sorted lists).  LR lanes, the right-hand sides rounded up to a power
// of two, share a point: a warp takes 32 / LR points at a time, the lanes of a
// point read the same list entry (one broadcast) and consecutive staged values,
// and own their 4 output components outright -- no atomics, each moment entry read
// once per launch, each output written once.  In FP64, SPL groups of LR lanes share a
// point's list entry by entry and add their sums by shuffles.
//
// What bounds it: the latency of the list entries, and in FP64 the multiply-
// adds, so lanes without a right-hand side (7 of 8 with LR = 8 and one vector)
// cost as much as the others.  One block per box left the chip empty on trees with
// few boxes.  Measured: 1,920 unknowns, 32 boxes, FP64, one vector
// 0.397 -> 0.078 ms; 48,000 unknowns, FP64, 8 vectors 2.75 -> 1.31 (two passes per 32
// points before); the nonuniform tree with 22 leaves of 41^3 points on its top
// level, 64 vectors 166 -> 5.8.  FP64 with lists shared by SPL groups (8 to 16 lanes a
// point; half or twice as many measured slower on small or on large trees) and eight
// entries in flight, 1, 2, 4 and 8 vectors: 1,920 unknowns in one level 0.188 -> 0.032,
// 0.182 -> 0.051, 0.165 -> 0.053, 0.175 -> 0.094; 48,000 unknowns 0.398 -> 0.300, 0.528 -> 0.400,
// 0.816 -> 0.638, 1.28 -> 0.98.  FP32, 6,750 unknowns, one vector, eight in flight: 0.081 ->
// 0.064.
template <typename R, int LR>
struct AnterpCfg {
  // values per staged function: rows of 80 bytes (FP32) and 144 (FP64) spread the banks
  static constexpr int XS = LR < 8 ? LR : sizeof(R) == 4 ? 10 : 9;
};
constexpr int ANTERP_SMEM = 96 * 1024;

template <typename R, int LR, int SPL>
__global__ void __launch_bounds__(256) k_anterp(const R* __restrict__ gr, const R* __restrict__ gt,
                                                const int32_t* __restrict__ gptr_r,
                                                const int32_t* __restrict__ gptr_t,
                                                const int64_t* __restrict__ mr_off,
                                                const int64_t* __restrict__ mt_off,
                                                const int64_t* __restrict__ box_rwg_ptr,
                                                const int64_t* __restrict__ box_tri_ptr,
                                                const int32_t* __restrict__ out_box,
                                                const cpx_t<R>* __restrict__ xs, int64_t ldx,
                                                const cpx_t<R>* __restrict__ rho, int64_t ldr, int nr,
                                                cpx_t<R>* __restrict__ q, int sp, int ak, int at, int nsplit) {
  using T = cpx_t<R>;
  constexpr int XS = AnterpCfg<R, LR>::XS, PW = 32 / (LR * SPL);
  extern __shared__ __align__(16) unsigned char anterp_smem[];
  T* xsm = reinterpret_cast<T*>(anterp_smem);  // [ak][XS]
  T* rsm = xsm + (size_t)ak * XS;              // [at][XS]
  const int b = blockIdx.x / nsplit, part = blockIdx.x - b * nsplit;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int npts = sp * sp * sp;
  const int64_t k0 = box_rwg_ptr[b], t0 = box_tri_ptr[b];
  const int nk = (int)(box_rwg_ptr[b + 1] - k0), nt = (int)(box_tri_ptr[b + 1] - t0);
  const R* ger = gr + 4 * (nk > 0 ? mr_off[k0] / 3 : 0);
  const R* get = gt + 2 * (nt > 0 ? mt_off[t0] : 0);
  const int32_t* pr = gptr_r + (int64_t)b * (npts + 1);
  const int32_t* pq = gptr_t + (int64_t)b * (npts + 1);
  const int nchunk = max((nk + ak - 1) / ak, (nt + at - 1) / at);
  auto stage = [&](int c) {
    for (int i = tid; i < ak * nr; i += blockDim.x) {
      const int r = i / ak, kk = i - r * ak, k = c * ak + kk;
      if (k < nk) xsm[kk * XS + r] = xs[r * ldx + k0 + k];
    }
    for (int i = tid; i < at * nr; i += blockDim.x) {
      const int r = i / at, kk = i - r * at, k = c * at + kk;
      if (k < nt) rsm[kk * XS + r] = rho[r * ldr + t0 + k];
    }
  };
  if (nchunk == 1) {
    stage(0);
    __syncthreads();
  }
  const int r = lane & (LR - 1), lp = lane / LR & (SPL - 1), ps = lane / (LR * SPL);
  const int C = 4 * nr;
  const int per_pass = PW * (blockDim.x >> 5);
  // passes part, part + nsplit, ..: points near the surface, where the lists
  // are long, spread over the parts
  for (int pb = part * per_pass; pb < npts; pb += nsplit * per_pass) {
    const int p = pb + PW * warp + ps;
    const bool okp = p < npts;
    T a0 = mk<R>(0, 0), a1 = a0, a2 = a0, a3 = a0;
    int er = okp ? pr[p] + lp : 0, er1 = okp ? pr[p + 1] : 0;
    int et = okp ? pq[p] + lp : 0, et1 = okp ? pq[p + 1] : 0;
    for (int c = 0; c < nchunk; ++c) {
      if (nchunk > 1) {
        __syncthreads();
        stage(c);
        __syncthreads();
      }
      const int kc0 = c * ak, tc0 = c * at;
      auto load4 = [&](int64_t i, R& ek, R& m0, R& m1, R& m2) {
        const R* e = ger + 4 * i;
        if constexpr (sizeof(R) == 4) {
          const float4 v = *reinterpret_cast<const float4*>(e);
          ek = v.x, m0 = v.y, m1 = v.z, m2 = v.w;
        } else {
          const double2 v0 = *reinterpret_cast<const double2*>(e), v1 = *reinterpret_cast<const double2*>(e + 2);
          ek = v0.x, m0 = v0.y, m1 = v1.x, m2 = v1.y;
        }
      };
      auto mac3 = [&](int k, R m0, R m1, R m2) {
        const T xv = xsm[(k - kc0) * XS + r];
        a0.x = fma(m0, xv.x, a0.x);
        a0.y = fma(m0, xv.y, a0.y);
        a1.x = fma(m1, xv.x, a1.x);
        a1.y = fma(m1, xv.y, a1.y);
        a2.x = fma(m2, xv.x, a2.x);
        a2.y = fma(m2, xv.y, a2.y);
      };
      if (nchunk == 1) {
        // every entry belongs to this chunk: several list entries in flight.  Eight, the
        // last ones of a list predicated, in FP64 and with at most two lanes of
        // vectors; else four (48,000 unknowns, FP32, 8 vectors: 0.195 ms against 0.217)
        if constexpr (sizeof(R) == 8 || LR <= 2) {
          for (; er < er1; er += 8 * SPL) {
            R k_[8], x_[8], y_[8], z_[8];
#pragma unroll
            for (int t = 0; t < 8; ++t)
              if (er + t * SPL < er1) load4(er + t * SPL, k_[t], x_[t], y_[t], z_[t]);
#pragma unroll
            for (int t = 0; t < 8; ++t)
              if (er + t * SPL < er1) mac3((int)k_[t], x_[t], y_[t], z_[t]);
          }
        } else {
          for (; er + 3 * SPL < er1; er += 4 * SPL) {
            R k_[4], x_[4], y_[4], z_[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) load4(er + t * SPL, k_[t], x_[t], y_[t], z_[t]);
#pragma unroll
            for (int t = 0; t < 4; ++t) mac3((int)k_[t], x_[t], y_[t], z_[t]);
          }
        }
      }
      for (; er < er1; er += SPL) {
        R ek, m0, m1, m2;
        load4(er, ek, m0, m1, m2);
        if ((int)ek >= kc0 + ak) break;
        mac3((int)ek, m0, m1, m2);
      }
      auto load2 = [&](int64_t i, R& ek, R& m) {
        const R* e = get + 2 * i;
        if constexpr (sizeof(R) == 4) {
          const float2 v = *reinterpret_cast<const float2*>(e);
          ek = v.x, m = v.y;
        } else {
          const double2 v = *reinterpret_cast<const double2*>(e);
          ek = v.x, m = v.y;
        }
      };
      auto mac1 = [&](int k, R m) {
        const T v = rsm[(k - tc0) * XS + r];
        a3.x = fma(m, v.x, a3.x);
        a3.y = fma(m, v.y, a3.y);
      };
      if (nchunk == 1) {
        for (; et + 3 * SPL < et1; et += 4 * SPL) {
          R k_[4], m_[4];
#pragma unroll
          for (int t = 0; t < 4; ++t) load2(et + t * SPL, k_[t], m_[t]);
#pragma unroll
          for (int t = 0; t < 4; ++t) mac1((int)k_[t], m_[t]);
        }
      }
      for (; et < et1; et += SPL) {
        R ek, m;
        load2(et, ek, m);
        if ((int)ek >= tc0 + at) break;
        mac1((int)ek, m);
      }
    }
#pragma unroll
    for (int o = LR; o < LR * SPL; o *= 2) {
      const auto add = [&](T& a) {
        a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
        a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
      };
      add(a0), add(a1), add(a2), add(a3);
    }
    if (okp && r < nr && lp == 0) {
      T* qp = q + ((int64_t)(out_box ? out_box[b] : b) * npts + p) * C + r;
      qp[0] = a0;
      qp[nr] = a1;
      qp[2 * nr] = a2;
      qp[3 * nr] = a3;
    }
  }
}

template <typename R>
void launch_gather_build(const R* mr, const int32_t* mr_base, const int32_t* mr_ext, const int64_t* mr_off,
                         const R* mt, const int32_t* mt_base, const int32_t* mt_ext, const int64_t* mt_off,
                         const int64_t* box_rwg_ptr, const int64_t* box_tri_ptr, int64_t B, int sp,
                         int32_t* gptr_r, int32_t* gptr_t, R* gr, R* gt, cudaStream_t s) {
  if (B <= 0) return;
  const int64_t npts = (int64_t)sp * sp * sp;
  const size_t smem = sizeof(int32_t) * 2 * (size_t)(npts < GB_PTS ? npts : GB_PTS);
  if (smem > 48 * 1024) cudaFuncSetAttribute(k_gather_build<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k_gather_build<R><<<(unsigned)B, 256, smem, s>>>(mr, mr_base, mr_ext, mr_off, mt, mt_base, mt_ext, mt_off,
                                                   box_rwg_ptr, box_tri_ptr, sp, gptr_r, gptr_t, gr, gt);
}

template <typename R, int LR, int SPL>
static void run_anterp(const R* gr, const R* gt, const int32_t* gptr_r, const int32_t* gptr_t, const int64_t* mr_off,
                       const int64_t* mt_off, const int64_t* box_rwg_ptr, const int64_t* box_tri_ptr, int64_t B,
                       int max_rwg, int max_sc, const int32_t* out_box, const cpx_t<R>* xs, int64_t ldx,
                       const cpx_t<R>* rho, int64_t ldr, int nr, cpx_t<R>* q, int sp, cudaStream_t s) {
  const size_t row = AnterpCfg<R, LR>::XS * sizeof(cpx_t<R>);
  const int cap = (int)(ANTERP_SMEM / row);
  int ak = std::max(1, max_rwg), at = std::max(1, max_sc);
  if (ak + at > cap) ak = at = cap / 2;
  const size_t smem = (size_t)(ak + at) * row;
  static SmemAttr attr;
  smem_attr_once(k_anterp<R, LR, SPL>, ANTERP_SMEM, attr.v);
  // parts of a box's points, up to one pass each, until the blocks fill the
  // chip twice over (4 blocks of 8 warps per SM); a part stages the box again
  const int64_t npts = (int64_t)sp * sp * sp, passes = ceil_div(npts, 256 / (LR * SPL));
  const int nsplit = (int)std::max<int64_t>(1, std::min<int64_t>(passes, ceil_div(152 * 8, B)));
  k_anterp<R, LR, SPL><<<(unsigned)(B * nsplit), 256, smem, s>>>(gr, gt, gptr_r, gptr_t, mr_off, mt_off, box_rwg_ptr,
                                                                 box_tri_ptr, out_box, xs, ldx, rho, ldr, nr, q, sp,
                                                                 ak, at, nsplit);
}

template <typename R>
void launch_anterp(const R* gr, const R* gt, const int32_t* gptr_r, const int32_t* gptr_t, const int64_t* mr_off,
                   const int64_t* mt_off, const int64_t* box_rwg_ptr, const int64_t* box_tri_ptr, int64_t B,
                   int max_rwg, int max_sc, const int32_t* out_box, const cpx_t<R>* xs, int64_t ldx,
                   const cpx_t<R>* rho, int64_t ldr, int nr, cpx_t<R>* q, int sp, cudaStream_t s) {
  if (B <= 0 || nr <= 0) return;
#define EFIE_AN(L, S)                                                                                                \
  run_anterp<R, L, S>(gr, gt, gptr_r, gptr_t, mr_off, mt_off, box_rwg_ptr, box_tri_ptr, B, max_rwg, max_sc, out_box, \
                      xs, ldx, rho, ldr, nr, q, sp, s)
  if constexpr (sizeof(R) == 4) {  // FP32 sums keep their order
    if (nr == 1) EFIE_AN(1, 1);
    else if (nr == 2) EFIE_AN(2, 1);
    else if (nr <= 4) EFIE_AN(4, 1);
    else EFIE_AN(8, 1);
  } else {
    if (nr == 1) EFIE_AN(1, 8);
    else if (nr == 2) EFIE_AN(2, 4);
    else if (nr <= 4) EFIE_AN(4, 4);
    else EFIE_AN(8, 2);
  }
#undef EFIE_AN
}

// ---------------------------------------------------------------- interpolation
// yA[r][i] = sum_e sum_d m_d[e] r[b][pt(e)][d nr + r] for RWG i, and
// u[r][t] = sum_e m^phi[e] r[b][pt(e)][3 nr + r] for triangle t (FP64
// outputs).  RWG: lane = channel d nr + r of the vector part (3 nr <= 24 lanes),
// so every grid point is one coalesced read; the three components are summed by
// shuffles at the end.  A warp takes up to 32 / (3 nr) RWGs, `per` (21,870 RWGs, 3
// right-hand sides of a chunk: 0.73 -> 0.64 ms with 3 of them; few RWGs keep one
// per warp, for the latency of its loads).  Triangle:
// the charge part is nr values per point, so the warp takes 32/nr entries at
// a time, lane = (entry slot, r).
template <typename R>
__global__ void __launch_bounds__(256) k_interp(const R* __restrict__ mr, const int32_t* __restrict__ mr_base,
                                                const int32_t* __restrict__ mr_ext,
                                                const int64_t* __restrict__ mr_off,
                                                const int32_t* __restrict__ rwg_box, int64_t N,
                                                const R* __restrict__ mt, const int32_t* __restrict__ mt_base,
                                                const int32_t* __restrict__ mt_ext,
                                                const int64_t* __restrict__ mt_off,
                                                const int32_t* __restrict__ tri_box, int64_t Nt,
                                                const cpx_t<R>* __restrict__ rg, int sp, int nr,
                                                double2* __restrict__ yA, int64_t ldy, double2* __restrict__ u,
                                                int64_t ldu, int per) {
  using T = cpx_t<R>;
  const int lane = threadIdx.x & 31;
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = (N + per - 1) / per;
  if (w >= nw + Nt) return;
  const int npts = sp * sp * sp, C = 4 * nr;
  T acc = mk<R>(0, 0);
  if (w < nw) {
    const int slot = lane / (3 * nr), ch = lane - slot * 3 * nr;
    const int64_t i = w * per + slot;
    const bool act = slot < per && i < N;
    if (act) {
      const int b0 = mr_base[3 * i], b1 = mr_base[3 * i + 1], b2 = mr_base[3 * i + 2];
      const int e0 = mr_ext[3 * i], e1 = mr_ext[3 * i + 1], e2 = mr_ext[3 * i + 2];
      const R* m = mr + mr_off[i] + ch / nr;  // entry e at m[3 e]
      const T* gp = rg + (int64_t)rwg_box[i] * npts * C + ch;
      int e = 0;
      for (int a0 = 0; a0 < e0; ++a0)
        for (int a1 = 0; a1 < e1; ++a1) {
          const T* gl = gp + (int64_t)(((b0 + a0) * sp + b1 + a1) * sp + b2) * C;
          const R* ml = m + 3 * e;
#pragma unroll 4
          for (int a2 = 0; a2 < e2; ++a2) {
            const R mv = ml[3 * a2];
            const T gv = gl[a2 * C];
            acc.x = fma(mv, gv.x, acc.x);
            acc.y = fma(mv, gv.y, acc.y);
          }
          e += e2;
        }
    }
    R sx = acc.x + __shfl_down_sync(0xffffffffu, acc.x, nr) + __shfl_down_sync(0xffffffffu, acc.x, 2 * nr);
    R sy = acc.y + __shfl_down_sync(0xffffffffu, acc.y, nr) + __shfl_down_sync(0xffffffffu, acc.y, 2 * nr);
    if (act && ch < nr) yA[ch * ldy + i] = make_double2((double)sx, (double)sy);
  } else {
    const int64_t i = w - nw;
    const int b0 = mt_base[3 * i], b1 = mt_base[3 * i + 1], b2 = mt_base[3 * i + 2];
    const int e0 = mt_ext[3 * i], e1 = mt_ext[3 * i + 1], e2 = mt_ext[3 * i + 2];
    const int ne = e0 * e1 * e2;
    const int Q = 32 / nr;
    const int slot = lane / nr, r = lane - slot * nr;
    const R* m = mt + mt_off[i];
    const T* gp = rg + (int64_t)tri_box[i] * npts * C + 3 * nr + r;
    if (slot < Q && ne > 0) {
      int e = slot;
      int a0 = e / (e1 * e2), a1 = (e / e2) % e1, a2 = e % e2;
      for (; e < ne; e += Q) {
        const T gv = gp[(int64_t)(((b0 + a0) * sp + b1 + a1) * sp + b2 + a2) * C];
        const R mv = m[e];
        acc.x = fma(mv, gv.x, acc.x);
        acc.y = fma(mv, gv.y, acc.y);
        a2 += Q;
        while (a2 >= e2) {
          a2 -= e2;
          if (++a1 == e1) {
            a1 = 0;
            ++a0;
          }
        }
      }
    }
    R sx = acc.x, sy = acc.y;
    for (int o = 1; o < Q; ++o) {
      sx += __shfl_down_sync(0xffffffffu, acc.x, o * nr);
      sy += __shfl_down_sync(0xffffffffu, acc.y, o * nr);
    }
    if (lane < nr) u[lane * ldu + i] = make_double2((double)sx, (double)sy);
  }
}

// Eight right-hand sides in FP32 (32 channels): a half-warp per basis
// function, two per warp, each lane holding two adjacent channels (one 16-byte
// load per grid point).  RWG: lanes 0..11 cover the 24 vector channels;
// triangle: four entries at a time, four lanes each over the 8 charge channels.
// Entries run in one flat loop with the grid offset advanced incrementally, so
// the two halves stay in step and each has its own loads in flight.
__global__ void __launch_bounds__(256) k_interp8(const float* __restrict__ mr, const int32_t* __restrict__ mr_base,
                                                 const int32_t* __restrict__ mr_ext,
                                                 const int64_t* __restrict__ mr_off,
                                                 const int32_t* __restrict__ rwg_box, int64_t N,
                                                 const float* __restrict__ mt, const int32_t* __restrict__ mt_base,
                                                 const int32_t* __restrict__ mt_ext,
                                                 const int64_t* __restrict__ mt_off,
                                                 const int32_t* __restrict__ tri_box, int64_t Nt,
                                                 const float2* __restrict__ rg, int sp,
                                                 double2* __restrict__ yA, int64_t ldy, double2* __restrict__ u,
                                                 int64_t ldu) {
  constexpr int C = 32;
  const int lane = threadIdx.x & 31, hl = lane & 15;
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 4;  // one basis function per half-warp
  const bool valid = w < N + Nt;
  const int npts = sp * sp * sp;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  const bool is_rwg = valid && w < N;
  const int64_t i = is_rwg ? w : w - N;
  const int32_t* base = is_rwg ? mr_base : mt_base;
  const int32_t* ext = is_rwg ? mr_ext : mt_ext;
  int b0 = 0, b1 = 0, b2 = 0, e0 = 0, e1 = 0, e2 = 0;
  if (valid) {
    b0 = base[3 * i], b1 = base[3 * i + 1], b2 = base[3 * i + 2];
    e0 = ext[3 * i], e1 = ext[3 * i + 1], e2 = ext[3 * i + 2];
  }
  const int ne = e0 * e1 * e2;
  if (is_rwg) {
    const bool act = hl < 12;
    const int d = hl >> 2;
    const float* m = mr + mr_off[i] + d;
    const float2* gp = rg + (int64_t)rwg_box[i] * npts * C + 2 * (act ? hl : 0);
    int64_t off = (int64_t)((b0 * sp + b1) * sp + b2) * C;
    int a1 = 0, a2 = 0;
    for (int e = 0; e < ne; ++e) {
      if (act) {
        const float mv = m[3 * e];
        const float4 g = *reinterpret_cast<const float4*>(gp + off);
        acc.x = fmaf(mv, g.x, acc.x);
        acc.y = fmaf(mv, g.y, acc.y);
        acc.z = fmaf(mv, g.z, acc.z);
        acc.w = fmaf(mv, g.w, acc.w);
      }
      off += C;
      if (++a2 == e2) {
        a2 = 0;
        off += (int64_t)(sp - e2) * C;
        if (++a1 == e1) {
          a1 = 0;
          off += (int64_t)(sp - e1) * sp * C;
        }
      }
    }
  } else if (valid) {
    const int slot = hl >> 2, pr = hl & 3;
    const float* m = mt + mt_off[i];
    const float2* gp = rg + (int64_t)tri_box[i] * npts * C + 24 + 2 * pr;
    if (ne > 0) {
      int e = slot;
      int a0 = e / (e1 * e2), a1 = (e / e2) % e1, a2 = e % e2;
      for (; e < ne; e += 4) {
        const float4 g =
            *reinterpret_cast<const float4*>(gp + (int64_t)(((b0 + a0) * sp + b1 + a1) * sp + b2 + a2) * C);
        const float mv = m[e];
        acc.x = fmaf(mv, g.x, acc.x);
        acc.y = fmaf(mv, g.y, acc.y);
        acc.z = fmaf(mv, g.z, acc.z);
        acc.w = fmaf(mv, g.w, acc.w);
        a2 += 4;
        while (a2 >= e2) {
          a2 -= e2;
          if (++a1 == e1) {
            a1 = 0;
            ++a0;
          }
        }
      }
    }
  }
  // lanes hl < 4 sum lanes hl, hl+4, hl+8, hl+12 of their half-warp: the
  // three components of an RWG (lanes 12..15 hold zeros) or the four entry
  // slots of a triangle
  float4 t;
  t.x = __shfl_down_sync(0xffffffffu, acc.x, 4, 16);
  t.y = __shfl_down_sync(0xffffffffu, acc.y, 4, 16);
  t.z = __shfl_down_sync(0xffffffffu, acc.z, 4, 16);
  t.w = __shfl_down_sync(0xffffffffu, acc.w, 4, 16);
  float4 v = make_float4(acc.x + t.x, acc.y + t.y, acc.z + t.z, acc.w + t.w);
  t.x = __shfl_down_sync(0xffffffffu, v.x, 8, 16);
  t.y = __shfl_down_sync(0xffffffffu, v.y, 8, 16);
  t.z = __shfl_down_sync(0xffffffffu, v.z, 8, 16);
  t.w = __shfl_down_sync(0xffffffffu, v.w, 8, 16);
  v = make_float4(v.x + t.x, v.y + t.y, v.z + t.z, v.w + t.w);
  if (valid && hl < 4) {
    double2* out = is_rwg ? yA : u;
    const int64_t ld = is_rwg ? ldy : ldu;
    out[(int64_t)(2 * hl) * ld + i] = make_double2((double)v.x, (double)v.y);
    out[(int64_t)(2 * hl + 1) * ld + i] = make_double2((double)v.z, (double)v.w);
  }
}

template <typename R>
void launch_interp(const R* mr, const int32_t* mr_base, const int32_t* mr_ext, const int64_t* mr_off,
                   const int32_t* rwg_box, int64_t N, const R* mt, const int32_t* mt_base,
                   const int32_t* mt_ext, const int64_t* mt_off, const int32_t* tri_box, int64_t Nt,
                   const cpx_t<R>* r, int sp, int nr, double2* yA, int64_t ldy, double2* u,
                   int64_t ldu, cudaStream_t s) {
  // nr <= 8 (the far pipeline runs right-hand sides in chunks of at most 8)
  if constexpr (sizeof(R) == 4) {
    if (nr == 8) {
      const int64_t halves = N + Nt;
      k_interp8<<<(unsigned)ceil_div(halves * 16, 256), 256, 0, s>>>(
          (const float*)mr, mr_base, mr_ext, mr_off, rwg_box, N, (const float*)mt, mt_base, mt_ext, mt_off, tri_box,
          Nt, (const float2*)r, sp, yA, ldy, u, ldu);
      return;
    }
  }
  // RWGs per warp: as many as it has lanes for, while 32 warps per SM are left
  const int per = (int)std::max<int64_t>(1, std::min<int64_t>(32 / (3 * nr), N / (152 * 32)));
  int64_t warps = ceil_div(N, per) + Nt;
  int64_t blocks = ceil_div(warps * 32, 256);
  k_interp<R><<<(unsigned)blocks, 256, 0, s>>>(mr, mr_base, mr_ext, mr_off, rwg_box, N, mt, mt_base, mt_ext,
                                               mt_off, tri_box, Nt, r, sp, nr, yA, ldy, u, ldu, per);
}

// ---------------------------------------------------------------- translation MAC
// Rh[f][x][c] = sum_{y in IL(x)} Kh[f][off(x - y)] * Qh[f][y][c].
// Tiles group targets that share one source list (the children of a parent
// box on interaction-list levels, chunks of boxes on the top grid level);
// kidx[tile][j][a] holds the offset id of (target a, source j) or -1.  Each
// thread keeps XR targets x CR channels of one frequency in registers, so every
// loaded spectrum value feeds XR complex MACs and every kernel value CR.
// grid: (tile, frequency chunk); block: fpb frequencies x ntx target groups x
// C/CR channel groups.
template <typename R, int XR, int CR>
__global__ void k_mac_tiled(const cpx_t<R>* __restrict__ Qh, cpx_t<R>* __restrict__ Rh,
                            const cpx_t<R>* __restrict__ Kh, int64_t B, int C, int64_t O, int64_t nf,
                            const int64_t* __restrict__ tgt_ptr, const int32_t* __restrict__ tgt,
                            const int64_t* __restrict__ src_ptr, const int32_t* __restrict__ src,
                            const int64_t* __restrict__ kidx_off, const int32_t* __restrict__ kidx,
                            int fpb, int ntx, int64_t f0) {
  using T = cpx_t<R>;
  const int tile = blockIdx.x;
  const int ncg = C / CR;
  const int per_f = ntx * ncg;
  const int fl = threadIdx.x / per_f;
  const int rem = threadIdx.x - fl * per_f;
  const int tg = rem / ncg, cg = rem - (rem / ncg) * ncg;
  const int64_t f = f0 + (int64_t)blockIdx.y * fpb + fl;
  if (fl >= fpb || f >= nf) return;
  const int64_t t0 = tgt_ptr[tile], nt = tgt_ptr[tile + 1] - t0;
  const int64_t s0 = src_ptr[tile], ns = src_ptr[tile + 1] - s0;
  const int xb = tg * XR;
  if (xb >= nt) return;
  const int tpad = (int)(((nt + XR - 1) / XR) * XR);
  const int32_t* kb = kidx + kidx_off[tile] + xb;
  const T* Qf = Qh + f * B * C + cg * CR;
  const T* Kf = Kh + f * O;
  T acc[XR][CR];
#pragma unroll
  for (int a = 0; a < XR; ++a)
#pragma unroll
    for (int c = 0; c < CR; ++c) acc[a][c] = mk<R>(0, 0);
#pragma unroll 2
  for (int64_t j = 0; j < ns; ++j) {
    const int32_t y = __ldg(src + s0 + j);
    T q[CR];
#pragma unroll
    for (int c = 0; c < CR; ++c) q[c] = Qf[(int64_t)y * C + c];
    const int32_t* kr = kb + j * tpad;
#pragma unroll
    for (int a = 0; a < XR; ++a) {
      const int32_t id = __ldg(kr + a);
      if (id < 0) continue;
      const T kv = Kf[id];
#pragma unroll
      for (int c = 0; c < CR; ++c) cfma(acc[a][c], kv, q[c]);
    }
  }
#pragma unroll
  for (int a = 0; a < XR; ++a) {
    if (xb + a >= nt) break;
    T* out = Rh + f * B * C + (int64_t)tgt[t0 + xb + a] * C + cg * CR;
#pragma unroll
    for (int c = 0; c < CR; ++c) out[c] = acc[a][c];
  }
}

// Top grid level, 32 channels (8 right-hand sides), FP32: every block owns one
// tile of <= 128 targets and one frequency; chunks of YS sources are staged in
// shared memory by cp.async (kernel values gathered through the index tile,
// zero-filled for excluded pairs; spectra copied 16 bytes at a time), double
// buffered so the next chunk's gathers run while the current chunk is
// multiplied; each thread runs 8 targets x 4 channels out of shared memory.
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem, bool valid) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  const int sz = valid ? 8 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(sa), "l"(gmem), "r"(sz));
}
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, bool valid) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  const int sz = valid ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(sz));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

template <int YS>
__global__ void __launch_bounds__(128) k_mac_top32(const float2* __restrict__ Qh, float2* __restrict__ Rh,
                                                   const float2* __restrict__ Kh, int64_t B, int64_t O,
                                                   int64_t nf, const int64_t* __restrict__ tgt_ptr,
                                                   const int32_t* __restrict__ tgt,
                                                   const int64_t* __restrict__ src_ptr,
                                                   const int32_t* __restrict__ src,
                                                   const int64_t* __restrict__ kidx_off,
                                                   const int32_t* __restrict__ kidx, int64_t f0) {
  extern __shared__ __align__(16) unsigned char mac_smem[];
  float2(*Ks)[YS][128] = reinterpret_cast<float2(*)[YS][128]>(mac_smem);
  float2(*Qs)[YS][32] = reinterpret_cast<float2(*)[YS][32]>(mac_smem + 2 * sizeof(float2) * YS * 128);
  const int tile = blockIdx.x;
  const int64_t f = f0 + blockIdx.y;
  if (f >= nf) return;
  const int64_t t0 = tgt_ptr[tile], nt = tgt_ptr[tile + 1] - t0;
  const int64_t s0 = src_ptr[tile], ns = src_ptr[tile + 1] - s0;
  const int tpad = (int)(((nt + 7) / 8) * 8);
  const int32_t* kb = kidx + kidx_off[tile];
  const float2* Qf = Qh + f * B * 32;
  const float2* Kf = Kh + f * O;
  const int tg = threadIdx.x >> 3, cg = threadIdx.x & 7;
  const float2 zero = make_float2(0.f, 0.f);
  auto stage = [&](int buf, int64_t j0) {
    const int jn = (int)min((int64_t)YS, ns - j0);
    for (int e = threadIdx.x; e < YS * 128; e += 128) {
      const int j = e >> 7, a = e & 127;
      int32_t id = -1;
      if (j < jn && a < tpad) id = __ldg(kb + (j0 + j) * tpad + a);
      cp_async8(&Ks[buf][j][a], id >= 0 ? (const void*)(Kf + id) : (const void*)Kf, id >= 0);
    }
    for (int e = threadIdx.x; e < YS * 16; e += 128) {
      const int j = e >> 4, c2 = (e & 15) * 2;
      const bool ok = j < jn;
      const int32_t y = ok ? __ldg(src + s0 + j0 + j) : 0;
      cp_async16(&Qs[buf][j][c2], Qf + (int64_t)y * 32 + c2, ok);
    }
    cp_async_commit();
  };
  float2 acc[8][4];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[a][c] = zero;
  const int nchunks = (int)((ns + YS - 1) / YS);
  if (nchunks > 0) stage(0, 0);
  for (int ch = 0; ch < nchunks; ++ch) {
    const int buf = ch & 1;
    if (ch + 1 < nchunks) {
      stage(buf ^ 1, (int64_t)(ch + 1) * YS);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const int jn = (int)min((int64_t)YS, ns - (int64_t)ch * YS);
    if (tg * 8 < nt) {
      for (int j = 0; j < jn; ++j) {
        const float4 qa = *reinterpret_cast<const float4*>(&Qs[buf][j][cg * 4]);
        const float4 qb = *reinterpret_cast<const float4*>(&Qs[buf][j][cg * 4 + 2]);
        const float2 q[4] = {make_float2(qa.x, qa.y), make_float2(qa.z, qa.w), make_float2(qb.x, qb.y),
                             make_float2(qb.z, qb.w)};
#pragma unroll
        for (int a = 0; a < 8; ++a) {
          const float2 kv = Ks[buf][j][tg * 8 + a];
#pragma unroll
          for (int c = 0; c < 4; ++c) cfma(acc[a][c], kv, q[c]);
        }
      }
    }
    __syncthreads();
  }
  if (tg * 8 >= nt) return;
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    if (tg * 8 + a >= nt) break;
    float2* out = Rh + f * B * 32 + (int64_t)tgt[t0 + tg * 8 + a] * 32 + cg * 4;
    *reinterpret_cast<float4*>(out) = make_float4(acc[a][0].x, acc[a][0].y, acc[a][1].x, acc[a][1].y);
    *reinterpret_cast<float4*>(out + 2) = make_float4(acc[a][2].x, acc[a][2].y, acc[a][3].x, acc[a][3].y);
  }
}

// Translation from the interaction lists: a thread owns NU units of 16 bytes of one
// (frequency, target) and runs down the target's list, four pairs in flight; NU = 2
// takes the list entry and the kernel value once for twice the products.  The
// register tiles of k_mac_tiled visit every (source, target) slot of a tile, pairs or
// not (FP64 multiply-adds of excluded slots cost as much as the others), and leave
// most of the chip idle on few tiles and channels; a kernel with the kernel rows of
// eight frequencies in shared memory and 8 targets per thread waited for its dependent
// loads.  Sources ascend in all of them, so the sums are the same bit for bit.  What
// bounds it: L1 requests.  ms: 1,920 unknowns, FP64, one vector 0.076 -> 0.045; 6,750,
// FP32, one vector 0.065 -> 0.032; 48,000, FP32, leaf level, one vector 0.33 -> 0.16, 4
// vectors 0.81 -> 0.36, 8 vectors 0.76 -> 0.59; 48,000, FP64, 8 vectors, top level
// 31.1 -> 27.8.
template <typename R, int NU>
__global__ void __launch_bounds__(128) k_mac_list(const typename U16<R>::T* __restrict__ Qh,
                                                  typename U16<R>::T* __restrict__ Rh,
                                                  const cpx_t<R>* __restrict__ Kh, int64_t B, int U, int64_t O,
                                                  const int64_t* __restrict__ il_ptr,
                                                  const int32_t* __restrict__ il_src,
                                                  const int32_t* __restrict__ il_off, int64_t f0) {
  using T = typename U16<R>::T;
  const int64_t t = (int64_t)blockIdx.x * 128 + threadIdx.x;
  const int US = U / NU;
  const int64_t x = t / US, f = f0 + blockIdx.y;
  const int u = (int)(t - x * US);
  if (x >= B) return;
  const T* Qf = Qh + f * B * U + u;
  const cpx_t<R>* Kf = Kh + f * O;
  T acc[NU];
#pragma unroll
  for (int v = 0; v < NU; ++v) acc[v] = U16<R>::zero();
  const int64_t e1 = il_ptr[x + 1];
  int64_t e = il_ptr[x];
  const auto mac = [&](T& s, const cpx_t<R>& k, const T& q) {
    cpx_t<R> a = mk<R>(s.x, s.y);
    cfma(a, k, mk<R>(q.x, q.y));
    s.x = a.x, s.y = a.y;
    if constexpr (sizeof(R) == 4) {
      a = mk<R>(s.z, s.w);
      cfma(a, k, mk<R>(q.z, q.w));
      s.z = a.x, s.w = a.y;
    }
  };
  for (; e + 4 <= e1; e += 4) {
    cpx_t<R> k[4];
    T q[4][NU];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      k[i] = Kf[__ldg(il_off + e + i)];
      const T* qp = Qf + (int64_t)__ldg(il_src + e + i) * U;
#pragma unroll
      for (int v = 0; v < NU; ++v) q[i][v] = __ldg(qp + v * US);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int v = 0; v < NU; ++v) mac(acc[v], k[i], q[i][v]);
  }
  for (; e < e1; ++e) {
    const cpx_t<R> k = Kf[__ldg(il_off + e)];
    const T* qp = Qf + (int64_t)__ldg(il_src + e) * U;
#pragma unroll
    for (int v = 0; v < NU; ++v) mac(acc[v], k, __ldg(qp + v * US));
  }
#pragma unroll
  for (int v = 0; v < NU; ++v) Rh[(f * B + x) * U + u + v * US] = acc[v];
}

template <typename R>
void launch_mac(const cpx_t<R>* Qh, cpx_t<R>* Rh, const cpx_t<R>* Kh, int64_t B, int C, int64_t O,
                int64_t nf, int64_t ntiles, int max_tile_targets, const int64_t* tgt_ptr, const int32_t* tgt,
                const int64_t* src_ptr, const int32_t* src, const int64_t* kidx_off, const int32_t* kidx,
                const int64_t* il_ptr, const int32_t* il_src, const int32_t* il_off, cudaStream_t s) {
  if (B <= 0 || nf <= 0 || ntiles <= 0) return;
  // a negative tile size asks for the register-tile kernel (autotuner choice)
  const bool force_reg = max_tile_targets < 0;
  if (force_reg) max_tile_targets = -max_tile_targets;
  if (!force_reg && sizeof(R) == 4 && C == 32 && max_tile_targets > 8 && max_tile_targets <= 128) {
    constexpr int YS = 16;
    const size_t smem = 2 * sizeof(float2) * YS * (128 + 32);
    static SmemAttr attr;
    smem_attr_once(k_mac_top32<YS>, (int)smem, attr.v);
    for (int64_t f0 = 0; f0 < nf; f0 += 65535) {
      int64_t nfc = std::min<int64_t>(65535, nf - f0);
      dim3 grid((unsigned)ntiles, (unsigned)nfc);
      k_mac_top32<YS><<<grid, 128, smem, s>>>((const float2*)Qh, (float2*)Rh, (const float2*)Kh, B, O, nf, tgt_ptr,
                                              tgt, src_ptr, src, kidx_off, kidx, f0);
    }
    return;
  }
  // From the lists: in FP64 always; in FP32 on interaction-list tiles (at most 8
  // targets), on top levels of at most 64 boxes, and otherwise for 12 channels and
  // more that are no multiple of 8 (128 boxes, 21^3 frequencies, 12, 20 and 28
  // channels: 1.02, 1.72 and 2.21 ms in register tiles, 0.98, 1.47 and 1.89 from the
  // lists).  Wide tiles of 4 channels reuse each kernel value for more products (0.51 ms
  // against 0.57), and those of 8, 16 and 24 take 8 channels per thread (0.83, 1.27
  // and 1.78 ms with 4; 0.68, 1.15 and 1.51 with 8; 0.76, 1.14 and 1.64 from the lists).
  const bool wide = max_tile_targets > 8 && !(ntiles == 1 && max_tile_targets <= 64);
  const bool cr8 = sizeof(R) == 4 && C % 8 == 0 && !force_reg;
  if (!force_reg && (sizeof(R) == 8 || !wide || (C >= 12 && !cr8))) {
    const int U = C * (int)sizeof(cpx_t<R>) / 16;
    const auto run = [&](auto k, int nu) {
      const unsigned gx = (unsigned)ceil_div(B * (U / nu), 128);
      for (int64_t f0 = 0; f0 < nf; f0 += 65535)
        k<<<dim3(gx, (unsigned)std::min<int64_t>(65535, nf - f0)), 128, 0, s>>>(
            reinterpret_cast<const typename U16<R>::T*>(Qh), reinterpret_cast<typename U16<R>::T*>(Rh), Kh, B, U, O,
            il_ptr, il_src, il_off, f0);
    };
    // two units per thread where there are enough (FP32; 8 channels: 0.171 ms with
    // one on the leaf level of 21,870 unknowns, 0.181 with two; 16: 0.284 and 0.255)
    if constexpr (sizeof(R) == 4) {
      if (C >= 12 && U % 2 == 0) return run(k_mac_list<R, 2>, 2);
    }
    return run(k_mac_list<R, 1>, 1);
  }
  constexpr int XR = 8;
  const auto run = [&](auto k, int cr) {
    const int ncg = C / cr;
    const int ntx = (max_tile_targets + XR - 1) / XR;
    const int per_f = ntx * ncg;
    const int fpb = per_f >= 128 ? 1 : 128 / per_f;
    const int threads = fpb * per_f;
    const int64_t fchunk = (int64_t)65535 * fpb;
    for (int64_t f0 = 0; f0 < nf; f0 += fchunk) {
      int64_t nfc = std::min<int64_t>(fchunk, nf - f0);
      dim3 grid((unsigned)ntiles, (unsigned)ceil_div(nfc, fpb));
      k<<<grid, threads, 0, s>>>(Qh, Rh, Kh, B, C, O, nf, tgt_ptr, tgt, src_ptr, src, kidx_off, kidx, fpb, ntx, f0);
    }
  };
  if constexpr (sizeof(R) == 4) {
    if (cr8) return run(k_mac_tiled<R, XR, 8>, 8);
  }
  run(k_mac_tiled<R, XR, 4>, 4);
}

// ---------------------------------------------------------------- kernel samples
// Kc[o][i0][i1][i2] = g(o h + t Delta), t_d = i_d (i_d < shat) or i_d - n, FP64.
// Samples of the Green's function g(D) = exp(-jkR) / (4 pi R) (comp < 0) or
// of one entry of its Hessian d_a d_b g (comp 0..5: ab = 00, 01, 02, 11, 12,
// 22; the dyadic factorization of Sec. VI-C) at D = o h + t Delta, with
//   d_a d_b g = g2 r_a r_b + (g1 / R) (delta_ab - r_a r_b),
//   g1 = dg/dR = -(jk + 1/R) g,  g2 = d2g/dR2 = ((jk + 1/R)^2 + 1/R^2) g,
// r = D / R.
__global__ void k_kernel_samples(double2* __restrict__ Kc, const int32_t* __restrict__ offsets,
                                 int64_t o0, int64_t no, int n, int shat, double h, double Delta,
                                 double k, int comp) {
  const int64_t n3 = (int64_t)n * n * n;
  const int64_t total = no * n3;
  const int ca = comp < 0 ? 0 : (comp < 3 ? 0 : (comp < 5 ? 1 : 2));
  const int cb = comp < 0 ? 0 : (comp < 3 ? comp : (comp < 5 ? comp - 2 : 2));
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t o = idx / n3, e = idx - o * n3;
    int i0 = (int)(e / (n * n)), i1 = (int)((e / n) % n), i2 = (int)(e % n);
    int t0 = i0 < shat ? i0 : i0 - n, t1 = i1 < shat ? i1 : i1 - n, t2 = i2 < shat ? i2 : i2 - n;
    const int32_t* ov = offsets + 3 * (o0 + o);
    double d[3] = {ov[0] * h + t0 * Delta, ov[1] * h + t1 * Delta, ov[2] * h + t2 * Delta};
    double R = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    double sn, cs;
    sincos(k * R, &sn, &cs);
    double fct = 1.0 / (12.566370614359172953850573533118 * R);
    const double2 g = make_double2(cs * fct, -sn * fct);
    if (comp < 0) {
      Kc[idx] = g;
      continue;
    }
    // a = 1/R + jk; g1 = -a g; g2 = (a^2 + 1/R^2) g = (2/R^2 - k^2 + 2jk/R) g
    const double iR = 1.0 / R;
    const double2 a = make_double2(iR, k);
    const double2 g1 = make_double2(-(a.x * g.x - a.y * g.y), -(a.x * g.y + a.y * g.x));
    const double2 c2 = make_double2(2.0 * iR * iR - k * k, 2.0 * k * iR);
    const double2 g2 = make_double2(c2.x * g.x - c2.y * g.y, c2.x * g.y + c2.y * g.x);
    const double rr = d[ca] * d[cb] * iR * iR;
    const double dl = (ca == cb ? 1.0 : 0.0) - rr;
    Kc[idx] = make_double2(g2.x * rr + g1.x * iR * dl, g2.y * rr + g1.y * iR * dl);
  }
}

// Dyadic translation (Sec. VI-C): for every frequency, target box x and
// right-hand side c, R[x][a] = sum_{y in IL(x)} sum_b H_ab(x - y) Q[y][b] over
// the three vector components a, b (H symmetric: six spectra, ab = 00, 01,
// 02, 11, 12, 22); the fourth component of R is set to zero.  Q and R are
// [n^3][B][4 nr] (component-major channels), K[ab] are [n^3][O].  One thread
// per (frequency, box, right-hand side), the interaction lists of the level.
template <typename R>
__global__ void k_mac_dyad(const cpx_t<R>* __restrict__ Q, cpx_t<R>* __restrict__ Rout, KH6<R> K, int64_t B,
                           int nr, int64_t nf, int64_t O, const int64_t* __restrict__ il_ptr,
                           const int32_t* __restrict__ il_src, const int32_t* __restrict__ il_off) {
  using T = cpx_t<R>;
  const int64_t C = 4 * nr;
  const int64_t total = nf * B * nr;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(idx % nr);
    const int64_t x = (idx / nr) % B, f = idx / (nr * B);
    T acc[3] = {mk<R>(0, 0), mk<R>(0, 0), mk<R>(0, 0)};
    for (int64_t e = il_ptr[x]; e < il_ptr[x + 1]; ++e) {
      const T* q = Q + (f * B + il_src[e]) * C + c;
      const T q0 = q[0], q1 = q[nr], q2 = q[2 * nr];
      const int64_t ko = f * O + il_off[e];
      const T h00 = K.k[0][ko], h01 = K.k[1][ko], h02 = K.k[2][ko];
      const T h11 = K.k[3][ko], h12 = K.k[4][ko], h22 = K.k[5][ko];
      cfma(acc[0], h00, q0);
      cfma(acc[0], h01, q1);
      cfma(acc[0], h02, q2);
      cfma(acc[1], h01, q0);
      cfma(acc[1], h11, q1);
      cfma(acc[1], h12, q2);
      cfma(acc[2], h02, q0);
      cfma(acc[2], h12, q1);
      cfma(acc[2], h22, q2);
    }
    T* r = Rout + (f * B + x) * C + c;
    r[0] = acc[0];
    r[nr] = acc[1];
    r[2 * nr] = acc[2];
    r[3 * nr] = mk<R>(0, 0);
  }
}

template <typename R>
void launch_mac_dyad(const cpx_t<R>* Q, cpx_t<R>* Rout, KH6<R> K, int64_t B, int nr, int64_t nf, int64_t O,
                     const int64_t* il_ptr, const int32_t* il_src, const int32_t* il_off, cudaStream_t s) {
  const int64_t total = nf * B * nr;
  if (total <= 0) return;
  int64_t blocks = ceil_div(total, 256);
  if (blocks > 152 * 64) blocks = 152 * 64;
  k_mac_dyad<R><<<(unsigned)blocks, 256, 0, s>>>(Q, Rout, K, B, nr, nf, O, il_ptr, il_src, il_off);
}
template void launch_mac_dyad<float>(const float2*, float2*, KH6<float>, int64_t, int, int64_t, int64_t,
                                     const int64_t*, const int32_t*, const int32_t*, cudaStream_t);
template void launch_mac_dyad<double>(const double2*, double2*, KH6<double>, int64_t, int, int64_t, int64_t,
                                      const int64_t*, const int32_t*, const int32_t*, cudaStream_t);

void launch_kernel_samples(double2* Kc, const int32_t* offsets, int64_t o0, int64_t no, int n,
                           int shat, double h, double Delta, double k, int comp, cudaStream_t s) {
  int64_t total = no * (int64_t)n * n * n;
  if (total <= 0) return;
  int64_t blocks = ceil_div(total, 256);
  if (blocks > 152 * 64) blocks = 152 * 64;
  k_kernel_samples<<<(unsigned)blocks, 256, 0, s>>>(Kc, offsets, o0, no, n, shat, h, Delta, k, comp);
}

template <typename R>
__global__ void k_convert(const double2* __restrict__ in, cpx_t<R>* __restrict__ out, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = mk<R>((R)in[i].x, (R)in[i].y);
}
template <typename R>
void launch_convert(const double2* in, cpx_t<R>* out, int64_t n, cudaStream_t s) {
  if (n <= 0) return;
  int64_t blocks = ceil_div(n, 256);
  if (blocks > 152 * 64) blocks = 152 * 64;
  k_convert<R><<<(unsigned)blocks, 256, 0, s>>>(in, out, n);
}

// ---------------------------------------------------------------- vectors
__global__ void k_permute_in(const double2* __restrict__ x, int64_t ldx, const int32_t* __restrict__ perm,
                             int64_t N, int nr, double2* __restrict__ xs) {
  int64_t total = N * nr;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t r = idx / N, i = idx - r * N;
    xs[r * N + i] = x[r * ldx + perm[i]];
  }
}
void launch_permute_in(const double2* x, int64_t ldx, const int32_t* perm, int64_t N, int nr,
                       double2* xs, cudaStream_t s) {
  int64_t total = N * nr;
  if (total <= 0) return;
  int64_t blocks = ceil_div(total, 256);
  if (blocks > 152 * 64) blocks = 152 * 64;
  k_permute_in<<<(unsigned)blocks, 256, 0, s>>>(x, ldx, perm, N, nr, xs);
}

// rho[r][t] = sum over the 3 RWGs of triangle t of sign * x (Sigma^T x, FP64)
__global__ void k_charges(const double2* __restrict__ xs, int64_t ldx, const int32_t* __restrict__ tri_rwg,
                          const int8_t* __restrict__ tri_sgn, int64_t Nt, int nr, double2* __restrict__ rho,
                          int64_t ldr) {
  int64_t total = Nt * nr;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t r = idx / Nt, t = idx - r * Nt;
    double2 a = make_double2(0, 0);
    for (int q = 0; q < 3; ++q) {
      int32_t i = tri_rwg[3 * t + q];
      if (i < 0) continue;
      double2 v = xs[r * ldx + i];
      double sg = (double)tri_sgn[3 * t + q];
      a.x += sg * v.x;
      a.y += sg * v.y;
    }
    rho[r * ldr + t] = a;
  }
}
void launch_charges(const double2* xs, int64_t ldx, const int32_t* tri_rwg, const int8_t* tri_sgn,
                    int64_t Nt, int nr, double2* rho, int64_t ldr, cudaStream_t s) {
  int64_t total = Nt * nr;
  if (total <= 0) return;
  int64_t blocks = ceil_div(total, 256);
  if (blocks > 152 * 64) blocks = 152 * 64;
  k_charges<<<(unsigned)blocks, 256, 0, s>>>(xs, ldx, tri_rwg, tri_sgn, Nt, nr, rho, ldr);
}

// y[r][m] = cA * yA[r][i] + cV * (w[r][t+] - w[r][t-]), m = perm[i]; with
// rts null (direct factorization) the scalar part is w[r][i] itself.
// yAn, wn (optional): near-field parts kept apart from the far parts yA, w
__global__ void k_combine(const double2* __restrict__ yA, int64_t ldA, const double2* __restrict__ w,
                          int64_t ldw, const double2* __restrict__ yAn, const double2* __restrict__ wn,
                          const int32_t* __restrict__ perm, const int32_t* __restrict__ rts,
                          int64_t N, int nr, double2 cA, double2 cV, double2* __restrict__ y, int64_t ldy,
                          double2* __restrict__ yAo, double2* __restrict__ yVo) {
  int64_t total = N * nr;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t r = idx / N, i = idx - r * N;
    double2 a = yA[r * ldA + i];
    double2 v;
    if (rts) {
      // star factorization: the charge part of RWG i is w(c+) - w(c-)
      double2 wp = w[r * ldw + rts[2 * i]], wm = w[r * ldw + rts[2 * i + 1]];
      if (yAn) {
        a = cadd(a, yAn[r * ldA + i]);
        wp = cadd(wp, wn[r * ldw + rts[2 * i]]);
        wm = cadd(wm, wn[r * ldw + rts[2 * i + 1]]);
      }
      v = make_double2(wp.x - wm.x, wp.y - wm.y);
    } else {
      // direct factorization: the scalar part is per RWG already
      v = w[r * ldw + i];
      if (yAn) {
        a = cadd(a, yAn[r * ldA + i]);
        v = cadd(v, wn[r * ldw + i]);
      }
    }
    int64_t m = perm[i];
    if (y) y[r * ldy + m] = cadd(cmul(cA, a), cmul(cV, v));
    if (yAo) yAo[r * ldy + m] = a;
    if (yVo) yVo[r * ldy + m] = v;
  }
}
void launch_combine(const double2* yA, int64_t ldA, const double2* w, int64_t ldw, const double2* yAn,
                    const double2* wn, const int32_t* rwg_perm, const int32_t* rwg_tri_sorted, int64_t N, int nr,
                    double2 cA, double2 cV, double2* y, int64_t ldy, double2* yAout, double2* yVout,
                    cudaStream_t s) {
  int64_t total = N * nr;
  if (total <= 0) return;
  int64_t blocks = ceil_div(total, 256);
  if (blocks > 152 * 64) blocks = 152 * 64;
  k_combine<<<(unsigned)blocks, 256, 0, s>>>(yA, ldA, w, ldw, yAn, wn, rwg_perm, rwg_tri_sorted, N, nr, cA, cV,
                                             y, ldy, yAout, yVout);
}

// Plane-wave RHS: per RWG, both triangles with a degree-10 collapsed rule (up to
// RHS_DIRECT waves, and boxes with more than 1,472 triangles).
__constant__ double c_q6[3][36];
__global__ void k_rhs_pw(const double* __restrict__ V, const int32_t* __restrict__ T,
                         const double* __restrict__ area, const int32_t* __restrict__ tri_pm,
                         const int32_t* __restrict__ free_pm, int64_t N, double k,
                         const double* __restrict__ khat, const double* __restrict__ pol, int nr,
                         double2* __restrict__ rhs, int64_t ld) {
  int64_t total = N * nr;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t r = idx / N, m = idx - r * N;
    const double* kh = khat + 3 * r;
    const double* pl = pol + 3 * r;
    double2 acc = make_double2(0, 0);
    for (int s = 0; s < 2; ++s) {
      int t = tri_pm[2 * m + s];
      const double* xf = V + 3 * free_pm[2 * m + s];
      double sc = (s == 0 ? 1.0 : -1.0) / (2.0 * area[t]);
      const double* a = V + 3 * T[3 * t];
      const double* b = V + 3 * T[3 * t + 1];
      const double* c = V + 3 * T[3 * t + 2];
      for (int q = 0; q < 36; ++q) {
        double xi = c_q6[0][q], eta = c_q6[1][q], w = c_q6[2][q] * 2.0 * area[t];
        double x[3];
        for (int d = 0; d < 3; ++d) x[d] = a[d] + xi * (b[d] - a[d]) + eta * (c[d] - a[d]);
        double ph = -k * (kh[0] * x[0] + kh[1] * x[1] + kh[2] * x[2]);
        double sn, cs;
        sincos(ph, &sn, &cs);
        double fp = 0;
        for (int d = 0; d < 3; ++d) fp += (x[d] - xf[d]) * pl[d];
        fp *= sc * w;
        acc.x += fp * cs;
        acc.y += fp * sn;
      }
    }
    rhs[r * ld + m] = acc;
  }
}
// Plane waves by leaf box: the triangles of the box's RWGs (its triangle set)
// are integrated once per wave and combined into the RWGs, instead of 72 sines and
// cosines per RWG.  For one triangle and wave, with x = c + (xi - 1/3) e1 +
// (eta - 1/3) e2 (c the centroid), alpha = -k khat.e1 and beta = -k khat.e2, the points
// of the collapsed 6 x 6 rule, xi = u_a, eta = (1 - u_a)(1/2 +- t_b), have the phases
//   phi_c + psi_a +- t_b gamma_a,  psi_a = (u_a - 1/3)(alpha - beta / 2),  gamma_a = (1 - u_a) beta,
// so a row a of six points needs one complex exponential of psi_a and the
// rule's even and odd sums C = sum_b w_b cos(t_b gamma), S = sum_b w_b t_b sin(t_b gamma),
// which are power series in gamma^2 with fixed coefficients.  Elements are a
// fraction of a wavelength, so Taylor series of eight terms leave less than
// 3e-16 for |gamma| <= 1 and |psi| <= 0.6; beyond (elements above lambda / 7) the row
// calls cos and sin.  Same rule, same points as k_rhs_pw, up to rounding.
//
// What bounds it: the FP64 pipe, about 350 operations per triangle and wave (2 per
// clock and SM).  38,720 triangles, 360 waves: 126 -> 12.0 ms.
__constant__ double c_pw_u[6], c_pw_w[6], c_pw_t[3], c_pw_v[3], c_pw_c[8], c_pw_s[8];

__device__ __forceinline__ double pw_poly8(const double* c, double x) {
  double r = c[7];
#pragma unroll
  for (int n = 6; n >= 0; --n) r = fma(r, x, c[n]);
  return r;
}
__global__ void __launch_bounds__(128) k_rhs_box(const RhsGeom g, const double* __restrict__ khat,
                                                 const double* __restrict__ pol, int nr, int W,
                                                 double2* __restrict__ rhs, int64_t ld) {
  extern __shared__ double2 pw_smem[];  // [triangle][wave][F0, G1]
  const int64_t t0 = g.tset_ptr[blockIdx.x], i0 = g.box_rwg_ptr[blockIdx.x];
  const int ntri = (int)(g.tset_ptr[blockIdx.x + 1] - t0), nrwg = (int)(g.box_rwg_ptr[blockIdx.x + 1] - i0);
  const int r0 = blockIdx.y * W, nw = min(W, nr - r0);
  const double third = 1.0 / 3.0;
  // Taylor coefficients of cos and sin(x) / x in x^2
  const double tc[8] = {1.0, -1.0 / 2, 1.0 / 24, -1.0 / 720, 1.0 / 40320, -1.0 / 3628800, 1.0 / 479001600,
                        -1.0 / 87178291200.0};
  const double ts[8] = {1.0, -1.0 / 6, 1.0 / 120, -1.0 / 5040, 1.0 / 362880, -1.0 / 39916800, 1.0 / 6227020800.0,
                        -1.0 / 1307674368000.0};
  for (int e = threadIdx.x; e < ntri * nw; e += blockDim.x) {
    const int w = e / ntri, t = e - w * ntri, tri = g.tset[t0 + t];
    const double* kh = khat + 3 * (r0 + w);
    const double* pl = pol + 3 * (r0 + w);
    const double* va = g.V + 3 * (int64_t)g.T[3 * tri];
    const double* vb = g.V + 3 * (int64_t)g.T[3 * tri + 1];
    const double* vc = g.V + 3 * (int64_t)g.T[3 * tri + 2];
    double phi = 0, alpha = 0, beta = 0, p1 = 0, p2 = 0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double a = va[d], e1 = vb[d] - a, e2 = vc[d] - a;
      phi = fma(kh[d], a + third * (e1 + e2), phi);
      alpha = fma(kh[d], e1, alpha);
      beta = fma(kh[d], e2, beta);
      p1 = fma(pl[d], e1, p1);
      p2 = fma(pl[d], e2, p2);
    }
    phi *= -g.k, alpha *= -g.k, beta *= -g.k;
    const double delta = alpha - 0.5 * beta;
    const bool series = fabs(beta) <= 1.0 && fabs(delta) <= 0.9;
    double2 F0 = make_double2(0, 0), Fx = F0, Fe = F0;
#pragma unroll 1
    for (int a = 0; a < 6; ++a) {
      const double u = c_pw_u[a], gam = (1.0 - u) * beta, psi = (u - third) * delta;
      double C, S, cs, sn;
      if (series) {
        const double g2 = gam * gam, q2 = psi * psi;
        C = pw_poly8(c_pw_c, g2);
        S = gam * pw_poly8(c_pw_s, g2);
        cs = pw_poly8(tc, q2);
        sn = psi * pw_poly8(ts, q2);
      } else {
        C = S = 0;
        for (int b = 0; b < 3; ++b) {
          double sb, cb;
          sincos(c_pw_t[b] * gam, &sb, &cb);
          C = fma(c_pw_v[b], cb, C);
          S = fma(c_pw_v[b] * c_pw_t[b], sb, S);
        }
        sincos(psi, &sn, &cs);
      }
      const double wa = c_pw_w[a], wc = wa * C, we = wa * (1.0 - u), p = 0.5 * we * C, q = we * S;
      F0.x = fma(wc, cs, F0.x);
      F0.y = fma(wc, sn, F0.y);
      Fx.x = fma(u * wc, cs, Fx.x);
      Fx.y = fma(u * wc, sn, Fx.y);
      Fe.x = fma(p, cs, fma(-q, sn, Fe.x));
      Fe.y = fma(p, sn, fma(q, cs, Fe.y));
    }
    double sp, cp;
    sincos(phi, &sp, &cp);
    const double2 G = make_double2(p1 * Fx.x + p2 * Fe.x, p1 * Fx.y + p2 * Fe.y);
    pw_smem[2 * (t * W + w)] = make_double2(F0.x * cp - F0.y * sp, F0.x * sp + F0.y * cp);
    pw_smem[2 * (t * W + w) + 1] = make_double2(G.x * cp - G.y * sp, G.x * sp + G.y * cp);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < nrwg * nw; e += blockDim.x) {
    const int w = e / nrwg, i = e - w * nrwg;
    const int64_t m = g.rwg_perm[i0 + i];
    const double* pl = pol + 3 * (r0 + w);
    double2 acc = make_double2(0, 0);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int t = g.rwg_tl[2 * (i0 + i) + s];
      const double* a = g.V + 3 * (int64_t)g.T[3 * g.tset[t0 + t]];
      const double* xf = g.V + 3 * (int64_t)g.free_pm[2 * m + s];
      const double d = (a[0] - xf[0]) * pl[0] + (a[1] - xf[1]) * pl[1] + (a[2] - xf[2]) * pl[2];
      const double2 F0 = pw_smem[2 * (t * W + w)], G = pw_smem[2 * (t * W + w) + 1];
      const double2 v = make_double2(fma(d, F0.x, G.x), fma(d, F0.y, G.y));
      acc = s == 0 ? v : csub(acc, v);
    }
    rhs[(int64_t)(r0 + w) * ld + m] = acc;
  }
}
int upload_rhs_rule(const double* q6) {
  // rows of the collapsed rule: xi = u_a, eta = (1 - u_a) v_b, weight w_a v_b-weight;
  // v_b = 1/2 -+ t_b in pairs of equal weight
  double u[6], w[6], t[3], v[3], c[8], sc[8];
  for (int a = 0; a < 6; ++a) {
    u[a] = q6[6 * a];
    w[a] = 0;
    for (int b = 0; b < 6; ++b) w[a] += q6[72 + 6 * a + b];
  }
  for (int b = 0; b < 3; ++b) {
    t[b] = q6[36 + 3 + b] / (1.0 - u[0]) - 0.5;
    v[b] = 2.0 * q6[72 + 3 + b] / w[0];
  }
  double fc = 1.0, fs = 1.0;  // (2n)!, (2n + 1)! with the sign
  for (int n = 0; n < 8; ++n) {
    if (n) fc *= -(2.0 * n) * (2.0 * n - 1.0), fs *= -(2.0 * n) * (2.0 * n + 1.0);
    c[n] = sc[n] = 0;
    for (int b = 0; b < 3; ++b) {
      c[n] += v[b] * std::pow(t[b], 2 * n) / fc;
      sc[n] += v[b] * std::pow(t[b], 2 * n + 2) / fs;
    }
  }
  const bool ok = cudaMemcpyToSymbol(c_q6, q6, sizeof(double) * 108) == cudaSuccess &&
                  cudaMemcpyToSymbol(c_pw_u, u, sizeof(u)) == cudaSuccess &&
                  cudaMemcpyToSymbol(c_pw_w, w, sizeof(w)) == cudaSuccess &&
                  cudaMemcpyToSymbol(c_pw_t, t, sizeof(t)) == cudaSuccess &&
                  cudaMemcpyToSymbol(c_pw_v, v, sizeof(v)) == cudaSuccess &&
                  cudaMemcpyToSymbol(c_pw_c, c, sizeof(c)) == cudaSuccess &&
                  cudaMemcpyToSymbol(c_pw_s, sc, sizeof(sc)) == cudaSuccess;
  return ok ? 0 : -1;
}
constexpr int RHS_DIRECT = 64;
void launch_rhs_planewave(const RhsGeom& g, const double* khat, const double* pol, int nr, double2* rhs, int64_t ld,
                          cudaStream_t s) {
  int64_t total = g.N * nr;
  if (total <= 0) return;
  // More waves than one pass of a product has vectors: by leaf box where its
  // triangles' integrals fit in shared memory, up to 8 waves at a time (46 KB: no
  // opt-in, four blocks per SM).  65 waves, 58,080 unknowns: 22.9 ms direct, 2.4 by
  // box.  The line is no crossover of times: fewer waves keep every bit of the direct
  // sums that callers have had, because an FP32 product rounds them as vectors, and a
  // last bit of a component on a rounding boundary moves that product by up to 3e-9.
  // Longer sweeps differ from the direct sums in their last bits, with the same error
  // against exact values (5.4e-15 against 5.3e-15).
  const int64_t per = 2 * sizeof(double2) * (int64_t)g.max_tset;
  const int W = (int)std::min<int64_t>(std::min(nr, 8), 46 * 1024 / std::max<int64_t>(per, 1));
  if (nr > RHS_DIRECT && W >= 1 && g.n_boxes > 0 && (nr + W - 1) / W <= 65535) {
    k_rhs_box<<<dim3((unsigned)g.n_boxes, (unsigned)((nr + W - 1) / W)), 128, (size_t)(W * per), s>>>(g, khat, pol, nr,
                                                                                                  W, rhs, ld);
    return;
  }
  int64_t blocks = ceil_div(total, 128);
  if (blocks > 152 * 64) blocks = 152 * 64;
  k_rhs_pw<<<(unsigned)blocks, 128, 0, s>>>(g.V, g.T, g.area, g.tri_pm, g.free_pm, g.N, g.k, khat, pol, nr, rhs, ld);
}

// ---------------------------------------------------------------- Krylov
// Block sum of 512 per-thread values in a fixed order (warp shuffles, then
// the 16 warp sums in ascending order); the result is valid in thread 0.
template <typename T>
__device__ __forceinline__ T block_sum512(T v, T* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) red[wid] = v;
  __syncthreads();
  T s = 0;
  if (threadIdx.x == 0)
    for (int i = 0; i < 16; ++i) s += red[i];
  return s;
}

// h[r][i] = sum_n conj(V[r][i][n]) w[r][n]; grid (nbasis, nr), 512 threads.
// One block per output and a fixed summation order: the Arnoldi coefficients,
// and so the iterates, are the same on every run.
__global__ void __launch_bounds__(512) k_multidot(const double2* __restrict__ Vb, int64_t ldv_r, int64_t ldv_i,
                                                  const double2* __restrict__ w, int64_t ldw, int64_t N,
                                                  const int* __restrict__ active, double2* __restrict__ h,
                                                  int nbasis) {
  const int i = blockIdx.x, r = blockIdx.y;
  if (active && !active[r]) {
    if (threadIdx.x == 0) h[(int64_t)r * nbasis + i] = make_double2(0, 0);
    return;
  }
  const double2* v = Vb + r * ldv_r + i * ldv_i;
  const double2* wr = w + r * ldw;
  double sx = 0, sy = 0;
  for (int64_t n = threadIdx.x; n < N; n += blockDim.x) {
    double2 a = v[n], b = wr[n];
    sx += a.x * b.x + a.y * b.y;
    sy += a.x * b.y - a.y * b.x;
  }
  __shared__ double rx[16], ry[16];
  sx = block_sum512(sx, rx);
  sy = block_sum512(sy, ry);
  if (threadIdx.x == 0) h[(int64_t)r * nbasis + i] = make_double2(sx, sy);
}
void launch_multidot(const double2* Vb, int64_t ldv_r, int64_t ldv_i, int nbasis, const double2* w,
                     int64_t ldw, int64_t N, int nr, const int* active, double2* h, cudaStream_t s) {
  if (nbasis <= 0 || nr <= 0) return;
  dim3 grid(nbasis, nr);
  k_multidot<<<grid, 512, 0, s>>>(Vb, ldv_r, ldv_i, w, ldw, N, active, h, nbasis);
}

// w[r][n] += sign * sum_i h[r][i] V[r][i][n]
__global__ void k_multiaxpy(const double2* __restrict__ Vb, int64_t ldv_r, int64_t ldv_i, int nbasis,
                            const double2* __restrict__ h, int hstride, double2* __restrict__ w,
                            int64_t ldw, int64_t N, int nr, const int* __restrict__ active, double sign) {
  int64_t total = N * nr;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t r = idx / N, n = idx - r * N;
    if (active && !active[r]) continue;
    double2 acc = make_double2(0, 0);
    // eight basis vectors in flight, summed in order
    const double2* v = Vb + r * ldv_r + n;
    const double2* hr = h + r * hstride;
    int i = 0;
    for (; i + 8 <= nbasis; i += 8) {
      double2 b[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) b[q] = v[(i + q) * ldv_i];
#pragma unroll
      for (int q = 0; q < 8; ++q) cfma(acc, hr[i + q], b[q]);
    }
    for (; i < nbasis; ++i) cfma(acc, hr[i], v[i * ldv_i]);
    double2 t = w[r * ldw + n];
    w[r * ldw + n] = make_double2(t.x + sign * acc.x, t.y + sign * acc.y);
  }
}
void launch_multiaxpy(const double2* Vb, int64_t ldv_r, int64_t ldv_i, int nbasis, const double2* h,
                      int hstride, double2* w, int64_t ldw, int64_t N, int nr, const int* active,
                      double sign, cudaStream_t s) {
  int64_t total = N * nr;
  if (total <= 0 || nbasis <= 0) return;
  const int th = total < 152 * 512 ? 64 : 256;  // short vectors over all SMs
  int64_t blocks = ceil_div(total, th);
  if (blocks > 152 * 64) blocks = 152 * 64;
  k_multiaxpy<<<(unsigned)blocks, th, 0, s>>>(Vb, ldv_r, ldv_i, nbasis, h, hstride, w, ldw, N, nr, active,
                                               sign);
}

// out = a x + b y over n complex entries (real a, b)
__global__ void k_lincomb(const double2* __restrict__ x, const double2* __restrict__ y, double a, double b,
                          double2* __restrict__ out, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double2 u = x[i], v = y[i];
    out[i] = make_double2(a * u.x + b * v.x, a * u.y + b * v.y);
  }
}
void launch_lincomb(const double2* x, const double2* y, double a, double b, double2* out, int64_t n,
                    cudaStream_t s) {
  if (n <= 0) return;
  int64_t blocks = ceil_div(n, 256);
  if (blocks > 152 * 64) blocks = 152 * 64;
  k_lincomb<<<(unsigned)blocks, 256, 0, s>>>(x, y, a, b, out, n);
}

// out = a conj(x)
__global__ void k_conj_scale(const double2* __restrict__ x, double a, double2* __restrict__ out, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double2 v = x[i];
    out[i] = make_double2(a * v.x, -a * v.y);
  }
}
void launch_conj_scale(const double2* x, double a, double2* out, int64_t n, cudaStream_t s) {
  if (n <= 0) return;
  int64_t blocks = ceil_div(n, 256);
  if (blocks > 152 * 64) blocks = 152 * 64;
  k_conj_scale<<<(unsigned)blocks, 256, 0, s>>>(x, a, out, n);
}

// out[r] = sum_n |w[r][n]|^2; one 512-thread block per vector, fixed order
__global__ void __launch_bounds__(512) k_norms(const double2* __restrict__ w, int64_t ldw, int64_t N,
                                               double* out) {
  const int r = blockIdx.x;
  double s = 0;
  for (int64_t n = threadIdx.x; n < N; n += blockDim.x) {
    double2 a = w[r * ldw + n];
    s += a.x * a.x + a.y * a.y;
  }
  __shared__ double red[16];
  s = block_sum512(s, red);
  if (threadIdx.x == 0) out[r] = s;
}
void launch_norms(const double2* w, int64_t ldw, int64_t N, int nr, double* out, cudaStream_t s) {
  if (nr <= 0) return;
  k_norms<<<nr, 512, 0, s>>>(w, ldw, N, out);
}

// explicit instantiations
template void launch_up_fused<float>(const float2*, float2*, int64_t, int, int, int, const SparseMat<float>&,
                                     const int32_t*, cudaStream_t);
template void launch_up_fused<double>(const double2*, double2*, int64_t, int, int, int, const SparseMat<double>&,
                                      const int32_t*, cudaStream_t);
template void launch_down_fused<float>(const float2*, float2*, int64_t, int, int, int, const SparseMat<float>&,
                                       const int64_t*, const int8_t*, cudaStream_t);
template void launch_down_fused<double>(const double2*, double2*, int64_t, int, int, int, const SparseMat<double>&,
                                        const int64_t*, const int8_t*, cudaStream_t);
template void launch_mode_pair<float>(const float2*, View, float2*, View, int64_t, int, int, int, int, int, int,
                                      const float*, const float*, const int64_t*, const int64_t*, const int8_t*,
                                      const int8_t*, cudaStream_t);
template void launch_mode_pair<double>(const double2*, View, double2*, View, int64_t, int, int, int, int, int, int,
                                       const double*, const double*, const int64_t*, const int64_t*,
                                       const int8_t*, const int8_t*, cudaStream_t);
template bool launch_dft<float>(const float2*, View, float2*, View, int64_t, int, int, int, int, int, int,
                                const float2*, int, bool, cudaStream_t);
template bool launch_dft<double>(const double2*, View, double2*, View, int64_t, int, int, int, int, int, int,
                                 const double2*, int, bool, cudaStream_t);
template void launch_mode<float>(const float2*, View, float2*, View, int64_t, int, int, int, int, int, int,
                                 const void*, const void*, bool, const int8_t*, const int64_t*, bool,
                                 cudaStream_t);
template void launch_mode<double>(const double2*, View, double2*, View, int64_t, int, int, int, int, int, int,
                                  const void*, const void*, bool, const int8_t*, const int64_t*, bool,
                                  cudaStream_t);
template void launch_gather_build<float>(const float*, const int32_t*, const int32_t*, const int64_t*,
                                         const float*, const int32_t*, const int32_t*, const int64_t*,
                                         const int64_t*, const int64_t*, int64_t, int, int32_t*, int32_t*, float*,
                                         float*, cudaStream_t);
template void launch_gather_build<double>(const double*, const int32_t*, const int32_t*, const int64_t*,
                                          const double*, const int32_t*, const int32_t*, const int64_t*,
                                          const int64_t*, const int64_t*, int64_t, int, int32_t*, int32_t*,
                                          double*, double*, cudaStream_t);
template void launch_anterp<float>(const float*, const float*, const int32_t*, const int32_t*, const int64_t*,
                                   const int64_t*, const int64_t*, const int64_t*, int64_t, int, int, const int32_t*,
                                   const float2*, int64_t, const float2*, int64_t, int, float2*, int, cudaStream_t);
template void launch_anterp<double>(const double*, const double*, const int32_t*, const int32_t*, const int64_t*,
                                    const int64_t*, const int64_t*, const int64_t*, int64_t, int, int, const int32_t*,
                                    const double2*, int64_t, const double2*, int64_t, int, double2*, int, cudaStream_t);
template void launch_interp<float>(const float*, const int32_t*, const int32_t*, const int64_t*, const int32_t*,
                                   int64_t, const float*, const int32_t*, const int32_t*, const int64_t*,
                                   const int32_t*, int64_t, const float2*, int, int, double2*, int64_t,
                                   double2*, int64_t, cudaStream_t);
template void launch_interp<double>(const double*, const int32_t*, const int32_t*, const int64_t*,
                                    const int32_t*, int64_t, const double*, const int32_t*, const int32_t*,
                                    const int64_t*, const int32_t*, int64_t, const double2*, int, int,
                                    double2*, int64_t, double2*, int64_t, cudaStream_t);
template void launch_mac<float>(const float2*, float2*, const float2*, int64_t, int, int64_t, int64_t, int64_t,
                                int, const int64_t*, const int32_t*, const int64_t*, const int32_t*,
                                const int64_t*, const int32_t*, const int64_t*, const int32_t*, const int32_t*, cudaStream_t);
template void launch_mac<double>(const double2*, double2*, const double2*, int64_t, int, int64_t, int64_t,
                                 int64_t, int, const int64_t*, const int32_t*, const int64_t*, const int32_t*,
                                 const int64_t*, const int32_t*, const int64_t*, const int32_t*, const int32_t*, cudaStream_t);
template void launch_convert<float>(const double2*, float2*, int64_t, cudaStream_t);
template void launch_convert<double>(const double2*, double2*, int64_t, cudaStream_t);

}  // namespace efie
