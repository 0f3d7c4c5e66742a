// FP64 translation on the tensor cores.
//
// R^[f][x][c] = sum_{y in IL(x)} K^[f][o(x - y)] Q^[f][y][c] in FP64 is bound by a pipe
// of two multiply-adds per clock and SM (2 clocks per complex one and SM).  For
// one frequency it is a (targets x sources) times (sources x channels) product,
// so it runs like the FP64 near field (near_mma.cu): kernel spectra and source
// spectra are cut into six 10-bit digits (60 bits below the largest of a
// frequency's kernel row, and of a frequency's channel) whose products are exact
// FP16 MMAs, 84 real multiply-adds at 1,024 per clock and SM.  Errors stay at
// those of FP64 sums (the oracle parity of the products is unchanged).
//
// A warp owns 16 consecutive boxes (Morton order) as targets and 8 NT channels
// of one frequency, and runs over the union of the targets' interaction lists, 8
// sources at a time, kernel values gathered by the offset index (excluded
// pairs are zeros).  Unions of 16 targets hold 40% pairs on the 4-wavelength
// sphere's leaf level; 128-target unions, which the FP32 form uses, 13%.  A thread
// gathers exactly the four kernel values and the digits of its own MMA
// fragments into a ring of its own by asynchronous copies: no barriers.
//
// Measured, 4-wavelength sphere, 8 vectors, ms: top level 31.1 -> 4.2 (27.8 from the
// lists in FP64 arithmetic), leaf level 7.7 -> 3.1 (6.7 for both with the digits in
// slabs, below); one vector 4.2 -> 1.2 and 1.2 -> 0.84.
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "device_api.cuh"
#include "digits.cuh"

namespace efie {

constexpr int MD_RD = 3;   // groups of 8 sources in the ring

// exponents of the kernel rows
__global__ void __launch_bounds__(128) k_spec_rowexp(const double2* __restrict__ K, int64_t O,
                                                     int16_t* __restrict__ kexp) {
  const double2* Kf = K + (int64_t)blockIdx.x * O;
  int mx = 0;
  for (int64_t o = threadIdx.x; o < O; o += blockDim.x) {
    const double2 v = Kf[o];
    mx = max(mx, max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff));
  }
  __shared__ int red[4];
  for (int d = 16; d > 0; d >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, d));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) kexp[blockIdx.x] = (int16_t)nm_row_exponent(max(max(red[0], red[1]), max(red[2], red[3])));
}

// the digits of the source spectra of one slab of frequencies, [f][box][c][6] (half2 real,
// imaginary): the first n0 frequencies at d0, the others at d1
struct MdSlab {
  uint32_t *d0, *d1;
  int n0;
  __device__ __forceinline__ uint32_t* at(int f, int64_t per_f) const {
    return f < n0 ? d0 + f * per_f : d1 + (f - n0) * per_f;
  }
};
// fills the slab that begins with the spectra Q, and qexp[f][c], the exponents over the
// boxes; one block per frequency, C <= 32 channels
__global__ void __launch_bounds__(256) k_spec_digits(const double2* __restrict__ Q, int64_t B, int C,
                                                     const MdSlab slab, int16_t* __restrict__ qexp) {
  __shared__ int mx[32];
  const int64_t f = blockIdx.x, n = B * C;
  const double2* Qf = Q + f * n;
  uint32_t* qd = slab.at(blockIdx.x, n * 6);
  if (threadIdx.x < 32) mx[threadIdx.x] = 0;
  __syncthreads();
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
    const double2 v = Qf[i];
    atomicMax(&mx[(int)(i % C)], max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff));
  }
  __syncthreads();
  if (threadIdx.x < C) {
    const int E = nm_exponent(mx[threadIdx.x]);
    qexp[f * C + threadIdx.x] = (int16_t)E;
    mx[threadIdx.x] = E;
  }
  __syncthreads();
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
    const int E = mx[(int)(i % C)];
    const double2 v = Qf[i];
    int a[6], b[6];
    nm_digits<6>(E == NM_ENAN ? 0 : nm_fixed(v.x, E), a);
    nm_digits<6>(E == NM_ENAN ? 0 : nm_fixed(v.y, E), b);
    uint2* o = reinterpret_cast<uint2*>(qd + i * 6);
#pragma unroll
    for (int s = 0; s < 3; ++s) o[s] = make_uint2(nm_pack(a[2 * s], b[2 * s]), nm_pack(a[2 * s + 1], b[2 * s + 1]));
  }
}

template <int N>
__device__ __forceinline__ void md_cp(void* dst, const void* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "n"(N), "r"(ok ? N : 0)
               : "memory");
}

template <int NT>
struct MdCfg {
  static constexpr int LANE = 64 + 48 * NT;               // bytes of a ring slot per lane
  static constexpr int SMEM = 128 * (MD_RD * LANE + 8 * NT * 8);
};

// grid: (groups of 4 row tiles x channel groups, frequency of the slab that begins at
// f0); idx [tile][kg][lane] =
// offset ids of (rows g, g + 8) x (sources t, t + 4), -1: none; src [tile][kg][8]
template <int NT>
__global__ void __launch_bounds__(128, NT == 1 ? 4 : 2)
k_mac_digits(const double2* __restrict__ K, const int16_t* __restrict__ kexp, const MdSlab slab,
             const int16_t* __restrict__ qexp, double2* __restrict__ Rh, int64_t B, int C, int64_t O, int ntiles,
             int ngr, const int32_t* __restrict__ kg_ptr, const int4* __restrict__ idx,
             const int32_t* __restrict__ src, int64_t f0) {
  constexpr int NS = 6, NG = 5, LANE = MdCfg<NT>::LANE;
  extern __shared__ __align__(16) unsigned char md_smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  // per warp: the kernel values [MD_RD][4][32] and the digits [MD_RD][NT][2][3][32], then the sums [8 NT][128]
  uint4* kv = reinterpret_cast<uint4*>(md_smem + warp * 32 * MD_RD * LANE) + lane;
  uint2* xv = reinterpret_cast<uint2*>(md_smem + warp * 32 * MD_RD * LANE + MD_RD * 4 * 32 * 16) + lane;
  double* acc = reinterpret_cast<double*>(md_smem + 128 * MD_RD * LANE) + tid;
  const int gr = blockIdx.x % ngr, tile = (int)(blockIdx.x / ngr) * 4 + warp;
  const int64_t f = f0 + blockIdx.y;
  if (tile >= ntiles) return;
  const int c0 = gr * 8 * NT;
  const double2* Kf = K + f * O;
  const uint32_t* qd = slab.at(blockIdx.y, B * C * 6);
  const uint32_t* Qf = qd + (c0 + g) * 6;
  const int E = kexp[f];
  const int k0 = kg_ptr[tile], nkg = kg_ptr[tile + 1] - k0;
#pragma unroll
  for (int v = 0; v < 8 * NT; ++v) acc[v * 128] = 0.0;
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
  bool chan[NT];
#pragma unroll
  for (int n = 0; n < NT; ++n) chan[n] = c0 + 8 * n + g < C;
  // indices of the next group to load, one group ahead of the copies
  int4 id = make_int4(-1, -1, -1, -1);
  int s0 = 0, s1 = 0;
  auto indices = [&](int kg) {
    if (kg < nkg) {
      id = __ldg(idx + (int64_t)(k0 + kg) * 32 + lane);
      s0 = __ldg(src + (int64_t)(k0 + kg) * 8 + t);
      s1 = __ldg(src + (int64_t)(k0 + kg) * 8 + t + 4);
    }
  };
  auto load = [&](int kg, int slot) {
    if (kg < nkg) {
      uint4* d = kv + slot * 4 * 32;
      md_cp<16>(d, Kf + (id.x < 0 ? 0 : id.x), id.x >= 0);
      md_cp<16>(d + 32, Kf + (id.y < 0 ? 0 : id.y), id.y >= 0);
      md_cp<16>(d + 64, Kf + (id.z < 0 ? 0 : id.z), id.z >= 0);
      md_cp<16>(d + 96, Kf + (id.w < 0 ? 0 : id.w), id.w >= 0);
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int y = h ? s1 : s0;
          const bool ok = y >= 0 && chan[n];
          const uint32_t* p = ok ? Qf + ((int64_t)y * C + 8 * n) * 6 : qd;
          uint2* o = xv + ((slot * NT + n) * 2 + h) * 3 * 32;
          md_cp<8>(o, p, ok);
          md_cp<8>(o + 32, p + 2, ok);
          md_cp<8>(o + 64, p + 4, ok);
        }
      indices(kg + 1);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  indices(0);
#pragma unroll
  for (int q = 0; q < MD_RD - 1; ++q) load(q, q);
  int slot = 0, nk = 0;
#pragma unroll 1
  for (int kg = 0; kg < nkg; ++kg) {
    load(kg + MD_RD - 1, slot == 0 ? MD_RD - 1 : slot - 1);
    asm volatile("cp.async.wait_group %0;\n" ::"n"(MD_RD - 1) : "memory");
    uint32_t a[NS][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint4 w = kv[(slot * 4 + q) * 32];
      int dr[NS], di[NS];
      nm_digits<NS>(E == NM_ENAN ? 0 : nm_fixed(__hiloint2double(w.y, w.x), E), dr);
      nm_digits<NS>(E == NM_ENAN ? 0 : nm_fixed(__hiloint2double(w.w, w.z), E), di);
#pragma unroll
      for (int s = 0; s < NS; ++s) a[s][q] = nm_pack(dr[s], di[s]);
    }
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      const uint2* xq = xv + (slot * NT + n) * 2 * 3 * 32;
      uint2 x[NS];
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        const uint2 p = xq[s * 32], q = xq[(3 + s) * 32];
        x[2 * s] = make_uint2(p.x, q.x);
        x[2 * s + 1] = make_uint2(p.y, q.y);
      }
#pragma unroll
      for (int part = 0; part < 2; ++part) {
        uint32_t b0[NS], b1[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) {
          b0[s] = part ? __byte_perm(x[s].x, 0, 0x1032) : x[s].x ^ 0x80000000u;
          b1[s] = part ? __byte_perm(x[s].y, 0, 0x1032) : x[s].y ^ 0x80000000u;
        }
#pragma unroll
        for (int w = 0; w < NG; ++w)
#pragma unroll
          for (int i = 0; i <= w; ++i) {
            if (w > 0 && i == w) continue;  // chained to (0, w) below
            float d[4];
            nm_mma(d, a[i], b0[w - i], b1[w - i], mg);
            if (w > 0 && i == 0) nm_mma(d, a[w], b0[0], b1[0], d);
#pragma unroll
            for (int v = 0; v < 4; ++v) run[n][w][part * 4 + v] += __float_as_int(d[v]);
          }
        float* fp = &fl[n][part * 4];
#pragma unroll
        for (int i = 0; i <= NG; ++i) nm_mma(fp, a[i], b0[NG - i], b1[NG - i], fp);
      }
    }
    slot = slot == MD_RD - 1 ? 0 : slot + 1;
    ++nk;
    if (kg + 1 < nkg && (kg + 1) % (NM_PIECE / 8) != 0) continue;
    // running sums into the FP64 accumulators, as in k_near_mma
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int c = c0 + 8 * n + 2 * t + (v & 1);
        const NmCol x = nm_col(c < C ? qexp[f * C + c] : 0);
        const double sc = nm_scale(E, x, 46);
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          const int q = part * 4 + v;
          int r_[NG];
#pragma unroll
          for (int w = 0; w < NG; ++w) {
            r_[w] = (int)((uint32_t)run[n][w][q] - MB * (uint32_t)(nk * (w > 0 ? w : 1)));
            run[n][w][q] = 0;
          }
          const long long T = ((long long)r_[0] << 30) + ((long long)r_[1] << 20) + ((long long)r_[2] << 10) + r_[3];
          const int low = r_[4] + __float2int_rn(fl[n][q] * 0.0009765625f);
          double* ap = acc + (n * 8 + q) * 128;
          *ap = fma(nm_raise((double)T, x), sc, fma(nm_raise((double)low, x), sc * 0.0009765625, *ap));
          fl[n][q] = 0.f;
        }
      }
    nk = 0;
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int64_t x = (int64_t)tile * 16 + g + (v < 2 ? 0 : 8);
      const int c = c0 + 8 * n + 2 * t + (v & 1);
      if (x < B && c < C) Rh[(f * B + x) * C + c] = make_double2(acc[(n * 8 + v) * 128], acc[(n * 8 + 4 + v) * 128]);
    }
}

void launch_spec_rowexp(const double2* K, int64_t nf, int64_t O, int16_t* kexp, cudaStream_t s) {
  if (nf > 0) k_spec_rowexp<<<(unsigned)nf, 128, 0, s>>>(K, O, kexp);
}
// The digits are 1.5 times the spectra, so they are made for as many frequencies as the
// two intermediates hold and used before the next ones: one or two slabs per level.  A buffer
// of their own for all frequencies took 0.93 GB of 3.74 on 48,000 unknowns with 8 vectors
// and was no faster (both levels 6.64 ms, slabs 6.66; slabs of one intermediate each 6.70).
int launch_mac_digits(const double2* Q, double2* Rh, const double2* K, const MacDigits& m, double2* tmp1,
                      double2* tmp2, int64_t ntmp, int64_t B, int C, int64_t O, int64_t nf, cudaStream_t s) {
  if (B <= 0 || nf <= 0 || m.ntiles <= 0) return 0;
  const int nt = C <= 8 ? 1 : 2, ngr = (C + 8 * nt - 1) / (8 * nt);
  const unsigned gx = (unsigned)(((m.ntiles + 3) / 4) * ngr);
  // the exponents first in tmp2
  int16_t* qexp = reinterpret_cast<int16_t*>(tmp2);
  const int64_t nexp = ceil_div(nf * C * (int64_t)sizeof(int16_t), 16), per_f = 24 * B * C;
  const int64_t fit0 = ntmp * 16 / per_f, fit1 = std::max<int64_t>(0, (ntmp - nexp) * 16 / per_f);
  const int64_t fit = std::min<int64_t>(65535, fit0 + fit1);
  const int64_t per = ceil_div(nf, ceil_div(nf, fit));
  const MdSlab slab{reinterpret_cast<uint32_t*>(tmp1), reinterpret_cast<uint32_t*>(tmp2 + nexp),
                    (int)std::min<int64_t>(per, fit0)};
  int launches = 0;
  for (int64_t f0 = 0; f0 < nf; f0 += per, launches += 2) {
    const unsigned n = (unsigned)std::min<int64_t>(per, nf - f0);
    k_spec_digits<<<n, 256, 0, s>>>(Q + f0 * B * C, B, C, slab, qexp + f0 * C);
    const dim3 grid(gx, n);
    if (nt == 1) {
      static SmemAttr attr;
      smem_attr_once(k_mac_digits<1>, MdCfg<1>::SMEM, attr.v);
      k_mac_digits<1><<<grid, 128, MdCfg<1>::SMEM, s>>>(K, m.kexp, slab, qexp, Rh, B, C, O, m.ntiles, ngr, m.kg_ptr,
                                                        m.idx, m.src, f0);
    } else {
      static SmemAttr attr;
      smem_attr_once(k_mac_digits<2>, MdCfg<2>::SMEM, attr.v);
      k_mac_digits<2><<<grid, 128, MdCfg<2>::SMEM, s>>>(K, m.kexp, slab, qexp, Rh, B, C, O, m.ntiles, ngr, m.kg_ptr,
                                                        m.idx, m.src, f0);
    }
  }
  return launches;
}

}  // namespace efie
