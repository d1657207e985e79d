// Grouped FP64 block GEMM on the tensor cores, by exact splitting.
//
// GB300 has 2 FP64 FMAs per SM and clock; its tensor cores do 1024 FP16
// products per SM and clock through mma.sync.  Following the error-free
// splitting of Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012),
// every operand row of a 32-long K chunk is scaled by a power of two (its
// largest element below 2^55) and rounded once to an integer of 56 bits,
// which is cut into seven signed base-256 digits -128..128 (FP16 holds them
// exactly).  The digit products of equal weight are summed by the tensor
// cores in FP32.  A sum over a chunk is an integer below 2^22 (at most 7 pairs x 32 x
// 2^14), and its accumulator starts at 1.5 x 2^23, so that every step is
// exact and the accumulator's bits are the integer.  The eight weights
// (34 digit pairs; pairs of weight 8 and more are below the rounding of the
// operands) are put together as one 64-bit integer, converted once and
// added to the FP64 sum of the output with one FMA.
//
// Accuracy: a chunk's operands and its sum are within 2^-56 of (largest
// element of the A row) x (largest of the B column); FP64 rounds at every
// one of the 32 FMAs instead.  On Gaussian, graded, near-diagonal and
// isometric operands the relative error against 64-bit-mantissa sums is
// 0.4 to 0.9 of the plain FMA loop's for K >= 8.
//
// Rows whose largest magnitude is not finite or outside 2^-323 .. 2^277
// (all-zero rows are fine) and coefficients outside 2^-73 .. 2^77 send
// their chunk through plain FMAs instead, so infinities, NaN and extreme
// scales give what the FMA loop gives.
//
// What bounds it: the three units that a chunk needs are about balanced --
// mma.sync 34 x 32 x 8 clocks over four sub-cores, two FP64 operations per
// output element, and the digit extraction (about 36 integer instructions
// per operand element) -- and none is full: with three CTAs an SM their
// latencies show (1.6 instructions a clock, tensor pipe 25 %, FP64 pipe 24 %
// in stage A of the CAS(16,16) M=512 H_eff product).  The 32 x 64 tile keeps
// the extraction at 3/64 of an element per product while sector blocks of a
// few tens waste little of it; K chunks of 32 are what the exact FP32 sums
// allow.  That H_eff product (39 GFLOP): 79 ms with FP64 FMAs, 21 ms here,
// 1.9 TFLOP/s against the FP64 pipe's 1.2.
#include <cuda_runtime.h>

#include <cuda_fp16.h>

#include "gbd_internal.h"

namespace gbd {

namespace {

constexpr int XM = kSplitTileM, XN = kSplitTileN, XK = kSplitChunk, XT = 128;
constexpr int NS = 7;                      // digits
constexpr int PK = 40;                     // raw pitch, K contiguous (doubles): 320 B, conflict-free 16 B reads
constexpr int PA = XM + 2, PB = XN + 2;    // raw pitch, K strided: rows of 272 / 528 B
constexpr int kRawA = XM * PK, kRawB = XN * PK;                  // doubles (both layouts fit)
static_assert(XK * PA <= kRawA && XK * PB <= kRawB, "raw tiles");
constexpr int kSlA = XM * 64, kSlB = XN * 64;                    // bytes of one digit plane (32 halves a row)
constexpr int kOffB = kRawA * 8, kOffSa = kOffB + kRawB * 8, kOffSb = kOffSa + NS * kSlA;
constexpr int kOffE = kOffSb + NS * kSlB;
constexpr int kSmem = kOffE + (XM + XN + 2) * 4;
constexpr float kMagic = 12582912.0f;      // 1.5 x 2^23: integers in +-2^22 added to it are its low mantissa bits
constexpr uint32_t kMagicBits = 0x4B400000u;

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// 8-byte asynchronous copy; zero fill when !in
__device__ __forceinline__ void copy8(uint32_t dst, const double* src, bool in) {
  const int n = in ? 8 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// 16-byte chunk c (0..3) of a digit row: rows two apart use different halves
// of a 128-byte line for the 8-byte digit stores, and the eight rows of an
// ldmatrix use eight different 16-byte bank groups
__device__ __forceinline__ int swz(int row, int c) { return c ^ (((row >> 1) & 1) << 1 | ((row >> 2) & 1)); }

// element (row, k) of a raw operand tile: K contiguous or K strided
template <int P>
__device__ __forceinline__ double raw_at(const double* raw, bool kcontig, int row, int k) {
  return kcontig ? raw[row * PK + k] : raw[k * P + row];
}

// Digit planes of one operand row, by four threads (kq = 0..3) with elements
// k = 16 h + 8 j + 2 kq + u of it each (h < nh, the 16-blocks in use).  The
// digits of element (h, j, u) go to position 16 h + 4 kq + 2 j + u: the same
// permutation of K for both operands.  Returns the row's scale exponent E
// (all |x| < 2^(E - 1023); 1023 for a zero row); bad = 1 when E is not usable.
template <int P>
__device__ __forceinline__ int split_row(const double* raw, bool kcontig, int row, int kq, int nh, uint8_t* planes,
                                         int plane, int& bad) {
  uint32_t lo[8], hi[8];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      double2 v = make_double2(0.0, 0.0);
      const int k = 16 * h + 8 * j + 2 * kq;
      if (h < nh) {
        if (kcontig) {
          v = *reinterpret_cast<const double2*>(raw + row * PK + k);
        } else {
          v.x = raw[k * P + row];
          v.y = raw[(k + 1) * P + row];
        }
      }
      const int i = 4 * h + 2 * j;
      lo[i] = (uint32_t)__double2loint(v.x);
      hi[i] = (uint32_t)__double2hiint(v.x);
      lo[i + 1] = (uint32_t)__double2loint(v.y);
      hi[i + 1] = (uint32_t)__double2hiint(v.y);
    }
  uint32_t mx = 0, any = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    mx = max(mx, hi[i] & 0x7FFFFFFFu);
    any |= lo[i];
  }
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
  int E = (int)(mx >> 20) + 1;
  const bool zero = mx == 0;
  bad = 0;
  if (mx < (700u << 20)) bad = (mx != 0 || any != 0);
  if (mx >= (1300u << 20)) bad = 1;
  const int sh0 = zero ? 5000 : E + 7;   // right shift of the left-aligned mantissa: sh0 - exponent
  const uint64_t bias = 2 * 0x0080808080808080ull + 1;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if (h >= nh) break;
    uint32_t pk[2][NS];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      uint32_t wl[2], wh[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const uint32_t xh = hi[4 * h + 2 * j + u], xl = lo[4 * h + 2 * j + u];
        const uint32_t mh = __funnelshift_l(xl, xh, 11) | 0x80000000u;
        const uint64_t m = ((uint64_t)mh << 32) | (uint32_t)(xl << 11);
        const uint32_t s = (uint32_t)(sh0 - (int)((xh >> 20) & 0x7FFu));
        uint64_t t;   // 2 |x| in units of the last digit; 0 for shifts of 64 and more
        asm("shr.u64 %0, %1, %2;" : "=l"(t) : "l"(m), "r"(s));
        const int64_t sg = (int64_t)((int32_t)xh >> 31);
        const uint64_t w = (uint64_t)((int64_t)((t ^ (uint64_t)sg) - (uint64_t)sg + bias)) >> 1;
        wl[u] = (uint32_t)w;
        wh[u] = (uint32_t)(w >> 32);
      }
      // half2 of digit i of the two elements: byte + 1024 as FP16, less 1152
#pragma unroll
      for (int i = 0; i < NS; ++i) {
        uint32_t b;
        if (i == 0) {
          b = __byte_perm(wh[0], wh[1], 0x7632) | 0x64006400u;
        } else {
          const int byte = NS - 1 - i;
          const uint32_t x0 = byte < 4 ? wl[0] : wh[0], x1 = byte < 4 ? wl[1] : wh[1];
          const uint32_t c = byte & 3;
          b = (__byte_perm(x0, x1, c | (c << 4) | ((c + 4) << 8) | ((c + 4) << 12)) & 0x00FF00FFu) | 0x64006400u;
        }
        const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&b), __half2half2(__ushort_as_half(0x6480)));
        pk[j][i] = *reinterpret_cast<const uint32_t*>(&d);
      }
    }
    uint8_t* dst = planes + row * 64 + swz(row, 2 * h + (kq >> 1)) * 16 + (kq & 1) * 8;
#pragma unroll
    for (int i = 0; i < NS; ++i) *reinterpret_cast<uint2*>(dst + i * plane) = make_uint2(pk[0][i], pk[1][i]);
  }
  return zero ? 1023 : E;
}

__global__ void __launch_bounds__(XT, 3)
gemm_f64_split_kernel(const GemmTerm* __restrict__ terms, const GemmOut* __restrict__ outs,
                      const GemmTile* __restrict__ tiles, int ntiles) {
  extern __shared__ __align__(128) uint8_t sm[];
  double* rawA = reinterpret_cast<double*>(sm);
  double* rawB = reinterpret_cast<double*>(sm + kOffB);
  uint8_t* slA = sm + kOffSa;
  uint8_t* slB = sm + kOffSb;
  int* expA = reinterpret_cast<int*>(sm + kOffE);
  int* expB = expA + XM;
  int* flag = expB + XN;   // [2]: a chunk needs plain FMAs
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = warp & 1, wn = warp >> 1;
  const uint32_t rawA_a = smem_addr(rawA), rawB_a = smem_addr(rawB);
  if (tid < 2) flag[tid] = 0;
  int par = 0;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const GemmTile tl = tiles[tile];
    const GemmOut o = outs[tl.out];
    const int m0 = tl.tm * XM, n0 = tl.tn * XN;
    const int mr = min(XM, o.M - m0), nr = min(XN, o.N - n0);
    double acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;

    // raw tiles of chunk k0 of term T: kc columns, zeros up to a multiple of 16
    auto fetch = [&](const GemmTerm& T, int k0) {
      const int kc = min(XK, T.K - k0), kz = (kc + 15) & ~15;
      if (!(T.flags & 1)) {
        const double* s = T.A + (int64_t)m0 * T.lda + k0;
        if (lane < kz)
          for (int r = warp; r < mr; r += 4)
            copy8(rawA_a + (r * PK + lane) * 8, s + (int64_t)r * T.lda + (lane < kc ? lane : 0), lane < kc);
      } else {
        const double* s = T.A + (int64_t)k0 * T.lda + m0;
        if (lane < mr)
          for (int k = warp; k < kz; k += 4)
            copy8(rawA_a + (k * PA + lane) * 8, s + (int64_t)(k < kc ? k : 0) * T.lda + lane, k < kc);
      }
      if (T.flags & 2) {
        const double* s = T.B + (int64_t)n0 * T.ldb + k0;
        if (lane < kz)
          for (int r = warp; r < nr; r += 4)
            copy8(rawB_a + (r * PK + lane) * 8, s + (int64_t)r * T.ldb + (lane < kc ? lane : 0), lane < kc);
      } else {
        const double* s = T.B + (int64_t)k0 * T.ldb + n0;
        for (int k = warp; k < kz; k += 4)
          for (int n = lane; n < nr; n += 32)
            copy8(rawB_a + (k * PB + n) * 8, s + (int64_t)(k < kc ? k : 0) * T.ldb + n, k < kc);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };

    // the chunk in work is (T, k0); (Tn) is the next term with columns
    int t = o.t0, k0 = 0;
    GemmTerm T{}, Tn{};
    auto skip_empty = [&](int& i, GemmTerm& X) {
      while (i < o.t1) {
        X = terms[i];
        if (X.K > 0) break;
        ++i;
      }
    };
    skip_empty(t, T);
    int tn = t + 1;
    if (t < o.t1) {
      skip_empty(tn, Tn);
      fetch(T, 0);
    }
    while (t < o.t1) {
      const int kc = min(XK, T.K - k0), nh = (kc + 15) >> 4;
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();   // raw tiles landed; every warp is done with the digit planes
      const bool ka = !(T.flags & 1), kb = T.flags & 2;
      const int ahi = __double2hiint(T.alpha);
      const int aexp = (ahi >> 20) & 0x7FF;
      const bool abad = aexp < 950 || aexp > 1100;
      {
        const int row = tid >> 2, kq = tid & 3;
        int bad;
        if ((row & ~7) < mr) {   // whole warps
          const int E = split_row<PA>(rawA, ka, row, kq, nh, slA, kSlA, bad);
          if (row < mr) {
            if (kq == 0) expA[row] = E;
            if (bad || abad) flag[par] = 1;
          }
        }
#pragma unroll 1
        for (int p = 0; p < XN; p += 32) {
          if (((p + row) & ~7) >= nr) break;
          const int E = split_row<PB>(rawB, kb, p + row, kq, nh, slB, kSlB, bad);
          if (p + row < nr) {
            if (kq == 0) expB[p + row] = E;
            if (bad) flag[par] = 1;
          }
        }
      }
      __syncthreads();
      const bool plain = flag[par] != 0;
      if (plain) {
        // the chunk by FP64 FMAs from the raw tiles
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int c8 = (wn + 2 * i) * 8;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int r = 16 * wm + (lane >> 2) + 8 * (j >> 1), c = c8 + 2 * (lane & 3) + (j & 1);
            if (r < mr && c < nr)
              for (int k = 0; k < kc; ++k)
                acc[i][j] = fma(raw_at<PA>(rawA, ka, r, k) * T.alpha, raw_at<PB>(rawB, kb, c, k), acc[i][j]);
          }
        }
        __syncthreads();
      }
      if (tid == 0) flag[par ^ 1] = 0;
      par ^= 1;
      // the next chunk's raw tiles arrive while this one multiplies
      const int ahi_cur = ahi, alo_cur = __double2loint(T.alpha);
      k0 += XK;
      if (k0 < T.K) {
        fetch(T, k0);
      } else {
        t = tn;
        k0 = 0;
        T = Tn;
        if (t < o.t1) {
          fetch(T, 0);
          ++tn;
          skip_empty(tn, Tn);
        }
      }
      if (plain || 16 * wm >= mr) continue;
      uint32_t a[2][NS][4];
      {
        const int row = 16 * wm + (lane & 15);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (h < nh) {
            const uint32_t ad = smem_addr(slA + row * 64 + swz(row, 2 * h + (lane >> 4)) * 16);
#pragma unroll
            for (int i = 0; i < NS; ++i) ldsm4(ad + i * kSlA, a[h][i]);
          }
        }
      }
      const int r0 = 16 * wm + (lane >> 2);
      const int e0 = expA[r0] - 2100, e1 = expA[r0 + 8] - 2100;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c8 = (wn + 2 * i) * 8;
        if (c8 >= nr) break;
        float s[8][4];
#pragma unroll
        for (int d = 0; d < 8; ++d)
#pragma unroll
          for (int j = 0; j < 4; ++j) s[d][j] = kMagic;
        const int row = c8 + (lane & 7);
        const uint32_t bd = smem_addr(slB + row * 64 + swz(row, lane >> 3) * 16);
#pragma unroll
        for (int jb = 0; jb < NS; ++jb) {
          uint32_t b[4];
          ldsm4(bd + jb * kSlB, b);
#pragma unroll
          for (int ia = 0; ia < NS; ++ia)
            if (ia + jb < 8) mma_f16(s[ia + jb], a[0][ia], b[0], b[1]);
          if (nh > 1) {
#pragma unroll
            for (int ia = 0; ia < NS; ++ia)
              if (ia + jb < 8) mma_f16(s[ia + jb], a[1][ia], b[2], b[3]);
          }
        }
        const int2 eb = *reinterpret_cast<const int2*>(expB + c8 + 2 * (lane & 3));
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          auto bits = [&](int d) { return (int)(__float_as_uint(s[d][j]) - kMagicBits); };
          // weights 2^40 .. 2^0, and the last two rounded to units
          const int q = bits(0) * 256 + bits(1);
          const int p = bits(2) * 256 + bits(3);
          const int l = bits(4) * 256 + bits(5) + ((bits(6) * 256 + bits(7) + 32768) >> 16);
          const int64_t v = ((int64_t)q << 32) + (int64_t)p * 65536 + l;
          const int e = (j < 2 ? e0 : e1) + ((j & 1) ? eb.y : eb.x);
          acc[i][j] = fma(__ll2double_rn(v), __hiloint2double(ahi_cur + (e << 20), alo_cur), acc[i][j]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = (wn + 2 * i) * 8 + 2 * (lane & 3);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = 16 * wm + (lane >> 2) + 8 * (j >> 1), cc = c + (j & 1);
        if (r >= mr || cc >= nr) continue;
        double* d = o.C + (int64_t)(m0 + r) * o.ldc + n0 + cc;
        *d = o.beta ? (*d + acc[i][j]) : acc[i][j];
      }
    }
  }
}

}  // namespace

int launch_gemm_f64_split(const GemmPlan& p, cudaStream_t s) {
  const int n = (int)p.split.size();
  if (n == 0) return 0;
  static const cudaError_t attr =
      cudaFuncSetAttribute(gemm_f64_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (attr != cudaSuccess) return -1;
  const int grid = n < 152 * 3 ? n : 152 * 3;
  gemm_f64_split_kernel<<<grid, XT, kSmem, s>>>(p.d_terms, p.d_outs, p.d_split, n);
  return 1;
}

}  // namespace gbd
