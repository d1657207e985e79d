// Grouped FP64 block GEMM on the tensor cores, by exact splitting.
//
// GB300 has 2 FP64 FMAs per SM and clock; its tensor cores do 1024 FP16
// products per SM and clock through mma.sync.  Following the error-free
// splitting of Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012),
// every operand row of a 32-long K chunk is scaled by a power of two (its
// largest element below 2^55) and rounded once to an integer of 56 bits,
// which is cut into seven signed base-256 digits -128..128 (FP16 holds them
// exactly).  The digit products of equal weight are summed by the tensor
// cores in FP32.  A sum over a chunk is an integer below 2^22 (at most 7
// pairs x 32 x 2^14), and its accumulator starts at 1.5 x 2^23, so that every
// step is exact and the accumulator's bits are the integer.  The eight weights
// (34 digit pairs; pairs of weight 8 and more are below the rounding of the
// operands) are put together as one 64-bit integer, converted once and
// added to the FP64 sum of the output with one FMA.
//
// Accuracy: with a = the largest element of the A row in the chunk and b = of
// the B column, an operand element is off by at most 2^-55 a (2^-55 b) and
// the sum of the chunk by another 2^-53 a b; FP64 rounds at every one of the
// 32 FMAs instead.  Where the large elements of a row meet the large ones
// of a column that is below the FMA loop's error.  Where they do not (grading
// in opposite directions, near-diagonal operands, disjoint places), the
// products are small against a b and would lose digits.  So for every output
// the strongest chunk is kept, sum |A||B| from the top digits (two more
// products in 70), next to the largest scale 2^e of a b that any chunk brought
// (chunks in which no nonzero element meets another do not count).  An output
// with (columns + 4) sum |A||B| below 2^14 digit units, less the square root
// of the number of its chunks, whose errors are independent, is formed again
// by FP64 FMAs (split_redo).  Outputs then are within (K + 4) 2^-53 |A||B| by
// element, as the FMA loop's are by its a priori bound.  Measured on Gaussian,
// graded (both ways, 0.5 to 8 decades), near-diagonal, sparse and 6-decade
// random operands, K = 3 to 3000: at most about half of that bound; root mean
// square 0.05 to 7 times 2^-53 |A||B| where the FMA loop has 0.4 to 23, and at
// most 6 times the loop's, where products graded apart stay just above the
// line.  The line is measured, repeated outputs of the H_eff product of
// CAS(16,16) M=512 (9.2 ms in all): without the root 2^12 0.9 ms, 2^13 2.3 and
// 2^14 7.4 (1.4 % of the outputs), with it 0.5; the check itself takes 0.3.
// Plans whose products are only summed into one number (an energy) leave it
// out: their error counts against the norm, where the digits' is 0.4 to 0.9
// of the FMA loop's on operands like a state's.
//
// Rows whose largest magnitude is not finite or outside 2^-323 .. 2^277
// (all-zero rows are fine) and coefficients outside 2^-73 .. 2^77 send
// their chunk through plain FMAs instead, so infinities, NaN and extreme
// scales give what the FMA loop gives.
//
// Four kernels.  split_operands cuts every operand block of a plan once (a
// block of the sigma build serves up to hundreds of products) into records
// that the second one copies as they are: per 32-column chunk and 64 rows, the
// seven digit planes, swizzled for ldmatrix, and the rows' exponents and masks
// of nonzero elements, all contiguous.  gemm_f64_split multiplies 64 x 64
// output tiles: one warp streams the records of all chunks of all terms of all
// tiles of its CTA through a ring of three stages by bulk copies, sixteen
// warps multiply.  Long chains are cut into pieces with partial sums;
// split_redo repeats weak outputs, split_sum adds the pieces in a fixed order.
// What bounds it: a 64 x 64 x 32 chunk takes 4350 clocks of mma.sync (34
// pairs) and 2048 clocks of FP64 FMAs, but the sub-blocks are small (35 % of
// a chunk's products are real in CAS(16,16) M=512, 58 % in CAS(20,20)
// M=1024), so that a warp has one 16 x 8 block per chunk and its latencies
// count: loading fragments, putting the weights together, the barriers.
// Four consumer warps a sub-core hide them best: 96 registers a thread, the B
// digits of a block and two planes of A in registers, the header left in
// shared memory and no division in a chunk.  The H_eff product of CAS(16,16)
// M=512 (39 GFLOP) takes 8.4 ms without the check by element (operands 0.8)
// and the one of CAS(20,20) M=1024 (432 GFLOP) 53 ms, FP64 FMAs 79 and 562 ms.
#include <algorithm>

#include <cuda_runtime.h>

#include <cuda_fp16.h>

#include "gbd_internal.h"
#include "mbarrier.h"
#include "smem_limit.h"

namespace gbd {

namespace {

constexpr int XM = kSplitTile, XK = kSplitChunk;
constexpr int NS = 7;                           // digits
constexpr int kWarps = 16, XT = 32 * kWarps + 32;   // 17 warps: at most 5 on a sub-core, 96 registers
constexpr int kStages = 3;
constexpr int kPlane = XM * 64;                 // bytes of a digit plane in a stage: 64 rows of 32 halves
constexpr int kTail = kSplitTail;               // bytes behind a row's digits: exponent, mask of nonzero elements
constexpr int kRec = NS * kPlane + XM * kTail;  // a stage's operand: 7 planes and the tails
constexpr int kHead = 64;                       // bytes of a stage's header
constexpr int kSmem = kStages * (2 * kRec + kHead) + 2 * kStages * 8 + 16;
constexpr float kMagic = 12582912.0f;           // 1.5 x 2^23: integers in +-2^22 added to it are its low mantissa bits
constexpr uint32_t kMagicBits = 0x4B400000u;
constexpr int kBadExp = 1 << 28;                // exponent of a row that the digits cannot hold
constexpr int kStrong = 14;                     // the line of a weak output, in powers of two of digit units
constexpr uint32_t kNoScale = 0x80008000u;      // no chunk yet

__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldsm2(uint32_t addr, uint32_t (&r)[2]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// the first product of a sum: the accumulator's start is the constant operand
__device__ __forceinline__ void mma_f16_first(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(kMagic));
}
// digit products of 16 columns into the sums of the eight weights (FIRST:
// their first): B's seven planes in registers, A's read one ahead
template <bool FIRST>
__device__ __forceinline__ void weights(float (&f)[8][4], uint32_t ad, uint32_t bd) {
  uint32_t b[NS][2], a[2][4];
  ldsm4(ad, a[0]);
#pragma unroll
  for (int x = 0; x < NS; ++x) ldsm2(bd + x * kPlane, b[x]);
#pragma unroll
  for (int ia = 0; ia < NS; ++ia) {
    if (ia + 1 < NS) ldsm4(ad + (ia + 1) * kPlane, a[(ia + 1) & 1]);
#pragma unroll
    for (int jb = 0; jb < NS; ++jb) {
      if (ia + jb >= 8) continue;
      if (FIRST && (ia == 0 || (ia == 1 && jb == 6))) mma_f16_first(f[ia + jb], a[ia & 1], b[jb][0], b[jb][1]);
      else mma_f16(f[ia + jb], a[ia & 1], b[jb][0], b[jb][1]);
    }
  }
}
// sums of |top digit of A| |top digit of B| over 16 columns: |A||B| in units of
// 2^96 of the last digits' (the largest element's top digit is 64 to 128)
__device__ __forceinline__ void magnitudes(float (&m)[4], uint32_t ad, uint32_t bd) {
  uint32_t a[4], b[2];
  ldsm4(ad, a);
  ldsm2(bd, b);
#pragma unroll
  for (int i = 0; i < 4; ++i) a[i] &= 0x7FFF7FFFu;
  mma_f16(m, a, b[0] & 0x7FFF7FFFu, b[1] & 0x7FFF7FFFu);
}
// Byte offset of 16-byte piece c of a digit row: rows of 64 bytes (32 columns,
// c 0..3) or 32 bytes (chunks of at most 16 columns, c 0..1).  The eight rows
// of an ldmatrix use eight different 16-byte bank groups.
__device__ __forceinline__ int piece(int row, int c, int nh) {
  return nh == 2 ? row * 64 + (c ^ (((row >> 1) & 1) << 1 | ((row >> 2) & 1))) * 16
                 : row * 32 + (c ^ ((row >> 2) & 1)) * 16;
}
__device__ __forceinline__ int pad8(int rows) { return (rows + 7) & ~7; }

// ---------------------------------------------------------------- operand records
// One warp per 8 rows of one chunk: four threads (kq = 0..3) per row, each
// with the elements k = 16 h + 8 j + 2 kq + u; the digits of element (h, j, u)
// go to position 16 h + 4 kq + 2 j + u, the same permutation of K for every
// operand.  Bound by its integer work (about 36 instructions an element) and
// by HBM (8 bytes read, 14 written).
__global__ void __launch_bounds__(256) split_operands_kernel(const SplitOperand* __restrict__ ops, int nops,
                                                             int64_t nitems, uint8_t* __restrict__ digits,
                                                             int* __restrict__ next, uint2* __restrict__ weak) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *next = 0;   // the product kernel's work counter
    if (weak) weak->x = 0;
  }
  const int lane = threadIdx.x & 31, kq = lane & 3;
  const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
  const int64_t w = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  int64_t it = nitems * w / nw;
  const int64_t end = nitems * (w + 1) / nw;
  if (it >= end) return;
  int lo_o = 0, hi_o = nops - 1;
  while (lo_o < hi_o) {
    const int mid = (lo_o + hi_o + 1) >> 1;
    if (ops[mid].first <= it) lo_o = mid; else hi_o = mid - 1;
  }
  SplitOperand O = ops[lo_o];
  for (; it < end; ++it) {
    const int rp = pad8(O.rows), groups = rp >> 3, chunks = (O.K + XK - 1) / XK;
    if (it - O.first >= (int64_t)groups * chunks) {   // items of an operand are never empty
      O = ops[++lo_o];
      --it;
      continue;
    }
    const int loc = (int)(it - O.first), chunk = loc / groups, row = (loc - chunk * groups) * 8 + (lane >> 2);
    const int k0 = chunk * XK, kc = min(XK, O.K - k0), nh = (kc + 15) >> 4;
    uint32_t lo[8], hi[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = 16 * (i >> 2) + 8 * ((i >> 1) & 1) + 2 * kq + (i & 1);
      double v = 0.0;
      if (row < O.rows && k < kc)
        v = O.kstrided ? O.src[(int64_t)(k0 + k) * O.ld + row] : O.src[(int64_t)row * O.ld + k0 + k];
      lo[i] = (uint32_t)__double2loint(v);
      hi[i] = (uint32_t)__double2hiint(v);
    }
    uint32_t mx = 0, any = 0, nz = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      mx = max(mx, hi[i] & 0x7FFFFFFFu);
      any |= lo[i];
      nz |= (hi[i] & 0x7FFFFFFFu) | lo[i] ? 1u << (8 * kq + i) : 0u;
    }
    nz |= __shfl_xor_sync(0xffffffffu, nz, 1);
    nz |= __shfl_xor_sync(0xffffffffu, nz, 2);
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    any |= __shfl_xor_sync(0xffffffffu, any, 1);
    any |= __shfl_xor_sync(0xffffffffu, any, 2);
    const bool zero = mx == 0;
    int E = zero ? 1023 : (int)(mx >> 20) + 1;   // all |x| < 2^(E - 1023)
    if (mx < (700u << 20) ? (mx != 0 || any != 0) : mx >= (1300u << 20)) E = kBadExp;
    const int sh0 = zero ? 5000 : (int)(mx >> 20) + 8;   // right shift of the left-aligned mantissa: sh0 - exponent
    const uint64_t bias = 0x0080808080808080ull;
    const int tile = row / XM, trow = row - tile * XM, rt = min(XM, rp - tile * XM);
    const int plane = rt * nh * 32;
    // chunks before this one are full: rp rows of 7 x 64 + 4 bytes
    uint8_t* rec = digits + O.off + (int64_t)chunk * rp * (NS * 64 + kTail) + (int64_t)tile * XM * (NS * nh * 32 + kTail);
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
          const uint64_t r = (t + 1) >> 1;   // to nearest, before the sign: either sign rounds alike
          const uint64_t q = (r ^ (uint64_t)sg) - (uint64_t)sg + bias;
          wl[u] = (uint32_t)q;
          wh[u] = (uint32_t)(q >> 32);
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
      uint8_t* dst = rec + piece(trow, 2 * h + (kq >> 1), nh) + (kq & 1) * 8;
#pragma unroll
      for (int i = 0; i < NS; ++i) *reinterpret_cast<uint2*>(dst + i * plane) = make_uint2(pk[0][i], pk[1][i]);
    }
    if (kq == 0) *reinterpret_cast<int2*>(rec + NS * plane + trow * kTail) = make_int2(E, (int)nz);
  }
}

// ---------------------------------------------------------------- products
struct Head {          // what the consumers need of one chunk, 64 bytes
  double* C;           // output tile (or partial slot), written after the last chunk
  double alpha;
  int32_t ldc, mr, nr, flags;   // kFirst | kLast | kBeta | kEnd
  int32_t nh, kc, term, k0;     // 16-column halves; columns, GemmTerm and first column of the chunk
  int32_t m0, n0, work, slack;  // work, slack: its SplitWork and that one's slack
};
static_assert(sizeof(Head) == kHead, "stage header");
enum { kFirst = 1, kLast = 2, kBeta = 4, kEnd = 8 };

template <bool kGuard>
__global__ void __launch_bounds__(XT, 1)
gemm_f64_split_kernel(const GemmTerm* __restrict__ terms, const GemmOut* __restrict__ outs,
                      const SplitTerm* __restrict__ sterms, const SplitWork* __restrict__ work, int nwork,
                      const uint8_t* __restrict__ digits, double* __restrict__ part, uint2* __restrict__ weak,
                      int* err, int* next) {
  extern __shared__ __align__(128) uint8_t sm[];
  // stage s: record of A, record of B; the headers and barriers behind them
  Head* heads = reinterpret_cast<Head*>(sm + kStages * 2 * kRec);
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + kStages * (2 * kRec + kHead));
  uint64_t* empty = full + kStages;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], kWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (warp == kWarps) {
    // ---------------- producer: lane 0 keeps the books, lanes 0-15 copy the
    // seven planes and the exponents of both operands (planes keep one pitch in
    // the stage, so that the consumers' addresses are constants apart)
    int s = 0;
    uint32_t ph = 0;
    bool ok = true;
    // the first piece of work by block, the others as they are free: pieces
    // differ by an order of magnitude in length (dealt out in turn, the
    // busiest SM of a CAS(16,16) stage A worked 1.3 times as long as the mean)
    int wnext = 0;
    for (int w = blockIdx.x; w < nwork && ok; w = __shfl_sync(0xffffffffu, wnext, 0)) {
      if (lane == 0) wnext = (int)gridDim.x + atomicAdd(next, 1);   // needed after this piece
      const SplitWork W = work[w];
      const GemmOut o = outs[W.out];
      Head h;
      h.work = w;
      h.slack = W.slack;
      h.m0 = W.tm * XM;
      h.n0 = W.tn * XM;
      h.mr = min(XM, o.M - h.m0);
      h.nr = min(XM, o.N - h.n0);
      h.C = W.slot >= 0 ? part + (int64_t)W.slot * XM * XM : o.C + (int64_t)h.m0 * o.ldc + h.n0;
      h.ldc = W.slot >= 0 ? XM : o.ldc;
      const int beta = W.slot < 0 && o.beta ? kBeta : 0;
      const int ra = pad8(h.mr), rb = pad8(h.nr);
      const int side = lane >> 3, x = lane & 7;   // this lane's copy: operand (0, 1) and plane (7: exponents)
      const int rows = side ? rb : ra, row0 = side ? h.n0 : h.m0;
      int t = W.t0, k0 = W.k0;
      SplitTerm T = sterms[t];
      for (int i = 0; i < W.steps; ++i) {
        while (k0 >= T.K) {   // also past terms without columns
          T = sterms[++t];
          k0 = 0;
        }
        h.kc = min(XK, T.K - k0);
        h.nh = (h.kc + 15) >> 4;
        h.flags = (i == 0 ? kFirst : 0) | (i == W.steps - 1 ? kLast | beta : 0);
        h.term = T.term;
        h.alpha = T.alpha;
        h.k0 = k0;
        const int chunk = k0 / XK, row_bytes = NS * h.nh * 32 + kTail;
        ok = mbar_wait(&empty[s], ph ^ 1, err);
        if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
        uint8_t* st = sm + s * 2 * kRec;
        if (lane == 0) {
          heads[s] = h;
          mbar_expect_tx(&full[s], (uint32_t)((ra + rb) * row_bytes));
        }
        __syncwarp();
        if (lane < 16) {
          // the operand may have more rows than the output: its tile's planes are `pitch` apart
          const int have = side ? T.rb : T.ra, pitch = min(XM, have - row0) * h.nh * 32;
          const uint8_t* rec = digits + (side ? T.b : T.a) + (int64_t)chunk * have * (NS * 64 + kTail) +
                               (int64_t)row0 * row_bytes;
          bulk_copy(st + side * kRec + x * kPlane, rec + x * pitch, x < NS ? rows * h.nh * 32 : rows * kTail, &full[s]);
        }
        if (++s == kStages) { s = 0; ph ^= 1; }
        k0 += XK;
      }
    }
    if (ok && mbar_wait(&empty[s], ph ^ 1, err)) {
      if (lane == 0) {
        heads[s].flags = kEnd;
        mbar_arrive(&full[s]);
      }
    } else {
      // stages armed but never consumed: let their copies land before the CTA exits
      for (int i = 0; i < kStages; ++i)
        for (uint32_t it = 0; it < (1u << 20) && !mbar_try(&full[i], i < s ? ph : ph ^ 1); ++it) {
        }
    }
    return;
  }
  // ---------------- consumers
  constexpr int kN8 = 2;   // 8-column groups of a warp: 8 of a tile over 16 / 4 warps
  double acc[kN8][4];
  // of every output, as powers of two: the strongest chunk's |A||B| (high half)
  // and the largest scale with the line on it (low half)
  uint32_t scale[kN8][4];
  int s = 0;
  uint32_t ph = 0;
  for (;;) {
    if (!mbar_wait(&full[s], ph, err)) break;
    const Head& h = heads[s];   // read where it is needed: registers are short
    const int flags = h.flags;
    if (flags & kEnd) break;
    const uint8_t* ra = sm + s * 2 * kRec;
    const uint8_t* rb = ra + kRec;
    const int nh = h.nh;
    // warps: row groups of 16, and the 8-column groups dealt out among the
    // warps of a row group, so that small tiles keep most warps at work
    // (warp / nm and kWarps / nm for nm = 1..4 from packed constants)
    const int nm = (h.mr + 15) >> 4, sh = 8 * (nm - 1);
    const int nb = warp * (int)(0x10162040u >> sh & 0xFFu) >> 6, per = (int)(0x04050810u >> sh & 0xFFu), g = warp - nb * nm;
    const int n8 = (h.nr + 7) >> 3;
    const bool on = nb < per && nb < n8;
    if (flags & kFirst) {
#pragma unroll
      for (int i = 0; i < kN8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j] = 0.0;
          scale[i][j] = kNoScale;
        }
    }
    if (on) {
      const int2* tailA = reinterpret_cast<const int2*>(ra + NS * kPlane);
      const int2* tailB = reinterpret_cast<const int2*>(rb + NS * kPlane);
      const int r0 = 16 * g + (lane >> 2);
      // rows and columns outside the tile hold whatever the stage held before: never stored
      const bool ok0 = r0 < h.mr, ok1 = r0 + 8 < h.mr;
      const int2 none = make_int2(1023, 0);
      const int2 xa = ok0 ? tailA[r0] : none, xb = ok1 ? tailA[r0 + 8] : none;
      const int x0 = xa.x, x1 = xb.x;
      const int ahi = __double2hiint(h.alpha), alo = __double2loint(h.alpha), aexp = (ahi >> 20) & 0x7FF;
      const bool badA = x0 == kBadExp || x1 == kBadExp || aexp < 950 || aexp > 1100;
      const float columns = (float)(h.kc + 4);
      const int arow = 16 * g + (lane & 15);
      const uint32_t ad0 = smem_addr(ra + piece(arow, lane >> 4, nh));
      const uint32_t ad1 = smem_addr(ra + piece(arow, 2 + (lane >> 4), 2));   // second half, full chunks only
#pragma unroll
      for (int i = 0; i < kN8; ++i) {
        const int c8 = (nb + i * per) * 8;
        if (c8 >= h.nr) break;
        const int c = c8 + 2 * (lane & 3);
        const int2 ya = c < h.nr ? tailB[c] : none, yb = c + 1 < h.nr ? tailB[c + 1] : none;
        const int y0 = ya.x, y1 = yb.x;
        // one half of the columns at a time: 14 registers of B digits and 8
        // of A leave room for four warps a sub-core
        float f[8][4];
        const int brow = c8 + (lane & 7), bc = (lane >> 3) & 1;
        // exponents of the four outputs' (columns + 4) sum |A||B|, a byte each:
        // before the products, whose sums leave no registers for it (after
        // them the two stages of CAS(16,16) M=512 took 8.6 ms instead of 7.9)
        uint32_t strong = 0;
        if (kGuard) {
          float mag[4] = {0.0f, 0.0f, 0.0f, 0.0f};
          magnitudes(mag, ad0, smem_addr(rb + piece(brow, bc, nh)));
          if (nh == 2) magnitudes(mag, ad1, smem_addr(rb + piece(brow, 2 + bc, 2)));
#pragma unroll
          for (int j = 0; j < 4; ++j) strong |= __float_as_uint(mag[j] * columns) >> 23 << (8 * j);
        }
        weights<true>(f, ad0, smem_addr(rb + piece(brow, bc, nh)));
        if (nh == 2) weights<false>(f, ad1, smem_addr(rb + piece(brow, 2 + bc, 2)));
        // asked for only now, so that the exponents arrive during the products
        if (__any_sync(0xffffffffu, badA || y0 == kBadExp || y1 == kBadExp)) {
          // the chunk of these 16 x 8 outputs by FP64 FMAs from the operands themselves
          const GemmTerm T = terms[h.term];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int r = r0 + 8 * (j >> 1), cc = c + (j & 1);
            if (r >= h.mr || cc >= h.nr) continue;
            const int64_t m = h.m0 + r, n = h.n0 + cc;
            for (int k = h.k0; k < h.k0 + h.kc; ++k) {
              const double av = T.flags & 1 ? T.A[(int64_t)k * T.lda + m] : T.A[m * T.lda + k];
              const double bv = T.flags & 2 ? T.B[n * T.ldb + k] : T.B[(int64_t)k * T.ldb + n];
              acc[i][j] = fma(av * T.alpha, bv, acc[i][j]);
            }
          }
          continue;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          // the sums are the accumulators' bits less kMagicBits, 2^8 apart from
          // 2^40 down to 2^0, the last two rounded to units; the constants of
          // two weights are taken off together (all of it modulo 2^32)
          auto two = [&](int d) { return __float_as_uint(f[d][j]) * 256u + __float_as_uint(f[d + 1][j]); };
          const int p = (int)(two(2) - kMagicBits * 257u);
          const int l = (int)(two(4) - kMagicBits * 257u) + ((int)(two(6) - (kMagicBits * 257u - 32768u)) >> 16);
          const int64_t v = (int64_t)p * 65536 + l + (int64_t)((uint64_t)(two(0) - kMagicBits * 257u) << 32);
          const int e = (j < 2 ? x0 : x1) + ((j & 1) ? y1 : y0) - 2100;
          if (kGuard && ((j < 2 ? xa.y : xb.y) & ((j & 1) ? yb.y : ya.y)) != 0)
            scale[i][j] = __vmaxs2(scale[i][j], (uint32_t)(e + aexp) * 0x10001u +
                                                    __byte_perm(strong, 0, 0x4044 | j << 8) + 127 + kStrong);
          acc[i][j] = fma(__ll2double_rn(v), __hiloint2double(ahi + (int)((uint32_t)e << 20), alo), acc[i][j]);
        }
      }
    }
    if ((flags & kLast) && on) {
      const int slack = h.slack;
      uint32_t marks = 0;   // lane 4 i + j: the lanes whose output (i, j) is weak
#pragma unroll
      for (int i = 0; i < kN8; ++i) {
        const int c = (nb + i * per) * 8 + 2 * (lane & 3);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int r = 16 * g + (lane >> 2) + 8 * (j >> 1), cc = c + (j & 1);
          bool store = r < h.mr && cc < h.nr;
          if (kGuard) {
            const bool redo = store && ((int)scale[i][j] >> 16) + slack < (int)(short)(scale[i][j] & 0xFFFFu);
            const uint32_t lanes = __ballot_sync(0xffffffffu, redo);
            if (lane == 4 * i + j) marks = lanes;
            store = store && !redo;
          }
          if (!store) continue;
          double* d = h.C + (int64_t)r * h.ldc + cc;
          *d = flags & kBeta ? (*d + acc[i][j]) : acc[i][j];
        }
      }
      if (kGuard) {
        const uint32_t any = __ballot_sync(0xffffffffu, marks != 0);
        if (any) {
          uint32_t at = 0;
          if (lane == 0) at = atomicAdd(&weak->x, (uint32_t)__popc(any));
          at = __shfl_sync(0xffffffffu, at, 0) + 1 + __popc(any & ((1u << lane) - 1));
          if (marks) weak[at] = make_uint2(marks, (uint32_t)h.work * kWeakPlaces + warp * 4 * kN8 + lane);
        }
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s]);
    if (++s == kStages) { s = 0; ph ^= 1; }
  }
}

// The outputs marked weak, by FP64 FMAs from the operands themselves: a warp
// takes a mark (a place of a consumer warp, 32 lanes) four outputs at a time,
// a lane every 32nd product of a term, its partial sums added as a tree.
// Bound by the FP64 pipe where the chains are short (stage A of the H_eff
// product of CAS(16,16): 80 % busy, with the trees) and by the latency of the
// terms' records and loads where they are long, hence four outputs at once and
// the next term's record asked for early: one at a time, from a bit map of
// marks, took 2.3 times as long there and 5.7 times on the small plans of
// CAS(13,11) orbital RDMs.  Now 0.5 ms of that product's two stages, and 2.4 ms
// in the 48 launches of the 1-/2-RDM there (the call 65-66 -> 67 ms).
__global__ void __launch_bounds__(256, 3)
split_redo_kernel(const GemmTerm* __restrict__ terms, const GemmOut* __restrict__ outs,
                  const SplitTerm* __restrict__ sterms, const SplitWork* __restrict__ work, double* __restrict__ part,
                  const uint2* __restrict__ weak) {
  const int lane = threadIdx.x & 31;
  const uint32_t n = weak->x;
  for (uint32_t e = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < n; e += gridDim.x * blockDim.x >> 5) {
    const uint2 mark = weak[e + 1];
    const SplitWork W = work[mark.y / kWeakPlaces];
    const GemmOut o = outs[W.out];
    // the consumer warp's place in the tile
    const int place = mark.y % kWeakPlaces, warp = place >> 3, i = place >> 2 & 1, j = place & 3;
    const int nm = (min(XM, o.M - W.tm * XM) + 15) >> 4, nb = warp / nm, per = kWarps / nm, g = warp - nb * nm;
    const int r0 = 16 * g + 8 * (j >> 1), c0 = (nb + i * per) * 8 + (j & 1);
    for (uint32_t lanes = mark.x; lanes;) {
      int r[4], c[4], have = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {   // fewer than four: the last one again, not stored
        const int l = __ffs(lanes) - 1;
        r[q] = l < 0 ? r[q ? q - 1 : 0] : r0 + (l >> 2);
        c[q] = l < 0 ? c[q ? q - 1 : 0] : c0 + 2 * (l & 3);
        have += l >= 0;
        lanes &= lanes - 1;
      }
      double s[4] = {0.0, 0.0, 0.0, 0.0};
      GemmTerm T = terms[sterms[W.t0].term];
      for (int left = W.steps, t = W.t0, k = W.k0; left > 0;) {
        const int steps = min(left, (T.K - k + XK - 1) / XK), len = min(T.K - k, steps * XK);
        const int sa = T.flags & 1 ? T.lda : 1, ra = T.flags & 1 ? 1 : T.lda;
        const int sb = T.flags & 2 ? 1 : T.ldb, cb = T.flags & 2 ? T.ldb : 1;
        const double* a = T.A + (int64_t)W.tm * XM * ra + (int64_t)(k + lane) * sa;
        const double* b = T.B + (int64_t)W.tn * XM * cb + (int64_t)(k + lane) * sb;
        const double al = T.alpha;
        left -= steps;
        k = 0;
        if (left > 0) T = terms[sterms[++t].term];   // on its way during this term's products
        const bool unit = fabs(al) == 1.0, minus = al < 0.0;   // signs cost no FP64 instruction
        for (int x = lane; x < len; x += 32, a += 32 * (int64_t)sa, b += 32 * (int64_t)sb) {
          double av[4], bv[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            av[q] = a[(int64_t)r[q] * ra];
            bv[q] = b[(int64_t)c[q] * cb];
          }
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (q < have) s[q] = fma(unit ? (minus ? -av[q] : av[q]) : av[q] * al, bv[q], s[q]);
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (q >= have) break;
        for (int d = 16; d > 0; d >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], d);
        if (lane == 0) {
          double* d = W.slot >= 0 ? part + (int64_t)W.slot * XM * XM + r[q] * XM + c[q]
                                  : o.C + (int64_t)(W.tm * XM + r[q]) * o.ldc + W.tn * XM + c[q];
          *d = W.slot < 0 && o.beta ? *d + s[q] : s[q];
        }
      }
    }
  }
}

// Tiles whose chain was cut: the pieces' partial sums in their order, a lane
// per output (16 blocks a tile: with one, a plan of few tiles and a hundred
// pieces each waited 300 us for its loads).
__global__ void __launch_bounds__(256)
split_sum_kernel(const GemmOut* __restrict__ outs, const SplitSum* __restrict__ sums, const double* __restrict__ part) {
  const SplitSum S = sums[blockIdx.x];
  const GemmOut o = outs[S.out];
  const int x = blockIdx.y * 256 + threadIdx.x, r = x / XM, c = x - r * XM;
  const int m = S.tm * XM + r, n = S.tn * XM + c;
  if (m >= o.M || n >= o.N) return;
  const double* p = part + (int64_t)S.slot * XM * XM + x;
  double v = 0.0;
#pragma unroll 8
  for (int i = 0; i < S.count; ++i) v += p[(int64_t)i * XM * XM];
  double* d = o.C + (int64_t)m * o.ldc + n;
  *d = o.beta ? *d + v : v;
}

}  // namespace

int launch_gemm_f64_split(const GemmPlan& p, int num_sms, int* err, cudaStream_t s) {
  const int n = (int)p.swork.size();
  if (n == 0) return 0;
  const bool guard = p.d_weak != nullptr;
  const auto kernel = guard ? gemm_f64_split_kernel<true> : gemm_f64_split_kernel<false>;
  if (!allow_shared_memory(kernel, kSmem)) return -1;
  const int64_t blocks = (p.split_items + 7) / 8;
  split_operands_kernel<<<(int)std::min<int64_t>(blocks, 16 * num_sms), 256, 0, s>>>(
      p.d_operands, (int)p.operands.size(), p.split_items, p.d_digits, err + 1, p.d_weak);
  kernel<<<n < num_sms ? n : num_sms, XT, kSmem, s>>>(p.d_terms, p.d_outs, p.d_sterms, p.d_swork, n, p.d_digits,
                                                      p.d_part, p.d_weak, err, err + 1);
  if (guard)
    split_redo_kernel<<<3 * num_sms, 256, 0, s>>>(p.d_terms, p.d_outs, p.d_sterms, p.d_swork, p.d_part, p.d_weak);
  if (!p.ssums.empty()) split_sum_kernel<<<dim3(p.ssums.size(), XM * XM / 256), 256, 0, s>>>(p.d_outs, p.d_ssums, p.d_part);
  return 2 + guard + !p.ssums.empty();
}

}  // namespace gbd
