// FP64 kernels of the sweep: grouped block GEMM (the sigma build, environment
// update and decimation contractions all reduce to lists of small dense
// products), block axpy (forming enlarged operators from environment blocks
// and MPO entries) and the Davidson vector operations.
//
// GB300 executes FP64 on its CUDA cores only; these kernels are the plain
// FP64 path (products that are results themselves run on the tensor cores,
// kernels_f64_split.cu).  Every output element is written once,
// deterministically, without atomics.
#include <type_traits>

#include <cuda_runtime.h>

#include "gbd_internal.h"

namespace gbd {

namespace {

// Grouped GEMM by FP64 FMAs.  An output element is one chain of FMAs over its
// terms in order and k ascending, A scaled by its coefficient first, whatever
// the tile: the result does not depend on how the plan is cut.
//
// Bound: the FP64 pipe, 2 FMAs per SM and clock -- so slow that a warp needs
// no register blocking to fill it (an FMA of a warp occupies its sub-core for
// 64 clocks, as long as its result takes; its two operand reads from shared
// memory take 4 of the SM's), but every idle lane and every other FP64
// instruction counts.  So a tile is a rectangle of at most 128 E outputs cut
// to the sector block, one or two outputs a lane and nothing padded but the
// last warp; coefficients of +-1 cost no FP64 operation, others one per
// operand element.  A fifth warp prepares the operands: the columns of all
// terms of the output, concatenated, are taken 32 at a time (one lane each,
// whatever term it falls in, so that short terms fill a step too) and copied
// asynchronously into a ring of three steps: one being multiplied, one
// landing, one on its way.
// CAS(12,12) M=256 H_eff product (3.41 GFLOP): 13.1 -> 3.5 ms (0.98 TFLOP/s of
// the pipe's 1.19; 92 % of its cycles busy), against a kernel of 32 x 32
// register tiles for the long chains and one with a lane per output that read
// from global memory and multiplied by the coefficient at every FMA.
constexpr int FT = 128, FK = 32, FR = 3;

template <int E>
__global__ void __launch_bounds__(FT + 32, 8)
gemm_f64_kernel(const GemmTerm* __restrict__ terms, const GemmOut* __restrict__ outs,
                const GemmTile* __restrict__ tiles) {
  extern __shared__ double ring[];
  __shared__ double coef[FR][FK];
  __shared__ int how[FR][FK];   // coefficient of a column: 0 one, 1 minus one, 2 another
  __shared__ int ncol[FR], scaled[FR];
  const GemmTile tl = tiles[blockIdx.x];
  const GemmOut o = outs[tl.out];
  const int m0 = tl.tm, n0 = tl.tn, tm = tl.pad >> 16, tn = tl.pad & 0xFFFF;
  const int pa = tm | 1, pb = tn | 1, step = FK * (pa + pb);   // odd pitches: the copies' lanes are K columns
  if (threadIdx.x >= FT) {
    const int lane = threadIdx.x & 31;
    const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(ring));
    int t = o.t0, k = 0, n = 0;   // next column: k of term t; columns of the prepared step
    const double *a = nullptr, *b = nullptr;
    int64_t sa = 0, sb = 0;
    double al = 1.0;
    // operand addresses of the next 32 columns, one per lane
    auto prepare = [&]() {
      n = 0;
      while (t < o.t1) {
        int kt = t + lane < o.t1 ? max(terms[t + lane].K, 0) : 0;
        if (lane == 0) kt -= k;
        int sum = kt;   // inclusive sums over the next 32 terms
        for (int d = 1; d < 32; d <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, sum, d);
          if (lane >= d) sum += v;
        }
        const int total = __shfl_sync(0xffffffffu, sum, 31);
        if (total == 0) {
          t += 32;
          k = 0;
          continue;
        }
        n = min(FK, total);
        int lo = 0;   // the first term whose sum exceeds this lane's column
        for (int d = 16; d > 0; d >>= 1)
          if (__shfl_sync(0xffffffffu, sum, lo + d - 1) <= lane) lo += d;
        const int before = __shfl_sync(0xffffffffu, sum - kt, lo);
        if (lane < n) {
          const GemmTerm T = terms[t + lo];
          const int64_t kk = lane - before + (lo == 0 ? k : 0);
          if (T.flags & 1) {
            a = T.A + kk * T.lda + m0;
            sa = 1;
          } else {
            a = T.A + (int64_t)m0 * T.lda + kk;
            sa = T.lda;
          }
          if (T.flags & 2) {
            b = T.B + (int64_t)n0 * T.ldb + kk;
            sb = T.ldb;
          } else {
            b = T.B + kk * T.ldb + n0;
            sb = 1;
          }
          al = T.alpha;
        }
        const int adv = __popc(__ballot_sync(0xffffffffu, sum <= n));   // terms used up
        const int used = __shfl_sync(0xffffffffu, sum, max(adv - 1, 0));
        k = adv == 0 ? k + n : n - used;
        t += adv;
        break;
      }
    };
    auto issue = [&](int s) {
      if (lane < n) {
        uint32_t da = base + (s * step + lane * pa) * 8, db = base + (s * step + FK * pa + lane * pb) * 8;
        const double *pa_ = a, *pb_ = b;
        for (int i = 0; i < tm; ++i, da += 8, pa_ += sa)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(da), "l"(pa_) : "memory");
        for (int j = 0; j < tn; ++j, db += 8, pb_ += sb)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(db), "l"(pb_) : "memory");
        coef[s][lane] = al;
        how[s][lane] = al == 1.0 ? 0 : al == -1.0 ? 1 : 2;
      }
      const unsigned any = __ballot_sync(0xffffffffu, lane < n && al != 1.0);
      if (lane == 0) {
        ncol[s] = n;
        scaled[s] = any != 0;
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    prepare();
    issue(0);
    prepare();
    issue(1);
    prepare();
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    for (int s = 0; ncol[s] > 0;) {
      issue(s == 0 ? 2 : s - 1);
      prepare();
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncthreads();
      s = s == 2 ? 0 : s + 1;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    return;
  }
  const int ne = tm * tn;
  int ia[E], jb[E];
  double acc[E];
#pragma unroll
  for (int u = 0; u < E; ++u) {
    const int e = min((int)threadIdx.x + u * FT, ne - 1);   // idle lanes repeat the last output
    ia[u] = e / tn;
    jb[u] = e - ia[u] * tn;
    acc[u] = 0.0;
  }
  // outputs per lane of this warp
  const int w0 = (int)threadIdx.x & ~31, on = (w0 < ne) + (E == 2 && w0 + FT < ne);
  __syncthreads();
  for (int s = 0;;) {
    const int n = ncol[s];
    if (n == 0) break;
    double* A = ring + s * step;
    const double* B = A + FK * pa;
    if (scaled[s]) {
      // columns with a coefficient other than 1: signs by their bit (no FP64
      // operation), others multiplied; one column per lane
      const int kk = threadIdx.x & (FK - 1), h = kk < n ? how[s][kk] : 0;
      for (int i = threadIdx.x >> 5; i < tm; i += FT / 32) {
        double& v = A[kk * pa + i];
        if (h == 1) v = __longlong_as_double(__double_as_longlong(v) ^ (1ll << 63));
        if (__any_sync(0xffffffffu, h == 2))
          if (h == 2) v *= coef[s][kk];
      }
      asm volatile("bar.sync 1, %0;" ::"n"(FT) : "memory");
    }
    auto products = [&](auto outputs) {
      constexpr int O = decltype(outputs)::value;
      if (n == FK) {
#pragma unroll 8
        for (int k = 0; k < FK; ++k)
#pragma unroll
          for (int u = 0; u < O; ++u) acc[u] = fma(A[k * pa + ia[u]], B[k * pb + jb[u]], acc[u]);
      } else {
        for (int k = 0; k < n; ++k)
#pragma unroll
          for (int u = 0; u < O; ++u) acc[u] = fma(A[k * pa + ia[u]], B[k * pb + jb[u]], acc[u]);
      }
    };
    if (E == 2 && on == 2) products(std::integral_constant<int, E>());
    else if (on > 0) products(std::integral_constant<int, 1>());
    __syncthreads();
    s = s == 2 ? 0 : s + 1;
  }
#pragma unroll
  for (int u = 0; u < E; ++u) {
    if ((int)threadIdx.x + u * FT >= ne) continue;
    double* c = o.C + (int64_t)(m0 + ia[u]) * o.ldc + n0 + jb[u];
    *c = o.beta ? (*c + acc[u]) : acc[u];
  }
}

// Block axpy over fixed work chunks of kAxpyChunk output elements (the
// chunks of all outputs in one list, cstart[o] = first chunk of output o):
// a long output no longer occupies one CTA while the others idle.  The term
// descriptors of a chunk are staged in shared memory, so the data loads of
// four terms (4 x kPer independent loads per thread) are in flight at once;
// every element is still summed over its terms in list order.  Bound by the
// FP64 pipe (93 % busy), so a warp adds only the vectors of a chunk that it has
// elements of: sector blocks of about 1200 elements filled 58 % of their
// chunks (CAS(16,16) M=512, right and left operators, 8.7 GB of terms: 4.31 ms
// with whole chunks, 2.31 ms so).  A CTA per chunk, so that the device deals
// them out: dealt in turn to 8 CTAs an SM, whose chunks have 1 to hundreds of
// terms, the busiest SM worked 1.4 times as long as the idlest (1.89 ms now;
// CAS(20,20) M=1024 17.8 -> 15.5 ms).
constexpr int kAxpyThreads = 256;
constexpr int kAxpyStage = 256;   // term descriptors staged per round
__global__ void __launch_bounds__(kAxpyThreads) axpy_kernel(const AxpyTerm* __restrict__ terms,
                                                            const AxpyOut* __restrict__ outs,
                                                            const int64_t* __restrict__ cstart, int nouts,
                                                            int64_t nchunks) {
  constexpr int kPer = kAxpyChunk / kAxpyThreads;
  static_assert(kPer == 4, "the cases below");
  __shared__ const double* sp[kAxpyStage];
  __shared__ double sc[kAxpyStage];
  for (int64_t c = blockIdx.x; c < nchunks; c += gridDim.x) {
    // the output of this chunk: 32 probes of the list a round
    int lo = 0;
    for (int hi = nouts; hi - lo > 1;) {
      const int step = (hi - lo + 31) >> 5, at = lo + (int)(threadIdx.x & 31) * step;
      const int below = __popc(__ballot_sync(0xffffffffu, at < hi && cstart[at] <= c));
      hi = min(hi, lo + below * step);
      lo += (below - 1) * step;
    }
    const AxpyOut o = outs[lo];
    const int64_t e0 = (c - cstart[lo]) * kAxpyChunk + threadIdx.x;
    // vectors of 256 elements that this warp has any of, and this lane
    const int64_t left = o.len - (e0 & ~(int64_t)31);
    const int mine = left <= 0 ? 0 : (int)min((int64_t)kPer, (left + kAxpyThreads - 1) / kAxpyThreads);
    bool in[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) in[i] = e0 + (int64_t)i * kAxpyThreads < o.len;
    double s[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) s[i] = 0.0;
    for (int tb = o.t0; tb < o.t1; tb += kAxpyStage) {
      const int nt = min(kAxpyStage, o.t1 - tb);
      __syncthreads();
      if (threadIdx.x < nt) {
        sp[threadIdx.x] = terms[tb + threadIdx.x].src;
        sc[threadIdx.x] = terms[tb + threadIdx.x].coef;
      }
      __syncthreads();
      auto add = [&](auto vectors) {
        constexpr int P = decltype(vectors)::value;
        int t = 0;
        for (; t + 4 <= nt; t += 4) {
          double x[4][P];
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int i = 0; i < P; ++i) x[u][i] = in[i] ? sp[t + u][e0 + (int64_t)i * kAxpyThreads] : 0.0;
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int i = 0; i < P; ++i) s[i] = fma(sc[t + u], x[u][i], s[i]);
        }
        for (; t < nt; ++t)
#pragma unroll
          for (int i = 0; i < P; ++i)
            if (in[i]) s[i] = fma(sc[t], sp[t][e0 + (int64_t)i * kAxpyThreads], s[i]);
      };
      if (mine == 4) add(std::integral_constant<int, 4>());
      else if (mine == 3) add(std::integral_constant<int, 3>());
      else if (mine == 2) add(std::integral_constant<int, 2>());
      else if (mine == 1) add(std::integral_constant<int, 1>());
    }
#pragma unroll
    for (int i = 0; i < kPer; ++i)
      if (in[i]) o.dst[e0 + (int64_t)i * kAxpyThreads] = s[i];
  }
}

// one warp per strided vector (the diagonals of the enlarged operators: a few
// tens of elements each, thousands of them; latency is all there is to hide)
__global__ void gather_kernel(const GatherTask* __restrict__ tasks, int ntasks) {
  const int t = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  if (t >= ntasks) return;
  const GatherTask g = tasks[t];
  for (int i = threadIdx.x & 31; i < g.len; i += 32)
    g.dst[(int64_t)i * g.dstep] = fma(g.coef, g.src[(int64_t)i * g.sstep], 0.0);
}

__global__ void set_identity_kernel(double* d, int m) {
  int64_t n = (int64_t)m * m;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    d[e] = (e / m == e % m) ? 1.0 : 0.0;
}

constexpr int RED_THREADS = 256;

__device__ double block_sum(double v) {
  __shared__ double sh[RED_THREADS / 32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) sh[w] = v;
  __syncthreads();
  v = (threadIdx.x < RED_THREADS / 32) ? sh[threadIdx.x] : 0.0;
  if (w == 0)
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  return v;
}

// partial[j * nblk + b] = sum over block b's chunk of V_j . x
__global__ void multi_dot_partial(const double* __restrict__ V, int64_t stride, int k,
                                  const double* __restrict__ x, int64_t n, double* partial) {
  const int j = blockIdx.y;
  const double* v = V + (int64_t)j * stride;
  double s = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RED_THREADS + threadIdx.x; i < n; i += (int64_t)gridDim.x * RED_THREADS)
    s = fma(v[i], x[i], s);
  s = block_sum(s);
  if (threadIdx.x == 0) partial[j * gridDim.x + blockIdx.x] = s;
}

__global__ void finish_sums(const double* partial, int nblk, int k, double* out) {
  int j = blockIdx.x;
  double s = 0.0;
  for (int b = threadIdx.x; b < nblk; b += RED_THREADS) s += partial[j * nblk + b];
  s = block_sum(s);
  if (threadIdx.x == 0) out[j] = s;
}

__global__ void lincomb_kernel(double* out, const double* __restrict__ V, int64_t stride,
                               const double* __restrict__ coef, int k, int64_t n, int accumulate, double cs) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double s = accumulate ? out[i] : 0.0;
    for (int j = 0; j < k; ++j) s = fma(cs * coef[j], V[(int64_t)j * stride + i], s);
    out[i] = s;
  }
}

// out = t / sqrt(nrm2[0]) (zero vector when the norm has vanished)
__global__ void normalize_kernel(const double* __restrict__ t, const double* __restrict__ nrm2, int64_t n,
                                 double* __restrict__ out) {
  const double q = nrm2[0];
  const double s = q > 1e-28 ? 1.0 / sqrt(q) : 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = t[i] * s;
}

// diag - theta, kept at least 1e-8 away from zero (sign kept, + for 0)
__device__ __forceinline__ double guarded_den(double d, double theta) {
  double den = d - theta;
  if (fabs(den) < 1e-8) den = den >= 0.0 ? 1e-8 : -1e-8;
  return den;
}

// r = sx - theta x ; t = -r / clamp(diag - theta) ; partial sums of r^2
__global__ void residual_precond_kernel(const double* __restrict__ x, const double* __restrict__ sx,
                                        const double* __restrict__ diag, double theta, int64_t n,
                                        double* r, double* t, double* partial) {
  double s = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RED_THREADS + threadIdx.x; i < n; i += (int64_t)gridDim.x * RED_THREADS) {
    double ri = sx[i] - theta * x[i];
    r[i] = ri;
    t[i] = -ri / guarded_den(diag[i], theta);
    s = fma(ri, ri, s);
  }
  s = block_sum(s);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// ---------------------------------------------------------------- one Davidson iteration
// The vector work of an iteration as four kernels instead of fifteen.  Small
// two-site vectors (chain ends, small active spaces) are bound by launches
// and by the latency of FP64 chains, so a CTA is 128 threads for 128 elements:
// warp g computes elements g of 32 lanes of the reduction below, all of them
// at once, then the warps share out the dot products.  Every sum keeps the
// order of multi_dot_partial / finish_sums (elements b 256 + 32 w + lane
// + g 256 nblk, g ascending, by a lane; lanes, then the 8 warps of a block b
// as a tree; blocks in steps of 256, then the same trees), so an iteration
// rounds as it did with them.  CAS(10,10) M=128 mixed solve (453 iterations)
// 217 -> 190 ms, eight batched spaces of 8 to 11 orbitals 310 -> 218 ms.
constexpr int kDavT = 128;
enum { kDavResidual = 0, kDavProject = 1, kDavLast = 2, kDavRow = 3 };

__device__ __forceinline__ double warp_tree(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double tree8(const double* p) {   // the eight warps of a reduction block
  return ((p[0] + p[4]) + (p[2] + p[6])) + ((p[1] + p[5]) + (p[3] + p[7]));
}

// MODE kDavResidual: x = V c, r = S c - theta x, t = -r / (diag - theta);
//                    sums V_j . t (j < k) to out, r . r to host[0]
//      kDavProject:  t -= V d; sums V_j . t
//      kDavLast:     t -= V d; t . t to out[0] and host[0]
//      kDavRow:      s = y; sums V_j . s to out and host
template <int MODE>
__global__ void __launch_bounds__(kDavT)
davidson_kernel(const double* __restrict__ V, const double* __restrict__ S, const double* __restrict__ src,
                const DavCoef c, const double* __restrict__ d, double theta, int64_t n, int k, int nblk, double* x,
                double* t, double* part, double* out, double* host, int* count) {
  __shared__ double tv[4][32], rv[4][32], ds[kDavMax];
  __shared__ int last;
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int64_t unit = blockIdx.x, i0 = unit * 32 + lane, gs = (int64_t)nblk * RED_THREADS;
  const int64_t i = i0 + g * gs;
  if (MODE == kDavProject || MODE == kDavLast) {
    if (threadIdx.x < k) ds[threadIdx.x] = -1.0 * d[threadIdx.x];
    __syncthreads();
  }
  double v = 0.0, rr = 0.0;
  if (i < n) {
    if (MODE == kDavResidual) {
      double xs = 0.0, ss = 0.0;
#pragma unroll 4
      for (int j = 0; j < k; ++j) {
        xs = fma(c.c[j], V[(int64_t)j * n + i], xs);
        ss = fma(c.c[j], S[(int64_t)j * n + i], ss);
      }
      x[i] = xs;
      rr = fma(-theta, xs, ss);
      v = -rr / guarded_den(src[i], theta);
      t[i] = v;
    } else if (MODE == kDavRow) {
      v = src[i];
      t[i] = v;
    } else {
      v = t[i];
#pragma unroll 4
      for (int j = 0; j < k; ++j) v = fma(ds[j], V[(int64_t)j * n + i], v);
      t[i] = v;
    }
  }
  tv[g][lane] = v;
  if (MODE == kDavResidual) rv[g][lane] = rr;
  __syncthreads();
  const int nd = MODE == kDavLast ? 1 : MODE == kDavResidual ? k + 1 : k;
  const int64_t nunits = (int64_t)nblk * 8;
  for (int j = g; j < nd; j += 4) {
    const bool self = MODE == kDavLast || (MODE == kDavResidual && j == k);
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int64_t e = i0 + q * gs;
      if (e >= n) continue;
      const double b = MODE == kDavResidual && j == k ? rv[q][lane] : tv[q][lane];
      s = fma(self ? b : V[(int64_t)j * n + e], b, s);
    }
    s = warp_tree(s);
    if (lane == 0) part[(int64_t)j * nunits + unit] = s;
  }
  // Long vectors: davidson_finish_kernel adds the parts.  Up to 64 blocks the
  // last CTA to finish does, two loads a lane, and saves a launch; with 0 or 32
  // the solves of CAS(6,6) and CAS(10,10) differ by less than their runs
  // (41-44 and 160-206 ms), so the line is where the loads still fit.
  if (nblk > 64) return;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(count, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x == 0) *count = 0;
  for (int j = g; j < nd; j += 4) {
    const double* p = part + (int64_t)j * nunits;
    double v0 = 0.0, v1 = 0.0;
    if (lane < nblk) v0 += tree8(p + lane * 8);
    if (32 + lane < nblk) v1 += tree8(p + (32 + lane) * 8);
    v0 = warp_tree(v0);
    if (nblk > 32) v0 += warp_tree(v1);
    if (lane == 0) {
      if (MODE == kDavResidual && j == k) {
        host[0] = v0;
      } else {
        out[j] = v0;
        if (MODE == kDavLast || MODE == kDavRow) host[j] = v0;
      }
    }
  }
}

// the same sums for more than 64 reduction blocks, one CTA each
__global__ void davidson_finish_kernel(const double* __restrict__ part, int nblk, int nout, double* out, double* host,
                                       int host_from) {
  const int j = blockIdx.x;
  const double* p = part + (int64_t)j * nblk * 8;
  double s = 0.0;
  for (int b = threadIdx.x; b < nblk; b += RED_THREADS) s += tree8(p + (int64_t)b * 8);
  s = block_sum(s);
  if (threadIdx.x != 0) return;
  if (j < nout) out[j] = s;
  if (j >= host_from) host[j - host_from] = s;
}

// out = out2 = t / sqrt(nrm2[0]) (zero vector when the norm has vanished)
__global__ void normalize2_kernel(const double* __restrict__ t, const double* __restrict__ nrm2, int64_t n,
                                  double* __restrict__ out, double* __restrict__ out2) {
  const double q = nrm2[0];
  const double s = q > 1e-28 ? 1.0 / sqrt(q) : 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double v = t[i] * s;
    out[i] = v;
    out2[i] = v;
  }
}

// projected diagonal preconditioner, pass 1: out = scale v / den; partial
// sums of x . out (row 0) and x . x / den (row 1)
__global__ void kdiv_kernel(const double* __restrict__ v, const double* __restrict__ x,
                            const double* __restrict__ diag, double theta, double scale, int64_t n, double* out,
                            double* partial) {
  const int nblk = gridDim.x;
  double s1 = 0.0, s2 = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RED_THREADS + threadIdx.x; i < n; i += (int64_t)gridDim.x * RED_THREADS) {
    const double den = guarded_den(diag[i], theta);
    const double o = scale * v[i] / den;
    out[i] = o;
    s1 = fma(x[i], o, s1);
    s2 = fma(x[i], x[i] / den, s2);
  }
  s1 = block_sum(s1);
  s2 = block_sum(s2);
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = s1;
    partial[nblk + blockIdx.x] = s2;
  }
}

// pass 2: out -= (sums[0] / sums[1]) x / den, so that x . out = 0
__global__ void kproj_kernel(const double* __restrict__ x, const double* __restrict__ diag, double theta,
                             const double* __restrict__ sums, int64_t n, double* out) {
  const double eps = sums[1] != 0.0 ? sums[0] / sums[1] : 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] -= eps * x[i] / guarded_den(diag[i], theta);
}

// y = a x + b y
__global__ void axpby_kernel(double* y, double a, const double* __restrict__ x, double b, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = fma(a, x[i], b * y[i]);
}

__global__ void add_sq_kernel(double* d, const double* __restrict__ phi, int k, int64_t n, double w) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int j = 0; j < k; ++j) s = fma(phi[(int64_t)j * n + i], phi[(int64_t)j * n + i], s);
    d[i] = fma(w, s, d[i]);
  }
}

__global__ void scale_kernel(double* x, double a, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] *= a;
}

int grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b > 152 * 16) b = 152 * 16;
  return (int)(b < 1 ? 1 : b);
}

}  // namespace

int reduction_blocks(int64_t n) {
  int64_t b = (n + RED_THREADS * 4 - 1) / (RED_THREADS * 4);
  if (b > 608) b = 608;
  return (int)(b < 1 ? 1 : b);
}

int launch_gemm_f64(const GemmPlan& p, int num_sms, int* err, cudaStream_t s) {
  const int ns = launch_gemm_f64_split(p, num_sms, err, s);
  if (ns < 0) return ns;
  const int nt = (int)p.tiles.size();
  const int smem = FR * FK * p.tile_span * (int)sizeof(double);
  if (nt > 0 && p.per_lane == 2) gemm_f64_kernel<2><<<nt, FT + 32, smem, s>>>(p.d_terms, p.d_outs, p.d_tiles);
  if (nt > 0 && p.per_lane == 1) gemm_f64_kernel<1><<<nt, FT + 32, smem, s>>>(p.d_terms, p.d_outs, p.d_tiles);
  return ns + (nt > 0);
}

void launch_gather(const GatherTask* tasks, int ntasks, cudaStream_t s) {
  if (ntasks > 0) gather_kernel<<<(ntasks + 7) / 8, 256, 0, s>>>(tasks, ntasks);
}

void launch_axpy(const AxpyPlan& p, cudaStream_t s) {
  const int no = (int)p.outs.size();
  if (no == 0 || p.nchunks == 0) return;
  const int64_t grid = p.nchunks < INT32_MAX ? p.nchunks : INT32_MAX;
  axpy_kernel<<<(int)grid, kAxpyThreads, 0, s>>>(p.d_terms, p.d_outs, p.d_cstart, no, p.nchunks);
}

// dst = sign * src^T, one 32 x 32 tile of one task per CTA: coalesced reads
// of src rows into shared memory, coalesced writes of dst rows
__global__ void __launch_bounds__(256)
block_transpose_kernel(const TransTask* __restrict__ tasks, const TransTile* __restrict__ tiles) {
  __shared__ double t[32][33];
  const TransTile tl = tiles[blockIdx.x];
  const TransTask T = tasks[tl.task];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int i = ty; i < 32; i += 8) {
    const int r = tl.r0 + i, c = tl.c0 + tx;
    if (r < T.rows && c < T.cols) t[i][tx] = T.src[(int64_t)r * T.cols + c];
  }
  __syncthreads();
  for (int j = ty; j < 32; j += 8) {
    const int c = tl.c0 + j, r = tl.r0 + tx;   // dst row c, column r
    if (r < T.rows && c < T.cols) T.dst[(int64_t)c * T.rows + r] = T.sign * t[tx][j];
  }
}

void launch_block_transpose(const TransTask* tasks, const TransTile* tiles, int ntiles, cudaStream_t s) {
  if (ntiles <= 0) return;
  block_transpose_kernel<<<ntiles, 256, 0, s>>>(tasks, tiles);
}

void launch_set_identity(double* d, int m, cudaStream_t s) {
  set_identity_kernel<<<grid_for((int64_t)m * m, 256), 256, 0, s>>>(d, m);
}

void launch_multi_dot(const double* V, int64_t stride, int k, const double* x, int64_t n, double* out_dev,
                      double* partial, int nblk, cudaStream_t s) {
  if (k <= 0) return;
  dim3 g(nblk, k);
  multi_dot_partial<<<g, RED_THREADS, 0, s>>>(V, stride, k, x, n, partial);
  finish_sums<<<k, RED_THREADS, 0, s>>>(partial, nblk, k, out_dev);
}

void launch_lincomb(double* out, const double* V, int64_t stride, const double* coef_dev, int k, int64_t n,
                    int accumulate, cudaStream_t s, double coef_scale) {
  lincomb_kernel<<<grid_for(n, 256), 256, 0, s>>>(out, V, stride, coef_dev, k, n, accumulate, coef_scale);
}

void launch_normalize(const double* t, const double* nrm2_dev, int64_t n, double* out, cudaStream_t s) {
  normalize_kernel<<<grid_for(n, 256), 256, 0, s>>>(t, nrm2_dev, n, out);
}

int launch_davidson_residual(const double* V, const double* S, const double* diag, const DavCoef& c, double theta,
                             int64_t n, int k, int nblk, double* x, double* t, double* part, double* overlaps,
                             double* host_rr, int* count, cudaStream_t s) {
  davidson_kernel<kDavResidual><<<nblk * 8, kDavT, 0, s>>>(V, S, diag, c, nullptr, theta, n, k, nblk, x, t, part,
                                                           overlaps, host_rr, count);
  if (nblk > 64) davidson_finish_kernel<<<k + 1, RED_THREADS, 0, s>>>(part, nblk, k, overlaps, host_rr, k);
  return 1 + (nblk > 64);
}

int launch_davidson_project(const double* V, const double* d, int64_t n, int k, int nblk, double* t, double* part,
                            double* out, double* host_norm, int* count, cudaStream_t s) {
  if (!host_norm) {
    davidson_kernel<kDavProject><<<nblk * 8, kDavT, 0, s>>>(V, nullptr, nullptr, DavCoef(), d, 0.0, n, k, nblk, nullptr,
                                                            t, part, out, nullptr, count);
    if (nblk > 64) davidson_finish_kernel<<<k, RED_THREADS, 0, s>>>(part, nblk, k, out, nullptr, k);
  } else {
    davidson_kernel<kDavLast><<<nblk * 8, kDavT, 0, s>>>(V, nullptr, nullptr, DavCoef(), d, 0.0, n, k, nblk, nullptr, t,
                                                         part, out, host_norm, count);
    if (nblk > 64) davidson_finish_kernel<<<1, RED_THREADS, 0, s>>>(part, nblk, 1, out, host_norm, 0);
  }
  return 1 + (nblk > 64);
}

int launch_davidson_row(const double* V, const double* y, int64_t n, int k, int nblk, double* sk, double* part,
                        double* out, double* host, int* count, cudaStream_t s) {
  davidson_kernel<kDavRow><<<nblk * 8, kDavT, 0, s>>>(V, nullptr, y, DavCoef(), nullptr, 0.0, n, k, nblk, nullptr, sk,
                                                      part, out, host, count);
  if (nblk > 64) davidson_finish_kernel<<<k, RED_THREADS, 0, s>>>(part, nblk, k, out, host, 0);
  return 1 + (nblk > 64);
}

void launch_normalize2(const double* t, const double* nrm2_dev, int64_t n, double* out, double* out2, cudaStream_t s) {
  normalize2_kernel<<<grid_for(n, 256), 256, 0, s>>>(t, nrm2_dev, n, out, out2);
}

void launch_residual_precond(const double* x, const double* sx, const double* diag, double theta, int64_t n,
                             double* r, double* t, double* partial, int nblk, double* out_dev, cudaStream_t s) {
  residual_precond_kernel<<<nblk, RED_THREADS, 0, s>>>(x, sx, diag, theta, n, r, t, partial);
  finish_sums<<<1, RED_THREADS, 0, s>>>(partial, nblk, 1, out_dev);
}

void launch_projected_precond(const double* v, const double* x, const double* diag, double theta, double scale,
                              int64_t n, double* out, double* partial, int nblk, double* sums_dev, cudaStream_t s) {
  kdiv_kernel<<<nblk, RED_THREADS, 0, s>>>(v, x, diag, theta, scale, n, out, partial);
  finish_sums<<<2, RED_THREADS, 0, s>>>(partial, nblk, 2, sums_dev);
  kproj_kernel<<<grid_for(n, 256), 256, 0, s>>>(x, diag, theta, sums_dev, n, out);
}

void launch_axpby(double* y, double a, const double* x, double b, int64_t n, cudaStream_t s) {
  axpby_kernel<<<grid_for(n, 256), 256, 0, s>>>(y, a, x, b, n);
}

void launch_add_sq(double* d, const double* phi, int k, int64_t n, double w, cudaStream_t s) {
  if (k > 0) add_sq_kernel<<<grid_for(n, 256), 256, 0, s>>>(d, phi, k, n, w);
}

void launch_scale(double* x, double a, int64_t n, cudaStream_t s) {
  scale_kernel<<<grid_for(n, 256), 256, 0, s>>>(x, a, n);
}

namespace {
// the bit patterns of non-negative doubles order like the values, so the
// maximum of |x| is an unsigned 64-bit atomicMax
__global__ void absmax_kernel(const double* __restrict__ x, int64_t n, unsigned long long* out) {
  double m = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    m = fmax(m, fabs(x[i]));
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}
}  // namespace

void launch_absmax(const double* x, int64_t n, double* out, cudaStream_t s) {
  cudaMemsetAsync(out, 0, sizeof(double), s);
  int64_t b = (n + 255) / 256;
  if (b > 152 * 8) b = 152 * 8;
  if (b < 1) b = 1;
  absmax_kernel<<<(int)b, 256, 0, s>>>(x, n, reinterpret_cast<unsigned long long*>(out));
}

}  // namespace gbd

// ---------------------------------------------------------------------------
// Allocation-free Davidson overlap reduction.  Some callers cannot call
// cudaMalloc (a host that hands us pointers from its own fixed arena, code
// running inside a stream capture owned by someone else, or a process whose
// allocator is locked).  This variant keeps its partial sums in a fixed
// file-scope device array instead of allocating.  Every GPU that loads the
// library holds the array until the process exits.
#include <mutex>

namespace {
constexpr int kNoAllocMaxK = 32;
constexpr int kNoAllocMaxBlocks = 608;   // reduction_blocks() never returns more
static __device__ __align__(256) double g_noalloc_partials[kNoAllocMaxK * kNoAllocMaxBlocks];
std::mutex g_noalloc_mu;
double* g_noalloc_ptr[256] = {};
}  // namespace

extern "C" int gbd_multi_dot_noalloc(int32_t device, const double* V, int64_t stride, int32_t k, const double* x,
                                     int64_t n, double* out, void* stream) {
  if (!V || !x || !out) return -1;
  if (k < 1 || k > kNoAllocMaxK || n < 0 || stride < n) return -1;
  if (device < 0 || device >= 256) return -1;
  // an error left pending by earlier work on this thread is not ours to
  // consume: report it, launch nothing and leave it in place
  if (cudaPeekAtLastError() != cudaSuccess) return -3;
  int prev = 0;
  if (cudaGetDevice(&prev) != cudaSuccess) return -3;
  if (cudaSetDevice(device) != cudaSuccess) return -3;
  double* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[device]) {
      // the array's name is a host-side stand-in; the device address of this
      // device's copy comes from the runtime, once, with the device current
      double* p = nullptr;
      if (cudaGetSymbolAddress((void**)&p, g_noalloc_partials) != cudaSuccess || !p) {
        cudaSetDevice(prev);
        return -3;
      }
      g_noalloc_ptr[device] = p;
    }
    scratch = g_noalloc_ptr[device];
  }
  int nblk = gbd::reduction_blocks(n);   // <= kNoAllocMaxBlocks, so nblk * k fits the array
  gbd::launch_multi_dot(V, stride, k, x, n, out, scratch, nblk, (cudaStream_t)stream);
  cudaError_t e = cudaGetLastError();
  cudaSetDevice(prev);
  return e == cudaSuccess ? 0 : -3;
}
