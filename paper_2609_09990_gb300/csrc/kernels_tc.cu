// tcgen05 + TMA grouped GEMM for the reduced-precision sigma build (sm_103a).
//
// Persistent, warp-specialised CTA of 6 warps (one per SM):
//   warp 0   TMA producer: one thread streams the A and B boxes of every
//            K chunk of every term of the CTA's tiles into a ring of
//            shared-memory stages (128B-swizzled, mbarrier complete_tx);
//   warp 1   owns TMEM (512 columns = two 128x256 FP32 accumulators) and one
//            thread issues tcgen05.mma (M = 128, N = n_mma, K step 16 for
//            BF16 / 8 for TF32) and tcgen05.commit;
//   warps 2-5 epilogue: tcgen05.ld of the accumulator rows they may access
//            (TMEM lane quarter = warp id % 4), conversion, global stores.
// Two accumulators let the epilogue of tile i overlap the MMAs of tile i+1.
// TF32x3 and BF16x3 (accurate tiers) split every operand into hi + lo of
// that type and issue hi*hi + hi*lo + lo*hi into the same accumulator.
// Every mbarrier wait is bounded: on timeout the kernel raises *err, all
// roles stop issuing, and TMEM is released before the CTA exits.
//
// What bounds it: with blocks of a few dozen rows and a dozen short MMAs per
// K chunk (TF32x3) the issuing lane itself was the limit, ~1500 clocks per
// chunk whatever the tile width, while the loads waited for free stages.  So
// the issuer is as lean as it can be: the type is a template argument, the
// K steps are unrolled, the descriptors of a chunk are formed once and
// advanced by additions, and both issuing roles run in the lane that
// elect.sync names (600-750 clocks per chunk now).  Stage A was bound by its
// epilogue, whose 16-byte stores filled half a sector each: a lane stores 32
// bytes at a time.  All accumulators and roundings are those of before.
// Per sigma: CAS(16,16) M=512 12.9 -> 9.1 ms for 38 launches, CAS(20,20)
// M=1024 58.8 -> 45.2 ms for 40, a full solve of CAS(10,10) 19.5 -> 13.2 ms
// for 634.  Now stage A waits for its boxes (two stages of 96 KB at N = 256).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "convert_bits.h"
#include "mbarrier.h"
#include "smem_limit.h"
#include "tc_gemm.h"

namespace gbd {

namespace {

constexpr int kThreads = 192;
constexpr int kStageA = 128 * 128;          // bytes of one A box (128 rows x 128 B)
constexpr int kSmemBudget = 232448;         // dynamic shared memory per CTA
constexpr int kMaxStages = 8;

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(smem_addr(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_addr(bar))
      : "memory");
}

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart (SBO), SM100 descriptor version 1
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;                 // LBO (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;       // SBO
  d |= (uint64_t)1 << 46;                 // version
  d |= (uint64_t)2 << 61;                 // SWIZZLE_128B
  return d;
}

template <bool bf>
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  if (bf)
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
  else
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// true in one lane of a converged warp.  The issuing roles run in the elected
// lane: the compiler then knows that one thread is active and feeds the tensor
// core and TMA instructions their uniform operands directly.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xFFFFFFFF;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}

// 32 bytes, one full sector per lane (d is 32-byte aligned)
__device__ __forceinline__ void store32(void* d, const uint32_t* w) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(d), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]),
               "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}

// the CTA's tile i (an empty one past the end) and its first term
__device__ __forceinline__ TcTile tile_at(const TcLaunch& L, int i) {
  TcTile T{};
  if (i < L.ntiles) T = L.tiles[i];
  return T;
}
__device__ __forceinline__ TcTerm first_term(const TcLaunch& L, const TcTile& T) {
  TcTerm t{};
  if (T.t1 > T.t0) t = L.terms[T.t0];
  return t;
}

template <bool bf, bool x3>
__global__ void __launch_bounds__(kThreads, 1) tc_gemm_kernel(const __grid_constant__ TcMaps maps,
                                                             const TcLaunch L) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // B boxes of this launch are at most L.ncap rows; the ring holds as many
  // stages as fit (tc_stages)
  const int bstage = L.ncap * 128;
  const int stages = L.stages;
  const int stage_bytes = (kStageA + bstage) * (x3 ? 2 : 1);
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(base + stages * stage_bytes);
  uint64_t* empty = full + stages;
  uint64_t* tfull = empty + stages;     // [2]
  uint64_t* tempty = tfull + 2;         // [2]
  uint32_t* tslot = reinterpret_cast<uint32_t*>(tempty + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int kc = bf ? kTcKChunk16 : kTcKChunk32;     // K elements per stage
  constexpr int kstep = bf ? 16 : 8;                      // K per MMA

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tfull[a], 1);
      mbar_init(&tempty[a], 128);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_addr(tslot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  if (warp == 0 && elect_one()) {
    // ---------------- TMA producer
    int stage = 0;
    uint32_t ph = 0;
    bool ok = true;
    // descriptors are software-pipelined: the tile after the next, the next
    // tile's first term and the next term are in flight while the current
    // ones are issued (each is a trip to L2, and many tiles are one box long)
    TcTile Tc = tile_at(L, blockIdx.x), Tn = tile_at(L, blockIdx.x + gridDim.x);
    TcTerm first_n = first_term(L, Tc);
    for (int tile = blockIdx.x; tile < L.ntiles && ok; tile += gridDim.x) {
      const TcTile T = Tc;
      TcTerm tmn = first_n;
      Tc = Tn;
      first_n = first_term(L, Tn);
      Tn = tile_at(L, tile + 2 * (int)gridDim.x);
      const int bbytes = (16 << T.bsel) * 128;
      const uint32_t tx = (uint32_t)(kStageA + bbytes) * (x3 ? 2 : 1);
      for (int t = T.t0; t < T.t1 && ok; ++t) {
        const TcTerm tm = tmn;
        if (t + 1 < T.t1) tmn = L.terms[t + 1];
        for (int k0 = 0; k0 < tm.k; k0 += kc) {
          if (!mbar_wait(&empty[stage], ph ^ 1, L.err)) { ok = false; break; }
          uint8_t* sa = base + stage * stage_bytes;
          uint8_t* sb = sa + kStageA;
          // K-blocked operands step down by ays / bys rows per box,
          // the others step right by one box
          const int kb = k0 / kc;
          const int xa = tm.ax + (tm.ays ? 0 : k0), ya = tm.ay + T.m0 + kb * tm.ays;
          const int xb = tm.bx + (tm.bys ? 0 : k0), yb = tm.by + T.n0 + kb * tm.bys;
          mbar_expect_tx(&full[stage], tx);
          tma_load_2d(sa, &maps.a[0], xa, ya, &full[stage]);
          tma_load_2d(sb, &maps.b[0][T.bsel], xb, yb, &full[stage]);
          if (x3) {
            uint8_t* sa2 = sb + bstage;
            tma_load_2d(sa2, &maps.a[1], xa, ya, &full[stage]);
            tma_load_2d(sa2 + kStageA, &maps.b[1][T.bsel], xb, yb, &full[stage]);
          }
          if (++stage == stages) { stage = 0; ph ^= 1; }
        }
      }
    }
    // a chunk armed but never consumed (error path): let its copies land
    // before the CTA can exit
    if (!ok || *(volatile int*)L.err) {
      for (int s = 0; s < stages; ++s)
        for (uint32_t it = 0; it < (1u << 20) && !mbar_try(&full[s], ph); ++it) {
        }
    }
  } else if (warp == 1 && elect_one()) {
    // ---------------- MMA issuer
    int stage = 0;
    uint32_t ph = 0;
    int acc_i = 0;
    bool ok = true;
    const uint32_t fmt = bf ? 1u : 2u;
    TcTile Tc = tile_at(L, blockIdx.x), Tn = tile_at(L, blockIdx.x + gridDim.x);
    TcTerm first_n = first_term(L, Tc);
    for (int tile = blockIdx.x; tile < L.ntiles && ok; tile += gridDim.x, ++acc_i) {
      const TcTile T = Tc;
      TcTerm tmn = first_n;
      Tc = Tn;
      first_n = first_term(L, Tn);
      Tn = tile_at(L, tile + 2 * (int)gridDim.x);
      const int a = acc_i & 1;
      const uint32_t aph = (acc_i >> 1) & 1;
      if (!mbar_wait(&tempty[a], aph ^ 1, L.err)) { ok = false; break; }
      tc_fence_after();
      const uint32_t dt = tmem + (uint32_t)(a * 256);
      uint32_t first = 1;
      for (int t = T.t0; t < T.t1 && ok; ++t) {
        const TcTerm tm = tmn;
        if (t + 1 < T.t1) tmn = L.terms[t + 1];
        const uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(tm.neg & 1) << 13) |
                               ((uint32_t)(T.n_mma >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        for (int k0 = 0; k0 < tm.k; k0 += kc) {
          if (!mbar_wait(&full[stage], ph, L.err)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sa = smem_addr(base + stage * stage_bytes);
          const uint32_t sb = sa + kStageA;
          const int nk = min(kc, tm.k - k0) / kstep;
          const uint64_t ad = smem_desc(sa), bd = smem_desc(sb);
          const uint64_t ad2 = smem_desc(sb + bstage), bd2 = smem_desc(sb + bstage + kStageA);
#pragma unroll
          for (int kk = 0; kk < kc / kstep; ++kk) {   // 32 bytes of K: 2 units of the start address
            if (kk == nk) break;
            mma<bf>(dt, ad + 2 * kk, bd + 2 * kk, idesc, first ? 0u : 1u);
            if (x3) {
              mma<bf>(dt, ad + 2 * kk, bd2 + 2 * kk, idesc, 1u);   // hi * lo
              mma<bf>(dt, ad2 + 2 * kk, bd + 2 * kk, idesc, 1u);   // lo * hi
            }
            first = 0;
          }
          mma_commit(&empty[stage]);
          if (++stage == stages) { stage = 0; ph ^= 1; }
        }
      }
      mma_commit(&tfull[a]);
    }
  } else if (warp >= 2) {
    // ---------------- epilogue: TMEM -> registers -> global
    const int q = warp & 3;              // TMEM lane quarter this warp may read
    const int row = q * 32 + lane;       // accumulator row (A row within the tile)
    int acc_i = 0;
    // the tile after the next, and the next tile's output row (two dependent
    // loads), are fetched while the current one is stored
    auto member = [&](const TcTile& X) {
      return X.mode == kTcYTblk && row < X.m_valid ? L.ymem[X.out + row] : -1;
    };
    TcTile Tc = tile_at(L, blockIdx.x), Tn = tile_at(L, blockIdx.x + gridDim.x);
    int mem = member(Tc);
    TcYRow yn{};
    if (mem >= 0) yn = L.yrows[mem];
    for (int tile = blockIdx.x; tile < L.ntiles; tile += gridDim.x, ++acc_i) {
      const TcTile T = Tc;
      TcYRow yr = yn;
      Tc = Tn;
      mem = member(Tn);
      Tn = tile_at(L, tile + 2 * (int)gridDim.x);
      const bool has = T.t1 > T.t0;
      const bool live = row < T.m_valid;
      yr.base += (T.out + row - yr.first) * (int64_t)kc;
      const int a = acc_i & 1;
      const uint32_t aph = (acc_i >> 1) & 1;
      if (!mbar_wait(&tfull[a], aph, L.err)) break;
      tc_fence_after();
      if (mem >= 0) yn = L.yrows[mem];
      for (int c0 = 0; c0 < T.n_mma; c0 += 16) {
        float v[16];
        if (has) {
          tmem_ld16(tmem + (uint32_t)(a * 256 + c0) + ((uint32_t)(q * 32) << 16), v);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = 0.f;
        }
        if (!live) continue;
        if (T.mode == kTcYTblk) {
          // 16 contiguous output columns: section s, K offset k, block k / kc
          if (c0 >= T.n_valid) continue;
          const int c = T.n0 + c0;
          int koff = yr.koff[0], brk = T.rbreak[0];
#pragma unroll
          for (int u = 1; u < 4; ++u)
            if (c >= T.rbreak[u]) {
              koff = yr.koff[u];
              brk = T.rbreak[u];
            }
          if (koff < 0) continue;
          const int k = koff + (c - brk);
          const int64_t idx = yr.base + (int64_t)(k / kc) * yr.stride + (k % kc);
          if (bf) {
            uint32_t w[8], wl[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              __nv_bfloat162 p2 = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
              w[i] = *reinterpret_cast<uint32_t*>(&p2);
              __nv_bfloat162 l2 = __floats2bfloat162_rn(v[2 * i] - __low2float(p2), v[2 * i + 1] - __high2float(p2));
              wl[i] = *reinterpret_cast<uint32_t*>(&l2);
            }
            store32(reinterpret_cast<__nv_bfloat16*>(L.yt_hi) + idx, w);
            if (x3) store32(reinterpret_cast<__nv_bfloat16*>(L.yt_lo) + idx, wl);
          } else {
            uint32_t h[16], l[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float hi = to_tf32(v[i]);
              h[i] = __float_as_uint(hi);
              l[i] = __float_as_uint(to_tf32(v[i] - hi));
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              store32(reinterpret_cast<float*>(L.yt_hi) + idx + 8 * u, h + 8 * u);
              if (x3) store32(reinterpret_cast<float*>(L.yt_lo) + idx + 8 * u, l + 8 * u);
            }
          }
          continue;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int j = c0 + i;
          if (j >= T.n_valid) break;
          if (T.mode == kTcSigma) {
            double* o = L.f64 + T.out + (int64_t)j * T.ld + T.m0 + row;
            *o = T.beta ? (*o + (double)v[i]) : (double)v[i];
          } else {
            L.part[T.out + (int64_t)j * 128 + row] = v[i];
          }
        }
      }
      tc_fence_before();
      mbar_arrive(&tempty[a]);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

// ---------------------------------------------------------------- bounded waits
// The failure path of every mbarrier wait, on its own: one thread
// waits (with the same bounded helper) on a barrier that is completed only
// when `arrive` is set.  Without the arrival the wait runs out, raises
// *err and the kernel returns; nothing hangs and no memory is touched
// outside the barrier and the flag.
__global__ void bounded_wait_probe_kernel(int arrive, int* err, int* waited_ok) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (arrive) mbar_arrive(&bar);
    *waited_ok = mbar_wait(&bar, 0, err) ? 1 : 0;
  }
}

// the last of n records (n > 0) whose key, ascending from key(0) <= e, is at
// most e, found by a converged warp: 32 probes a round instead of one
template <class Key>
__device__ __forceinline__ int warp_find(int n, int64_t e, Key key) {
  const int lane = threadIdx.x & 31;
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int step = (hi - lo + 31) >> 5, i = lo + lane * step;
    const int k = __popc(__ballot_sync(0xffffffffu, i < hi && key(i) <= e));
    hi = min(hi, lo + k * step);
    lo += (k - 1) * step;
  }
  return lo;
}

// ---------------------------------------------------------------- split-K sum
// one thread per output element; the slots are summed in FP64 with eight
// interleaved partial sums combined in a fixed order (deterministic).  The
// eight loads of a round are independent, so a long slot list is not a
// chain of dependent memory latencies; a warp finds the task of its first
// element together.  Bound by the FP64 pipe, one addition a value: a conversion
// costs it as much, and one that is predicated off does too, hence widen and
// the loop exits.  CAS(20,20) M=1024, 227 slots of 1.1 M elements at most: 573
// -> 310 us; CAS(16,16) M=512, 137 of 0.29 M: 108 -> 71 us.
__global__ void tc_reduce_kernel(const TcRed* __restrict__ tasks, int ntasks, int64_t total,
                                 const float* __restrict__ part, double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  for (int64_t e0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; e0 < total;
       e0 += (int64_t)gridDim.x * blockDim.x) {
    int lo = warp_find(ntasks, e0, [&](int i) { return tasks[i].e0; });
    const int64_t e = e0 + lane;
    if (e >= total) break;
    while (lo + 1 < ntasks && tasks[lo + 1].e0 <= e) ++lo;
    const TcRed R = tasks[lo];
    const int loc = (int)(e - R.e0);
    const int j = loc / R.m_valid, i = loc - j * R.m_valid;
    const int64_t ss = (int64_t)128 * R.n_stride;
    const float* p = part + R.slot0 + (int64_t)j * 128 + i;
    double a[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    int s = 0;
    for (; s + 8 <= R.nslot; s += 8) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = p[(s + u) * ss];
#pragma unroll
      for (int u = 0; u < 8; ++u) a[u] += widen(v[u]);
    }
#pragma unroll
    for (int u = 0; u < 7; ++u) {   // the rest, as one round (no indexed array)
      if (s + u >= R.nslot) break;
      a[u] += widen(p[(s + u) * ss]);
    }
    out[R.out + (int64_t)j * R.ld + R.m0 + i] = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
  }
}

// ---------------------------------------------------------------- conversions
__device__ __forceinline__ void store_conv(double x, int prec, void* hi, void* lo, int64_t idx) {
  if (prec == kBF16 || prec == kBF16x3) {
    const __nv_bfloat16 h = __double2bfloat16(x);
    reinterpret_cast<__nv_bfloat16*>(hi)[idx] = h;
    if (prec == kBF16x3) reinterpret_cast<__nv_bfloat16*>(lo)[idx] = __double2bfloat16(x - (double)__bfloat162float(h));
  } else {
    const float h = to_tf32((float)x);
    reinterpret_cast<float*>(hi)[idx] = h;
    if (prec == kTF32x3) reinterpret_cast<float*>(lo)[idx] = to_tf32((float)(x - (double)h));
  }
}

// A block per sub-block.  Positions advance by additions (256 elements a step),
// divisions are once a task, and four loads of a thread are in flight together.
// Transposed sources (the conjugate channels) are read along their rows and
// turned in shared memory, so that the panel rows are written in runs too:
// single elements of 32 different sectors were the bound, then the five FP64
// instructions an element.  The four conversions of a CAS(20,20) M=1024 step:
// 13.0 -> 6.7 ms; additions for divisions alone 13.0, then without FP64 12.0,
// turned in shared memory 7.3.
__global__ void __launch_bounds__(256) tc_convert_kernel(const TcConv* __restrict__ tasks, int ntasks, int prec, void* hi,
                                                         void* lo, int64_t pitch) {
  constexpr int kU = 4, kBuf = 2048;
  __shared__ double buf[kBuf];
  const int sh = 63 - __clzll(pitch);   // K-blocked panels: pitch is a power of two
  for (int t = blockIdx.x; t < ntasks; t += gridDim.x) {
    const TcConv c = tasks[t];
    if (c.rows <= 0 || c.cols <= 0) continue;
    const bool unit = fabs(c.scale) == 1.0;
    const uint32_t flip = c.scale < 0.0 ? 0x80000000u : 0u;
    auto put = [&](int r, int col, double x) {
      col += c.c0;
      const int64_t dst = c.kstride > 0
                              ? (((int64_t)c.r0 + (int64_t)(col >> sh) * c.kstride + r) << sh) + (col & ((1 << sh) - 1))
                              : (int64_t)(c.r0 + r) * pitch + col;
      const uint32_t xh = (uint32_t)__double2hiint(x) ^ flip, xl = (uint32_t)__double2loint(x);
      float h, l;
      uint16_t b;
      if (unit && prec == kTF32x3 && split_tf32(xh, xl, &h, &l)) {
        reinterpret_cast<float*>(hi)[dst] = h;
        reinterpret_cast<float*>(lo)[dst] = l;
      } else if (unit && prec == kBF16 && round_bf16(xh, xl, &b)) {
        reinterpret_cast<uint16_t*>(hi)[dst] = b;
      } else {
        store_conv(c.scale * x, prec, hi, lo, dst);
      }
    };
    // elements (o, i) of an outer x inner rectangle, i fastest, 256 apart; four at a time
    auto walk = [&](int outer, int inner, auto load, auto use) {
      const int so = 256 / inner, si = 256 - so * inner;
      int o = threadIdx.x / inner, i = threadIdx.x - o * inner;
      while (o < outer) {
        double x[kU];
        int oo[kU], ii[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          oo[u] = o;
          ii[u] = i;
          if (o < outer) x[u] = load(o, i);
          o += so;
          i += si;
          if (i >= inner) {
            i -= inner;
            ++o;
          }
        }
#pragma unroll
        for (int u = 0; u < kU; ++u)
          if (oo[u] < outer) use(oo[u], ii[u], x[u]);
      }
    };
    if (!c.trans || c.rows > kBuf / 8) {
      const int inner = c.trans ? c.rows : c.cols, outer = c.trans ? c.cols : c.rows;
      walk(outer, inner, [&](int o, int i) { return c.src[(int64_t)o * c.ld_src + i]; },
           [&](int o, int i, double x) { put(c.trans ? i : o, c.trans ? o : i, x); });
      continue;
    }
    const int per = ((kBuf / c.rows) - 1) | 1;   // columns at a time, odd: no bank conflicts
    for (int c0 = 0; c0 < c.cols; c0 += per) {
      const int nc = min(per, c.cols - c0);
      walk(nc, c.rows, [&](int o, int i) { return c.src[(int64_t)(c0 + o) * c.ld_src + i]; },
           [&](int o, int i, double x) { buf[i * per + o] = x; });
      __syncthreads();
      walk(c.rows, nc, [&](int r, int o) { return buf[r * per + o]; },
           [&](int r, int o, double x) { put(r, c0 + o, x); });
      __syncthreads();
    }
  }
}

__global__ void tc_convert_psi_kernel(const double* __restrict__ psi, const TcPsiSector* __restrict__ sec, int nsec,
                                      int64_t total, int prec, void* hi, void* lo, int64_t pitch) {
  const int lane = threadIdx.x & 31;
  for (int64_t e0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; e0 < total;
       e0 += (int64_t)gridDim.x * blockDim.x) {
    int si = warp_find(nsec, e0, [&](int i) { return sec[i].src_off; });
    const int64_t e = e0 + lane;
    if (e >= total) break;
    while (si + 1 < nsec && sec[si + 1].src_off <= e) ++si;
    const TcPsiSector S = sec[si];
    const int64_t el = e - S.src_off;
    // (a sector of 2^32 elements and more would need the long division)
    const int r = el >> 32 ? (int)(el / S.cols) : (int)((uint32_t)el / (uint32_t)S.cols);
    const int c = (int)(el - (int64_t)r * S.cols);
    int cp = S.cpad[0], cb = S.cbreak[0], rp = S.rpad[0], rb = S.rbreak[0];
#pragma unroll
    for (int u = 1; u < 4; ++u) {
      if (c >= S.cbreak[u]) {
        cp = S.cpad[u];
        cb = S.cbreak[u];
      }
      if (r >= S.rbreak[u]) {
        rp = S.rpad[u];
        rb = S.rbreak[u];
      }
    }
    store_conv(psi[e], prec, hi, lo, ((int64_t)S.r0 + rp + (r - rb)) * pitch + cp + (c - cb));
  }
}

}  // namespace

void launch_tc_reduce(const TcRed* tasks, int ntasks, int64_t total, const float* part, double* out,
                      cudaStream_t s) {
  if (ntasks <= 0 || total <= 0) return;
  int64_t b = (total + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  tc_reduce_kernel<<<(int)b, 256, 0, s>>>(tasks, ntasks, total, part, out);
}

bool bounded_wait_probe(int arrive, int* err_dev, int* ok_dev, cudaStream_t s) {
  bounded_wait_probe_kernel<<<1, 32, 0, s>>>(arrive, err_dev, ok_dev);
  return cudaGetLastError() == cudaSuccess;
}

int tc_stages(int prec, int ncap) {
  const int stage_bytes = (kStageA + ncap * 128) * (prec == kTF32x3 || prec == kBF16x3 ? 2 : 1);
  int s = (kSmemBudget - 1024 - 256) / stage_bytes;
  return s < kMaxStages ? s : kMaxStages;
}

int tc_smem_bytes(int prec, int ncap) {
  const int stages = tc_stages(prec, ncap);
  const int stage_bytes = (kStageA + ncap * 128) * (prec == kTF32x3 || prec == kBF16x3 ? 2 : 1);
  return 1024 + stages * stage_bytes + (2 * stages + 4) * 8 + 16;
}

bool launch_tc_gemm(const TcMaps& maps, const TcLaunch& L, int num_sms, cudaStream_t s) {
  if (L.ncap != 64 && L.ncap != 128 && L.ncap != 256) return false;
  if (L.stages != tc_stages(L.prec, L.ncap)) return false;
  if (L.ntiles <= 0) return true;
  const int smem = tc_smem_bytes(L.prec, L.ncap);
  using Kernel = void (*)(const TcMaps, const TcLaunch);
  static const Kernel kernels[4] = {tc_gemm_kernel<true, false>, tc_gemm_kernel<false, false>,
                                    tc_gemm_kernel<false, true>, tc_gemm_kernel<true, true>};   // by TcPrec
  if (L.prec < 0 || L.prec > 3) return false;
  if (!allow_shared_memory(kernels[L.prec], kSmemBudget)) return false;
  const int grid = L.ntiles < num_sms ? L.ntiles : num_sms;
  kernels[L.prec]<<<grid, kThreads, smem, s>>>(maps, L);
  return true;
}

void launch_tc_convert(const TcConv* tasks, int ntasks, int prec, void* hi, void* lo, int64_t pitch,
                       cudaStream_t s) {
  if (ntasks <= 0) return;
  tc_convert_kernel<<<ntasks < 152 * 16 ? ntasks : 152 * 16, 256, 0, s>>>(tasks, ntasks, prec, hi, lo, pitch);
}

void launch_tc_convert_psi(const double* psi, const TcPsiSector* sec, int nsec, int64_t total, int prec, void* hi,
                           void* lo, int64_t pitch, cudaStream_t s) {
  if (total <= 0) return;
  int64_t b = (total + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  tc_convert_psi_kernel<<<(int)b, 256, 0, s>>>(psi, sec, nsec, total, prec, hi, lo, pitch);
}

// tensor maps: 2D, inner dimension = pitch (K), box = 128 bytes x box_rows,
// 128-byte swizzle, zero fill outside the panel
bool tc_encode_panel(CUtensorMap* m, int elem_bytes, const void* base, uint64_t pitch, uint64_t rows,
                     uint32_t box_rows) {
  using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static EncodeFn fn = nullptr;
  if (!fn) {
    cudaDriverEntryPointQueryResult q;
    void* p = nullptr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !p)
      return false;
    fn = reinterpret_cast<EncodeFn>(p);
  }
  const CUtensorMapDataType dt = elem_bytes == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
  cuuint64_t dims[2] = {pitch, rows < 1 ? 1 : rows};
  cuuint64_t strides[1] = {pitch * (cuuint64_t)elem_bytes};
  cuuint32_t box[2] = {(cuuint32_t)(128 / elem_bytes), box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(m, dt, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace gbd
