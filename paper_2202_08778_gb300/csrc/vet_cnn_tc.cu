// vet_cnn_tc.cu -- the learned closure's 3x3x3 convolutions on the 5th
// generation tensor cores (tcgen05, accumulators in tensor memory).
//
// Implicit GEMM over columns of 8 x 16 cells (x, y) marched along z.  Each
// input slice of a column (with its halo, 10 x 18 cells) is staged once and
// serves the three output slices it touches in one go: their accumulators are
// neighbouring column blocks of tensor memory and the weights of the three dz
// taps are stacked along N, so that one tcgen05.mma.kind::f16 (BF16 x BF16 ->
// FP32) per (dy, dx) tap and 16-channel step has M = 128 cells, N = 3 C_out,
// K = 16.  Why: an M = 128, K = 16 MMA reads 4 KB of A from shared memory
// and takes about 46 clocks whatever N up to 64, so one MMA per tap and output
// slice (N = 32) reached 0.35 of the tensor rate; stacking issues a third of
// the MMAs for the same products.  Every output still adds its taps in the
// order dz, dy, dx, channel step: results are the same bits.
// Both operands sit in shared memory in the canonical K-major layout without
// swizzle: "core matrices" of 8 rows x 16 bytes stored contiguously, addressed
// by a descriptor (start, leading byte offset LBO between core matrices along
// K, stride byte offset SBO between 8-row groups along M or N).
//   A (activations): a slice's halo as [16-byte channel chunk][halo cell][16 B],
//     so that 8 cells consecutive in x form one core matrix at every tap
//     shift: start = the tap's first halo cell, LBO = one chunk plane
//     (180 x 16 B), SBO = one halo row in y (10 x 16 B).
//   B (weights): [dy, dx][channel chunk][dz = +1, 0, -1][C_out][16 B],
//     LBO = 3 C_out x 16 B, SBO = 8 x 16 B.
// Tensor memory: a ring of 512 / C_out output slices (all 512 columns, one
// CTA per SM), each zeroed by the epilogue that read it; a window of three
// slices that wraps around the ring's end is issued as two sets of MMAs.
// 128^3, ncu: 32 -> 32 channels 261 -> 95 us, 16 -> 32 150 -> 77 us, 32 -> 16
// 248 -> 95 us; the network on one 128^3 grid 1144 -> 588 us.
#include <cstdint>

#include <cuda_bf16.h>

#include "vet_cnn.h"

namespace vet {
namespace cnn {
namespace {

constexpr int TX = 8, TY = 16;             // output tile of a slice (x, y)
constexpr int HX = 10, HY = 18;            // input halo of a slice
constexpr int HN = HX * HY;                // 180 halo cells
constexpr int kRing = 6;                   // staged input slices (even: two loader groups take turns)
constexpr uint32_t kTmemCols = 512;
constexpr long long kWaitPolls = 1LL << 24;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ float silu(float z) { return __fdividef(z, 1.0f + __expf(-z)); }
__device__ __forceinline__ float silu_grad(float z) {
  const float s = __fdividef(1.0f, 1.0f + __expf(-z));
  return s * (1.0f + z * (1.0f - s));
}

// Shared-memory matrix descriptor (tcgen05): start address, LBO and SBO in
// 16-byte units, descriptor version 1 (bits 46-47), no swizzle (bits 61-63 = 0).
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// Instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A and B BF16
// (bits 7-9 and 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at bits
// 17-22, M >> 4 at bits 24-28.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// D += A B; the descriptors as (low, high) words.
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                         uint32_t idesc) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 a, b;\n setp.ne.b32 p, 1, 0;\n mov.b64 a, {%1, %2};\n mov.b64 b, {%3, %4};\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}\n" ::"r"(d_tmem),
      "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc));
}

// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(r));
  return r != 0;
}
// A value that is the same on every lane, known as such to the compiler.
__device__ __forceinline__ uint32_t uniform(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t *bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return done != 0;
}

__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, uint32_t src_bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}

// 16 (or 8) consecutive FP32 columns of this thread's tensor-memory lane,
// which are then set to zero for the next output slice that takes them.
template <int N>
__device__ __forceinline__ void tmem_take(uint32_t taddr, float (&v)[N]);
template <>
__device__ __forceinline__ void tmem_take<16>(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(taddr),
               "r"(0u)
               : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
template <>
__device__ __forceinline__ void tmem_take<8>(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(taddr), "r"(0u) : "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// Loads (no wait) and stores of 16 columns.
__device__ __forceinline__ void tmem_load16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_store16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
               "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
               "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
               : "memory");
}
__device__ __forceinline__ void tmem_zero16(uint32_t taddr) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(taddr),
               "r"(0u)
               : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// A run of n output slices za .. za + n - 1 of one column.
struct Run {
  int v, ty, tx, za, n;
};

// A CTA's share of the work: output slices [t, end) of the launch, numbered
// column by column with z fastest, cut into runs at the column ends.  Run r of
// n slices takes n + 2 steps, one per input slice za - 1 .. za + n (those
// outside the volume are steps without a load or an MMA).
struct Cursor {
  long long t, end;
  int step;
  Run run;
  __device__ __forceinline__ void load(const Vol &V) {
    if (t >= end) return;
    const int ntx = (V.nx + TX - 1) / TX, nty = (V.ny + TY - 1) / TY;
    long long col = t / V.nz;
    run.za = (int)(t - col * V.nz);
    run.n = (int)min((long long)(V.nz - run.za), end - t);
    run.tx = (int)(col % ntx);
    col /= ntx;
    run.ty = (int)(col % nty);
    run.v = (int)(col / nty);
  }
  __device__ __forceinline__ Cursor(long long t0, long long t1, const Vol &V) : t(t0), end(t1), step(0), run{0, 0, 0, 0, 0} {
    load(V);
  }
  __device__ __forceinline__ bool live() const { return t < end; }
  __device__ __forceinline__ int z_in() const { return run.za - 1 + step; }
  // true when the next step starts another run
  __device__ __forceinline__ bool advance(const Vol &V) {
    if (++step < run.n + 2) return false;
    t += run.n;
    step = 0;
    load(V);
    return true;
  }
};

template <int C_IN>
__host__ __device__ constexpr size_t slice_bytes() {
  return (size_t)C_IN / 8 * HN * 16;
}

// warp 0 issues the MMAs, warp 1 prepares them
constexpr int kFirstLoader = 64;
constexpr int kLoaders = 128;             // warps 2-5, 6-9: halo loads of the even and odd steps
constexpr int kFirstEpi = kFirstLoader + 2 * kLoaders;
constexpr int kEpiGroup = 256;            // warps 10-17, 18-25: epilogue of the even and odd output slices
constexpr int kTcThreads = kFirstEpi + 2 * kEpiGroup;

// Halo loads of one thread (cp.async, zero outside the volume): its up to
// six 16-byte pieces sit at the same place in every slice of a column, so
// the offsets are computed once per run.
template <int C_IN>
struct HaloLoader {
  static constexpr int NCI = C_IN / 8, K = (HN * NCI + kLoaders - 1) / kLoaders;
  long long off[K];  // elements from the slice's first cell; negative: outside
  const __nv_bfloat16 *base;
  long long plane;
  __device__ __forceinline__ void set(const __nv_bfloat16 *__restrict__ x, const Vol &V, const Run &r) {
    plane = (long long)V.ny * V.nx * C_IN;
    base = x + (long long)r.v * V.nz * plane;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int h = ((int)threadIdx.x - kFirstLoader) % kLoaders + k * kLoaders, hc = h / NCI, c = h - hc * NCI;
      const int y = r.ty * TY + hc / HX - 1, xx = r.tx * TX + hc % HX - 1;
      off[k] = y >= 0 && y < V.ny && xx >= 0 && xx < V.nx ? ((long long)y * V.nx + xx) * C_IN + c * 8 : -1;
    }
  }
  __device__ __forceinline__ void load(uint32_t dst, const __nv_bfloat16 *__restrict__ x, int z) const {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int h = ((int)threadIdx.x - kFirstLoader) % kLoaders + k * kLoaders, hc = h / NCI, c = h - hc * NCI;
      if (h < HN * NCI)
        cp_async16(dst + (uint32_t)((c * HN + hc) * 16), off[k] >= 0 ? base + z * plane + off[k] : x, off[k] >= 0 ? 16u : 0u);
    }
  }
};

// What the issuing warp does next: the MMAs of one input slice into a window
// of neighbouring output slices (idesc 0: none), then the commits.
struct alignas(16) MmaCommand {
  uint32_t d, a, b, idesc;     // accumulator; low words of the descriptors; 0xffffffff: the end
  uint32_t done, ready;              // shared addresses of the barriers to commit to (0: none)
  uint32_t flags, pad;               // weight gradient: kFlush..
};

// Named-barrier hand-over between the preparing and the issuing warp.
__device__ __forceinline__ void pair_sync(int id) { asm volatile("barrier.cta.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void pair_arrive(int id) { asm volatile("barrier.cta.arrive %0, 64;" ::"r"(id) : "memory"); }
constexpr int kBarLoad = 1, kBarEpi = 3, kBarReady = 5, kBarFree = 7;  // named barriers, two of each

// The 9 x (C_IN / 16) MMAs of a command, issued by one lane of a converged
// warp.  Descriptor start addresses are 16-byte units in their low 14 bits,
// so moving an operand by b bytes adds b / 16 to the descriptor's low word (no
// carry: shared memory < 256 KB).  The instruction takes its operands from
// uniform registers: the bases are made uniform once and every tap is a
// constant away (a base kept in ordinary registers is moved over for each
// MMA: 94 clocks between MMAs, not 56).  `midway` runs between two halves of
// the MMAs, while the tensor pipe has work queued.
template <int C_IN, int C_OUT, typename F>
__device__ __forceinline__ void issue_slice(const MmaCommand &c, uint32_t a_hi, uint32_t b_hi, F midway) {
  constexpr int NCI = C_IN / 8;
  const uint32_t idesc = uniform(c.idesc), d = uniform(c.d), al = uniform(c.a), bl = uniform(c.b);
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    if (idesc && elect_one()) {
#pragma unroll
      for (int tap = half ? 5 : 0; tap < (half ? 9 : 5); ++tap) {
#pragma unroll
        for (int ks = 0; ks < NCI / 2; ++ks)
          mma_bf16(d, al + (uint32_t)(2 * ks * HN + (tap / 3) * HX + tap % 3), a_hi,
                   bl + (uint32_t)((tap * NCI + 2 * ks) * 3 * C_OUT), b_hi, idesc);
      }
    }
    __syncwarp();
    if (half == 0) midway();
  }
}

// One thread's part of the output slices of a run: cell r of the 128,
// channels [c0, c0 + C_OUT / 2).
template <int C_OUT, int EPI>
struct Epilogue {
  static constexpr int NC = C_OUT / 2;
  static_assert(EPI != EPI_F32 || kOutRow % NC == 0, "whole halves are stored");
  long long at, plane;  // element of this thread's first channel in the run's slice 0, and per slice
  bool in;
  float bias[EPI == EPI_SILU_BWD ? 1 : NC];
  int4 p[EPI == EPI_SILU_BWD ? NC / 8 : 1];
  __device__ __forceinline__ void set(const Vol &V, const Run &run, int r, int c0) {
    const int xx = run.tx * TX + (r & 7), y = run.ty * TY + (r >> 3);
    constexpr int kRow = EPI == EPI_F32 ? kOutRow : C_OUT;  // stored channels
    in = xx < V.nx && y < V.ny && c0 < kRow;
    plane = (long long)V.ny * V.nx * kRow;
    at = ((((long long)run.v * V.nz + run.za) * V.ny + y) * V.nx + xx) * kRow + c0;
  }
  // the pre-activations the backward epilogue needs, ahead of the wait
  __device__ __forceinline__ void prefetch(const __nv_bfloat16 *__restrict__ pre_in, int j) {
    if constexpr (EPI == EPI_SILU_BWD) {
      if (!in) return;
#pragma unroll
      for (int i = 0; i < NC / 8; ++i) p[i] = reinterpret_cast<const int4 *>(pre_in + at + j * plane)[i];
    }
  }
  __device__ __forceinline__ void store(const float (&acc)[NC], __nv_bfloat16 *__restrict__ pre_out,
                                        void *__restrict__ out, int j) {
    if (!in) return;
    const long long e = at + j * plane;
    if constexpr (EPI == EPI_F32) {
      float4 *dst = reinterpret_cast<float4 *>(reinterpret_cast<float *>(out) + e);
#pragma unroll
      for (int i = 0; i < NC / 4; ++i)
        dst[i] = make_float4(acc[4 * i] + bias[4 * i], acc[4 * i + 1] + bias[4 * i + 1], acc[4 * i + 2] + bias[4 * i + 2],
                             acc[4 * i + 3] + bias[4 * i + 3]);
    } else {
      __align__(16) __nv_bfloat162 o2[NC / 2];
      if constexpr (EPI == EPI_SILU) {
        __align__(16) __nv_bfloat162 p2[NC / 2];
#pragma unroll
        for (int i = 0; i < NC / 2; ++i) {
          const float z0 = acc[2 * i] + bias[2 * i], z1 = acc[2 * i + 1] + bias[2 * i + 1];
          p2[i] = __floats2bfloat162_rn(z0, z1);
          o2[i] = __floats2bfloat162_rn(silu(z0), silu(z1));
        }
        if (pre_out) {
          int4 *pd = reinterpret_cast<int4 *>(pre_out + e);
#pragma unroll
          for (int i = 0; i < NC / 8; ++i) pd[i] = reinterpret_cast<const int4 *>(p2)[i];
        }
      } else {  // EPI_SILU_BWD
        const __nv_bfloat162 *p2 = reinterpret_cast<const __nv_bfloat162 *>(p);
#pragma unroll
        for (int i = 0; i < NC / 2; ++i)
          o2[i] = __floats2bfloat162_rn(acc[2 * i] * silu_grad(__bfloat162float(p2[i].x)),
                                        acc[2 * i + 1] * silu_grad(__bfloat162float(p2[i].y)));
      }
      int4 *od = reinterpret_cast<int4 *>(reinterpret_cast<__nv_bfloat16 *>(out) + e);
#pragma unroll
      for (int i = 0; i < NC / 8; ++i) od[i] = reinterpret_cast<const int4 *>(o2)[i];
    }
  }
};

// Bounded wait of one thread on an mbarrier phase, giving up early when
// another role has aborted (*abort set).
__device__ __forceinline__ bool wait_or_abort(uint64_t *bar, uint32_t parity, volatile int *abort) {
  for (long long i = 0; i < kWaitPolls; ++i) {
    if (mbar_try(bar, parity)) return true;
    if ((i & 1023) == 1023 && *abort != 0) return false;
  }
  return false;
}

// Named barrier over nthreads threads (whole warps) that also tells each
// whether ok held for all of them: no shared-memory access.
__device__ __forceinline__ bool group_all(int id, int nthreads, bool ok) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.and.pred q, %2, %3, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)ok), "r"(id), "r"(nthreads)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Warp-specialised pipeline over the steps of this CTA's share (all roles walk
// the same steps; step g uses ring buffer g % kRing, output o of the share,
// counted over its runs, tensor-memory block o % (512 / C_OUT)).
//   Loader groups, step g (even and odd ones): wait done[g - kRing] (the
//     buffer is free); start the slice's loads; the loads of the group's step
//     before have landed by then: fence them to the async proxy and arrive on
//     full.
//   MMA preparation, step g: wait full[g % kRing] and empty[block] of the
//     output that joins, work out the window, hand a command to
//   MMA issuer: issue the slice's MMAs; commit them to done[g % kRing] and to
//     ready[block] of the output slice they complete.  Two warps, since the
//     waits and the bookkeeping of a step (about 700 clocks on one warp) are
//     more than the MMAs queued meanwhile (six, 340 clocks) hide.
//   Epilogue groups, output o (even and odd ones): wait ready[block]; read,
//     zero and store it (warp w: tensor-memory lanes 32 (w % 4) ..,
//     channels of half w / 4); arrive on empty[block].
// The MMAs read their operands at the full 128 bytes per clock of shared
// memory (56 clocks for N = 96: 4 KB of A, 3 KB of B), so every other access
// to it takes their time: one thread of a role polls a barrier and hands the
// verdict to the others by a named barrier, and a warp arrives once.
// What bounds a step (95 us: about 1640 clocks, of which the MMAs take 1225 with
// their commits and windows cut in two): the hand-overs between the roles.
// Every wait is bounded; a role that gives up sets `abort`, which ends the
// other roles' waits too.
template <int C_IN, int C_OUT, int EPI>
__global__ void __launch_bounds__(kTcThreads, 1)
    conv3d_tc_kernel(const __nv_bfloat16 *__restrict__ x, const __nv_bfloat16 *__restrict__ W,
                     const float *__restrict__ b, Vol V, __nv_bfloat16 *__restrict__ pre_out,
                     const __nv_bfloat16 *__restrict__ pre_in, void *__restrict__ out, int *status) {
  constexpr int NCI = C_IN / 8, NC = C_OUT / 2;
  constexpr int kSlots = (int)kTmemCols / C_OUT;
  constexpr uint32_t A_LBO = HN * 16, A_SBO = HX * 16;
  constexpr uint32_t B_LBO = 3 * C_OUT * 16, B_SBO = 8 * 16;
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char *sA = smem;                                   // kRing x [NCI][HN][16 B]
  unsigned char *sB = smem + kRing * slice_bytes<C_IN>();     // [9][NCI][3][C_OUT][16 B]
  __shared__ __align__(8) uint64_t full[kRing], done[kRing], ready[kSlots], empty[kSlots];
  __shared__ MmaCommand commands[2];
  __shared__ uint32_t tmem_base_slot;
  __shared__ volatile int abort_flag;
  __shared__ int n_committed, n_next[2];  // steps whose MMAs were committed; first even and odd step the loaders did not see complete

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  after_previous();
  let_next_launch();
  for (int h = threadIdx.x; h < 27 * C_OUT * NCI; h += blockDim.x) {
    const int c = h % NCI, co = (h / NCI) % C_OUT, tap = h / (NCI * C_OUT);
    const int4 val = reinterpret_cast<const int4 *>(W + ((size_t)tap * C_OUT + co) * C_IN)[c];
    const int yx = tap % 9, k = 2 - tap / 9;
    *reinterpret_cast<int4 *>(sB + ((((size_t)yx * NCI + c) * 3 + k) * C_OUT + co) * 16) = val;
  }
  if (threadIdx.x == 0) {
    for (int k = 0; k < kRing; ++k) {
      mbar_init(&full[k], kLoaders / 32);
      mbar_init(&done[k], 1);
    }
    for (int k = 0; k < kSlots; ++k) {
      mbar_init(&ready[k], 1);
      mbar_init(&empty[k], kEpiGroup / 32);
    }
    abort_flag = 0;
    n_committed = n_next[0] = 0;
    n_next[1] = 1;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_proxy_async();
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = tmem_base_slot;
  const long long nt = (long long)V.n * ((V.ny + TY - 1) / TY) * ((V.nx + TX - 1) / TX) * V.nz;
  const long long t0 = nt * blockIdx.x / gridDim.x, t1 = nt * (blockIdx.x + 1) / gridDim.x;
  const uint32_t a_base = smem_u32(sA), b_base = smem_u32(sB);
  auto wait = [&](uint64_t *bar, uint32_t parity) {  // one thread
    if (wait_or_abort(bar, parity, &abort_flag)) return true;
    atomicOr(status, 16);
    abort_flag = 1;
    return false;
  };
  auto wait_warp = [&](uint64_t *bar, uint32_t parity) {  // every lane of a warp, one verdict
    return __all_sync(0xffffffffu, wait(bar, parity));
  };
  // the accumulators start at zero: each epilogue warp its lanes' quarter of the columns
  if (warp >= kFirstEpi / 32) {
    const int w = warp - kFirstEpi / 32;
    const uint32_t t = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((w >> 2) * ((int)kTmemCols / 4));
    for (int k = 0; k < (int)kTmemCols / 4; k += 16)
      asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(
                       t + (uint32_t)k),
                   "r"(0u)
                   : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();

  if (warp == 0) {
    // ---- MMA issuer: the next command is fetched halfway through the current one
    const uint32_t a_hi = uniform((uint32_t)(smem_desc(a_base, A_LBO, A_SBO) >> 32));
    const uint32_t b_hi = uniform((uint32_t)(smem_desc(b_base, B_LBO, B_SBO) >> 32));
    MmaCommand cur, nxt;
    int k = 0;
    auto fetch = [&]() {
      pair_sync(kBarReady + (k & 1));
      nxt = commands[k & 1];
      pair_arrive(kBarFree + (k & 1));
      ++k;
    };
    fetch();
    while (nxt.d != 0xffffffffu) {
      cur = nxt;
      fence_after_sync();
      issue_slice<C_IN, C_OUT>(cur, a_hi, b_hi, fetch);
      if (elect_one()) {
        if (cur.done) mma_commit(cur.done);
        if (cur.ready) mma_commit(cur.ready);
      }
      __syncwarp();
    }
  } else if (warp == 1) {
    // ---- MMA preparation: waits for a step's slice and accumulator, works out its window
    const uint32_t a_lo = (uint32_t)smem_desc(a_base, A_LBO, A_SBO), b_lo = (uint32_t)smem_desc(b_base, B_LBO, B_SBO);
    int o_run = 0;         // the run's first output, counted over the share
    int s = 0, lap = 0;    // step g = lap kRing + s
    int freed = kSlots;    // outputs below this index have a block to take
    int k = 0;             // commands sent
    auto send = [&](uint32_t d, uint32_t a, uint32_t b2, uint32_t idesc, uint32_t dn, uint32_t rd) {
      if (k >= 2) pair_sync(kBarFree + (k & 1));
      if (lane == 0) commands[k & 1] = MmaCommand{d, a, b2, idesc, dn, rd, 0, 0};
      __syncwarp();
      fence_before_sync();
      pair_arrive(kBarReady + (k & 1));
      ++k;
    };
    for (Cursor cu(t0, t1, V); cu.live();) {
      bool ok = wait_warp(&full[s], (uint32_t)lap & 1u);
      if (ok && cu.step < cu.run.n && o_run + cu.step >= freed) {
        // the next four blocks at once: each group reads its outputs in order,
        // so the last one of either parity vouches for the other
        const uint32_t ph = (uint32_t)(freed / kSlots - 1) & 1u;
        ok = wait_warp(&empty[(freed + 2) % kSlots], ph) && wait_warp(&empty[(freed + 3) % kSlots], ph);
        freed += 4;
      }
      if (!ok) break;
      fence_after_sync();
      const int z = cu.z_in();
      const uint32_t dn = smem_u32(&done[s]), rd = cu.step >= 2 ? smem_u32(&ready[(o_run + cu.step - 2) % kSlots]) : 0u;
      if (z >= 0 && z < V.nz) {
        // outputs z - 1 .. z + 1 that lie in the run; a window around the ring's end in two parts
        const int lo = max(cu.step - 2, 0), hi = min(cu.step, cu.run.n - 1);
        const int cnt = hi - lo + 1, slot = (o_run + lo) % kSlots, head = min(cnt, kSlots - slot);
        const uint32_t ad = a_lo + (uint32_t)(s * (int)(slice_bytes<C_IN>() / 16));
        const uint32_t bd = b_lo + (uint32_t)((lo - (cu.step - 2)) * C_OUT);
        constexpr uint32_t kBlock = (uint32_t)(C_OUT >> 3) << 17;  // of the descriptor's N
        const uint32_t id1 = idesc_bf16(128, C_OUT) - kBlock;
        if (head < cnt) send(tmem + (uint32_t)(slot * C_OUT), ad, bd, id1 + (uint32_t)head * kBlock, 0u, 0u);
        const int from = head < cnt ? head : 0;
        send(tmem + (uint32_t)((slot + from) % kSlots * C_OUT), ad, bd + (uint32_t)(from * C_OUT),
             id1 + (uint32_t)(cnt - from) * kBlock, dn, rd);
      } else {
        send(tmem, 0u, 0u, 0u, dn, rd);
      }
      if (++s == kRing) {
        s = 0;
        ++lap;
      }
      if (lane == 0) n_committed = lap * kRing + s;
      const int n = cu.run.n;
      if (cu.advance(V)) o_run += n;
    }
    send(0xffffffffu, 0u, 0u, 0u, 0u, 0u);
  } else if (warp < kFirstEpi / 32) {
    // ---- loaders
    const int grp = ((int)threadIdx.x - kFirstLoader) / kLoaders;
    const bool poller = ((int)threadIdx.x - kFirstLoader) % kLoaders == 0;
    HaloLoader<C_IN> hl;
    Cursor ld(t0, t1, V);
    if (ld.live()) hl.set(x, V, ld.run);
    auto next = [&]() {
      if (ld.advance(V) && ld.live()) hl.set(x, V, ld.run);
    };
    auto landed = [&](int g) {  // this warp's part of step g's slice
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[g % kRing]);
    };
    if (grp && ld.live()) next();
    int g = grp;
    for (; ld.live(); g += 2) {
      if (g >= kRing) {
        if (!group_all(kBarLoad + grp, kLoaders, !poller || wait(&done[g % kRing], (uint32_t)(g / kRing - 1) & 1u))) break;
        if (poller) n_next[grp] = g - kRing + 2;
      }
      const int z = ld.z_in();
      if (z >= 0 && z < V.nz) hl.load(a_base + (uint32_t)((g % kRing) * slice_bytes<C_IN>()), x, z);
      asm volatile("cp.async.commit_group;" ::: "memory");
      if (g >= 2) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        landed(g - 2);
      }
      next();
      if (ld.live()) next();
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (g >= 2) landed(g - 2);
  } else {
    // ---- epilogue
    const int w = warp - kFirstEpi / 32, grp = w / (kEpiGroup / 32);
    const int sp = warp & 3, c0 = ((w >> 2) & 1) * NC;  // tensor-memory lane quarter, first channel
    const int r = 32 * sp + lane;                    // this thread's cell of the slice
    const uint32_t t_lane = tmem + ((uint32_t)(32 * sp) << 16) + (uint32_t)c0;
    // the group's polling thread: a warp on another sub-partition than the MMAs'
    const bool poller = w % (kEpiGroup / 32) == 1 && lane == 0;
    Epilogue<C_OUT, EPI> ep;
    if constexpr (EPI != EPI_SILU_BWD) {
#pragma unroll
      for (int i = 0; i < NC; ++i) ep.bias[i] = b[c0 + i];
    }
    int o = 0;
    bool ok = true;
    for (Cursor cu(t0, t1, V); ok && cu.live();) {
      ep.set(V, cu.run, r, c0);
      const int n = cu.run.n;
      for (int j = (o + grp) & 1; j < n; j += 2) {
        const int slot = (o + j) % kSlots;
        ep.prefetch(pre_in, j);
        ok = group_all(kBarEpi + grp, kEpiGroup, !poller || wait(&ready[slot], (uint32_t)((o + j) / kSlots) & 1u));
        if (!ok) break;
        fence_after_sync();
        float acc[NC];
        tmem_take<NC>(t_lane + (uint32_t)(slot * C_OUT), acc);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[slot]);
        ep.store(acc, pre_out, out, j);
        __syncwarp();
      }
      o += n;
      cu.step = n + 1;  // to the next run
      cu.advance(V);
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();
  fence_before_sync();
  __syncthreads();
  if (abort_flag && threadIdx.x == 0) {
    // committed MMAs may still run: wait (bounded) for every step committed
    // but not yet seen complete before tensor and shared memory are released
    for (int q = 0; q < 2; ++q)
      for (int g = n_next[q]; g < n_committed; g += 2)
        for (long long n = 0; n < kWaitPolls && !mbar_try(&done[g % kRing], (uint32_t)(g / kRing) & 1u); ++n) {
        }
  }
  __syncthreads();
  if (warp == 0) {
    fence_after_sync();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// ---------------------------------------------------------- weight gradient
// gW[dz, dy, dx][co][ci] += sum_cells g[cell][co] x[cell + (dx, dy, dz)][ci],
// gb[co] += sum_cells g[cell][co]: a contraction over cells.  Same march along
// the columns; per slice of g (8 x 16 cells) and dy one tcgen05.mma per 16
// cells, with
//   M = (dx, co), 3 C_out of 128 rows: the cells c of the column's tile read
//     g[c - dx], from three copies of the g slice shifted in x (a tap's shift
//     in y is an offset of whole rows in the copies),
//   N = (dz, ci), 3 C_in: three neighbouring slices of x in their ring,
//   K = 16 cells, two rows of the tile,
// both operands MN-major (8 channels of a cell are the 16 contiguous bytes, the
// cells of a row follow each other): core matrices of 8 cells x 16 bytes, SBO
// between 8-channel chunks, LBO between rows of 8 cells.  The tensor core's
// FP32 accumulation truncates, so chains are kept to kFlushSlices slices (16
// MMAs): the accumulators of a dy (3 C_in columns) are then added, rounded, to
// sums that live in the rest of tensor memory and, for what does not fit there,
// in registers, while the MMAs of the other two dy run (chains over a CTA's
// whole share were off by 1.4e-5 on 4 x 64^3).  The sums are added to gW
// at the share's end by 16-byte reductions.
// What the MMAs need: their operands' 24 x 56 clocks a slice (C_in = 32), 40 us on
// 4 x 64^3; measured there, ncu: 32 -> 32 channels 327 -> 110 us, 32 -> 16 260 -> 88 us,
// 16 -> 32 210 -> 84 us (before: a tap at a time by mma.sync into
// shared-memory accumulators, the tensor pipe 28% busy).  What is left over: the
// hand-overs of a step and the sums (20 us).
constexpr int kWgRing = 4;   // staged g slices (even: two loader groups take turns)
constexpr int kWgX = 8;      // staged x slices: a step's slice is read by it and the next two
static_assert(kWgRing + 2 <= kWgX, "the wait for a g buffer must cover the x buffer");
constexpr int kWgSum = 128;  // warps 10-13: sums of the accumulators
constexpr int kWgBias = 64;  // warps 14, 15: bias sums
constexpr int kWgThreads = kFirstLoader + 2 * kLoaders + kWgSum + kWgBias;
constexpr int kFlushSlices = 2;
constexpr uint32_t kFlush = 1, kAfterFlush = 2, kFlushOdd = 4;  // command flags: a chain ends / starts here; parity
constexpr int kGRows = TY + 2;                      // rows of a g copy: y - 1 .. y + 16
constexpr int kGPlane = kGRows * TX * 16, kXPlane = TY * TX * 16;  // bytes of one channel chunk

template <int C_IN, int C_OUT>
__host__ __device__ constexpr size_t wg_g_bytes() {
  return (size_t)3 * (C_OUT / 8) * kGPlane;
}
template <int C_IN, int C_OUT>
__host__ __device__ constexpr size_t wg_x_bytes() {
  return (size_t)(C_IN / 8) * kXPlane;
}
// The M = 128 MMAs read 16 chunks from the last g buffer on: its own 3 C_out / 8
// and what follows (the x ring), whose rows of the result nobody reads.
template <int C_IN, int C_OUT>
__host__ __device__ constexpr size_t wg_smem() {
  return kWgRing * wg_g_bytes<C_IN, C_OUT>() + kWgX * wg_x_bytes<C_IN, C_OUT>();
}

// Loads of one thread, in 16-byte pieces from a slice's first cell (negative:
// outside the volume, zero).
template <int C_IN, int C_OUT>
struct WgradLoader {
  static constexpr int NCI = C_IN / 8, NCO = C_OUT / 8;
  static constexpr int NG = 3 * NCO * kGRows * TX, NX = NCI * TY * TX;
  static constexpr int KG = (NG + kLoaders - 1) / kLoaders, KX = NX / kLoaders;
  static_assert(NX % kLoaders == 0, "x pieces divide evenly");
  int og[KG], ox[KX];
  const __nv_bfloat16 *gb, *xb;
  long long plane;  // cells of a slice
  __device__ __forceinline__ void set(const __nv_bfloat16 *__restrict__ x, const __nv_bfloat16 *__restrict__ g, const Vol &V,
                                      const Run &r, int tid) {
    plane = (long long)V.ny * V.nx;
    gb = g + (long long)r.v * V.nz * plane * C_OUT;
    xb = x + (long long)r.v * V.nz * plane * C_IN;
#pragma unroll
    for (int k = 0; k < KG; ++k) {
      // a warp's lanes take whole cells: [dx][row][x][chunk]
      const int h = tid + k * kLoaders, c = h % NCO, xc = (h / NCO) % TX, row = (h / (NCO * TX)) % kGRows;
      const int xx = r.tx * TX + xc - (h / (NCO * TX * kGRows) - 1), y = r.ty * TY + row - 1;
      og[k] = xx >= 0 && xx < V.nx && y >= 0 && y < V.ny ? (y * V.nx + xx) * NCO + c : -1;
    }
#pragma unroll
    for (int k = 0; k < KX; ++k) {
      const int h = tid + k * kLoaders, c = h % NCI, xc = (h / NCI) % TX, row = h / (NCI * TX);
      const int xx = r.tx * TX + xc, y = r.ty * TY + row;
      ox[k] = xx < V.nx && y < V.ny ? (y * V.nx + xx) * NCI + c : -1;
    }
  }
  __device__ __forceinline__ void load_g(uint32_t dst, int z, int tid) const {
    const __nv_bfloat16 *src = gb + z * plane * C_OUT;
#pragma unroll
    for (int k = 0; k < KG; ++k) {
      const int h = tid + k * kLoaders;
      if (NG % kLoaders == 0 || h < NG)
        cp_async16(dst + (uint32_t)((h / (NCO * TX * kGRows) * NCO + h % NCO) * kGPlane + (h / NCO) % (TX * kGRows) * 16), og[k] >= 0 ? src + (long long)og[k] * 8 : gb, og[k] >= 0 ? 16u : 0u);
    }
  }
  __device__ __forceinline__ void load_x(uint32_t dst, int z, int tid) const {
    const __nv_bfloat16 *src = xb + z * plane * C_IN;
#pragma unroll
    for (int k = 0; k < KX; ++k)
      cp_async16(dst + (uint32_t)((tid + k * kLoaders) % NCI * kXPlane + (tid + k * kLoaders) / NCI * 16), ox[k] >= 0 ? src + (long long)ox[k] * 8 : xb,
                 ox[k] >= 0 ? 16u : 0u);
  }
};

// dst[0..3] += v by one reduction.
__device__ __forceinline__ void red_add4(float *dst, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// Roles as in conv3d_tc_kernel; step g of a run loads x slice za - 1 + step and,
// from step 2 on, g slice za + step - 2, whose MMAs it issues.
template <int C_IN, int C_OUT>
__global__ void __launch_bounds__(kWgThreads, 1)
    wgrad_tc_kernel(const __nv_bfloat16 *__restrict__ x, const __nv_bfloat16 *__restrict__ gpre, Vol V,
                    float *__restrict__ gW, float *__restrict__ gb, int *status) {
  constexpr int NCO = C_OUT / 8;
  // accumulators in columns [0, kAcc); the sums of the first kTm of them in
  // [kAcc, kAcc + kTm), of the others in registers
  constexpr int kAcc = 9 * C_IN, kDy = 3 * C_IN, kTm = kAcc < (int)kTmemCols - kAcc ? kAcc : (int)kTmemCols - kAcc;
  static_assert(kTm % 16 == 0 && kDy % 16 == 0, "whole pieces of 16 columns");
  constexpr size_t kG = wg_g_bytes<C_IN, C_OUT>(), kX = wg_x_bytes<C_IN, C_OUT>();
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[kWgRing], done[kWgRing], ready[3], zeroed[3];
  __shared__ MmaCommand commands[2];
  __shared__ uint32_t tmem_base_slot;
  __shared__ volatile int abort_flag;
  __shared__ int n_committed, n_next[2];
  __shared__ float sBias[C_OUT];

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  after_previous();
  if (threadIdx.x < C_OUT) sBias[threadIdx.x] = 0.f;
  if (threadIdx.x == 0) {
    for (int k = 0; k < kWgRing; ++k) {
      mbar_init(&full[k], kLoaders / 32);
      mbar_init(&done[k], 1);
    }
    for (int k = 0; k < 3; ++k) {
      mbar_init(&ready[k], 1);
      mbar_init(&zeroed[k], kWgSum / 32);
    }
    abort_flag = 0;
    n_committed = n_next[0] = 0;
    n_next[1] = 1;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_proxy_async();
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = tmem_base_slot;
  const long long nt = (long long)V.n * ((V.ny + TY - 1) / TY) * ((V.nx + TX - 1) / TX) * V.nz;
  const long long t0 = nt * blockIdx.x / gridDim.x, t1 = nt * (blockIdx.x + 1) / gridDim.x;
  const uint32_t g_base = smem_u32(smem), x_base = g_base + (uint32_t)(kWgRing * kG);
  auto wait = [&](uint64_t *bar, uint32_t parity) {  // one thread
    if (wait_or_abort(bar, parity, &abort_flag)) return true;
    atomicOr(status, 16);
    abort_flag = 1;
    return false;
  };
  constexpr int kFirstSum = (kFirstLoader + 2 * kLoaders) / 32;
  constexpr int kFirstBias = kFirstSum + kWgSum / 32;
  if (warp >= kFirstSum && warp < kFirstBias) {  // the accumulators and their sums start at zero
    for (int k = 0; k < (int)kTmemCols; k += 16) tmem_zero16(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)k);
    tmem_wait_st();
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();

  if (warp == 0) {
    // ---- MMA issuer
    const uint32_t a_hi = uniform((uint32_t)(smem_desc(g_base, 128, kGPlane) >> 32));
    const uint32_t b_hi = uniform((uint32_t)(smem_desc(x_base, 128, kXPlane) >> 32));
    MmaCommand cur, nxt;
    int k = 0;
    auto fetch = [&]() {
      pair_sync(kBarReady + (k & 1));
      nxt = commands[k & 1];
      pair_arrive(kBarFree + (k & 1));
      ++k;
    };
    fetch();
    bool ok = true;  // once a wait gave up, commands are taken and not carried out
    while (nxt.d != 0xffffffffu) {
      cur = nxt;
      fence_after_sync();
      const uint32_t idesc = uniform(cur.idesc), d = uniform(cur.d), al = uniform(cur.a), bl = uniform(cur.b),
                     flags = uniform(cur.flags);
#pragma unroll
      for (int dy = 0; dy < 3; ++dy) {
        if (flags & kAfterFlush) {
          ok = ok && __all_sync(0xffffffffu, wait(&zeroed[dy], flags & kFlushOdd ? 1u : 0u));
          fence_after_sync();
        }
        if (idesc && ok && elect_one()) {
#pragma unroll
          for (int ks = 0; ks < TY / 2; ++ks)
            mma_bf16(d + (uint32_t)(dy * kDy), al + (uint32_t)((2 * ks + 2 - dy) * TX), a_hi, bl + (uint32_t)(2 * ks * TX), b_hi,
                     idesc);
          if (flags & kFlush) mma_commit(smem_u32(&ready[dy]));
        }
        __syncwarp();
        if (dy == 1) fetch();
      }
      if (cur.done && ok && elect_one()) mma_commit(cur.done);
      __syncwarp();
    }
  } else if (warp == 1) {
    // ---- MMA preparation
    const uint32_t a_lo = (uint32_t)smem_desc(g_base, 128, kGPlane), b_lo = (uint32_t)smem_desc(x_base, 128, kXPlane);
    int g = 0, k = 0;
    auto send = [&](uint32_t d, uint32_t a, uint32_t b2, uint32_t idesc, uint32_t dn, uint32_t flags) {
      if (k >= 2) pair_sync(kBarFree + (k & 1));
      if (lane == 0) commands[k & 1] = MmaCommand{d, a, b2, idesc, dn, 0u, flags, 0u};
      __syncwarp();
      fence_before_sync();
      pair_arrive(kBarReady + (k & 1));
      ++k;
    };
    int i = 0;  // g slices done
    for (Cursor cu(t0, t1, V); cu.live(); ++g) {
      const int s = g % kWgRing;
      if (!__all_sync(0xffffffffu, wait(&full[s], (uint32_t)(g / kWgRing) & 1u))) break;
      fence_after_sync();
      const int step = cu.step, zg = cu.run.za + step - 2;
      const uint32_t dn = smem_u32(&done[s]);
      if (step >= 2) {
        // x slices zg - 1 .. zg + 1 in the volume; a window around the ring's end in two parts
        const int lo = zg > 0 ? 0 : 1, hi = zg < V.nz - 1 ? 2 : 1, cnt = hi - lo + 1;
        const int first = (g - 2 + lo) % kWgX, head = min(cnt, kWgX - first);
        const uint32_t ad = a_lo + (uint32_t)(s * (int)(kG / 16));
        const uint32_t fl = i % kFlushSlices == kFlushSlices - 1 || i == (int)(t1 - t0) - 1 ? kFlush : 0u;
        uint32_t af = i && i % kFlushSlices == 0 ? kAfterFlush | ((i / kFlushSlices - 1) & 1 ? kFlushOdd : 0u) : 0u;
        // bits 15, 16: both operands MN-major
        const uint32_t id0 = idesc_bf16(128, 0) | (1u << 15) | (1u << 16);
        constexpr uint32_t kBlock = (uint32_t)(C_IN >> 3) << 17;
        if (head < cnt) {
          send(tmem + (uint32_t)(lo * C_IN), ad, b_lo + (uint32_t)(first * (int)(kX / 16)), id0 + (uint32_t)head * kBlock, 0u, af);
          af = 0u;
        }
        const int from = head < cnt ? head : 0;
        send(tmem + (uint32_t)((lo + from) * C_IN), ad, b_lo + (uint32_t)((first + from) % kWgX * (int)(kX / 16)),
             id0 + (uint32_t)(cnt - from) * kBlock, dn, fl | af);
        ++i;
      } else {
        send(tmem, 0u, 0u, 0u, dn, 0u);
      }
      if (lane == 0) n_committed = g + 1;
      cu.advance(V);
    }
    send(0xffffffffu, 0u, 0u, 0u, 0u, 0u);
  } else if (warp < kFirstSum) {
    // ---- loaders
    const int grp = ((int)threadIdx.x - kFirstLoader) / kLoaders, tid = ((int)threadIdx.x - kFirstLoader) % kLoaders;
    WgradLoader<C_IN, C_OUT> wl;
    Cursor ld(t0, t1, V);
    if (ld.live()) wl.set(x, gpre, V, ld.run, tid);
    auto next = [&]() {
      if (ld.advance(V) && ld.live()) wl.set(x, gpre, V, ld.run, tid);
    };
    auto landed = [&](int g) {
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[g % kWgRing]);
    };
    if (grp && ld.live()) next();
    int g = grp;
    for (; ld.live(); g += 2) {
      if (g >= 2) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        landed(g - 2);
      }
      if (g >= kWgRing) {
        if (!group_all(kBarLoad + grp, kLoaders, tid != 0 || wait(&done[g % kWgRing], (uint32_t)(g / kWgRing - 1) & 1u))) break;
        if (tid == 0) n_next[grp] = g - kWgRing + 2;
      }
      const int z = ld.z_in();
      if (z >= 0 && z < V.nz) wl.load_x(x_base + (uint32_t)((g % kWgX) * kX), z, tid);
      if (ld.step >= 2) wl.load_g(g_base + (uint32_t)((g % kWgRing) * kG), z - 1, tid);
      asm volatile("cp.async.commit_group;" ::: "memory");
      next();
      if (ld.live()) next();
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (g >= 2) landed(g - 2);
  } else if (warp < kFirstBias) {
    // ---- sums of the accumulators
    const int tid = (int)threadIdx.x - 32 * kFirstSum;
    const uint32_t t_lane = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
    constexpr int kRegs = kAcc > kTm ? kAcc - kTm : 1;
    float sum[kRegs];
#pragma unroll
    for (int q = 0; q < kRegs; ++q) sum[q] = 0.f;
    const int flushes = (int)((t1 - t0 + kFlushSlices - 1) / kFlushSlices);
    bool ok = true;
    for (int f = 0; f < flushes && ok; ++f) {
#pragma unroll
      for (int dy = 0; dy < 3; ++dy) {
        ok = ok && group_all(kBarEpi, kWgSum, tid != 0 || wait(&ready[dy], (uint32_t)f & 1u));
        if (!ok) break;
        fence_after_sync();
#pragma unroll
        for (int q = dy * kDy; q < (dy + 1) * kDy; q += 16) {
          uint32_t v[16], u[16];
          tmem_load16(t_lane + (uint32_t)q, v);
          if (q < kTm) {
            tmem_load16(t_lane + (uint32_t)(kAcc + q), u);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 16; ++e) u[e] = __float_as_uint(__uint_as_float(u[e]) + __uint_as_float(v[e]));
            tmem_store16(t_lane + (uint32_t)(kAcc + q), u);
          } else {
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 16; ++e) sum[q >= kTm ? q - kTm + e : 0] += __uint_as_float(v[e]);
          }
          tmem_zero16(t_lane + (uint32_t)q);
        }
        tmem_wait_st();
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&zeroed[dy]);
      }
    }
    if (ok) {
      const int row = 32 * (warp & 3) + lane, dx = row / C_OUT, co = row - dx * C_OUT;
#pragma unroll
      for (int q = 0; q < kAcc; q += 16) {
        const int dy = q / kDy, dz = (q - dy * kDy) / C_IN, ci = q % C_IN;
        uint32_t u[16];
        if (q < kTm) {
          tmem_load16(t_lane + (uint32_t)(kAcc + q), u);
          tmem_wait_ld();
        } else {
#pragma unroll
          for (int e = 0; e < 16; ++e) u[e] = __float_as_uint(sum[q >= kTm ? q - kTm + e : 0]);
        }
        float *dst = gW + ((long long)(dz * 9 + dy * 3 + dx) * C_OUT + co) * C_IN + ci;
        if (dx < 3) {
#pragma unroll
          for (int e = 0; e < 16; e += 4)
            red_add4(dst + e, __uint_as_float(u[e]), __uint_as_float(u[e + 1]), __uint_as_float(u[e + 2]), __uint_as_float(u[e + 3]));
        }
        __syncwarp();
      }
    }
  } else {
    // ---- bias sums: thread = (channel chunk, cells j, j + kWgBias / NCO, ...) of every g slice
    const int tid = (int)threadIdx.x - 32 * kFirstBias, c = tid % NCO;
    float acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0.f;
    for (Cursor cu(t0, t1, V); cu.live();) {
      const long long plane = (long long)V.ny * V.nx;
#pragma unroll 1
      for (int j = tid / NCO; j < TX * TY; j += kWgBias / NCO) {
        const int xx = cu.run.tx * TX + j % TX, y = cu.run.ty * TY + j / TX;
        if (xx >= V.nx || y >= V.ny) continue;
        const int4 *src = reinterpret_cast<const int4 *>(
                              gpre + ((((long long)cu.run.v * V.nz + cu.run.za) * V.ny + y) * V.nx + xx) * C_OUT) +
                          c;
        // eight reads in flight: these warps' own chain of reads, not the MMAs,
        // can be the last to end (four in flight: a training step of 4 x 64^3
        // cells 942 us, eight 924; sixteen spill, 972)
#pragma unroll 8
        for (int z = 0; z < cu.run.n; ++z) {
          const int4 q = src[z * plane * NCO];
          const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&q);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float2 f = __bfloat1622float2(h[i]);
            acc[2 * i] += f.x;
            acc[2 * i + 1] += f.y;
          }
        }
      }
      cu.step = cu.run.n + 1;  // to the next run
      cu.advance(V);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) atomicAdd(&sBias[c * 8 + i], acc[i]);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();
  fence_before_sync();
  __syncthreads();
  if (threadIdx.x < C_OUT && !abort_flag) atomicAdd(gb + threadIdx.x, sBias[threadIdx.x]);
  if (abort_flag && threadIdx.x == 0) {
    // committed MMAs may still run (see conv3d_tc_kernel)
    for (int q = 0; q < 2; ++q)
      for (int g = n_next[q]; g < n_committed; g += 2)
        for (long long n = 0; n < kWaitPolls && !mbar_try(&done[g % kWgRing], (uint32_t)(g / kWgRing) & 1u); ++n) {
        }
  }
  __syncthreads();
  if (warp == 0) {
    fence_after_sync();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

}  // namespace

size_t conv_tc_smem_bytes(int cin, int cout) { return kRing * ((size_t)cin / 8 * HN * 16) + (size_t)27 * cout * cin * 2; }

template <int C_IN, int C_OUT, int EPI>
cudaError_t conv3d_tc(const __nv_bfloat16 *x, const __nv_bfloat16 *W, const float *b, const Vol &V,
                      __nv_bfloat16 *pre_out, const __nv_bfloat16 *pre_in, void *out, int *status, cudaStream_t st) {
  const size_t sm = conv_tc_smem_bytes(C_IN, C_OUT);
  const void *fn = (const void *)conv3d_tc_kernel<C_IN, C_OUT, EPI>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  const long long nt = (long long)V.n * ((V.ny + TY - 1) / TY) * ((V.nx + TX - 1) / TX) * V.nz;
  if (nt < 1) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // one CTA per SM (it takes all of tensor memory), equal shares of the slices
  const long long g = nt < sms ? nt : sms;
  return launch_after(conv3d_tc_kernel<C_IN, C_OUT, EPI>, dim3((unsigned)g), kTcThreads, sm, st, x, W, b, V, pre_out, pre_in,
                      out, status);
}

template <int C_IN, int C_OUT>
cudaError_t wgrad(const __nv_bfloat16 *x, const __nv_bfloat16 *gpre, const Vol &V, float *gW, float *gb, int *status,
                  cudaStream_t st) {
  constexpr size_t sm = wg_smem<C_IN, C_OUT>();
  static_assert((kWgRing - 1) * wg_g_bytes<C_IN, C_OUT>() + 16 * kGPlane <= sm, "the MMAs' 16 chunks stay in shared memory");
  const void *fn = (const void *)wgrad_tc_kernel<C_IN, C_OUT>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  const long long nt = (long long)V.n * ((V.ny + TY - 1) / TY) * ((V.nx + TX - 1) / TX) * V.nz;
  if (nt < 1) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long long g = nt < sms ? nt : sms;
  return launch_after(wgrad_tc_kernel<C_IN, C_OUT>, dim3((unsigned)g), kWgThreads, sm, st, x, gpre, V, gW, gb, status);
}

#define VET_TC_INST(CI, CO, EPI)                                                                                  \
  template cudaError_t conv3d_tc<CI, CO, EPI>(const __nv_bfloat16 *, const __nv_bfloat16 *, const float *,       \
                                              const Vol &, __nv_bfloat16 *, const __nv_bfloat16 *, void *, int *, \
                                              cudaStream_t);
VET_TC_INST(16, 32, EPI_SILU)
VET_TC_INST(32, 32, EPI_SILU)
VET_TC_INST(32, 16, EPI_F32)
VET_TC_INST(16, 32, EPI_SILU_BWD)
VET_TC_INST(32, 32, EPI_SILU_BWD)

#define VET_WG_INST(CI, CO)                                                                                    \
  template cudaError_t wgrad<CI, CO>(const __nv_bfloat16 *, const __nv_bfloat16 *, const Vol &, float *, float *, \
                                     int *, cudaStream_t);
VET_WG_INST(16, 32)
VET_WG_INST(32, 32)
VET_WG_INST(32, 16)

}  // namespace cnn
}  // namespace vet
