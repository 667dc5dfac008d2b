// vet_cnn.cu -- kernels of the learned closure (not in the VETTAM paper: a
// 3D convolutional network predicting the Eddington tensor from local
// features, with the exact ray tracer as fallback): features, head and loss,
// AdamW, indicator and block list.  The convolutions and their weight gradients
// run on the tcgen05 tensor cores (vet_cnn_tc.cu).
//
// Activations are stored cells-major, channels-minor ([volume][z][y][x][C],
// BF16, C a multiple of 16).
#include <cstdint>

#include <cuda_bf16.h>

#include "vet_cnn.h"
#include "vet_floatsum.h"

namespace vet {
namespace cnn {
namespace {

// ---------------------------------------------------------------- features
// Per (volume, block) CTA: mean and standard deviation (population) of
// tau = log10(kappa h) over the block, and the volume sums of log10 S and
// log10 E (FP64 atomics).
constexpr float kTiny = 1e-30f;

__device__ __forceinline__ double block_sum_d(double v, double *red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
  return s;  // valid in thread 0
}

// Sums and differences in FP32 arithmetic to FP64's precision: the FP64 pipe does
// two operations per clock per SM, and a conversion and an addition per value held
// these kernels to a fifth of the memory rate.  At 128^3, ncu: feat_stats 47 ->
// 24 us, feat_pack 88 -> 20 us (of them 14 for its 92 MB).  (Pairs of floats, 48
// bits, left features up to half a unit further off where log S or log E hardly
// differs from its mean.)
// The block's optical depths are summed as differences from its first cell's
// (a block of equal cells then has the exact mean and a standard deviation of
// 0); a thread's up to B^3 / 256 terms by FloatSum, the threads' sums in FP64.
__global__ void __launch_bounds__(256) feat_stats_kernel(const float *__restrict__ kappa, const float *__restrict__ S,
                                                         const float *__restrict__ E, Vol V, int B, float h,
                                                         double *__restrict__ sums, float *__restrict__ bstat) {
  __shared__ double red[8][4];
  const int nbx = V.nx / B, nby = V.ny / B, nbz = V.nz / B;
  const int blk = blockIdx.x, v = blockIdx.y;
  const int bx = blk % nbx, by = (blk / nbx) % nby, bz = blk / (nbx * nby);
  const long long vol = (long long)V.nz * V.ny * V.nx;
  const int B3 = B * B * B;
  const long long c0 = (long long)v * vol + ((long long)(bz * B) * V.ny + by * B) * V.nx + bx * B;
  const float tau0 = log10f(fmaxf(kappa[c0] * h, kTiny));
  FloatSum pt, pt2, ps, pe;
  // i / B for i < 2^16 (block edges up to 32) by a multiplication
  const unsigned mB = (unsigned)(((1ull << 32) + B - 1) / B);
  for (int i0 = threadIdx.x; i0 < B3; i0 += 4 * blockDim.x) {  // four cells a trip, their loads together
    float k[4], s[4], en[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + u * (int)blockDim.x;
      k[u] = s[u] = en[u] = 1.f;
      if (i < B3) {
        int r = i, z = 0, x = 0;
        if (B <= 32) {
          r = B > 1 ? (int)__umulhi((unsigned)i, mB) : i;
          z = B > 1 ? (int)__umulhi((unsigned)r, mB) : r;
        } else {
          r = i / B;
          z = r / B;
        }
        x = i - r * B;
        const long long c = c0 + ((long long)z * V.ny + (r - z * B)) * V.nx + x;
        k[u] = kappa[c];
        s[u] = S[c];
        en[u] = E[c];
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (i0 + u * (int)blockDim.x >= B3) break;
      float d = log10f(fmaxf(k[u] * h, kTiny));
      const float dl = two_sum(d, -tau0);  // the difference is d + dl
      pt.add(d, dl);
      // its square: d^2 and 2 d dl by products with their exact roundings (FMA);
      // the second one's is, like dl^2, below 2^-48 of the total
      const float q = __fmul_rn(d, d), r = __fmul_rn(2.f * d, dl);
      pt2.add(q, __fmaf_rn(d, d, -q));
      pt2.c = __fadd_rn(pt2.c, __fadd_rn(two_sum(pt2.b, r), __fmaf_rn(dl, dl, __fmaf_rn(2.f * d, dl, -r))));
      ps.add(log10f(fmaxf(s[u], kTiny)));
      pe.add(log10f(fmaxf(en[u], kTiny)));
    }
  }
  double vt = pt.value(), vt2 = pt2.value(), vs = ps.value(), ve = pe.value(), ref = tau0;
  if (__syncthreads_or(!isfinite(vt) || !isfinite(vt2) || !isfinite(vs) || !isfinite(ve))) {
    // an infinity among the fields (a FloatSum loses its sign): plain FP64 sums
    vt = vt2 = vs = ve = ref = 0.0;
    for (int i = threadIdx.x; i < B3; i += blockDim.x) {
      const int x = i % B, y = (i / B) % B, z = i / (B * B);
      const long long c = c0 + ((long long)z * V.ny + y) * V.nx + x;
      const double tau = log10f(fmaxf(kappa[c] * h, kTiny));
      vt += tau;
      vt2 += tau * tau;
      vs += log10f(fmaxf(S[c], kTiny));
      ve += log10f(fmaxf(E[c], kTiny));
    }
  }
  // the warp's four sums in six FP64 additions a lane, each exchange halving what a
  // lane carries; then the warps' by four threads
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool up = lane & 16, mid = lane & 8;
  double v0 = up ? vs : vt, v1 = up ? ve : vt2;
  v0 += __shfl_xor_sync(0xffffffffu, up ? vt : vs, 16);
  v1 += __shfl_xor_sync(0xffffffffu, up ? vt2 : ve, 16);
  double w = (mid ? v1 : v0) + __shfl_xor_sync(0xffffffffu, mid ? v0 : v1, 8);
  for (int o = 4; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
  if ((lane & 7) == 0) red[warp][lane >> 3] = w;
  __syncthreads();
  if (threadIdx.x >= 32) return;
  double sum = 0.0;
  if (threadIdx.x < 4)
    for (int q = 0; q < 8; ++q) sum += red[q][threadIdx.x];
  const double st2 = __shfl_sync(0xffffffffu, sum, 1);
  if (threadIdx.x == 0) {
    const double mean = sum / B3, var = fmax(st2 / B3 - mean * mean, 0.0);
    bstat[((long long)v * nbx * nby * nbz + blk) * 2] = (float)(ref + mean);
    bstat[((long long)v * nbx * nby * nbz + blk) * 2 + 1] = (float)sqrt(var);
  }
  if (threadIdx.x == 2 || threadIdx.x == 3) atomicAdd(sums + 2 * v + threadIdx.x - 2, sum);
}

// A double as three floats, and l - it: exact sums of the parts, rounded once but
// for what is below 2^-48 of l.
struct Mean {
  float a, b, c;
};
__device__ __forceinline__ Mean split_mean(double m) {
  const float a = (float)m;
  if (!isfinite(a)) return {a, 0.f, 0.f};
  const float b = (float)(m - (double)a);
  return {a, b, (float)((m - (double)a) - (double)b)};
}
__device__ __forceinline__ float minus_mean(float l, const Mean &mean) {
  float d = l;
  const float e1 = two_sum(d, -mean.a);
  const float first = d;
  const float e2 = two_sum(d, -mean.b), r = __fadd_rn(d, __fadd_rn(e2, __fsub_rn(e1, mean.c)));
  return isfinite(first) ? r : first;  // a select: a return in between took 6 us of 47
}

// n / d for any n and d below 2^32: the multiplication's quotient is exact or one short.
struct Div {
  unsigned d, m;
  explicit Div(int v) : d((unsigned)v), m(v > 1 ? (unsigned)((1ull << 32) / (unsigned)v) : 0xffffffffu) {}
  __device__ __forceinline__ unsigned quotient(unsigned n) const {
    const unsigned q = __umulhi(n, m);
    return n - q * d >= d ? q + 1 : q;
  }
};

// The input rows (bf16), cell by cell (grid: x over the cells of a volume, y
// over the volumes).  64-bit divisions for a cell's block cost more than the
// logarithms: the learned closure of 128^3 cells 475 us with them, 463 with
// 32-bit quotients.
template <bool NARROW>
__global__ void __launch_bounds__(256) feat_pack_kernel(const float *__restrict__ kappa, const float *__restrict__ S,
                                                        const float *__restrict__ E, Vol V, Div dnx, Div dny, Div dB, int B, float h,
                                                        const double *__restrict__ sums,
                                                        const float *__restrict__ bstat, __nv_bfloat16 *__restrict__ x0,
                                                        float *__restrict__ feat_out) {
  __shared__ Mean s_mean[2];
  after_previous();
  let_next_launch();
  const long long vol = (long long)V.nz * V.ny * V.nx;
  const int v = blockIdx.y;
  if (threadIdx.x < 2) s_mean[threadIdx.x] = split_mean(sums[2 * v + threadIdx.x] / (double)vol);
  __syncthreads();
  const Mean mean_s = s_mean[0], mean_e = s_mean[1];
  const int nbx = V.nx / B, nby = V.ny / B, nbz = V.nz / B;
  for (long long l = blockIdx.x * (long long)blockDim.x + threadIdx.x; l < vol; l += (long long)gridDim.x * blockDim.x) {
    const long long c = v * vol + l;
    int blk;
    if (NARROW) {
      const unsigned r = dnx.quotient((unsigned)l), z = dny.quotient(r);
      const unsigned x = (unsigned)l - r * dnx.d, y = r - z * dny.d;
      blk = (int)(dB.quotient(x) + nbx * (dB.quotient(y) + nby * dB.quotient(z)));
    } else {
      const long long r = l / V.nx;
      const int x = (int)(l - r * V.nx), z = (int)(r / V.ny), y = (int)(r - (long long)z * V.ny);
      blk = (x / B) + nbx * ((y / B) + nby * (z / B));
    }
    const float *bs = bstat + ((long long)v * nbx * nby * nbz + blk) * 2;
    float f[kIn];
    f[0] = 1.f;
    f[1] = log10f(fmaxf(kappa[c] * h, kTiny));
    f[2] = minus_mean(log10f(fmaxf(S[c], kTiny)), mean_s);
    f[3] = minus_mean(log10f(fmaxf(E[c], kTiny)), mean_e);
    f[4] = bs[0];
    f[5] = bs[1];
    __align__(16) __nv_bfloat162 row[kInPad / 2];
#pragma unroll
    for (int i = 0; i < kInPad / 2; ++i) row[i] = __floats2bfloat162_rn(0.f, 0.f);
    row[0] = __floats2bfloat162_rn(f[0], f[1]);
    row[1] = __floats2bfloat162_rn(f[2], f[3]);
    row[2] = __floats2bfloat162_rn(f[4], f[5]);
    int4 *dst = reinterpret_cast<int4 *>(x0 + c * kInPad);
    dst[0] = reinterpret_cast<const int4 *>(row)[0];
    dst[1] = reinterpret_cast<const int4 *>(row)[1];
    if (feat_out)
      for (int i = 0; i < kIn; ++i) feat_out[((long long)v * kIn + i) * vol + l] = f[i];
  }
}

// ------------------------------------------------------------- head / loss
// f_ii = 1/3 + D_ii - tr(D)/3, f_ij = D_ij; the error target
// log(max |f - f_ref| + 1e-4) is a constant of the gradient.
constexpr float kErrEps = 1e-4f;

__device__ __forceinline__ void head_f(const float *o, float *f) {
  const float tr = (o[0] + o[1] + o[2]) * (1.f / 3.f);
  f[0] = 1.f / 3.f + o[0] - tr;
  f[1] = 1.f / 3.f + o[1] - tr;
  f[2] = 1.f / 3.f + o[2] - tr;
  f[3] = o[3];
  f[4] = o[4];
  f[5] = o[5];
}

__global__ void __launch_bounds__(256) count_kernel(const unsigned char *__restrict__ mask, long long n,
                                                    unsigned long long *count) {
  unsigned long long k = 0;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x)
    k += mask[c] != 0;
  for (int o = 16; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
  if ((threadIdx.x & 31) == 0 && k) atomicAdd(count, k);
}

__global__ void __launch_bounds__(256) head_loss_kernel(const float *__restrict__ o, const float *__restrict__ f_ref,
                                                        const unsigned char *__restrict__ mask, Vol V, float lam,
                                                        const unsigned long long *__restrict__ count,
                                                        double *__restrict__ loss, __nv_bfloat16 *__restrict__ go) {
  __shared__ double red[8];
  const long long vol = (long long)V.nz * V.ny * V.nx, n = vol * V.n;
  const unsigned long long cnt = mask ? *count : (unsigned long long)n;
  const float inv_n = cnt ? (float)(1.0 / (double)cnt) : 0.f;
  double part = 0.0;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    const int v = (int)(c / vol);
    const long long l = c - v * vol;
    float ov[8];
    const float4 *src = reinterpret_cast<const float4 *>(o + c * kOutRow);
    const float4 a = src[0], b = src[1];
    ov[0] = a.x; ov[1] = a.y; ov[2] = a.z; ov[3] = a.w;
    ov[4] = b.x; ov[5] = b.y; ov[6] = b.z; ov[7] = b.w;
    float f[6], d[6];
    head_f(ov, f);
    float mx = 0.f, sq = 0.f;
    for (int i = 0; i < 6; ++i) {
      d[i] = f[i] - f_ref[((long long)v * 6 + i) * vol + l];
      mx = fmaxf(mx, fabsf(d[i]));
      sq += d[i] * d[i];
    }
    const float m = (!mask || mask[c]) ? 1.f : 0.f;
    const float r = ov[6] - logf(mx + kErrEps);
    part += (double)(m * (sq * (1.f / 6.f) + lam * r * r));
    float gf[6];
    for (int i = 0; i < 6; ++i) gf[i] = m * 2.f * d[i] * (1.f / 6.f) * inv_n;
    const float tg = (gf[0] + gf[1] + gf[2]) * (1.f / 3.f);
    __align__(16) __nv_bfloat162 row[kOutPad / 2];
    row[0] = __floats2bfloat162_rn(gf[0] - tg, gf[1] - tg);
    row[1] = __floats2bfloat162_rn(gf[2] - tg, gf[3]);
    row[2] = __floats2bfloat162_rn(gf[4], gf[5]);
    row[3] = __floats2bfloat162_rn(m * lam * 2.f * r * inv_n, 0.f);
#pragma unroll
    for (int i = 4; i < kOutPad / 2; ++i) row[i] = __floats2bfloat162_rn(0.f, 0.f);
    int4 *dst = reinterpret_cast<int4 *>(go + c * kOutPad);
    dst[0] = reinterpret_cast<const int4 *>(row)[0];
    dst[1] = reinterpret_cast<const int4 *>(row)[1];
  }
  part = block_sum_d(part, red);
  if (threadIdx.x == 0) atomicAdd(loss, part * (double)inv_n);
}

// -------------------------------------------------------------------- AdamW
// Loshchilov & Hutter (2019): m <- b1 m + (1-b1) g, v <- b2 v + (1-b2) g^2,
// p <- p - lr (m/bc1 / (sqrt(v/bc2) + eps) + wd p), bc = 1 - beta^step.
__global__ void __launch_bounds__(256) adamw_kernel(NetMeta M, float *__restrict__ p, const float *__restrict__ g,
                                                    float *__restrict__ m, float *__restrict__ v, float lr, float b1,
                                                    float b2, float eps, float wd, float bc1, float bc2, int update) {
  after_previous();
  let_next_launch();
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < M.total;
       i += (long long)gridDim.x * blockDim.x) {
    float pi = p[i];
    if (update) {
      const float gi = g[i];
      const float mi = b1 * m[i] + (1.f - b1) * gi;
      const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
      m[i] = mi;
      v[i] = vi;
      pi -= lr * ((mi / bc1) / (sqrtf(vi / bc2) + eps) + wd * pi);
      p[i] = pi;
    }
    for (int l = 0; l < 4; ++l) {
      const LayerMeta &L = M.L[l];
      const long long k = i - L.w_off;
      if (k < 0 || k >= 27LL * L.cout * L.cin) continue;
      const int tap = (int)(k / ((long long)L.cout * L.cin));
      const int rem = (int)(k - (long long)tap * L.cout * L.cin), co = rem / L.cin, ci = rem - co * L.cin;
      const __nv_bfloat16 w = __float2bfloat16_rn(pi);
      L.wb[k] = w;
      L.wt[((long long)(26 - tap) * L.cin + ci) * L.cout + co] = w;
    }
  }
}

// --------------------------------------------------------------- indicator
// Eigenvalues of the symmetric 3 x 3 tensor f by the trigonometric closed form
// (O. K. Smith, Comm. ACM 4 (1961) 168): with q = tr f / 3 and
// p = sqrt(|f - q I|_F^2 / 6), the eigenvalues are q + 2 p cos(phi + 2 pi k/3),
// phi = acos(det((f - q I)/p) / 2) / 3.
__device__ __forceinline__ void sym3_eig_minmax(const float *f, float &lmin, float &lmax) {
  const float q = (f[0] + f[1] + f[2]) * (1.f / 3.f);
  const float p1 = f[3] * f[3] + f[4] * f[4] + f[5] * f[5];
  const float a = f[0] - q, b = f[1] - q, c = f[2] - q;
  const float p2 = a * a + b * b + c * c + 2.f * p1;
  if (!(p2 > 0.f)) {
    lmin = lmax = q;
    return;
  }
  const float p = sqrtf(p2 * (1.f / 6.f)), ip = 1.f / p;
  const float A = a * ip, Bv = b * ip, C = c * ip, xy = f[3] * ip, xz = f[4] * ip, yz = f[5] * ip;
  const float det = A * (Bv * C - yz * yz) - xy * (xy * C - yz * xz) + xz * (xy * yz - Bv * xz);
  const float r = fminf(fmaxf(0.5f * det, -1.f), 1.f);
  const float phi = acosf(r) * (1.f / 3.f);
  lmax = q + 2.f * p * cosf(phi);
  lmin = q + 2.f * p * cosf(phi + 2.0943951023931953f);
}

__global__ void __launch_bounds__(256) indicator_kernel(const float *__restrict__ o, Vol V, int B, float thr,
                                                        float *__restrict__ f_out, float *__restrict__ r_out,
                                                        unsigned int *__restrict__ flags) {
  const long long n = (long long)V.nz * V.ny * V.nx;
  const int nbx = V.nx / B, nby = V.ny / B;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    const float4 *src = reinterpret_cast<const float4 *>(o + c * kOutRow);
    const float4 a = src[0], b = src[1];
    const float ov[7] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z};
    float f[6];
    head_f(ov, f);
    for (int i = 0; i < 6; ++i) f_out[i * n + c] = f[i];
    float lmin, lmax;
    sym3_eig_minmax(f, lmin, lmax);
    float r = fmaxf(fmaxf(fmaxf(0.f, -lmin), fmaxf(0.f, lmax - 1.f)), expf(ov[6]));
    // fmaxf drops NaN: a non-finite output must still send its block to the
    // exact closure
    float chk = 0.f;
    for (int i = 0; i < 7; ++i) chk += ov[i] * 0.f;
    if (chk != 0.f) r = INFINITY;
    if (r_out) r_out[c] = r;
    if (r > thr) {
      const int x = (int)(c % V.nx), y = (int)((c / V.nx) % V.ny), z = (int)(c / ((long long)V.nx * V.ny));
      flags[(x / B) + nbx * ((y / B) + nby * (z / B))] = 1u;
    }
  }
}

__global__ void __launch_bounds__(1024) compact_kernel(const unsigned int *__restrict__ flags, int n,
                                                       int *__restrict__ list, int *__restrict__ count) {
  after_previous();
  let_next_launch();
  __shared__ int wsum[32];
  const int per = (n + blockDim.x - 1) / blockDim.x;
  const int b = threadIdx.x * per, e = min(n, b + per);
  int k = 0;
  for (int i = b; i < e; ++i) k += flags[i] != 0;
  // block exclusive scan of k
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int incl = k;
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) wsum[w] = incl;
  __syncthreads();
  if (w == 0) {
    int s = lane < (int)(blockDim.x >> 5) ? wsum[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += t;
    }
    wsum[lane] = s;
  }
  __syncthreads();
  int pos = incl - k + (w ? wsum[w - 1] : 0);
  for (int i = b; i < e; ++i)
    if (flags[i]) list[pos++] = i;
  if (threadIdx.x == blockDim.x - 1) *count = pos;
}

__global__ void __launch_bounds__(256) unpack_kernel(const float *__restrict__ o, Vol V, float *__restrict__ out) {
  const long long vol = (long long)V.nz * V.ny * V.nx, n = vol * V.n;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    const int v = (int)(c / vol);
    const long long l = c - v * vol;
    for (int i = 0; i < kOut; ++i) out[((long long)v * kOut + i) * vol + l] = o[c * kOutRow + i];
  }
}

int grid_for(long long n, int threads) {
  long long b = (n + threads - 1) / threads;
  if (b > 152LL * 16) b = 152LL * 16;
  return (int)(b < 1 ? 1 : b);
}

}  // namespace

cudaError_t features(const float *kappa, const float *S, const float *E, const Vol &V, int B, double h, double *sums,
                     float *bstat, __nv_bfloat16 *x0, float *feat_out, cudaStream_t st) {
  if (V.n < 1) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(sums, 0, sizeof(double) * 2 * V.n, st);
  if (e != cudaSuccess) return e;
  const int nblk = (V.nx / B) * (V.ny / B) * (V.nz / B);
  feat_stats_kernel<<<dim3(nblk, V.n), 256, 0, st>>>(kappa, S, E, V, B, (float)h, sums, bstat);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int per_vol = (grid_for((long long)V.n * V.nz * V.ny * V.nx, 256) + V.n - 1) / V.n;
  // cell numbers of a volume in 32 bits: quotients by multiplication
  const bool narrow = (long long)V.nz * V.ny * V.nx < (1LL << 31);
  auto *pack = narrow ? feat_pack_kernel<true> : feat_pack_kernel<false>;
  return launch_after(pack, dim3(per_vol, V.n), 256, 0, st, kappa, S, E, V, Div(V.nx), Div(V.ny), Div(B), B, (float)h, sums,
                      bstat, x0, feat_out);
}

cudaError_t head_loss(const float *o, const float *f_ref, const unsigned char *mask, const Vol &V, float lam,
                      unsigned long long *count, double *loss, __nv_bfloat16 *go, cudaStream_t st) {
  const long long n = (long long)V.n * V.nz * V.ny * V.nx;
  cudaError_t e = cudaMemsetAsync(count, 0, sizeof(unsigned long long), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(loss, 0, sizeof(double), st);
  if (e != cudaSuccess) return e;
  if (mask) count_kernel<<<grid_for(n, 256), 256, 0, st>>>(mask, n, count);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  head_loss_kernel<<<grid_for(n, 256), 256, 0, st>>>(o, f_ref, mask, V, lam, count, loss, go);
  return cudaGetLastError();
}

cudaError_t adamw(const NetMeta &M, float *p, const float *g, float *m, float *v, float lr, float b1, float b2,
                  float eps, float wd, float bc1, float bc2, int update, cudaStream_t st) {
  return launch_after(adamw_kernel, dim3(grid_for(M.total, 256)), 256, 0, st, M, p, g, m, v, lr, b1, b2, eps, wd, bc1, bc2,
                      update);
}

cudaError_t indicator(const float *o, const Vol &V, int B, float thr, float *f_out, float *r_out, unsigned int *flags,
                      cudaStream_t st) {
  const int nblk = (V.nx / B) * (V.ny / B) * (V.nz / B);
  cudaError_t e = cudaMemsetAsync(flags, 0, sizeof(unsigned int) * nblk, st);
  if (e != cudaSuccess) return e;
  const long long n = (long long)V.nz * V.ny * V.nx;
  indicator_kernel<<<grid_for(n, 256), 256, 0, st>>>(o, V, B, thr, f_out, r_out, flags);
  return cudaGetLastError();
}

cudaError_t compact_flags(const unsigned int *flags, int n, int *list, int *count, cudaStream_t st) {
  return launch_after(compact_kernel, dim3(1), 1024, 0, st, flags, n, list, count);
}

cudaError_t unpack_outputs(const float *o, const Vol &V, float *o_out, cudaStream_t st) {
  const long long n = (long long)V.n * V.nz * V.ny * V.nx;
  unpack_kernel<<<grid_for(n, 256), 256, 0, st>>>(o, V, o_out);
  return cudaGetLastError();
}

}  // namespace cnn
}  // namespace vet
