// vet_point.cu -- direct radiation of a point source (paper Sec. 2.2.6):
// the energy and momentum a source of luminosity L at x_s deposits in every
// cell, from the optical depth along the straight ray from x_s through the
// cell centre (long characteristics, the limit of the paper's hybrid
// tracer):
//   tau_*    sum kappa * length over the cells the ray crosses from x_s to
//            where it enters cell c (0 if the source lies in c),
//   dr       the ray's length inside c (from its entry, or from x_s),
//   Edot     L e^{-tau_*} (1 - e^{-kappa_c dr}) / (4 pi r^2 dr), r = |x_c - x_s|,
//            with 1 - e^{-x} = -expm1(-x): the small-tau Taylor form needs
//            no switch,
//   pdot     Edot (x_c - x_s) / r (c = 1).
// A ray point on a cell face lies in the cell the ray enters next; a cell
// whose centre is the source gets zeros.
//
// One thread per cell, a warp's cells in a brick (8 x 2 x 2 where the grid has
// the extents): the rays of a warp start at the same point, stay close and
// cross nearly the same number of planes.  Geometry in cell units (planes at
// integers); every plane crossing is computed from the source position, not
// accumulated, so a crossing's error is a few ulp of its own distance.  The
// walk's crossings, about |di| + |dj| + |dk|, are counted before it starts, and
// it runs in groups of four whose kappa reads are in flight together.
//
// Bound by instruction issue (76% of the slots, 27 instructions a crossing):
// 128^3 cells take 2.3e8 crossings; kappa and the results are 42 MB, 6 us.  One
// row of x a warp, a test of the end and of the grid's bounds at every step and
// selects for the axes took 760 us; without the tests, in bricks, 252; with the
// crossed axis' update under a predicate instead of selects 215 (bricks of 4 x 4
// x 2 212, of 16 x 2 x 1 222; groups of six or eight crossings the same).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>

#include <cuda_runtime.h>

#include "vet.h"

namespace {

struct PointArgs {
  int nx, ny, nz;
  float h;
  float xs[3];  // source, cell units
  float L;
  // a warp's brick is 2^w cells along each axis, a CTA's 2^c warps (sums 5 and 3)
  int w[3], c[3];
  int tx, ty;  // CTAs along x and y
};

// Largest extent whose walks need no check of the grid's bounds, below.
constexpr int kPlainExtent = 65536;

// Extents up to kPlainExtent (CHECK = false, at most 2^31 - 1 cells): a walk
// takes exactly the crossings between the source's cell and the target's, and
// stays between them.  The ray leaves the target's slab of any axis at least
// half a cell beyond the target's centre and enters it by half a cell before, so
// that a crossing past the target lies at least one cell behind t_in, and the
// crossings' rounding (5 ulp of at most 1.8 x 65536 cells: 0.04) cannot bring it
// forward.  Larger grids check every read.
template <bool CHECK>
__global__ void __launch_bounds__(256) point_kernel(PointArgs a, const float *__restrict__ kappa,
                                                   float *__restrict__ Edot, float *__restrict__ pdot) {
  using Idx = std::conditional_t<CHECK, long long, int>;
  using Plane = std::conditional_t<CHECK, int, float>;  // exact either way: kPlainExtent < 2^24
  const long long ncell = (long long)a.nx * a.ny * a.nz;
  const int n[3] = {a.nx, a.ny, a.nz};
  const int tile[3] = {(int)(blockIdx.x % a.tx), (int)(blockIdx.x / a.tx % a.ty), (int)(blockIdx.x / a.tx / a.ty)};
  int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, cc[3];
  bool inside = true;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    cc[q] = (((tile[q] << a.c[q]) + (warp & ((1 << a.c[q]) - 1))) << a.w[q]) + (lane & ((1 << a.w[q]) - 1));
    lane >>= a.w[q];
    warp >>= a.c[q];
    inside = inside && cc[q] < n[q];
  }
  if (!inside) return;
  const long long c = ((long long)cc[2] * a.ny + cc[1]) * a.nx + cc[0];
  float v[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) v[q] = cc[q] + 0.5f - a.xs[q];
  const float r = sqrtf(fmaf(v[0], v[0], fmaf(v[1], v[1], v[2] * v[2])));
  if (!(r > 0.f)) {
    Edot[c] = 0.f;
    if (pdot) pdot[c] = pdot[ncell + c] = pdot[2 * ncell + c] = 0.f;
    return;
  }
  float d[3], inv[3], in_q[3];
  float t_in = 0.f, t_out = INFINITY;  // the target cell's parameter interval (slabs)
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    d[q] = v[q] / r;
    inv[q] = d[q] != 0.f ? 1.f / d[q] : INFINITY;
    in_q[q] = 0.f;
    if (d[q] != 0.f) {
      const float t1 = (cc[q] - a.xs[q]) * inv[q], t2 = (cc[q] + 1 - a.xs[q]) * inv[q];
      in_q[q] = fminf(t1, t2);
      t_in = fmaxf(t_in, in_q[q]);
      t_out = fminf(t_out, fmaxf(t1, t2));
    }
  }
  const float dr = t_out - t_in;
  // The walk from the source cell to the entry of the target cell: the next
  // crossing tm of each axis is kept, at plane pl, and only the axis just
  // crossed has its next crossing recomputed from the source position.  A step
  // runs from the last crossing to the next, and none starts at t_in - 1e-5 or
  // later: of an axis' crossings between the two cells only the last, at in_q,
  // can lie there.
  const float t_end = t_in - 1e-5f;
  Plane pl[3], s[3];
  float tm[3];
  Idx e[3] = {1, (Idx)a.nx, (Idx)a.nx * a.ny}, idx = 0;
  int steps = 1;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int cs = min((int)floorf(a.xs[q]), n[q] - 1);  // rounded to 32 bits, a source may lie on the upper boundary
    const bool up = d[q] > 0.f;
    steps += abs(cc[q] - cs) - (cc[q] != cs && !(in_q[q] < t_end) ? 1 : 0);
    idx += cs * e[q];
    e[q] = up ? e[q] : -e[q];
    s[q] = (Plane)(up ? 1 : -1);
    pl[q] = (Plane)(cs + (up ? 1 : 0));
    tm[q] = d[q] != 0.f ? (pl[q] - a.xs[q]) * inv[q] : INFINITY;
  }
  if (!(t_end > 0.f)) steps = 0;
  float t = 0.f, tau = 0.f;
  auto step = [&](float &kv, float &len) {
    if constexpr (!CHECK) {
      // the clamp below never acts here: the last step ends at the first of the
      // crossings from t_end on, and the target's own is one of them
      const float t0 = t;
      kv = __ldg(kappa + idx);
      asm("{\n .reg .pred p, q, r;\n .reg .f32 u;\n"
          " min.f32 u, %4, %5;\n min.f32 %0, u, %6;\n"
          " setp.eq.f32 p, %4, %0;\n setp.eq.and.f32 q|r, %5, %0, !p;\n"
          " @p add.f32 %1, %1, %8;\n @p sub.f32 u, %1, %11;\n @p mul.f32 %4, u, %14;\n @p add.s32 %7, %7, %17;\n"
          " @q add.f32 %2, %2, %9;\n @q sub.f32 u, %2, %12;\n @q mul.f32 %5, u, %15;\n @q add.s32 %7, %7, %18;\n"
          " @r add.f32 %3, %3, %10;\n @r sub.f32 u, %3, %13;\n @r mul.f32 %6, u, %16;\n @r add.s32 %7, %7, %19;\n}\n"
          : "=&f"(t), "+f"(pl[0]), "+f"(pl[1]), "+f"(pl[2]), "+f"(tm[0]), "+f"(tm[1]), "+f"(tm[2]), "+r"(idx)
          : "f"(s[0]), "f"(s[1]), "f"(s[2]), "f"(a.xs[0]), "f"(a.xs[1]), "f"(a.xs[2]), "f"(inv[0]), "f"(inv[1]),
            "f"(inv[2]), "r"(e[0]), "r"(e[1]), "r"(e[2]));
      len = t - t0;
      return;
    }
    const float tn = fminf(fminf(tm[0], tm[1]), tm[2]);
    const bool p0 = tm[0] == tn, p1 = !p0 && tm[1] == tn, p2 = !p0 && !p1;
    const float te = fminf(tn, t_in);
    len = te - t;
    t = te;
    bool in = true;
    if constexpr (CHECK) {
#pragma unroll
      for (int q = 0; q < 3; ++q) in = in && (unsigned)(pl[q] - (s[q] > 0)) < (unsigned)n[q];
    }
    kv = in ? __ldg(kappa + idx) : 0.f;
    len = in ? len : 0.f;
    if (p0) {
      pl[0] += s[0];
      tm[0] = (pl[0] - a.xs[0]) * inv[0];
      idx += e[0];
    }
    if (p1) {
      pl[1] += s[1];
      tm[1] = (pl[1] - a.xs[1]) * inv[1];
      idx += e[1];
    }
    if (p2) {
      pl[2] += s[2];
      tm[2] = (pl[2] - a.xs[2]) * inv[2];
      idx += e[2];
    }
  };
  for (; steps >= 4; steps -= 4) {
    float kv[4], len[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) step(kv[u], len[u]);
#pragma unroll
    for (int u = 0; u < 4; ++u) tau = fmaf(kv[u], len[u], tau);
  }
  {
    float kv[3] = {0.f, 0.f, 0.f}, len[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int u = 0; u < 3; ++u)
      if (u < steps) step(kv[u], len[u]);
#pragma unroll
    for (int u = 0; u < 3; ++u) tau = fmaf(kv[u], len[u], tau);
  }
  const float taus = tau * a.h, drl = dr * a.h, rl = r * a.h;
  const float tc = kappa[c] * drl;
  const float E = a.L * expf(-taus) * (-expm1f(-tc)) / (4.f * 3.14159265358979f * rl * rl * drl);
  Edot[c] = E;
  if (pdot) {
    pdot[c] = E * d[0];
    pdot[ncell + c] = E * d[1];
    pdot[2 * ncell + c] = E * d[2];
  }
}

bool on_device(const void *p) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" __attribute__((visibility("default"))) vet_status vet_point_source(const vet_grid *grid, const double xs[3],
                                                                                double L, const float *kappa,
                                                                                float *Edot_out, float *pdot_out,
                                                                                void *stream) {
  if (!grid || !xs || !kappa || !Edot_out) return VET_EINVAL;
  if (grid->nx < 1 || grid->ny < 1 || grid->nz < 1 || !(grid->h > 0.0) || !std::isfinite(L)) return VET_EINVAL;
  const int n[3] = {grid->nx, grid->ny, grid->nz};
  PointArgs a;
  a.nx = n[0];
  a.ny = n[1];
  a.nz = n[2];
  a.h = (float)grid->h;
  a.L = (float)L;
  for (int q = 0; q < 3; ++q) {
    const double u = xs[q] / grid->h;
    if (!(u >= 0.0 && u < n[q])) return VET_EINVAL;  // the source must lie in the grid
    a.xs[q] = (float)u;
  }
  if (!on_device(kappa) || !on_device(Edot_out) || (pdot_out && !on_device(pdot_out))) return VET_EINVAL;
  // bricks no wider than the grid's planes: 8 x 2 x 2 cells a warp, 16 x 4 x 4 a CTA
  for (int q = 1; q < 3; ++q) {
    a.w[q] = n[q] > 1;
    a.c[q] = n[q] > 2;
  }
  a.w[0] = 5 - a.w[1] - a.w[2];
  a.c[0] = 3 - a.c[1] - a.c[2];
  long long tiles[3];
  for (int q = 0; q < 3; ++q) tiles[q] = (n[q] + (1LL << (a.w[q] + a.c[q])) - 1) >> (a.w[q] + a.c[q]);
  a.tx = (int)tiles[0];
  a.ty = (int)tiles[1];
  const long long ctas = tiles[0] * tiles[1] * tiles[2];
  const bool plain = std::max({n[0], n[1], n[2]}) <= kPlainExtent && (long long)n[0] * n[1] * n[2] <= INT32_MAX;
  auto kernel = plain ? point_kernel<false> : point_kernel<true>;
  kernel<<<(unsigned)ctas, 256, 0, (cudaStream_t)stream>>>(a, kappa, Edot_out, pdot_out);
  return cudaGetLastError() == cudaSuccess ? VET_OK : VET_ECUDA;
}
