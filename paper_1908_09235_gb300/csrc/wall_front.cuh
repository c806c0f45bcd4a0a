// The wall pass of the step before, and the channel ends, as the first CTAs of a large lattice's step
// kernel (csrc/step_vec.cu, csrc/step_march.cu).
//
// As a launch of its own the pass stands between two steps and leaves the GPU idle but for a few
// warps: it waits for the last tile of one step and the first tile of the next waits for it, 3 to 5
// us a step.  Here its CTAs come first in the grid, do the pass on the source lattice in place and
// count themselves done; tiles start at once, and only what reads nodes it writes waits for the
// count.  CTAs are dispatched in the order of their index, so the pass is under way before anything
// waits for it; the wait is bounded all the same.  Marching kernel, FP16 4096^2 / 2048^2: 148.1 / 47.7
// us a step against 154.7 / 50.8 with the pass apart (149.9 / 46.7 without walls).
#pragma once
#include "tma.cuh"
#include "wall.cuh"

namespace lbm {
namespace wall {

// CTA id of the front, nt threads; flags: the node flags.
template <typename S>
__device__ __forceinline__ void front_cta(const DevParams& p, const FrontWalls& w,
                                          const uint8_t* flags, int id, int tid, int nt) {
  if (id >= w.ctas) {
    pdl_wait();
    return;
  }
  if (id < w.wall_ctas) {
    const int gt = id * nt + tid, b = gt >> 3, k = gt & 7;
    const auto q = load_link<typename Pop<S>::C>(b, k, b < w.nb, w.bnode, w.boff, w.ldir, w.recipe);
    pdl_wait();
    wall_values<S>(p, b, k, b < w.nb, q, Lat<S>{nullptr, w.f, p.N, p.rho_ref}, w.rho, w.ux, w.uy,
                   w.carry, InPlace<S>{w.f, p.N, w.carry}, nullptr, 0xffffffffu);
  } else {
    open_row<S>(p, (id - w.wall_ctas) * nt + tid, w.f, flags, w.u_in);  // waits too
  }
  __syncthreads();
  if (tid == 0) {
    if (id == 0) *w.reset = 0;  // of the next step; nobody uses it in this one
    // the CTA's stores before the count, for plain loads and for tensor copies of the readers
    __threadfence();
    asm volatile("fence.proxy.async;" ::: "memory");
    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(w.done) : "memory");
  }
}

// Whether a tile of nodes x0 .. x0 + tw - 1, y0 .. y0 + th - 1, with its ring, may read what the front
// writes.  Boundary nodes are within sqrt(2) of a circle, so the distances of the ringed tile's nearest
// and farthest points from its centre must lie on either side of it, give or take 2.
__device__ __forceinline__ bool front_touches(const FrontWalls& w, int x0, int y0, int tw, int th,
                                              int nx, int ny) {
  bool hit = w.everywhere || (w.flat && (y0 <= 3 || y0 + th >= ny - 3)) ||
             (w.open_x && (x0 == 0 || x0 + tw >= nx));
  const float hx = 0.5f * float(tw + 1), hy = 0.5f * float(th + 1);
#pragma unroll
  for (int i = 0; i < FrontWalls::kCircles; ++i) {
    if (i >= w.n_circles) break;
    const float dx = fabsf(float(x0 - 1) + hx - w.cx[i]), dy = fabsf(float(y0 - 1) + hy - w.cy[i]);
    const float nx_ = fmaxf(dx - hx, 0.f), ny_ = fmaxf(dy - hy, 0.f), fx = dx + hx, fy = dy + hy;
    const float lo = fmaxf(w.r[i] - 2.f, 0.f), hi = w.r[i] + 2.f;
    hit = hit || (nx_ * nx_ + ny_ * ny_ <= hi * hi && fx * fx + fy * fy >= lo * lo);
  }
  return hit;
}

// One thread waits until the front is done; the caller's barrier comes after.  At most about limit_ns
// (that of every bounded wait: a front has microseconds of work, but another process's time slice may
// come between), and not at all once a wait of any tile has given up: that sets kErrTimeout in *err,
// which fails the lattice's next blocking read (lbm_mass, lbm_fields, lbm_force, lbm_save_state), since
// the tile goes on without the walls.
__device__ __forceinline__ void front_wait(const FrontWalls& w, int* err,
                                           unsigned long long limit_ns = tma::kWaitNs) {
  const unsigned long long t0 = tma::global_ns();
  for (long long i = 0; i < (1LL << 32); ++i) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(w.done) : "memory");
    if (v >= w.ctas) break;
    if ((i & 63) == 63) {
      if (*reinterpret_cast<volatile int*>(err) & kErrTimeout) break;
      if (tma::global_ns() - t0 > limit_ns) {
        atomicOr(err, kErrTimeout);
        break;
      }
    }
  }
  asm volatile("fence.proxy.async;" ::: "memory");
}

}  // namespace wall
}  // namespace lbm
