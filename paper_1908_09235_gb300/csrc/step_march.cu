// The fused per-node pass of one time step (as csrc/step_vec.cu: the same per-node arithmetic, the
// same bits) for large two-phase lattices in FP16 deviations, by warps that march up strips.
//
// A CTA is one warp.  It owns a strip of 128 columns and kRows rows, four consecutive nodes per lane,
// and goes through its rows one by one: psi of row y + 1 from the row just arrived, collision of row
// y with psi of rows y - 1, y, y + 1 in registers, streaming of row y.  No CTA barrier stands between
// loads and arithmetic, neighbours in x come by two shuffles per row, and there is no psi ring to
// stage and index: 222 thread instructions per fluid node (2048^2) against the vector kernel's 273, whose
// issue bounded the FP16 step (40 B per node, 0.5 of HBM).  Rows arrive in kSlots shared-memory slots by tensor copies
// (two per row, issued by one lane; every wait is bounded), so the loads in flight cost no registers.  psi of the columns
// beside the strip is computed at the start, one (row, side) per lane.
//
// Strips are short: the first and last row's neighbours cost (kRows + 2) / kRows of the psi work, but
// the rows that the resident warps have in work should lie close together in memory.  4096^2, us a
// step without walls, rows 4 / 5 / 6 / 7 / 8 / 10 / 28: 158 / 154 / 151 / 150 / 153 / 157 / 191 (the
// vector kernel 183); 2048^2 46.9 / 46.1 / 47.1 / 46.6 / 48.2 / 50.5 / 64 (50).  Two slots: 154, four:
// 158; at most 12 warps an SM: 165; the loop unrolled over the three slots, which saves its moves but
// not the instruction cache: 184.  FP32 deviations the same way: 201-220 against 195 us, so not theirs.
#include "step_core.cuh"
#include "tma.cuh"
#include "wall_front.cuh"

namespace lbm {

namespace {

using namespace step_core;

constexpr int SWD = 128;               // strip width
constexpr int kRows = 7;               // rows of a strip
constexpr int kMaxRows = 14;           // two sides of kMaxRows + 2 rows fit the lanes of a warp
constexpr int kSlots = 3;              // rows in shared memory: y, y + 1 and one on its way
constexpr int kWarps = 14;             // resident warps per SM the registers allow for
constexpr int kRowBytes = SWD * 4 + 8 * SWD * 2;  // the FP32 rest plane, then eight FP16 planes
static_assert(kRows <= kMaxRows, "side psi in one register");

// the lane's four values of plane a in a slot
__device__ __forceinline__ void read4(const unsigned char* s, int a, int lane, float (&o)[4]) {
  if (a == 0) {
    const float4 v = *reinterpret_cast<const float4*>(s + lane * 16);
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
  } else {
    const uint2 u = *reinterpret_cast<const uint2*>(s + SWD * 4 + (a - 1) * SWD * 2 + lane * 8);
    const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
    const float2 hi = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
    o[0] = lo.x; o[1] = lo.y; o[2] = hi.x; o[3] = hi.y;
  }
}

// Stores of values already rounded to the format (n % 4 == 0 for four, even for two; two and one:
// moving planes).
__device__ __forceinline__ __half* moving_at(void* b, int a, int N, int n) {
  return Pop<__half>::moving(b, N) + (a - 1) * N + n;
}
__device__ __forceinline__ void store4(void* b, int a, int N, int n, float v0, float v1, float v2,
                                       float v3) {
  n = LBM_CHK(n, N - 3);
  if (a == 0) {
    *reinterpret_cast<float4*>(static_cast<float*>(b) + n) = make_float4(v0, v1, v2, v3);
  } else {
    const __half2 lo = __floats2half2_rn(v0, v1), hi = __floats2half2_rn(v2, v3);
    uint2 u;
    u.x = *reinterpret_cast<const uint32_t*>(&lo);
    u.y = *reinterpret_cast<const uint32_t*>(&hi);
    *reinterpret_cast<uint2*>(moving_at(b, a, N, n)) = u;
  }
}
__device__ __forceinline__ void store2(void* b, int a, int N, int n, float v0, float v1) {
  *reinterpret_cast<__half2*>(moving_at(b, a, N, LBM_CHK(n, N - 1))) = __floats2half2_rn(v0, v1);
}
__device__ __forceinline__ void store1(void* b, int a, int N, int n, float v) {
  *moving_at(b, a, N, LBM_CHK(n, N)) = __float2half_rn(v);
}

// FRONT: the first block rows are the wall pass of the step before (csrc/wall_front.cuh).
template <int EOS, bool FRONT>
__global__ void __launch_bounds__(32, kWarps)
    step_march_kernel(const __grid_constant__ DevParams p, const void* fa, void* __restrict__ fb,
                      const uint8_t* __restrict__ flags, float* __restrict__ rho_m,
                      float* __restrict__ ux_m, float* __restrict__ uy_m,
                      const __grid_constant__ CUtensorMap map,
                      const __grid_constant__ CUtensorMap map2, int* __restrict__ err,
                      const __grid_constant__ FrontWalls front) {
  using S = __half;
  using L = float2;
  constexpr int R = kSlots;
  __shared__ __align__(128) unsigned char slots[R][kRowBytes];
  __shared__ __align__(8) uint64_t bars[R];
  const int lane = threadIdx.x;
  const int nx = p.nx, ny = p.ny, N = p.N;
  const Consts<float>& k = p.cf;
  const float rho_ref = k.rho_ref, psi_w = k.psi_wall;
  int by = blockIdx.y, strips = gridDim.y;
  if constexpr (FRONT) {
    if (by < front.rows) {
      wall::front_cta<S>(p, front, flags, by * gridDim.x + blockIdx.x, lane, 32);
      return;
    }
    by -= front.rows;
    strips -= front.rows;
  }
  const int x0 = blockIdx.x * SWD;
  // rows y0 .. y1 - 1 (the strips' heights differ by one at most)
  const int y0 = (int)((long long)by * ny / strips);
  const int y1 = (int)((long long)(by + 1) * ny / strips);
  const int nv = min(32, (nx - x0) >> 2);  // lanes with nodes inside the lattice
  const bool lane_ok = lane < nv, first = lane == 0, last = lane == nv - 1;
  const int col = x0 + 4 * (lane_ok ? lane : 0);
  const int col_l = x0 == 0 ? nx - 1 : x0 - 1, col_r = x0 + 4 * nv == nx ? 0 : x0 + 4 * nv;
  auto wrapy = [ny](int y) { return y < 0 ? y + ny : (y >= ny ? y - ny : y); };

  if (lane == 0) {
    for (int s = 0; s < R; ++s) tma::mbar_init(&bars[s], 1);
    tma::fence_mbar_init();
  }
  __syncwarp();
  // flags of the rows a step ahead (fixed data)
  auto row_flags = [&](int y) {
    return *reinterpret_cast<const uint32_t*>(flags + LBM_CHK(wrapy(y) * nx + col, N - 3));
  };
  uint32_t fl_c = row_flags(y0 - 1), fl_n = row_flags(y0);
  pdl_wait();
  if constexpr (FRONT) {
    if (wall::front_touches(front, x0, y0, SWD, y1 - y0, nx, ny)) {
      if (lane == 0) wall::front_wait(front, err);
      __syncwarp();
    }
  }
  // row y goes to slot (y - y0 + 1) % R
  auto fetch = [&](int y, int s) {
    if (lane == 0) {
      tma::mbar_expect_tx(&bars[s], kRowBytes);
      tma::tma_load_2d(slots[s], &map, &bars[s], x0, wrapy(y));
      tma::tma_load_3d(slots[s] + SWD * 4, &map2, &bars[s], x0, wrapy(y), 0);
    }
  };
  for (int s = 0; s < R; ++s)
    if (y0 - 1 + s <= y1) fetch(y0 - 1 + s, s);

  // psi beside the strip: lane 2 r + side has row y0 - 1 + r (kMaxRows + 2 rows)
  float side = 0.f;
  if (y0 - 1 + (lane >> 1) <= y1) {
    const int n = wrapy(y0 - 1 + (lane >> 1)) * nx + (lane & 1 ? col_r : col_l);
    float g[9];
#pragma unroll
    for (int a = 0; a < 9; ++a) g[a] = Pop<S>::load(fa, a, N, n);
    side = (flags[LBM_CHK(n, N)] & FLAG_SOLID) ? psi_w
                                               : psi_of<float, EOS>(k, density_of<true, EOS>(rho_ref, g));
  }

  // psi of a row: [0] left neighbour, [1 .. 4] own, [5] right neighbour; and the own densities
  uint32_t phase = 0;
  bool ok = true;
  auto psi_row = [&](int r, int s, uint32_t fl, float (&ps)[6], L (&rho)[2]) {
    // (after one wait that gave up, the rest of the copies in flight get a short one)
    ok = tma::mbar_wait_bounded(&bars[s], (phase >> s) & 1u, ok ? tma::kWaitNs : 1000000ull) && ok;
    phase ^= 1u << s;
    L sum[2];
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      float t[4];
      read4(slots[s], a, lane, t);
      const L lo = make_float2(t[0], t[1]), hi = make_float2(t[2], t[3]);
      sum[0] = a == 0 ? lo : r_add(sum[0], lo);
      sum[1] = a == 0 ? hi : r_add(sum[1], hi);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) rho[q] = r_add(splat<L>(rho_ref), sum[q]);
    const bool solids = __any_sync(0xffffffffu, fl & 0x01010101u * FLAG_SOLID);
    if (solids) {
      if (fl & FLAG_SOLID) rho[0].x = 1.f;
      if (fl >> 8 & FLAG_SOLID) rho[0].y = 1.f;
      if (fl >> 16 & FLAG_SOLID) rho[1].x = 1.f;
      if (fl >> 24 & FLAG_SOLID) rho[1].y = 1.f;
    }
    const L a = psi_of<float, EOS>(k, rho[0]), b = psi_of<float, EOS>(k, rho[1]);
    ps[1] = a.x; ps[2] = a.y; ps[3] = b.x; ps[4] = b.y;
    if (solids) {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (fl >> (8 * e) & FLAG_SOLID) ps[1 + e] = psi_w;
    }
    ps[0] = __shfl_up_sync(0xffffffffu, ps[4], 1);
    ps[5] = __shfl_down_sync(0xffffffffu, ps[1], 1);
    const float beside = __shfl_sync(0xffffffffu, side, 2 * r + (first ? 0 : 1));
    if (first) ps[0] = beside;
    if (nv == 1) {  // one lane: both sides
      const float right = __shfl_sync(0xffffffffu, side, 2 * r + 1);
      if (last) ps[5] = right;
    } else if (last) {
      ps[5] = beside;
    }
  };

  float pm[6], pc[6], pp[6];
  L rc[2], rn[2];
  psi_row(0, 0, fl_c, pm, rc);  // row y0 - 1: psi only
  psi_row(1, 1 % R, fl_n, pc, rc);
  fl_c = fl_n;
  fl_n = row_flags(y0 + 1);
  // slot 0 is free
  int free_row = y0 - 1 + R;  // next row to fetch
  __syncwarp();
  if (free_row <= y1) {
    if (lane == 0) tma::fence_proxy_async();
    fetch(free_row, 0);
  }
  ++free_row;
  int sc = 1 % R;  // slot of row y
  for (int y = y0; y < y1; ++y) {
    const int sn = sc + 1 == R ? 0 : sc + 1;
    psi_row(y + 2 - y0, sn, fl_n, pp, rn);
    const uint32_t fl_a = y + 2 <= y1 ? row_flags(y + 2) : 0u;
    // row y's populations; its slot is free then
    L f[2][9];
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      float t[4];
      read4(slots[sc], a, lane, t);
      f[0][a] = make_float2(t[0], t[1]);
      f[1][a] = make_float2(t[2], t[3]);
    }
    __syncwarp();
    if (free_row <= y1) {
      if (lane == 0) tma::fence_proxy_async();
      fetch(free_row, sc);
    }
    ++free_row;
    if (free_row == y1 + 1) pdl_trigger();
    const bool macros = __any_sync(0xffffffffu, lane_ok && (fl_c & 0x01010101u * FLAG_MACRO));
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int c = 1 + 2 * q;  // index of the pair's first node in a psi row
      const L d13 = make_float2(r_sub(pc[c + 1], pc[c - 1]), r_sub(pc[c + 2], pc[c]));
      const L d24 = r_sub(make_float2(pp[c], pp[c + 1]), make_float2(pm[c], pm[c + 1]));
      const L d57 = make_float2(r_sub(pp[c + 1], pm[c - 1]), r_sub(pp[c + 2], pm[c]));
      const L d86 = make_float2(r_sub(pm[c + 1], pp[c - 1]), r_sub(pm[c + 2], pp[c]));
      const float x = float(col + 2 * q);
      L st[9], ux, uy;
      collide_node<S, EOS, L>(p, k, f[q], rc[q], rc[q], d13, d24, d57, d86,
                              make_float2(pc[c], pc[c + 1]), make_float2(x, x + 1.f),
                              splat<L>(float(y)), st, ux, uy);
      if (macros) {  // for the wall pass
#pragma unroll
        for (int e = 0; e < 2; ++e)
          if (lane_ok && (fl_c >> (16 * q + 8 * e) & FLAG_MACRO)) {
            const int n = LBM_CHK(y * nx + col + 2 * q + e, N);
            rho_m[n] = e ? rc[q].y : rc[q].x;
            ux_m[n] = e ? ux.y : ux.x;
            uy_m[n] = e ? uy.y : uy.x;
          }
      }
#pragma unroll
      for (int a = 0; a < 9; ++a) f[q][a] = st[a];
    }
    // streaming: whole vectors of the destination columns the strip owns; at its edges partial ones
    // and single elements into the neighbouring strips' columns
    const int row0 = y * nx, rowp = (y + 1 == ny ? 0 : y + 1) * nx,
              rowm = (y == 0 ? ny - 1 : y - 1) * nx;
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      const int d = ey(a) > 0 ? rowp : (ey(a) < 0 ? rowm : row0);
      const float v0 = f[0][a].x, v1 = f[0][a].y, v2 = f[1][a].x, v3 = f[1][a].y;
      if (ex(a) == 0) {
        if (lane_ok) store4(fb, a, N, d + col, v0, v1, v2, v3);
      } else if (ex(a) > 0) {
        const float in = __shfl_up_sync(0xffffffffu, v3, 1);
        if (lane_ok && !first) store4(fb, a, N, d + col, in, v0, v1, v2);
        if (first) {
          store1(fb, a, N, d + col + 1, v0);
          store2(fb, a, N, d + col + 2, v1, v2);
        }
        if (last) store1(fb, a, N, d + col_r, v3);
      } else {
        const float in = __shfl_down_sync(0xffffffffu, v0, 1);
        if (lane_ok && !last) store4(fb, a, N, d + col, v1, v2, v3, in);
        if (last) {
          store2(fb, a, N, d + col, v1, v2);
          store1(fb, a, N, d + col + 2, v3);
        }
        if (first) store1(fb, a, N, d + col_l, v0);
      }
    }
#pragma unroll
    for (int e = 0; e < 6; ++e) {
      pm[e] = pc[e];
      pc[e] = pp[e];
    }
    rc[0] = rn[0];
    rc[1] = rn[1];
    fl_c = fl_n;
    fl_n = fl_a;
    sc = sn;
  }
  // every copy issued has been waited for; a wait that gave up is reported
  if (__any_sync(0xffffffffu, !ok) && lane == 0) atomicOr(err, kErrTimeout);
}

// Self-test of the front's wait: one thread waits for w.ctas counts of w.done.
__global__ void front_wait_selftest_kernel(const __grid_constant__ FrontWalls w, int* err,
                                           unsigned long long limit_ns) {
  wall::front_wait(w, err, limit_ns);
}

template <int EOS>
cudaError_t launch_march_t(const MarchMaps& maps, const DevParams& p, const void* fa, void* fb, const uint8_t* flags,
                           double* rho_m, double* ux_m, double* uy_m, int* err, cudaStream_t s,
                           const FrontWalls* front) {
  const CUtensorMap& map = *reinterpret_cast<const CUtensorMap*>(maps.rest);
  const CUtensorMap& map2 = *reinterpret_cast<const CUtensorMap*>(maps.moving);
  dim3 grid((p.nx + SWD - 1) / SWD, (p.ny + kRows - 1) / kRows);
  if (!front)
    return launch_pdl(step_march_kernel<EOS, false>, grid, dim3(32), s, p, fa, fb, flags,
                      (float*)rho_m, (float*)ux_m, (float*)uy_m, map, map2, err, FrontWalls{});
  FrontWalls w = *front;
  w.wall_ctas = w.ctas = (8 * w.nb + 31) / 32;
  w.rows = (w.ctas + grid.x - 1) / grid.x;
  grid.y += w.rows;
  return launch_pdl(step_march_kernel<EOS, true>, grid, dim3(32), s, p, fa, fb, flags,
                    (float*)rho_m, (float*)ux_m, (float*)uy_m, map, map2, err, w);
}

}  // namespace

// From the size on where the scalar tiles, which do the wall pass too, stop being the faster ones
// (step.cu, pick_step_tiles); rows of 16 bytes.
bool step_march_supported(int precision, int eos, int nx, int ny) {
  return precision == LBM_FP16_DEV && eos != LBM_EOS_NONE && nx % 8 == 0 &&
         (long long)nx * ny > 152LL * 8192;
}

cudaError_t launch_front_wait_selftest(int* done, int target, int* err, unsigned long long limit_ns,
                                       cudaStream_t s) {
  FrontWalls w{};
  w.done = done;
  w.ctas = target;
  front_wait_selftest_kernel<<<1, 1, 0, s>>>(w, err, limit_ns);
  return cudaGetLastError();
}

bool make_march_maps(MarchMaps* maps, const void* fa, int nx, int ny) {
  static_assert(sizeof(MarchMaps) == 2 * sizeof(CUtensorMap), "a tensor map each");
  return make_ring_tensor_maps_fp16(maps->rest, maps->moving, fa, nx, ny, SWD, SWD);
}

cudaError_t launch_step_march(const MarchMaps& maps, const DevParams& p, const void* fa, void* fb, const uint8_t* flags,
                              double* rho_m, double* ux_m, double* uy_m, int* err, cudaStream_t s,
                              const FrontWalls* front) {
  if (p.eos == LBM_EOS_EXP)
    return launch_march_t<LBM_EOS_EXP>(maps, p, fa, fb, flags, rho_m, ux_m, uy_m, err, s, front);
  return launch_march_t<LBM_EOS_CS>(maps, p, fa, fb, flags, rho_m, ux_m, uy_m, err, s, front);
}

}  // namespace lbm
