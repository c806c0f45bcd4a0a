// The fused per-node pass of one time step (Sec. 2.1, Sec. 3.2):
//   density and velocity (Eq. 5), pseudopotential force (Eq. 16) from psi of the 8 neighbours,
//   BGK collision with Guo forcing (Eqs. 2, 4), streaming (Eq. 3).
//
// Layout: two lattices of 9 planes [a][j][i] (structure of arrays).  The source lattice holds
// f(x, t) at x; each fluid node writes f*_a(x, t) to x + e_a of the destination lattice (push),
// including into solid nodes, whose slots then hold the outgoing populations the boundary pass
// reads.  Every population is read once and written once per step.
//
// A CTA covers a 32 x (8 RY) tile; each thread keeps the 9 populations of its RY nodes in
// registers.  psi of the tile and of a one-node ring around it goes to shared memory (ring nodes
// recompute their density from their own 9 populations), so the force needs no second pass over
// memory.  RY = 4 rows per thread for FP32 arithmetic, 2 for FP64 (register budget).  Lattices that
// do not fill the GPU so take smaller tiles (pick_step_tiles).
#include "step_core.cuh"

namespace lbm {

namespace {

using namespace step_core;

// CTAs per SM the tile kernels are compiled for (register budget 65536 / (256 x this)), as
// measured on the batched workload: FP32 storage, 3 for 32-row tiles (at 4 they spill; 5% slower)
// and 4 for shorter ones; FP16 storage, 4 (at 3 its 32-row tiles ran 11% slower); FP64, 2.
template <typename S, int RY>
constexpr int tile_ctas() {
  return sizeof(S) == 8 ? 2 : (sizeof(S) == 4 && RY == 4 ? 3 : 4);
}

// TXN x TYN threads, RY rows per thread.
template <typename S, int EOS, bool FIELDS, int TXN, int TYN, int RY>
__global__ void __launch_bounds__(TXN* TYN, tile_ctas<S, RY>() * (TX * TYT) / (TXN * TYN))
    step_kernel(DevParams p, const void* __restrict__ fa, void* __restrict__ fb,
                const uint8_t* __restrict__ flags, double* __restrict__ rho_m,
                double* __restrict__ ux_m, double* __restrict__ uy_m) {
  using C = typename StoreTraits<S>::C;
  __shared__ C psi_s[TYN * RY + 2][TXN + 2];
  step_tile<S, EOS, FIELDS, RY, TYN, TXN, true>(p, fa, fb, flags, rho_m, ux_m, uy_m,
                                                blockIdx.x * TXN, blockIdx.y * TYN * RY, psi_s);
}

// The same tile, whose source lattice has not had its wall pass yet (WallIn).  MODE: step_tile's WALL;
// 1 may use 128 registers (the CTAs of a small lattice do not fill the SMs anyway).
template <typename S, int EOS, int TXN, int TYN, int RY, int MODE>
__global__ void __launch_bounds__(TXN* TYN,
                                  (MODE == 1 ? 2 : tile_ctas<S, RY>()) * (TX * TYT) / (TXN * TYN))
    step_wall_kernel(const __grid_constant__ DevParams p, const void* __restrict__ fa,
                     void* __restrict__ fb, const uint8_t* __restrict__ flags,
                     double* __restrict__ rho_m, double* __restrict__ ux_m,
                     double* __restrict__ uy_m, const __grid_constant__ WallIn wi) {
  using C = typename StoreTraits<S>::C;
  __shared__ C psi_s[TYN * RY + 2][TXN + 2];
  extern __shared__ __align__(16) unsigned char wall_smem[];
  step_tile<S, EOS, false, RY, TYN, TXN, true, MODE>(
      p, fa, fb, flags, rho_m, ux_m, uy_m, blockIdx.x * TXN, blockIdx.y * TYN * RY, psi_s, &wi,
      blockIdx.y * gridDim.x + blockIdx.x, wall_smem);
}

// Many lattices in one launch: a persistent grid works through a queue of tiles (domain, x0,
// y0).  With claim == nullptr each CTA takes every gridDim.x-th tile; otherwise CTAs claim the
// next tile from the device counter *claim (reset to 0 by the advance kernel after every step),
// one atomic per tile, taken while the previous tile is still being worked on.  Tiles of domains
// whose step budget is spent are skipped.  RY (rows per thread, so the tile height 8 RY) and the
// queue are chosen by the batch's tuner.
template <typename S, int EOS, int RY>
__global__ void __launch_bounds__(TX* TYT, tile_ctas<S, RY>())
    batch_step_kernel(const BatchDomain* __restrict__ doms, const int4* __restrict__ tiles,
                      const int* __restrict__ n_tiles, int* __restrict__ claim) {
  using C = typename StoreTraits<S>::C;
  __shared__ C psi_s[TYT * RY + 2][TX + 2];
  __shared__ int next_s[2];  // claimed tiles, double-buffered across the end-of-tile barrier
  const bool lead = threadIdx.x == 0 && threadIdx.y == 0;
  const int nt = *n_tiles;
  int t = blockIdx.x;
  if (claim) {
    if (lead) next_s[0] = atomicAdd(claim, 1);
    __syncthreads();
    t = next_s[0];
  }
  for (int k = 1; t < nt; ++k) {
    if (claim && lead) next_s[k & 1] = atomicAdd(claim, 1);
    const int4 tile = tiles[t];  // (domain, x0, y0, -)
    const BatchDomain& D = doms[tile.x];
    if (D.steps_left > 0) {
      const int cur = D.cur;
      step_tile<S, EOS, false, RY>(D.p, D.f[cur], D.f[cur ^ 1], D.flags, D.rho_m, D.ux_m,
                                   D.uy_m, tile.y, tile.z, psi_s);
    }
    __syncthreads();  // psi_s is reused by the next tile; next_s[k & 1] is visible
    t = claim ? next_s[k & 1] : t + gridDim.x;
  }
}


template <typename S, int EOS, int TXN, int TYN, int RY>
cudaError_t launch_shape(const DevParams& p, const void* fa, void* fb, const uint8_t* flags,
                         double* rho_m, double* ux_m, double* uy_m, bool fields_only,
                         cudaStream_t s) {
  constexpr int TH = TYN * RY;
  const dim3 block(TXN, TYN), grid((p.nx + TXN - 1) / TXN, (p.ny + TH - 1) / TH);
  if (fields_only) {
    step_kernel<S, EOS, true, TXN, TYN, RY>
        <<<grid, block, 0, s>>>(p, fa, fb, flags, rho_m, ux_m, uy_m);
    return cudaGetLastError();
  }
  return launch_pdl(step_kernel<S, EOS, false, TXN, TYN, RY>, grid, block, s, p, fa, fb, flags,
                    rho_m, ux_m, uy_m);
}

template <typename S, int EOS>
cudaError_t launch_t(const DevParams& p, const void* fa, void* fb, const uint8_t* flags,
                     double* rho_m, double* ux_m, double* uy_m, bool fields_only,
                     cudaStream_t s) {
  // (FP64 without psi has no ring to share: one row a thread, 2048^2 525 against 545 us)
  constexpr int RY = sizeof(S) == 8 && EOS == LBM_EOS_NONE ? 1 : StoreTraits<S>::RY;
  return launch_shape<S, EOS, TX, TYT, RY>(p, fa, fb, flags, rho_m, ux_m, uy_m, fields_only, s);
}

template <typename S>
cudaError_t launch_s(const DevParams& p, const void* fa, void* fb, const uint8_t* flags,
                     double* rho_m, double* ux_m, double* uy_m, bool fields_only,
                     cudaStream_t s) {
  switch (p.eos) {
    case LBM_EOS_EXP:
      return launch_t<S, LBM_EOS_EXP>(p, fa, fb, flags, rho_m, ux_m, uy_m, fields_only, s);
    case LBM_EOS_CS:
      return launch_t<S, LBM_EOS_CS>(p, fa, fb, flags, rho_m, ux_m, uy_m, fields_only, s);
    default:
      return launch_t<S, LBM_EOS_NONE>(p, fa, fb, flags, rho_m, ux_m, uy_m, fields_only, s);
  }
}

template <typename S, int EOS, int TXN, int TYN, int RY, int MODE>
cudaError_t launch_wall_shape(const DevParams& p, const void* fa, void* fb, const uint8_t* flags,
                              double* rho_m, double* ux_m, double* uy_m, const WallIn* wi,
                              cudaStream_t s) {
  constexpr int TH = TYN * RY;
  const dim3 block(TXN, TYN), grid((p.nx + TXN - 1) / TXN, (p.ny + TH - 1) / TH);
  if (!wi)
    return launch_pdl(step_kernel<S, EOS, false, TXN, TYN, RY>, grid, block, s, p, fa, fb, flags,
                      rho_m, ux_m, uy_m);
  const size_t smem = wall::tile_wall_bytes<typename Pop<S>::C>(wi->max_links, wi->max_nodes,
                                                                (TXN + 2) * (TH + 2));
  return launch_pdl_smem(step_wall_kernel<S, EOS, TXN, TYN, RY, MODE>, grid, block, smem, s, p, fa, fb,
                         flags, rho_m, ux_m, uy_m, *wi);
}

struct TileShape {
  int w, ty, ry, mode;  // threads in x and y, rows per thread, step_tile's WALL
};
constexpr TileShape kShapes[] = {{16, 4, 1, 1}, {16, 8, 1, 1}, {32, 8, 1, 1},
                                 {32, 8, 1, 2}, {32, 8, 2, 2}, {32, 8, 4, 2}};
// Whether pick_step_tiles gives shape k to lattices of a format with or without psi; the others are not
// compiled.
template <typename S, int EOS>
constexpr bool shape_taken(int k) {
  constexpr bool psi = EOS != LBM_EOS_NONE;
  if (sizeof(S) == 8) return k == 0 || k == 1 || (psi && k == 4);
  return k == 2 || (psi && k == 3) || k == 4 || (sizeof(S) == 4 && k == 5);
}

template <typename S, int EOS>
cudaError_t launch_tiles_t(int shape, const DevParams& p, const void* fa, void* fb,
                           const uint8_t* flags, double* rho_m, double* ux_m, double* uy_m,
                           const WallIn* wi, cudaStream_t s) {
#define LBM_SHAPE(k)                                                                           \
  if constexpr (shape_taken<S, EOS>(k))                                                        \
    if (shape == k)                                                                            \
      return launch_wall_shape<S, EOS, kShapes[k].w, kShapes[k].ty, kShapes[k].ry, kShapes[k].mode>( \
          p, fa, fb, flags, rho_m, ux_m, uy_m, wi, s)
  LBM_SHAPE(0);
  LBM_SHAPE(1);
  LBM_SHAPE(2);
  LBM_SHAPE(3);
  LBM_SHAPE(4);
  LBM_SHAPE(5);
#undef LBM_SHAPE
  return cudaErrorInvalidValue;
}

template <typename S>
cudaError_t launch_tiles_s(int shape, const DevParams& p, const void* fa, void* fb,
                           const uint8_t* flags, double* rho_m, double* ux_m, double* uy_m,
                           const WallIn* wi, cudaStream_t s) {
  switch (p.eos) {
    case LBM_EOS_EXP:
      return launch_tiles_t<S, LBM_EOS_EXP>(shape, p, fa, fb, flags, rho_m, ux_m, uy_m, wi, s);
    case LBM_EOS_CS:
      return launch_tiles_t<S, LBM_EOS_CS>(shape, p, fa, fb, flags, rho_m, ux_m, uy_m, wi, s);
    default:
      return launch_tiles_t<S, LBM_EOS_NONE>(shape, p, fa, fb, flags, rho_m, ux_m, uy_m, wi, s);
  }
}

template <typename S, int EOS, int RY>
cudaError_t launch_batch_t(const BatchDomain* doms, const int4* tiles, const int* n_tiles,
                           int* claim, int grid, cudaStream_t s) {
  batch_step_kernel<S, EOS, RY><<<grid, dim3(TX, TYT), 0, s>>>(doms, tiles, n_tiles, claim);
  return cudaGetLastError();
}

template <typename S, int RY>
cudaError_t launch_batch_e(int eos, const BatchDomain* doms, const int4* tiles, const int* n_tiles,
                           int* claim, int grid, cudaStream_t s) {
  switch (eos) {
    case LBM_EOS_EXP:
      return launch_batch_t<S, LBM_EOS_EXP, RY>(doms, tiles, n_tiles, claim, grid, s);
    case LBM_EOS_CS: return launch_batch_t<S, LBM_EOS_CS, RY>(doms, tiles, n_tiles, claim, grid, s);
    default: return launch_batch_t<S, LBM_EOS_NONE, RY>(doms, tiles, n_tiles, claim, grid, s);
  }
}

template <typename S>
cudaError_t launch_batch_s(int eos, int ry, const BatchDomain* doms, const int4* tiles,
                           const int* n_tiles, int* claim, int grid, cudaStream_t s) {
  if (ry == 1) return launch_batch_e<S, 1>(eos, doms, tiles, n_tiles, claim, grid, s);
  if (ry == 2) return launch_batch_e<S, 2>(eos, doms, tiles, n_tiles, claim, grid, s);
  if constexpr (sizeof(typename Pop<S>::C) == 4) {
    if (ry == 4) return launch_batch_e<S, 4>(eos, doms, tiles, n_tiles, claim, grid, s);
  }
  return cudaErrorInvalidValue;
}

template <typename S>
int batch_grid_s(int eos, int ry) {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const void* fn = nullptr;
  auto pick = [&](auto k) { fn = reinterpret_cast<const void*>(k); };
  if (ry == 1) pick(batch_step_kernel<S, LBM_EOS_CS, 1>);
  else if (ry == 2) pick(batch_step_kernel<S, LBM_EOS_CS, 2>);
  else if constexpr (sizeof(typename Pop<S>::C) == 4) pick(batch_step_kernel<S, LBM_EOS_CS, 4>);
  if (!fn || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, TX * TYT, 0) != cudaSuccess) {
    cudaGetLastError();
    per = 2;
  }
  (void)eos;
  return sms * (per > 0 ? per : 1);
}

}  // namespace

int batch_tile_rows(int ry) { return TYT * ry; }
int batch_tile_cols() { return TX; }

int batch_step_grid(int precision, int eos, int ry) {
  if (precision == LBM_FP32_DEV) return batch_grid_s<float>(eos, ry);
  if (precision == LBM_FP16_DEV) return batch_grid_s<__half>(eos, ry);
  return batch_grid_s<double>(eos, ry);
}

cudaError_t launch_batch_step(int precision, int eos, int ry, const BatchDomain* doms,
                              const int4* tiles, const int* n_tiles, int* claim, int grid,
                              cudaStream_t s) {
  if (precision == LBM_FP32_DEV)
    return launch_batch_s<float>(eos, ry, doms, tiles, n_tiles, claim, grid, s);
  if (precision == LBM_FP16_DEV)
    return launch_batch_s<__half>(eos, ry, doms, tiles, n_tiles, claim, grid, s);
  return launch_batch_s<double>(eos, ry, doms, tiles, n_tiles, claim, grid, s);
}

// By nodes per SM (152), from us a step with the wall pass inside the step kernel / apart from it
// (vector kernel, or scalar tiles where the width or format asks for them), droplet on a cylinder
// (single phase in brackets):
//   FP32  100^2 4.5 / 6.2 (4.2 / 5.0)   345^2 5.3 / 6.4 (4.6 / 5.6)   512^2 7.0 / 7.9 (5.8 / 6.3)
//         724^2 9.2 / 12.2 (7.9 / 8.0)  1024^2 15.1 / 18.0 (11.3 / 11.2)  1448^2 33.7 / 36.1
//         2048^2 61.6 / 58.0            2047^2 61.7 / 64.2 (scalar tiles apart)
//   FP16  345^2 5.7 / 8.0               1024^2 16.7 / 16.9            2047^2 63.6 / 62.6
//   FP64  100^2 9.7 / 21.7 (6.7 / 15.2) 300x350 30.1 / 39.8 (17.6 / 26.8)  1024^2 225.6 / 228.8
// (The same in the vector kernel's tiles lost where it is the faster one: its registers leave no room,
// 4096^2 FP32 207.9 / 199.9, FP16 192.4 / 187.8, single-phase FP16 139.1 / 124.1.)
// Few nodes want small tiles, so that every SM has some: FP64 100^2 9.7 (16 x 4), 9.9 (16 x 8), 13.5
// (32 x 8), 22.7 us (32 x 16); 600^2 94.8, 84.6, 83.6, 86.0 us; FP32 400^2 6.1 (32 x 8, walls
// inline), 6.7 (apart), 7.0 us (32 x 16), 600^2 10.0, 8.7, 8.1 us.
int pick_step_tiles(int precision, int eos, int nx, int ny, int* tw, int* th) {
  const long long per_sm = ((long long)nx * ny + 151) / 152;
  const bool psi = eos != LBM_EOS_NONE, vec = step_vec_supported(precision, nx, ny);
  int shape = -1;
  if (precision == LBM_FP64) {
    if (per_sm <= (psi ? 256 : 1024)) shape = 0;
    else if (!psi || per_sm <= 2560) shape = 1;
    else shape = 4;
    // a second set of FP64 moments is 24 bytes a node: only where a step is short
    if (per_sm > 16384) shape = -1;
  } else if (per_sm <= (psi ? 1280 : (precision == LBM_FP16_DEV ? 2048 : 2560))) {
    shape = 2;
  } else if (psi || !vec) {
    if (psi && per_sm <= 2048) shape = 3;
    else if (per_sm <= 8192) shape = 4;
    else if (precision == LBM_FP32_DEV) shape = !vec || per_sm <= 16384 ? 5 : -1;
    else shape = !vec && per_sm <= 16384 ? 4 : -1;
  }
  if (shape < 0) return -1;
  *tw = kShapes[shape].w;
  *th = kShapes[shape].ty * kShapes[shape].ry;
  return shape;
}

bool tiles_do_ends(int shape) { return shape >= 0 && kShapes[shape].mode == 1; }

cudaError_t launch_step_tiles(int shape, int precision, const DevParams& p, const void* fa,
                              void* fb, const uint8_t* flags, double* rho_m, double* ux_m,
                              double* uy_m, const WallIn* wi, cudaStream_t s) {
  if (precision == LBM_FP32_DEV)
    return launch_tiles_s<float>(shape, p, fa, fb, flags, rho_m, ux_m, uy_m, wi, s);
  if (precision == LBM_FP16_DEV)
    return launch_tiles_s<__half>(shape, p, fa, fb, flags, rho_m, ux_m, uy_m, wi, s);
  return launch_tiles_s<double>(shape, p, fa, fb, flags, rho_m, ux_m, uy_m, wi, s);
}

// Every lattice of the marching kernel, and the single-phase FP32 ones that the vector kernel takes, at
// every size the tiles above leave.  Single phase, us a step in front / apart, one cylinder of r = nx/80
// (r = 0.15 of the side):
//             640^2                   1024^2                    1600 x 1000               2048^2
//   closed    7.1 / 6.9 (7.6 / 7.1)   9.7 / 11.1 (11.3 / 11.3)  17.1 / 18.7 (17.7 / 19.0) 46.2 / 49.2 (47.1 / 50.4)
//   channel   12.7 / 8.7 (13.8 / 9.4) 16.2 / 13.3 (19.0 / 13.5) 20.2 / 21.5 (21.9 / 21.6) 49.8 / 51.9 (50.8 / 55.0)
// So a closed lattice gains from about 0.6 M nodes on (large cylinder: 1 M), and a channel only from about
// 1.5 M (large cylinder: between 2 and 4 M): its inlet is FP64 work of ny rows, which the front's few
// 256-thread CTAs do on as few SMs (by itself it runs in one-warp CTAs).  Below that the rule is not the fastest; all of these are faster than three launches
// in plain stream order (channels 15.5, 20.1, 29.6, 60.2).
bool step_front_supported(int precision, int eos, int nx, int ny, const void* f0, const void* f1) {
  MarchMaps maps;
  if (step_march_supported(precision, eos, nx, ny))
    return make_march_maps(&maps, f0, nx, ny) && make_march_maps(&maps, f1, nx, ny);
  return precision == LBM_FP32_DEV && eos == LBM_EOS_NONE && step_vec_supported(precision, nx, ny);
}

cudaError_t launch_step_front(int precision, const DevParams& p, const void* fa, void* fb,
                              const uint8_t* flags, double* rho_m, double* ux_m, double* uy_m,
                              FrontWalls front, int* err, cudaStream_t s) {
  if (step_march_supported(precision, p.eos, p.nx, p.ny)) {
    MarchMaps maps;
    if (!make_march_maps(&maps, fa, p.nx, p.ny)) return cudaErrorNotSupported;
    return launch_step_march(maps, p, fa, fb, flags, rho_m, ux_m, uy_m, err, s, &front);
  }
  return launch_step_vec(precision, p, fa, fb, flags, rho_m, ux_m, uy_m, false, s, true, err,
                         &front);
}

cudaError_t launch_step(int precision, const DevParams& p, const void* fa, void* fb,
                        const uint8_t* flags, double* rho_m, double* ux_m, double* uy_m,
                        bool fields_only, cudaStream_t s, int path, int* err) {
  MarchMaps maps;
  if ((path == 0 || path == 4) && !fields_only && err &&
      step_march_supported(precision, p.eos, p.nx, p.ny) &&
      make_march_maps(&maps, fa, p.nx, p.ny))
    return launch_step_march(maps, p, fa, fb, flags, rho_m, ux_m, uy_m, err, s);
  // FP64 is bound by the FP64 pipe, where the scalar tiling (fewer ring psi per node) is faster
  const bool vec = path == 3 || ((path == 0 || path == 4) && precision != LBM_FP64);
  if (vec && step_vec_supported(precision, p.nx, p.ny))
    return launch_step_vec(precision, p, fa, fb, flags, rho_m, ux_m, uy_m, fields_only, s,
                           (path == 0 || path == 4) && err != nullptr, err);
  if (precision == LBM_FP32_DEV)
    return launch_s<float>(p, fa, fb, flags, rho_m, ux_m, uy_m, fields_only, s);
  if (precision == LBM_FP16_DEV)
    return launch_s<__half>(p, fa, fb, flags, rho_m, ux_m, uy_m, fields_only, s);
  return launch_s<double>(p, fa, fb, flags, rho_m, ux_m, uy_m, fields_only, s);
}

}  // namespace lbm
