// Curved-wall pass of one time step (Sec. 2.2, Sec. 3.1, Sec. 4.1): for every boundary node x_b
// and every cut link a (x_s = x_b + e_a solid, fraction q), the unknown incoming population
// f_abar(x_b, t+1) from the time-t values, then the per-node leakage of Eq. (15) and the
// correction of scheme A (Eq. 18) or the fictitious density of scheme B (Eq. 22) / Bao (Eq. 23).
//
// With the push layout of the step kernel (destination lattice B, source lattice A) the time-t
// values of a link are found at:
//   f*_a(x_b)    = B_a(x_s)        (pushed into the solid slot)
//   f*_abar(x_b) = B_abar(x_f)     f*_a(x_f) = B_a(x_b)      f*_a(x_ff) = B_a(x_f)
//   f*_abar(x_f) = B_abar(x_ff)    f_a(x_b) (pre-collision) = A_a(x_b)
// with x_f = x_b - e_a and x_ff = x_b - 2 e_a; rho and u at x_b and x_f come from the step
// kernel's macro arrays.  The pass writes B_abar(x_b) and, for scheme A, B_0(x_b); none of the
// slots it reads is written by another link, so the pass is race-free.
//
// Everything that depends only on q, tau and the scheme (chi of Eqs. 9-11, u_s of Eq. 10, the
// weights of Eqs. 12-14, which operands a link reads) is evaluated once at creation by
// link_setup_kernel into a per-link recipe, with the same operations the equations state; a step
// then costs each link a few loads and FMAs.  An 8-lane group handles a boundary node, one lane
// per link; per-node sums use fixed-order shuffles (bitwise reproducible).  Link values are
// computed in the step's arithmetic type (FP64 for FP64 storage, FP32 for the deviation
// formats); each boundary node's mass bookkeeping is FP64 for every format.  (FP64 link
// arithmetic for the deviation formats was measured: 4.3 us more per step at 4096^2 and 0.25 ms
// more per batched step of 512 lattices, on GB300's narrow FP64 pipe.)
#include "wall.cuh"

namespace lbm {

namespace {

using namespace wall;

// One thread per boundary node: the recipe of each of its links.
__global__ void link_setup_kernel(DevParams p, int nb, const int32_t* __restrict__ bnode,
                                  const int32_t* __restrict__ boff,
                                  const uint8_t* __restrict__ ldir, const double* __restrict__ lq,
                                  const uint8_t* __restrict__ flags, LinkRecipe r) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nb) return;
  const int nx = p.nx, ny = p.ny, N = p.N, scheme = p.scheme;
  const double tau = p.tau;
  const int n = bnode[b];
  const int i = n % nx, j = n / nx;
  for (int l = boff[b]; l < boff[b + 1]; ++l) {
    const int a = ldir[l], ab = opposite(a);
    const double q = lq[l];
    const int ns = wrap_once(j + ey(a), ny) * nx + wrap_once(i + ex(a), nx);
    const int nf = wrap_once(j - ey(a), ny) * nx + wrap_once(i - ex(a), nx);
    const int nff = wrap_once(j - 2 * ey(a), ny) * nx + wrap_once(i - 2 * ex(a), nx);
    const bool f_solid = flags[LBM_CHK(nf, N)] & FLAG_SOLID;
    const bool ff_solid = flags[LBM_CHK(nff, N)] & FLAG_SOLID;
    double c0 = 1.0, c1 = 0.0, c2 = 0.0, chi = 0.0, cus = 0.0;  // default: halfway bounce-back
    int x1 = -1, x2 = -1, uf = -1;
    uint8_t kind = 0;
    switch (scheme) {
      case LBM_FH:
      case LBM_MLS:
      case LBM_MOD_A:
      case LBM_MOD_B:
      case LBM_BAO:
        if (q < 0.5) {
          if (scheme == LBM_FH) {  // Eq. (9): u_s = u_b
            chi = (2.0 * q - 1.0) / (tau - 1.0);
            cus = 1.0;
            kind = kGhost;
          } else if (!f_solid) {   // Eq. (11): u_s = u(x_f)
            chi = (2.0 * q - 1.0) / (tau - 2.0);
            uf = nf;
            kind = kGhost;
          }                        // x_f solid: halfway bounce-back for this link
        } else {                   // Eq. (10) with u_w = 0
          chi = (2.0 * q - 1.0) / tau;
          cus = (q - 1.0) / q;
          kind = kGhost;
        }
        if (kind & kGhost) c0 = 1.0 - chi;  // Eq. (7) / Eq. (17)
        break;
      case LBM_BOUZIDI_L:
      case LBM_BOUZIDI_L_A:  // Eq. (12)
        if (q < 0.5) {
          if (!f_solid) {
            c0 = 2.0 * q;
            c1 = 1.0 - 2.0 * q;
            x1 = a * N + n;
          }
        } else {
          c0 = 1.0 / (2.0 * q);
          c1 = (2.0 * q - 1.0) / (2.0 * q);
          x1 = ab * N + nf;
        }
        break;
      case LBM_BOUZIDI_Q:  // Eq. (13)
        if (q < 0.5) {
          if (!f_solid) {
            if (ff_solid) {  // x_ff solid: linear Bouzidi
              c0 = 2.0 * q;
              c1 = 1.0 - 2.0 * q;
              x1 = a * N + n;
            } else {
              c0 = q * (1.0 + 2.0 * q);
              c1 = 1.0 - 4.0 * q * q;
              x1 = a * N + n;
              c2 = -(q * (1.0 - 2.0 * q));
              x2 = a * N + nf;
            }
          }
        } else if (f_solid) {  // x_f solid: linear Bouzidi
          c0 = 1.0 / (2.0 * q);
          c1 = (2.0 * q - 1.0) / (2.0 * q);
          x1 = ab * N + nf;
        } else {
          c0 = 1.0 / (q * (2.0 * q + 1.0));
          c1 = (2.0 * q - 1.0) / q;
          x1 = ab * N + nf;
          c2 = -((2.0 * q - 1.0) / (2.0 * q + 1.0));
          x2 = ab * N + nff;
        }
        break;
      case LBM_ZHAO_YONG:  // Eq. (14): post-collision f*_abar(x_b), pre-collision f_a(x_b)
        c0 = 0.0;
        c1 = 2.0 * q / (1.0 + 2.0 * q);
        x1 = ab * N + nf;
        c2 = 1.0 / (1.0 + 2.0 * q);
        x2 = a * N + n;
        kind = kFromA;
        break;
      default:
        break;
    }
    r.src[l] = a * N + ns;
    r.dst[l] = ab * N + n;
    r.x1[l] = x1;
    r.x2[l] = x2;
    r.uf[l] = uf;
    r.kind[l] = kind;
    r.c0[l] = c0;
    r.c1[l] = c1;
    r.c2[l] = c2;
    r.chi[l] = chi;
    r.cus[l] = cus;
    r.c0f[l] = float(c0);
    r.c1f[l] = float(c1);
    r.c2f[l] = float(c2);
    r.chif[l] = float(chi);
    r.cusf[l] = float(cus);
  }
}

template <typename T>
__global__ void tile_links_kernel(int n_nodes, const TileNode* __restrict__ nodes,
                                  const int32_t* __restrict__ first,
                                  const int32_t* __restrict__ boff,
                                  const uint8_t* __restrict__ ldir, LinkRecipe r,
                                  const int32_t* __restrict__ local, TileLink<T>* links) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n_nodes) return;
  const TileNode nd = nodes[k];
  for (int l = boff[nd.b], o = first[k]; l < boff[nd.b + 1]; ++l, ++o) {
    TileLink<T> q{};
    q.src = r.src[l];
    q.x1 = r.x1[l];
    q.x2 = r.x2[l];
    q.uf = r.uf[l];
    q.n = nd.n;
    q.info = ldir[l] | r.kind[l] << 4 | local[k] << 8;
    q.c0 = pick<T>(r.c0, r.c0f, l);
    q.c1 = pick<T>(r.c1, r.c1f, l);
    q.c2 = pick<T>(r.c2, r.c2f, l);
    q.chi = pick<T>(r.chi, r.chif, l);
    q.cus = pick<T>(r.cus, r.cusf, l);
    links[o] = q;
  }
}

// The wall pass: 8 lanes per boundary node.  CTAs from wall_ctas on (launched only in channel mode
// when no boundary node reads or writes what the channel ends touch) do the channel ends, one
// thread per row, so that the two need one launch.
template <typename S>
__global__ void __launch_bounds__(128) boundary_kernel(DevParams p, int nb,
                                                       const int32_t* __restrict__ bnode,
                                                       const int32_t* __restrict__ boff,
                                                       const uint8_t* __restrict__ ldir,
                                                       LinkRecipe r, const void* fa, void* fb,
                                                       const double* rho_m, const double* ux_m,
                                                       const double* uy_m, const double* carry_in,
                                                       double* carry_out,
                                                       double* __restrict__ force, int wall_ctas,
                                                       const uint8_t* __restrict__ flags,
                                                       double u_in, int* done) {
  if (done && blockIdx.x == 0 && threadIdx.x < 2) {  // the counters of FrontWalls start at 0
    pdl_wait();
    done[threadIdx.x] = 0;
  }
  if ((int)blockIdx.x >= wall_ctas) {
    open_row<S>(p, (blockIdx.x - wall_ctas) * blockDim.x + threadIdx.x, fb, flags, u_in);
    return;
  }
  const int gt = blockIdx.x * blockDim.x + threadIdx.x;
  const int b = gt >> 3, k = gt & 7;
  const auto q = load_link<typename Pop<S>::C>(b, k, b < nb, bnode, boff, ldir, r);
  // the link records are fixed for the lattice's lifetime; everything read below was written by
  // the kernels before this one
  pdl_wait();
  wall_values<S>(p, b, k, b < nb, q, Lat<S>{fa, fb, p.N, p.rho_ref}, rho_m, ux_m, uy_m, carry_in,
                 InPlace<S>{fb, p.N, carry_out}, force, 0xffffffffu);
}

template <typename S>
__global__ void __launch_bounds__(128) open_x_kernel(DevParams p, void* __restrict__ fb,
                                                     const uint8_t* __restrict__ flags,
                                                     double u_in) {
  open_row<S>(p, blockIdx.x * blockDim.x + threadIdx.x, fb, flags, u_in);
}

// Boundary nodes of many lattices: items are (domain, boundary node); a persistent grid of
// 8-lane groups walks them.  Lattices whose step budget is spent are skipped.
template <typename S>
// 12 CTAs per SM (40 registers, a few spilled): more resident 8-lane groups for the chains of
// dependent loads each item is (80 against 83 us per batched step FP32, 78 against 84 FP16)
__global__ void __launch_bounds__(128, 12) batch_boundary_kernel(const BatchDomain* __restrict__ doms,
                                                             const int2* __restrict__ items,
                                                             const int* __restrict__ n_items) {
  const int gt = blockIdx.x * blockDim.x + threadIdx.x;
  const int k = gt & 7;
  const unsigned mask = 0xffu << (threadIdx.x & 24);
  const int ni = *n_items;
  for (int i = gt >> 3; i < ni; i += (gridDim.x * blockDim.x) >> 3) {
    const int2 it = items[i];
    const BatchDomain& D = doms[it.x];
    if (D.steps_left <= 0) continue;  // uniform over the group
    const int cur = D.cur;
    const auto q = load_link<typename Pop<S>::C>(it.y, k, true, D.bnode, D.boff, D.ldir, D.recipe);
    wall_values<S>(D.p, it.y, k, true, q, Lat<S>{D.f[cur], D.f[cur ^ 1], D.p.N, D.p.rho_ref},
                   D.rho_m, D.ux_m, D.uy_m, D.carry, InPlace<S>{D.f[cur ^ 1], D.p.N, D.carry},
                   nullptr, mask);
  }
}

__global__ void batch_advance_kernel(BatchDomain* __restrict__ doms, int n, int* claim) {
  const int d = blockIdx.x * blockDim.x + threadIdx.x;
  if (d == 0) *claim = 0;  // the step kernel of the next step claims tiles from 0
  if (d < n && doms[d].steps_left > 0) {
    doms[d].cur ^= 1;
    --doms[d].steps_left;
    ++doms[d].steps_done;
  }
}

// CTAs of one warp while that leaves at most four on an SM: a group is a chain of dependent loads
// and (FP64) of narrow-pipe operations, so a few warps are best spread over as many SMs.
unsigned wall_threads(long long threads) { return threads <= 32LL * 152 * 4 ? 32 : 128; }

template <typename S>
cudaError_t launch_b(const DevParams& p, int nb, const int32_t* bnode, const int32_t* boff,
                     const uint8_t* ldir, LinkRecipe r, const void* fa, void* fb,
                     const double* rho_m, const double* ux_m, const double* uy_m,
                     const double* carry_in, double* carry_out, double* force,
                     const uint8_t* open_flags, double u_in, int* done, cudaStream_t s) {
  const long long threads = 8LL * nb;
  const unsigned nt = wall_threads(threads + (open_flags ? p.ny : 0));
  const unsigned wall = (unsigned)((threads + nt - 1) / nt);
  const unsigned ends = open_flags ? (p.ny + nt - 1) / nt : 0;
  return launch_pdl(boundary_kernel<S>, dim3(wall + ends), dim3(nt), s, p, nb, bnode, boff, ldir,
                    r, fa, fb, rho_m, ux_m, uy_m, carry_in, carry_out, force, (int)wall, open_flags,
                    u_in, done);
}

size_t align256(size_t v) { return (v + 255) / 256 * 256; }

}  // namespace

size_t link_recipe_bytes(long long nl) {
  return 5 * align256(nl * 4) + align256(nl) + 5 * align256(nl * 8) + 5 * align256(nl * 4);
}

void link_recipe_carve(char* base, long long nl, LinkRecipe* r) {
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* q = base + off;
    off += align256(bytes);
    return q;
  };
  r->src = (int32_t*)take(nl * 4);
  r->dst = (int32_t*)take(nl * 4);
  r->x1 = (int32_t*)take(nl * 4);
  r->x2 = (int32_t*)take(nl * 4);
  r->uf = (int32_t*)take(nl * 4);
  r->kind = (uint8_t*)take(nl);
  r->c0 = (double*)take(nl * 8);
  r->c1 = (double*)take(nl * 8);
  r->c2 = (double*)take(nl * 8);
  r->chi = (double*)take(nl * 8);
  r->cus = (double*)take(nl * 8);
  r->c0f = (float*)take(nl * 4);
  r->c1f = (float*)take(nl * 4);
  r->c2f = (float*)take(nl * 4);
  r->chif = (float*)take(nl * 4);
  r->cusf = (float*)take(nl * 4);
}

cudaError_t launch_link_setup(const DevParams& p, int nb, const int32_t* bnode,
                              const int32_t* boff, const uint8_t* ldir, const double* lq,
                              const uint8_t* flags, LinkRecipe r, cudaStream_t s) {
  if (nb <= 0) return cudaSuccess;
  link_setup_kernel<<<(nb + 127) / 128, 128, 0, s>>>(p, nb, bnode, boff, ldir, lq, flags, r);
  return cudaGetLastError();
}

size_t tile_link_bytes(int precision) {
  return precision == LBM_FP64 ? sizeof(TileLink<double>) : sizeof(TileLink<float>);
}

cudaError_t launch_tile_links(int precision, int n_nodes, const TileNode* nodes,
                              const int32_t* first, const int32_t* local, const int32_t* boff,
                              const uint8_t* ldir, LinkRecipe r, void* links, cudaStream_t s) {
  const int grid = (n_nodes + 127) / 128;
  if (precision == LBM_FP64)
    tile_links_kernel<double><<<grid, 128, 0, s>>>(n_nodes, nodes, first, boff, ldir, r, local,
                                                   (TileLink<double>*)links);
  else
    tile_links_kernel<float><<<grid, 128, 0, s>>>(n_nodes, nodes, first, boff, ldir, r, local,
                                                  (TileLink<float>*)links);
  return cudaGetLastError();
}

cudaError_t launch_batch_boundary(int precision, const BatchDomain* doms, const int2* items,
                                  const int* n_items, int grid, cudaStream_t s) {
  if (precision == LBM_FP32_DEV)
    batch_boundary_kernel<float><<<grid, 128, 0, s>>>(doms, items, n_items);
  else if (precision == LBM_FP16_DEV)
    batch_boundary_kernel<__half><<<grid, 128, 0, s>>>(doms, items, n_items);
  else
    batch_boundary_kernel<double><<<grid, 128, 0, s>>>(doms, items, n_items);
  return cudaGetLastError();
}

int batch_boundary_grid(int precision) {
  // every 8-lane group walks items one after the other, each a chain of dependent loads: fill
  // the GPU with as many resident groups as it takes
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const void* fn = precision == LBM_FP32_DEV ? (const void*)batch_boundary_kernel<float>
                   : precision == LBM_FP16_DEV ? (const void*)batch_boundary_kernel<__half>
                                               : (const void*)batch_boundary_kernel<double>;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, 128, 0) != cudaSuccess || per < 1) {
    cudaGetLastError();
    per = 8;
  }
  return sms * per;
}

cudaError_t launch_batch_advance(BatchDomain* doms, int n_doms, int* claim, cudaStream_t s) {
  if (n_doms <= 0) return cudaSuccess;
  batch_advance_kernel<<<(n_doms + 127) / 128, 128, 0, s>>>(doms, n_doms, claim);
  return cudaGetLastError();
}

cudaError_t launch_boundary(int precision, const DevParams& p, int nb, const int32_t* bnode,
                            const int32_t* boff, const uint8_t* ldir, LinkRecipe r,
                            const void* fa, void* fb, const double* rho_m, const double* ux_m,
                            const double* uy_m, const double* carry_in, double* carry_out,
                            double* force, const uint8_t* open_flags, double u_in, int* done,
                            cudaStream_t s) {
  if (nb <= 0) return cudaSuccess;
  if (precision == LBM_FP32_DEV)
    return launch_b<float>(p, nb, bnode, boff, ldir, r, fa, fb, rho_m, ux_m, uy_m, carry_in, carry_out, force,
                           open_flags, u_in, done, s);
  if (precision == LBM_FP16_DEV)
    return launch_b<__half>(p, nb, bnode, boff, ldir, r, fa, fb, rho_m, ux_m, uy_m, carry_in, carry_out, force,
                            open_flags, u_in, done, s);
  return launch_b<double>(p, nb, bnode, boff, ldir, r, fa, fb, rho_m, ux_m, uy_m, carry_in, carry_out, force,
                          open_flags, u_in, done, s);
}

cudaError_t launch_open_x(int precision, const DevParams& p, void* fb, const uint8_t* flags,
                          double u_in, cudaStream_t s) {
  const unsigned nt = wall_threads(p.ny);
  const dim3 grid((p.ny + nt - 1) / nt);
  if (precision == LBM_FP32_DEV)
    return launch_pdl(open_x_kernel<float>, grid, dim3(nt), s, p, fb, flags, u_in);
  if (precision == LBM_FP16_DEV)
    return launch_pdl(open_x_kernel<__half>, grid, dim3(nt), s, p, fb, flags, u_in);
  return launch_pdl(open_x_kernel<double>, grid, dim3(nt), s, p, fb, flags, u_in);
}

}  // namespace lbm
