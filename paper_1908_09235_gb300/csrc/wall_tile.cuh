// The wall pass of the step before, applied by a step kernel's tile to the populations it has loaded
// (csrc/step_core.cuh).  A wall pass of its own costs a small lattice a second dependent launch per
// step, 3.3 us (FP64: 5.3 us) beside a step kernel of 2.3-3.6 us; inside the tile its operands load
// while the tile's own populations do, and what is left is a few operations and CTA barriers, in
// tiles that hold boundary nodes only.
//
// A tile needs the values of its own boundary nodes and, for psi, of its ring's; ring nodes are
// computed by every tile that needs them, with the same operations on the same values, so nobody
// waits and nothing is written back.  One thread takes a link (not 8 lanes a node: on average 3.4
// of them have a link, and in FP64 a lane without one costs the narrow pipe as much), one thread a
// node's sums, over its links in the fixed tree order of the wall kernels, so the bits are theirs.
#pragma once
#include "wall.cuh"

namespace lbm {
namespace wall {

constexpr int kNodeSums = 8;  // links of a node at most

// Shared memory of a tile with at most nl links and nn nodes (dynamic; 16-byte aligned parts):
// two terms per link, then per node the ghost density and the nine values, then an entry per cell.
template <typename T>
__host__ __device__ constexpr size_t tile_terms_bytes(int nl) {
  return (size_t)nl * 16;
}
template <typename T>
__host__ __device__ constexpr size_t tile_wall_bytes(int nl, int nn, int cells) {
  return tile_terms_bytes<T>(nl) + ((size_t)nn * 10 * sizeof(T) + 15) / 16 * 16 +
         (size_t)cells * 4;
}

// Sum of eight terms in the order of group8_sum's lane 0; links beyond n count as zero.
template <typename T>
__device__ __forceinline__ T tree8(const T* v, int stride, int n) {
  T t[kNodeSums];
#pragma unroll
  for (int k = 0; k < kNodeSums; ++k) t[k] = k < n ? v[k * stride] : T(0);
  return ((t[0] + t[4]) + (t[2] + t[6])) + ((t[1] + t[5]) + (t[3] + t[7]));
}

// NT threads, thread c.
template <typename S, int NT>
struct TileWalls {
  using T = typename Pop<S>::C;
  static constexpr int U = NT >= 256 ? 1 : 2;  // links a thread keeps in registers

  int4 head;  // first link, links, first node, nodes of the tile
  T* terms;   // [link][2] T, or [link] double
  T* rho_g;
  T* f;       // [node][9]
  uint32_t* cell;  // per cell with a boundary node: its node | directions with a wall value << 16
  Link<T> link[U];
  int node[U];  // a link's node in the tile
  TileNode own;  // node c of the tile

  // the record of link l (in the tile), kept apart from the recipe arrays so that one dependent
  // load brings it
  __device__ __forceinline__ void record(const WallIn& w, int l, Link<T>& q, int& nd) const {
    q = Link<T>{false, 0, 1, 0, 0, -1, -1, -1, 0, T(1), T(0), T(0), T(0), T(0)};
    nd = 0;
    if (l >= head.y) return;
    const TileLink<T>& r = reinterpret_cast<const TileLink<T>*>(w.links)[head.x + l];
    q.act = true;
    q.n = r.n;
    q.a = r.info & 15;
    q.kind = (r.info >> 4) & 15;
    nd = r.info >> 8;
    q.src = r.src;
    q.x1 = r.x1;
    q.x2 = r.x2;
    q.uf = r.uf;
    q.c0 = r.c0;
    q.c1 = r.c1;
    q.c2 = r.c2;
    q.chi = r.chi;
    q.cus = r.cus;
  }

  __device__ __forceinline__ void carve(const WallIn& w, unsigned char* smem) {
    terms = reinterpret_cast<T*>(smem);
    rho_g = reinterpret_cast<T*>(smem + tile_terms_bytes<T>(w.max_links));
    f = rho_g + w.max_nodes;
    cell = reinterpret_cast<uint32_t*>(smem + tile_terms_bytes<T>(w.max_links) +
                                       ((size_t)w.max_nodes * 10 * sizeof(T) + 15) / 16 * 16);
  }

  // before the wait for the kernel before: the tables and the first records (fixed data)
  __device__ __forceinline__ void begin(const WallIn& w, int t, int c, unsigned char* smem) {
    head = w.heads[t];
    if (head.w == 0) return;
    carve(w, smem);
    if (c < head.w) own = w.nodes[head.z + c];
    for (int i = c; i < head.w; i += NT) {
      const int m = (i == c ? own : w.nodes[head.z + i]).cell, at = m & kCellMask;
      cell[LBM_CHK(at, w.cells)] = uint32_t(i | (m >> kMaskShift & 511) << 16);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) record(w, c + u * NT, link[u], node[u]);
  }

  // after it; every thread of the CTA.  On return (after a barrier) f holds the values.
  __device__ __forceinline__ void run(const DevParams& p, const WallIn& w, const void* fa, int c) {
    if (head.w == 0) return;
    constexpr bool DEV = Pop<S>::dev;
    const Lat<S> L{nullptr, fa, p.N, p.rho_ref};
    const bool fict = fictitious(p.scheme), rest = writes_rest<S>(p.scheme);
    Operands<T> o[U];
#pragma unroll
    for (int u = 0; u < U; ++u) o[u] = load_operands<S>(p, link[u], L, w.rho, w.ux, w.uy);
    if (fict) {
      auto put_terms = [&](int l, const Link<T>& q, const Operands<T>& x) {
        if (q.act) fict_terms(p.scheme, q, x, terms[2 * l], terms[2 * l + 1]);
      };
#pragma unroll
      for (int u = 0; u < U; ++u) put_terms(c + u * NT, link[u], o[u]);
      for (int l = c + U * NT; l < head.y; l += NT) {
        Link<T> q;
        int nd;
        record(w, l, q, nd);
        put_terms(l, q, load_operands<S>(p, q, L, w.rho, w.ux, w.uy));
      }
      // the node's density, where no link has a ghost term, is read beside the sums
      T rho0 = T(0);
      if (c < head.w) rho0 = __ldcg(reinterpret_cast<const T*>(w.rho) + own.n);
      __syncthreads();
      for (int i = c; i < head.w; i += NT) {
        const TileNode nd = i == c ? own : w.nodes[head.z + i];
        const int l0 = nd.links >> 8, nl = nd.links & 255;
        const T num = tree8(terms + 2 * l0, 2, nl), den = tree8(terms + 2 * l0 + 1, 2, nl);
        if (i != c) rho0 = __ldcg(reinterpret_cast<const T*>(w.rho) + nd.n);
        rho_g[i] = den != T(0) ? num / den : rho0;
      }
    }
    T f0_d = T(0);
    double residue = 0.0;
    if (rest && c < head.w) {
      f0_d = Pop<S>::load_t(fa, own.n, p.N);
      if (DEV) residue = __ldcg(w.carry_in + own.b);
    }
    if (fict) __syncthreads();
    double* dterms = reinterpret_cast<double*>(terms);  // [link]; the fictitious terms are read
    auto put_value = [&](int l, int nd, const Link<T>& q, const Operands<T>& x) {
      if (!q.act) return;
      const T v = to_store<S>(p, q, x, link_value(q, x, fict ? rho_g[nd] : x.rho_b));
      const T st = Pop<S>::rounded(opposite(q.a), v);
      f[nd * 9 + opposite(q.a)] = st;
      if (rest) dterms[l] = double(x.fo_d) - double(st);
    };
#pragma unroll
    for (int u = 0; u < U; ++u) put_value(c + u * NT, node[u], link[u], o[u]);
    for (int l = c + U * NT; l < head.y; l += NT) {
      Link<T> q;
      int nd;
      record(w, l, q, nd);
      put_value(l, nd, q, load_operands<S>(p, q, L, w.rho, w.ux, w.uy));
    }
    __syncthreads();
    if (rest) {
      for (int i = c; i < head.w; i += NT) {
        const TileNode nd = i == c ? own : w.nodes[head.z + i];
        if (i != c) {
          f0_d = Pop<S>::load_t(fa, nd.n, p.N);
          if (DEV) residue = __ldcg(w.carry_in + nd.b);
        }
        const double dm = tree8(dterms + (nd.links >> 8), 1, nd.links & 255);
        double left;
        f[i * 9] = rest_value<T>(f0_d, dm, residue, left);
        if (DEV && (nd.cell & kOwnedNode)) w.carry_out[nd.b] = left;
      }
      __syncthreads();
    }
  }

  // the values of the boundary node at a cell, in place of what was loaded
  __device__ __forceinline__ void take(const DevParams& p, int at, T (&g)[9]) const {
    const uint32_t e = cell[at];
    const int i0 = e & 0xffff, i = LBM_CHK(i0, head.w), m = e >> 16;
#pragma unroll
    for (int a = 1; a < 9; ++a)
      if (m >> a & 1) g[a] = f[i * 9 + a];
    if (writes_rest<S>(p.scheme)) g[0] = f[i * 9];
  }
};

// All of it in a call of its own: a kernel that runs several CTAs per SM one after the other keeps the
// registers of its own work, which this one's would spill (1024^2 FP32: 18.9 us a step inlined), and
// its few tiles with walls lose the overlap of the loads instead.
template <typename S, int NT>
__device__ __noinline__ void tile_walls_apart(const DevParams& p, const WallIn& w, const void* fa,
                                              int t, int c, unsigned char* smem) {
  TileWalls<S, NT> walls;
  walls.begin(w, t, c, smem);
  walls.run(p, w, fa, c);
}

}  // namespace wall
}  // namespace lbm
