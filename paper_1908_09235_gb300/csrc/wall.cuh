// The arithmetic of the wall pass for one boundary node (Sec. 2.2, Sec. 3.1, Sec. 4.1), shared by
// the wall kernels (csrc/boundary.cu) and by the step kernels that apply it to their source lattice
// (csrc/wall_tile.cuh).  Both are compiled without multiply-add contraction, so a node gets the
// same bits in each.
#pragma once
#include "d2q9.cuh"

namespace lbm {
namespace wall {

constexpr uint8_t kFromA = 1;   // X2 is read from lattice A (pre-collision)
constexpr uint8_t kGhost = 2;   // the link has the ghost-node term chi f_eq(x_s)

// e_a . (x, y)
template <typename T>
__device__ __forceinline__ T edot(int a, T x, T y) {
  const T u = ex(a) == 0 ? T(0) : (ex(a) > 0 ? x : -x);
  return ey(a) == 0 ? u : (ey(a) > 0 ? u + y : u - y);
}

// The bracket of Eqs. (8), (20), (22): w_a [1 + 3 e_a.u_s + 4.5 (e_a.u_b)^2 - 1.5 u_b.u_b].
template <typename T>
__device__ __forceinline__ T bracket(int a, T usx, T usy, T ubx, T uby) {
  const T eub = edot(a, ubx, uby);
  return wgt<T>(a) * (T(1) + T(3) * edot(a, usx, usy) + T(4.5) * eub * eub -
                      T(1.5) * (ubx * ubx + uby * uby));
}

template <typename S>
struct Lat {
  const void* src;  // lattice A: f(t)
  const void* dst;  // lattice B: streamed values of step t
  int N;
  double rho_ref;
};

// Sum over the 8 lanes of a node's group in a fixed tree order (bitwise reproducible); `mask`
// holds the 8 lanes of the group.
template <typename T>
__device__ __forceinline__ T group8_sum(T v, unsigned mask) {
  v += __shfl_xor_sync(mask, v, 4);
  v += __shfl_xor_sync(mask, v, 2);
  v += __shfl_xor_sync(mask, v, 1);
  return v;
}

template <typename T>
__device__ __forceinline__ T pick(const double* d, const float* f, int l) {
  if constexpr (sizeof(T) == 8) return d[l]; else return f[l];
}

// A link's record (fixed for the lattice's lifetime) as lane k of its boundary node's 8-lane group
// holds it; act: the lane has a link.
template <typename T>
struct Link {
  bool act;
  int n, a, src, dst, x1, x2, uf;
  uint8_t kind;
  T c0, c1, c2, chi, cus;
};

template <typename T>
__device__ __forceinline__ Link<T> load_link(int b, int k, bool node_ok,
                                             const int32_t* __restrict__ bnode,
                                             const int32_t* __restrict__ boff,
                                             const uint8_t* __restrict__ ldir,
                                             const LinkRecipe& r) {
  Link<T> q{false, 0, 1, 0, 0, -1, -1, -1, 0, T(1), T(0), T(0), T(0), T(0)};
  int l0 = 0, nl = 0;
  if (node_ok) {
    q.n = bnode[b];
    l0 = boff[b];
    nl = boff[b + 1] - l0;
  }
  q.act = node_ok && k < nl;
  if (q.act) {
    const int l = l0 + k;
    q.a = ldir[l];
    q.src = r.src[l];
    q.dst = r.dst[l];
    q.x1 = r.x1[l];
    q.x2 = r.x2[l];
    q.uf = r.uf[l];
    q.kind = r.kind[l];
    q.c0 = pick<T>(r.c0, r.c0f, l);
    q.c1 = pick<T>(r.c1, r.c1f, l);
    q.c2 = pick<T>(r.c2, r.c2f, l);
    q.chi = pick<T>(r.chi, r.chif, l);
    q.cus = pick<T>(r.cus, r.cusf, l);
  }
  return q;
}

// What a link's wall value depends on, as read after the step: the outgoing population, stored (fo_d)
// and whole (fo), the other operands and the bracket (0 without a ghost term).
template <typename T>
struct Operands {
  T fo_d, fo, X1, X2, br, rho_b;
};

template <typename S>
__device__ __forceinline__ Operands<typename Pop<S>::C> load_operands(
    const DevParams& p, const Link<typename Pop<S>::C>& q, const Lat<S>& L, const double* rho_m,
    const double* ux_m, const double* uy_m) {
  using T = typename Pop<S>::C;
  const int N = L.N;
  // moment arrays: FP64 for FP64 storage, FP32 (in the same memory) for the deviation formats
  const T* rhoT = reinterpret_cast<const T*>(rho_m);
  const T* uxT = reinterpret_cast<const T*>(ux_m);
  const T* uyT = reinterpret_cast<const T*>(uy_m);
  // deviations d_ for the FP32 formats: f = d_ + w rho_ref
  const T wr = Pop<S>::dev ? wgt<T>(q.a) * p.k<T>().rho_ref : T(0);
  Operands<T> o{T(0), wr, T(0), T(0), T(0), T(1)};
  if (!q.act) return o;
  o.rho_b = __ldcg(rhoT + LBM_CHK(q.n, N));
  o.fo_d = Pop<S>::load_t(L.dst, q.src, N);  // outgoing f*_a(x_b, t)
  o.fo = o.fo_d + wr;
  if (q.x1 >= 0) o.X1 = Pop<S>::load_t(L.dst, q.x1, N) + wr;
  if (q.x2 >= 0) o.X2 = Pop<S>::load_t((q.kind & kFromA) ? L.src : L.dst, q.x2, N) + wr;
  if (q.kind & kGhost) {
    const T ubx = __ldcg(uxT + q.n), uby = __ldcg(uyT + q.n);
    T usx = q.cus * ubx, usy = q.cus * uby;
    if (q.uf >= 0) {
      usx = __ldcg(uxT + LBM_CHK(q.uf, N));
      usy = __ldcg(uyT + q.uf);
    }
    o.br = bracket<T>(q.a, usx, usy, ubx, uby);
  }
  return o;
}

// Terms of the fictitious density, Eq. (22) (scheme B) or Eq. (23) (Bao): rho_s = sum num / sum den
// over the links with a ghost term (the others are halfway bounce-back: chi = 0).
template <typename T>
__device__ __forceinline__ void fict_terms(int scheme, const Link<T>& q, const Operands<T>& o,
                                           T& num, T& den) {
  const bool gh = q.act && (q.kind & kGhost);
  num = gh ? (scheme == LBM_MOD_B ? q.chi * o.fo : o.fo) : T(0);
  den = gh ? (scheme == LBM_MOD_B ? q.chi * o.br : o.br) : T(0);
}

// The incoming population (whole) from the ghost density rho_g, Eqs. (7)-(14), (17), (20).
template <typename T>
__device__ __forceinline__ T link_value(const Link<T>& q, const Operands<T>& o, T rho_g) {
  T val = q.c0 * o.fo;
  if (q.x1 >= 0) val += q.c1 * o.X1;
  if (q.x2 >= 0) val += q.c2 * o.X2;
  if (q.act && (q.kind & kGhost)) val += q.chi * (rho_g * o.br);
  return val;
}

// The value to store for it: a pure bounce-back link (halfway bounce-back or a fallback) of a
// deviation format copies the stored one.
template <typename S>
__device__ __forceinline__ typename Pop<S>::C to_store(const DevParams& p,
                                                       const Link<typename Pop<S>::C>& q,
                                                       const Operands<typename Pop<S>::C>& o,
                                                       typename Pop<S>::C val) {
  using T = typename Pop<S>::C;
  if constexpr (!Pop<S>::dev) return val;
  const bool copy = !(q.kind & kGhost) && q.x1 < 0 && q.x2 < 0 && q.c0 == T(1);
  return copy ? o.fo_d : val - wgt<T>(q.a) * p.k<T>().rho_ref;
}

// The schemes that change the rest population: Eq. (18) in every format, and in the deviation formats
// those whose mass balance is kept exactly.
__device__ __forceinline__ bool corrects_rest(int scheme) {
  return scheme == LBM_MOD_A || scheme == LBM_BOUZIDI_L_A;
}
template <typename S>
__device__ __forceinline__ bool writes_rest(int scheme) {
  return corrects_rest(scheme) || (Pop<S>::dev && (scheme == LBM_MOD_B || scheme == LBM_HBB));
}
__device__ __forceinline__ bool fictitious(int scheme) {
  return scheme == LBM_MOD_B || scheme == LBM_BAO;
}

// The new rest population and FP64 residue of a node whose links' imbalance (outgoing less
// incoming) is dm: Eq. (18); for the deviation formats with the residue of the step before, and
// what rounding leaves of it.
template <typename T>
__device__ __forceinline__ T rest_value(T f0_d, double dm, double residue, double& left) {
  left = 0.0;
  if constexpr (sizeof(T) == 8) return f0_d + dm;
  const double want = double(f0_d) + dm + residue;
  if (want == double(f0_d)) return f0_d;
  const T st = T(want);
  left = want - double(st);
  return st;
}

// Inlet of the channel mode (Sec. 4.2) at a node of column 0: the populations entering from the left
// (1, 5, 8) follow from the prescribed velocity (u_in, 0) and the known ones by Zou and He's rule,
//   rho = (f0 + f2 + f4 + 2 (f3 + f6 + f7)) / (1 - u_in),  f1 = f3 + 2/3 rho u_in,
//   f5 = f7 - (f2 - f4)/2 + rho u_in / 6,  f8 = f6 + (f2 - f4)/2 + rho u_in / 6,
// in FP64 on the full populations (stored value + w rho_ref); get(a): the stored value, put(a, v):
// the new one, to be rounded to the format.
template <typename Get, typename Set>
__device__ __forceinline__ void inlet(double rho_ref, double u_in, Get get, Set set) {
  auto whole = [&](int a) { return get(a) + wgt<double>(a) * rho_ref; };
  const double f0 = whole(0), f2 = whole(2), f3 = whole(3), f4 = whole(4), f6 = whole(6),
               f7 = whole(7);
  const double rho = (f0 + f2 + f4 + 2.0 * (f3 + f6 + f7)) / (1.0 - u_in);
  set(1, f3 + 2.0 / 3.0 * rho * u_in - wgt<double>(1) * rho_ref);
  set(5, f7 - 0.5 * (f2 - f4) + rho * u_in / 6.0 - wgt<double>(5) * rho_ref);
  set(8, f6 + 0.5 * (f2 - f4) + rho * u_in / 6.0 - wgt<double>(8) * rho_ref);
}

// The wall values of a boundary node by the 8 lanes of its group, lane k one link (node_ok false: a
// padding group, which still takes part in the shuffles).  put.incoming(dst, a, v) and
// put.rest(n, v) take the unknown population f_a(x_b, t+1) and the corrected rest population and
// return the value as stored; put.carry(b, c) the node's new FP64 residue, read from carry.
// Arithmetic type T: FP64 for FP64 storage; FP32 for the deviation formats, whose mass bookkeeping
// is exact instead: each node's imbalance between the stored outgoing and incoming values is
// summed in FP64 and goes, with the previous step's FP64 rounding residue, into its rest
// population.  For schemes A and L-Bouzidi + A that is Eq. (18); for B (balanced by construction,
// Eq. 19) and halfway bounce-back it only returns the FP32 rounding.
template <typename S, typename Put>
__device__ __forceinline__ void wall_values(const DevParams& p, int b, int k, bool node_ok,
                                            const Link<typename Pop<S>::C>& q, const Lat<S>& L,
                                            const double* rho_m, const double* ux_m,
                                            const double* uy_m, const double* carry, Put put,
                                            double* __restrict__ force, unsigned mask) {
  using T = typename Pop<S>::C;
  constexpr bool DEV = Pop<S>::dev;
  const int scheme = p.scheme;
  const bool lane0 = node_ok && k == 0, rest = writes_rest<S>(scheme);
  const Operands<T> o = load_operands<S>(p, q, L, rho_m, ux_m, uy_m);
  T f0_d = T(0);
  double residue = 0.0;
  if (lane0 && rest) {
    f0_d = Pop<S>::load_t(L.dst, q.n, L.N);
    if (DEV) residue = __ldcg(carry + b);
  }
  T rho_g = o.rho_b;
  if (fictitious(scheme)) {
    T num, den;
    fict_terms(scheme, q, o, num, den);
    num = group8_sum(num, mask);
    den = group8_sum(den, mask);
    if (den != T(0)) rho_g = num / den;
  }
  const T val = link_value(q, o, rho_g);
  T in_d = T(0);
  if (q.act) in_d = put.incoming(q.dst, opposite(q.a), to_store<S>(p, q, o, val));
  if (force) {
    // Momentum exchange (Sec. 4.2, after Mei et al. 2002): through link a the wall receives
    // e_a (f*_a(x_b, t) + f_abar(x_b, t+1)), with the incoming value as stored; FP64 sums over
    // the node's links in the fixed group order, one (fx, fy) per boundary node.
    const double m =
        q.act ? double(o.fo_d) + double(in_d) + 2.0 * wgt<double>(q.a) * L.rho_ref : 0.0;
    const double fx = group8_sum(double(ex(q.a)) * m, mask);
    const double fy = group8_sum(double(ey(q.a)) * m, mask);
    if (lane0) {
      force[2 * b] = fx;
      force[2 * b + 1] = fy;
    }
  }
  if (rest) {
    // Eq. (15); exact in FP64 for the deviation formats (the w rho_ref parts cancel)
    const double dm = group8_sum(q.act ? double(o.fo_d) - double(in_d) : 0.0, mask);
    if (lane0) {
      double left;
      put.rest(q.n, rest_value<T>(f0_d, dm, residue, left));
      if (DEV) put.carry(b, left);
    }
  }
}

// The wall values written in place, into lattice B and the carry array.
template <typename S>
struct InPlace {
  using T = typename Pop<S>::C;
  void* f;
  int N;
  double* out;
  __device__ __forceinline__ T incoming(int dst, int a, T v) const {
    return Pop<S>::store_t(f, dst, N, v);
  }
  __device__ __forceinline__ T rest(int n, T v) const { return Pop<S>::store_t(f, n, N, v); }
  __device__ __forceinline__ void carry(int b, double c) const { out[b] = c; }
};

// Channel ends (Sec. 4.2), after streaming and the wall pass; one thread per row j: the inlet at
// i = 0, and at the outlet i = nx - 1 (fully developed flow) the populations entering from the right
// (3, 6, 7) equal those of column nx - 2.
template <typename S>
__device__ __forceinline__ void open_row(const DevParams& p, int j, void* __restrict__ fb,
                                         const uint8_t* __restrict__ flags, double u_in) {
  const int nx = p.nx, N = p.N;
  const bool in = j < p.ny;
  const int n0 = in ? j * nx : 0, n1 = n0 + nx - 1;
  const bool fluid0 = in && !(flags[n0] & FLAG_SOLID), fluid1 = in && !(flags[n1] & FLAG_SOLID);
  pdl_wait();
  if (fluid0)
    inlet(p.rho_ref, u_in, [&](int a) { return Pop<S>::load_e(fb, a * N + n0, N); },
          [&](int a, double v) { Pop<S>::store_e(fb, a * N + n0, N, v); });
  if (fluid1) {
    // copies of stored values: no rounding for any format
    Pop<S>::store_e(fb, 3 * N + n1, N, Pop<S>::load_e(fb, 3 * N + n1 - 1, N));
    Pop<S>::store_e(fb, 6 * N + n1, N, Pop<S>::load_e(fb, 6 * N + n1 - 1, N));
    Pop<S>::store_e(fb, 7 * N + n1, N, Pop<S>::load_e(fb, 7 * N + n1 - 1, N));
  }
}

}  // namespace wall
}  // namespace lbm
