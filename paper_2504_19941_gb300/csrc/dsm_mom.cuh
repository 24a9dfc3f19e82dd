// dsm_mom.cuh -- the stage-2 lattice Boltzmann step (Sec. II.B) on the moments
// that fix the populations, for lattices whose relaxation times are all 1.
// Included by dsm_lb_impl.cuh (two fluids) and used by dsm_multi.cu (N fluids).
//
// With tau = 1 the BGK collision replaces f_i by f_eq_i plus the forcing, and
// with tau_g = 1 and equal densities every population after a collision is a
// function of a few reals of its node:
//   f_i = w_i (1 + phi_i),  phi_i = dP + c_i.G + rho b(c_i.u)
//   g_i = w_i (A + C b(c_i.u))            (i != 0)
//   b(v) = v (3 + 9/2 v),  dP = pt - 1 - 3/2 rho u.u,  G = 3/2 F,
//   A = mu - 3/2 C u.u
// (F the total force; a solid node holds f_i = w_i, i.e. dP = G = u = 0).  The
// state is then (A, C) per free fluid, dP, u and G: 9 reals in 3D and 7 in 2D
// for two fluids, where the populations f alone are 19 and 9.  A step pulls
// these, adds up the streamed links
//   pt = 1 + sum_i w_i phi_i(x - c_i),  m = sum_i c_i w_i phi_i(x - c_i),
//   C = C(x) + sum_{i != 0} w_i (A + C b)(x - c_i) - (1 - w_0) A(x) - 3/2 C u.u(x)
// forms mu and F from C on the 1-neighbourhood and stores the new moments:
// there is no collision per direction left.  dP, m and b hold only the small
// parts of the populations, so their FP32 sums round at 1e-7 of the deviation
// from rest rather than of the rest weights.
//
// Everything that fixes a result is written with explicitly rounded
// operations (fm, ad, sb, ml below): the tile of a block, the planes of its run
// and the launch form (single or batched) cannot change it by a contraction.
#pragma once

#include <atomic>
#include <type_traits>

namespace dsm {

__device__ __forceinline__ float fm(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float ad(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sb(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float ml(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double fm(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double ad(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sb(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double ml(double a, double b) { return __dmul_rn(a, b); }

constexpr int MOM_NF = 3;  // most free fluids

// One buffer of the state.  3D: q1 quads (A, C, u_x, u_y), q2 quads
// (dP, G_x, G_y, G_z), w plane u_z, pe pairs (A_e, C_e) of each further free
// fluid (N pairs per fluid).  2D: q1 the same, q2 pairs (G_x, G_y), w plane dP.
template <class T>
struct MomBuf {
  T *q1, *q2, *w, *pe;
};

template <class T>
struct MomArgs {
  int nx, ny, nz;
  long long N, pitch;
  MomBuf<T> in, out;
  const T *sol;        // pairs (C1, L[C1]) of the frozen solid
  // of the nodes next to the solid, by node in 2D (lk: 0 elsewhere), in the order of
  // list in 3D:
  const unsigned *lk;  // bit i: x + c_i is solid
  const T *qpl;        // plane j - 1: link fraction of the wall link pulled in direction j
  const unsigned char *near;  // 3D: next to the solid
  unsigned *list;      // 3D: the nodes next to the solid, their count
  int *count;
  T *wall;             // 3D: quads, what their wall links add to (S, M)
  const T *c1;         // C1 (the kernel that makes the three above)
  int *err;
  T k[MOM_NF], ak[MOM_NF];  // kappa and alpha^2 kappa of the free fluids
  T kl, akl;                // the dependent fluid's
  T rho, irho, body[3], alpha_s;
  unsigned seed;       // MOM_SEED x the number of the step (mom_add)
};

// reals of one buffer per node, two fluids
__host__ __device__ constexpr int mom_reals(int kind) { return kind == 0 ? 7 : 9; }

template <class T>
struct alignas(2 * sizeof(T)) Duo {
  T v[2];
};

template <class T>
__device__ __forceinline__ T mom_b(T v) {  // b(v)
  return ml(v, fm(T(4.5), v, T(3)));
}
template <class T>
__device__ __forceinline__ T mom_bn(T v) {  // b(-v)
  return ml(v, fm(T(4.5), v, T(-3)));
}
// A step adds to each C a difference d, and two things in it would make an FP32
// lattice gain or lose liquid steadily (24^3, 10000 steps: -5.1e-5 of it; with f as
// populations, whose rounding shakes u and so d, -1.6e-5; as it is, 1e-8):
//   - Where C is near 1, d is mostly less than half a unit in C's last place and
//     would round away, while the nodes with small C that exchange with it keep what
//     they receive.  mom_add adds a fraction in (-1/2, 1/2) of that unit to d: C + d
//     rounded without bias.  The fraction is a hash of d and the step, no function of
//     the node, so that every form and tile of the step rounds alike and fields keep
//     their symmetries.  (One fraction for all nodes, the golden ratio's multiples over
//     the steps, gave 0.8 of the errors of short runs but lost 1.7e-6 in 5000 steps at
//     24^3, where the hash loses 1e-8; a hash only where |d| is below 4 units changed
//     neither the errors of short runs nor the loss.)
//   - A leaves a node as 1 - w_0 and arrives as the weights, which in FP32 do not add
//     up to it.  All of them are 2^k times the last one in any precision, so A leaves
//     as mom_out (24 in 3D, 20 in 2D) times that weight (in FP64, where the difference
//     is 1e-16 and a product more costs 1 %, as 1 - w_0 in the 3D step).
// 256 x 256 x 192: 275 -> 284 us per step for both.
template <class L>
__host__ __device__ constexpr int mom_out() {
  return L::D == 3 ? 24 : 20;
}
constexpr unsigned MOM_SEED = 0x85ebca77u;
__device__ __forceinline__ float mom_add(float c, float d, unsigned seed) {
  unsigned h = (__float_as_uint(d) ^ seed) * 0x9e3779b1u;
  h = (h ^ (h >> 15)) * 0x2c1b3c6du;
  const float r = sb(__uint_as_float((h >> 9) | 0x3f800000u), 1.5f);
  const unsigned m = __float_as_uint(c) & 0x7fffffffu;
  const float e = __uint_as_float((m - (m != 0u)) & 0x7f800000u);  // 2^23 units (below c)
  return ad(c, fm(e, ml(r, 1.1920928955078125e-7f), d));
}
__device__ __forceinline__ double mom_add(double c, double d, unsigned) { return ad(c, d); }

template <class T>
__device__ __forceinline__ T mom_well(T c) {
  return ml(ml(c, sb(T(1), c)), fm(T(-2), c, T(1)));
}

// A node's moments, for the few places that need single populations.
template <class T>
struct MomNode {
  T dP, u[3], G[3];
};
template <class L, class T>
__device__ __forceinline__ MomNode<T> mom_load(const MomBuf<T> &b, long long n) {
  MomNode<T> m;
  const Quad<T> a = reinterpret_cast<const Quad<T> *>(b.q1)[n];
  m.u[0] = a.v[2];
  m.u[1] = a.v[3];
  if (L::D == 3) {
    const Quad<T> q = reinterpret_cast<const Quad<T> *>(b.q2)[n];
    m.dP = q.v[0];
    m.G[0] = q.v[1];
    m.G[1] = q.v[2];
    m.G[2] = q.v[3];
    m.u[2] = b.w[n];
  } else {
    const Duo<T> q = reinterpret_cast<const Duo<T> *>(b.q2)[n];
    m.G[0] = q.v[0];
    m.G[1] = q.v[1];
    m.G[2] = m.u[2] = T(0);
    m.dP = b.w[n];
  }
  return m;
}
template <class L, class T>
__device__ __forceinline__ T mom_dot(int i, const T (&v)[3]) {  // c_i . v, i != 0
  T s = T(0);
  bool first = true;
#pragma unroll
  for (int e = 0; e < 3; e++) {
    const int c = e == 0 ? L::cx(i) : (e == 1 ? L::cy(i) : L::cz(i));
    if (c == 0) continue;
    if (first) s = c > 0 ? v[e] : -v[e];
    else s = c > 0 ? ad(s, v[e]) : sb(s, v[e]);
    first = false;
  }
  return s;
}
template <class L, class T>
__device__ __forceinline__ T mom_phi(const MomNode<T> &m, int i, T rho) {
  if (i == 0) return m.dP;
  return fm(rho, mom_b(mom_dot<L>(i, m.u)), ad(m.dP, mom_dot<L>(i, m.G)));
}

// The interpolated bounce-back (Sec. II.B) of a fluid node's wall links.  The
// link pulled from a solid node added exactly 0 (its moments are 0), so the
// node adds the interpolated value: the formulas are linear with coefficients
// that sum to 1, hence the same in phi as in f.  The link fractions do not
// change while the solid is frozen; mom_solid_kernel makes them once.  node(j):
// the moments at x + c_j (j = 0: the node itself).
// One wall link: v, the interpolated phi pulled in direction j, into S and M.
// own, far: the moments at x and at x + c_j.
template <class L, class T>
__device__ __forceinline__ void mom_wall_add(const MomArgs<T> &a, unsigned lk, int j, T q,
                                             const MomNode<T> &own, const MomNode<T> &far, T &S,
                                             T (&M)[3]) {
  const int i = L::opp(j);
  const T pi = mom_phi<L>(own, i, a.rho);
  T v = pi;
  if (q < T(0.5)) {
    if (!((lk >> j) & 1u)) {
      const T q2 = ml(T(2), q);
      v = fm(q2, pi, ml(sb(T(1), q2), mom_phi<L>(far, i, a.rho)));
    }
  } else {
    const T r = T(1) / (T(2) * q);
    v = fm(r, pi, ml(sb(T(1), r), mom_phi<L>(own, j, a.rho)));
  }
  const T wv = ml(T(L::w(j)), v);
  S = ad(S, wv);
  if (L::cx(j)) M[0] = L::cx(j) > 0 ? ad(M[0], wv) : sb(M[0], wv);
  if (L::cy(j)) M[1] = L::cy(j) > 0 ? ad(M[1], wv) : sb(M[1], wv);
  if (L::cz(j)) M[2] = L::cz(j) > 0 ? ad(M[2], wv) : sb(M[2], wv);
}
template <class L, class T, class Node>
__device__ __forceinline__ void mom_walls(const MomArgs<T> &a, unsigned lk, long long n,
                                          const Node &node, T &S, T (&M)[3]) {
  const MomNode<T> own = node(0);
#pragma unroll
  for (int j = 1; j < L::Q; j++) {
    if ((lk >> L::opp(j)) & 1u) {
      const T q = a.qpl[(long long)(j - 1) * a.pitch + n];
      MomNode<T> far = own;
      if (q < T(0.5) && !((lk >> j) & 1u)) far = node(j);
      mom_wall_add<L>(a, lk, j, q, own, far, S, M);
    }
  }
}

// 3D: the wall sums of every node next to the solid, ahead of the step.  In the
// step itself a wall node's loads (its link fractions, then the far nodes) would
// follow one another while its block waits at the plane's barrier.  Here a
// thread has all of a node's loads of one kind in flight: its index, link bits and
// the fractions of all its links (which lie in the order of the list: 1/2 where
// there is no link), then the node's moments and those at the far end of nine
// links each (at the node itself where the link needs none).
template <class T>
__device__ __forceinline__ void mom_wall_nodes(const MomArgs<T> &a, int first, int stride) {
  using L = Lat<1>;
  const int cnt = *a.count;
  for (int k = first; k < cnt; k += stride) {
    const int n = chk(a.err, (int)a.list[k], a.N);
    const unsigned lk = a.lk[k];
    T q[L::Q - 1];
#pragma unroll
    for (int j = 1; j < L::Q; j++) q[j - 1] = a.qpl[(long long)(j - 1) * a.pitch + k];
    const MomNode<T> own = mom_load<L>(a.in, n);
    const int x = n % a.nx, y = n / a.nx % a.ny, z = n / (a.nx * a.ny);
    Hood h;
    h.init(x, y, z, a.nx, a.ny, a.nz);
    h.guard(a.err);
    T S = T(0), M[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int j0 = 1; j0 < L::Q; j0 += 9) {
      MomNode<T> far[9];
#pragma unroll
      for (int e = 0; e < 9; e++) {
        const int j = j0 + e;
        far[e] = mom_load<L>(a.in, q[j - 1] < T(0.5) && !((lk >> j) & 1u) ? h.plus<L>(j) : n);
      }
#pragma unroll
      for (int e = 0; e < 9; e++) {
        const int j = j0 + e, i = L::opp(j);
        if ((lk >> i) & 1u) mom_wall_add<L>(a, lk, j, q[j - 1], own, far[e], S, M);
      }
    }
    Quad<T> r;
    r.v[0] = S;
    r.v[1] = M[0];
    r.v[2] = M[1];
    r.v[3] = M[2];
    reinterpret_cast<Quad<T> *>(a.wall)[n] = r;
  }
}
template <class T>
__global__ void __launch_bounds__(128) mom_wall_kernel(const __grid_constant__ MomArgs<T> a) {
  pdl_wait();
  mom_wall_nodes(a, blockIdx.x * 128 + threadIdx.x, gridDim.x * 128);
  pdl_next();
}

// mu, F and the new moments of one node from this step's C, its stencils and
// the streamed sums; the result in (A, dP, u, G).
template <class T, int NF>
struct MomOut {
  T A[NF], mu[NF], dP, u[3], G[3], uu;
};
template <int D, class T, int NF>
__device__ __forceinline__ MomOut<T, NF> mom_collide(const MomArgs<T> &a, T c1, T l1,
                                                     const T (&C)[NF], const T (&lap)[NF],
                                                     const T (&g)[NF][3], T S, const T (&M)[3]) {
  MomOut<T, NF> o;
  T s = c1, sl = l1;
#pragma unroll
  for (int f = 0; f < NF; f++) {
    s = ad(s, C[f]);
    sl = ad(sl, lap[f]);
  }
  // minus the dependent fluid's derivative: b(1 - s) = -b(s), L[1 - s] = -L[s]
  const T dl = fm(a.kl, mom_well(s), ml(-a.akl, sl));
  T F[3] = {T(0), T(0), T(0)}, bad = T(0);
#pragma unroll
  for (int f = 0; f < NF; f++) {
    o.mu[f] = fm(a.k[f], mom_well(C[f]), fm(-a.ak[f], lap[f], dl));
#pragma unroll
    for (int e = 0; e < D; e++) F[e] = f == 0 ? ml(o.mu[0], g[0][e]) : fm(o.mu[f], g[f][e], F[e]);
    bad = ad(bad, o.mu[f]);
  }
  const bool solid = c1 >= T(0.5);
#pragma unroll
  for (int e = 0; e < 3; e++) {
    if (e < D) {
      F[e] = fm(C[0], a.body[e], F[e]);
      o.u[e] = solid ? T(0) : ml(fm(T(0.5), F[e], M[e]), a.irho);
      o.G[e] = solid ? T(0) : ml(T(1.5), F[e]);
      bad = ad(bad, o.u[e]);
    } else {
      o.u[e] = o.G[e] = T(0);
    }
  }
  T uu = fm(o.u[1], o.u[1], ml(o.u[0], o.u[0]));
  if (D == 3) uu = fm(o.u[2], o.u[2], uu);
  const T h = ml(T(-1.5), uu);
  o.dP = solid ? T(0) : fm(a.rho, h, S);
#pragma unroll
  for (int f = 0; f < NF; f++) o.A[f] = fm(C[f], h, o.mu[f]);
  o.uu = uu;
  if (!isfinite(ad(bad, o.dP))) atomicOr(a.err, ERR_NONFINITE);
  return o;
}

// 16, 8 or 4 bytes to shared memory asynchronously.  (16 bytes bypass L1.)
template <int B>
__device__ __forceinline__ void cp_async_bytes(unsigned dst, const void *src) {
  if constexpr (B == 32) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst + 16),
                 "l"((const char *)src + 16)
                 : "memory");
  } else if constexpr (B == 16) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
  } else {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(dst), "l"(src), "n"(B)
                 : "memory");
  }
}

// ---------------------------------------------------------------------------
// 3D step.  A block marches a 32 x TY tile up a run of z planes, a thread
// carrying RY nodes of one column in y.  Each plane of the state over the tile
// and a two-node halo is staged once in a ring of three by asynchronous copies,
// two planes ahead of use.  A thread reads the in-plane points of its nodes from
// a plane once and adds their links to three targets: those with c_z = 1 to the
// node above, c_z = 0 to its own, c_z = -1 to the node below, whose partial sums
// stay in registers.  The C that plane q completes (target q - 1) goes to shared
// memory on the tile and a one-node halo (the first threads carry a second, halo
// node's C only); one plane later its points give the stencil's share for three
// nodes in the same way, and the node of plane q - 3 collides.  One barrier per
// plane.
//
// Bound by instruction issue and latency: 425 thread instructions per node, 59 %
// of issue slots used by 16 warps per SM, shared memory 62 % busy (256 x 256 x
// 96).  Two nodes per thread, because neighbouring rows share points: 100 shared
// wavefronts per 32 nodes instead of 136, and 0.242 against 0.282 ms per step at
// 256 x 256 x 192 (one node per thread, 3 blocks of 256 threads per SM at 80
// registers; at 64 registers it spilled: 0.413).  32 x 8 tiles of 128 threads,
// four per SM at 128 registers; 32 x 16 tiles, two per SM: 0.250.  Staged rows
// have a pitch of 37 quads, so that the halo columns' reads do not conflict.
// The kernel it replaced for these lattices (populations f, tensor-memory
// loads, dsm_zstep.cuh) takes 0.572 ms there: 196 B and 1189 instructions per
// node against 81 B and 425.
// With the wall pass, whole steps: 256 x 256 x 192 0.572 -> 0.284 ms, 101^3
// 76.4 -> 42.9 us.
// ---------------------------------------------------------------------------
constexpr int M3_X = 32, M3_HX = M3_X + 4, M3_HP = M3_HX + 1, M3_CX = M3_X + 2, M3_RING = 3;

template <class T, int NF, int TY>
struct M3Smem {
  static constexpr int HY = TY + 4, CY = TY + 2;
  static constexpr int NS = M3_HP * HY, NC = M3_CX * CY;
  static constexpr unsigned o2 = 4 * sizeof(T) * NS;          // q2 quads
  static constexpr unsigned ope = 8 * sizeof(T) * NS;         // further fluids' pairs
  static constexpr unsigned ow = (8 + 2 * (NF - 1)) * sizeof(T) * NS;  // u_z
  static constexpr unsigned slot = ((9 + 2 * (NF - 1)) * sizeof(T) * NS + 15) / 16 * 16;
  static constexpr unsigned cplane = sizeof(T) * NC;
  static constexpr unsigned cring = M3_RING * slot;           // two planes of C per fluid
  static constexpr unsigned total = cring + 2 * NF * cplane;
};

template <class T, int NF, int TY, int RY>
__device__ __forceinline__ void mom_run3(const MomArgs<T> &a, int x0, int y0, int z0, int z1,
                                         unsigned seed, unsigned char *sm) {
  using SM = M3Smem<T, NF, TY>;
  constexpr int NT = M3_X * TY / RY;
  constexpr int HP = M3_HP;  // staged row: nodes, pitch
  constexpr int PER = (SM::NS + NT - 1) / NT;
  constexpr T w0 = T(1.0 / 3.0), w1 = T(1.0 / 18.0), w2 = T(1.0 / 36.0);
  const int tx = threadIdx.x, ty = threadIdx.y * RY, tid = tx + M3_X * threadIdx.y;
  const int nx = a.nx, ny = a.ny, nz = a.nz;
  const int plane = nx * ny;
  auto wrap = [](int v, int n) {
    v %= n;
    return v < 0 ? v + n : v;
  };
  int off[PER];  // in-plane index of the staged nodes this thread copies
#pragma unroll
  for (int r = 0; r < PER; r++) {
    const int k = tid + r * NT;
    off[r] = wrap(x0 - 2 + k % HP, nx) + nx * wrap(y0 - 2 + k / HP, ny);
  }
  const unsigned sbase = (unsigned)__cvta_generic_to_shared(sm) + tid * (4 * sizeof(T));
  const unsigned wbase = (unsigned)__cvta_generic_to_shared(sm) + SM::ow + tid * sizeof(T);
  int pzo = wrap(z0 - 2, nz) * plane;  // the next plane to stage
  auto issue = [&](unsigned slot) {
#pragma unroll
    for (int r = 0; r < PER; r++) {
      if ((r + 1) * NT <= SM::NS || tid + r * NT < SM::NS) {
        const int n = chk(a.err, pzo + off[r], a.N);
        const unsigned d = sbase + slot + r * NT * (4 * sizeof(T));
        cp_async_bytes<4 * sizeof(T)>(d, reinterpret_cast<const Quad<T> *>(a.in.q1) + n);
        cp_async_bytes<4 * sizeof(T)>(d + SM::o2, reinterpret_cast<const Quad<T> *>(a.in.q2) + n);
#pragma unroll
        for (int e = 1; e < NF; e++)
          cp_async_bytes<2 * sizeof(T)>(
              (unsigned)__cvta_generic_to_shared(sm) + slot + SM::ope +
                  ((e - 1) * SM::NS + tid + r * NT) * 2 * sizeof(T),
              reinterpret_cast<const Duo<T> *>(a.in.pe) + (e - 1) * a.N + n);
        cp_async_bytes<sizeof(T)>(wbase + slot + r * NT * sizeof(T), a.in.w + n);
      }
    }
    pzo += plane;
    if (pzo == nz * plane) pzo = 0;
  };
  const int x = x0 + tx, y = y0 + ty;
  const int k0 = (ty + 2) * HP + tx + 2;          // own (first) node in a staged plane
  const int c0i = (ty + 1) * M3_CX + tx + 1;      // and in a C plane
  // the halo node whose C this thread carries too (the ring around the tile)
  constexpr int NE = SM::NC - M3_X * TY;
  static_assert(NE <= NT, "one halo node per thread");
  const bool extra = tid < NE;
  int ci = 0, cj = 0;
  if (extra) {
    if (tid < 2 * M3_CX) {
      ci = tid % M3_CX;
      cj = tid < M3_CX ? 0 : SM::CY - 1;
    } else {
      const int t = tid - 2 * M3_CX;
      ci = t < TY ? 0 : M3_CX - 1;
      cj = 1 + (t < TY ? t : t - TY);
    }
  }
  const int ke = (cj + 1) * HP + ci + 1, cei = cj * M3_CX + ci;

  // sums of a carried node -- order parameter: up, the links of the plane below
  // into it; mid, up + the links of its own plane; ck, its C
  struct GSum {
    T up[NF], mid[NF], ck[NF];
  };
  // streamed f: up, mid (mid.Z: up's S); d1, d2, complete: targets q - 2, q - 3
  struct FSum {
    T S, X, Y, Z;
  };
  struct Pt {  // a point of a plane: its quads
    T A[NF], C[NF], ux, uy;
  };
  auto point = [&](unsigned slot, int k) {
    Pt p;
    const Quad<T> q = *reinterpret_cast<const Quad<T> *>(sm + slot + k * (4 * sizeof(T)));
    p.A[0] = q.v[0];
    p.C[0] = q.v[1];
    p.ux = q.v[2];
    p.uy = q.v[3];
#pragma unroll
    for (int e = 1; e < NF; e++) {
      const Duo<T> d = *reinterpret_cast<const Duo<T> *>(
          sm + slot + SM::ope + ((e - 1) * SM::NS + k) * (2 * sizeof(T)));
      p.A[e] = d.v[0];
      p.C[e] = d.v[1];
    }
    return p;
  };
  auto hydro = [&](unsigned slot, int k) {
    return *reinterpret_cast<const Quad<T> *>(sm + slot + SM::o2 + k * (4 * sizeof(T)));
  };
  auto velz = [&](unsigned slot, int k) {
    return *reinterpret_cast<const T *>(sm + slot + SM::ow + k * sizeof(T));
  };
  FSum up[RY], mid[RY], d1[RY], d2[RY];
  GSum g[RY], ge[1];
#pragma unroll
  for (int j = 0; j < RY; j++) {
    up[j] = mid[j] = d1[j] = d2[j] = FSum{0, 0, 0, 0};
#pragma unroll
    for (int f = 0; f < NF; f++) g[j].up[f] = g[j].mid[f] = g[j].ck[f] = T(0);
  }
#pragma unroll
  for (int f = 0; f < NF; f++) ge[0].up[f] = ge[0].mid[f] = ge[0].ck[f] = T(0);

  // The links of plane `slot` around the R staged nodes k, k + HP, ..: adds
  // those with c_z = 1, 0, -1 to the sums of the targets above, in and below
  // the plane, and completes the one below (its C in Cd).  With v = c.u in the
  // plane, h = 9/2 u_z^2 and s = u_z (3 + 9 v), b(v +- u_z) = b(v) + h +- s: the
  // links c_z = +-1 of a point share all but the sign of one term, and so do
  // their sums.  Row by row, each point read once for all R nodes.
  auto links = [&](unsigned slot, int k, auto *gs, auto &Cd, auto joint, auto rows) {
    constexpr bool F = decltype(joint)::value;
    constexpr int R = decltype(rows)::value;
    T s0[R][NF], sE[R][NF], sQ[R][NF], gc[R][NF], out[R][NF], cn[R][NF];
    T f0[R], fH[R], fK[R], fD[R], Dx[R], Hx[R], Kx[R], Dy[R], Hy[R], Ky[R], dX[R], dY[R];
    T gP[R][NF], gR[R][NF], fP[R], fR[R], f00[R];
#pragma unroll
    for (int r = -1; r <= R; r++) {
      const int kr = k + r * HP;
      // the row's middle point: the node itself for j = r, its -y / +y neighbour
      // for j = r + 1 / r - 1
      {
        const Pt p = point(slot, kr);
        const T uz = velz(slot, kr);
        const T h = ml(ml(T(4.5), uz), uz);
        Quad<T> q;
        if (F) q = hydro(slot, kr);
#pragma unroll
        for (int j = 0; j < R; j++) {
          if (j == r) {
            const T z3 = ml(T(3), uz);
            const T uu = fm(uz, uz, fm(p.uy, p.uy, ml(p.ux, p.ux)));
#pragma unroll
            for (int f = 0; f < NF; f++) {
              const T away = sizeof(T) == 8 ? ml(T(1) - w0, p.A[f])
                                            : ml(T(mom_out<Lat<1>>()), ml(w2, p.A[f]));
              out[j][f] = fm(ml(T(1.5), p.C[f]), uu, away);
              gP[j][f] = ml(w1, fm(p.C[f], h, p.A[f]));
              gR[j][f] = ml(w1, ml(p.C[f], z3));
              cn[j][f] = p.C[f];
            }
            if (F) {
              fP[j] = ml(w1, fm(a.rho, h, q.v[0]));
              fR[j] = ml(w1, fm(a.rho, z3, q.v[3]));
              f00[j] = ml(w0, q.v[0]);
            }
          } else if (r - j == -1 || r - j == 1) {
            const bool lo = r < j;
            const T b = lo ? mom_b(p.uy) : mom_bn(p.uy);
            const T s = ml(uz, fm(lo ? T(9) : T(-9), p.uy, T(3)));
#pragma unroll
            for (int f = 0; f < NF; f++) {
              const T t = fm(p.C[f], b, p.A[f]);
              s0[j][f] = lo ? t : ad(s0[j][f], t);
              sE[j][f] = lo ? ml(p.C[f], h) : fm(p.C[f], h, sE[j][f]);
              sQ[j][f] = lo ? ml(p.C[f], s) : fm(p.C[f], s, sQ[j][f]);
            }
            if (F) {
              const T v = fm(a.rho, b, lo ? ad(q.v[0], q.v[2]) : sb(q.v[0], q.v[2]));
              const T H = fm(a.rho, h, v), K = fm(a.rho, s, q.v[3]);
              f0[j] = lo ? v : ad(f0[j], v);
              fH[j] = lo ? H : ad(fH[j], H);
              fK[j] = lo ? K : ad(fK[j], K);
              Dy[j] = lo ? v : sb(Dy[j], v);
              Hy[j] = lo ? H : sb(Hy[j], H);
              Ky[j] = lo ? K : sb(Ky[j], K);
            }
          }
        }
      }
      // its two side points: -x / +x neighbours for j = r, diagonals for the
      // nodes of the rows next to it
      {
        const Pt m = point(slot, kr - 1), p = point(slot, kr + 1);
        Quad<T> qm, qp;
        if (F) {
          qm = hydro(slot, kr - 1);
          qp = hydro(slot, kr + 1);
        }
        if (r >= 0 && r < R) {
          const int j = r;
          const T zm = velz(slot, kr - 1), zp = velz(slot, kr + 1);
          const T bm = mom_b(m.ux), bp = mom_bn(p.ux);
          const T hm = ml(ml(T(4.5), zm), zm), hp = ml(ml(T(4.5), zp), zp);
          const T sm_ = ml(zm, fm(T(9), m.ux, T(3))), sp_ = ml(zp, fm(T(-9), p.ux, T(3)));
#pragma unroll
          for (int f = 0; f < NF; f++) {
            s0[j][f] = ad(s0[j][f], ad(fm(m.C[f], bm, m.A[f]), fm(p.C[f], bp, p.A[f])));
            sE[j][f] = fm(m.C[f], hm, fm(p.C[f], hp, sE[j][f]));
            sQ[j][f] = fm(m.C[f], sm_, fm(p.C[f], sp_, sQ[j][f]));
          }
          if (F) {
            const T vm = fm(a.rho, bm, ad(qm.v[0], qm.v[1]));
            const T vp = fm(a.rho, bp, sb(qp.v[0], qp.v[1]));
            const T Hm = fm(a.rho, hm, vm), Hp = fm(a.rho, hp, vp);
            const T Km = fm(a.rho, sm_, qm.v[3]), Kp = fm(a.rho, sp_, qp.v[3]);
            f0[j] = ad(f0[j], ad(vm, vp));
            fH[j] = ad(fH[j], ad(Hm, Hp));
            fK[j] = ad(fK[j], ad(Km, Kp));
            Dx[j] = sb(vm, vp);
            Hx[j] = sb(Hm, Hp);
            Kx[j] = sb(Km, Kp);
          }
        }
#pragma unroll
        for (int j = 0; j < R; j++) {
          if (r - j == -1 || r - j == 1) {
            const bool lo = r < j;  // from the row below: c = (+, +), (-, +)
            const T bm = mom_b(lo ? ad(m.ux, m.uy) : sb(m.ux, m.uy));
            const T bp = mom_bn(lo ? sb(p.ux, p.uy) : ad(p.ux, p.uy));
#pragma unroll
            for (int f = 0; f < NF; f++) {
              const T t = ad(fm(m.C[f], bm, m.A[f]), fm(p.C[f], bp, p.A[f]));
              gc[j][f] = lo ? t : ad(gc[j][f], t);
            }
            if (F) {
              const T vm =
                  fm(a.rho, bm, ad(qm.v[0], lo ? ad(qm.v[1], qm.v[2]) : sb(qm.v[1], qm.v[2])));
              const T vp =
                  fm(a.rho, bp, sb(qp.v[0], lo ? sb(qp.v[1], qp.v[2]) : ad(qp.v[1], qp.v[2])));
              const T s = ad(vm, vp), d = sb(vm, vp);
              fD[j] = lo ? s : ad(fD[j], s);
              dX[j] = lo ? d : ad(dX[j], d);
              dY[j] = lo ? s : sb(dY[j], s);
            }
          }
        }
      }
      // node r - 1 has its three rows
      if (r >= 1) {
        const int j = r - 1;
#pragma unroll
        for (int f = 0; f < NF; f++) {
          const T P = fm(w2, ad(s0[j][f], sE[j][f]), gP[j][f]), Q = fm(w2, sQ[j][f], gR[j][f]);
          Cd[j][f] = mom_add(gs[j].ck[f], ad(gs[j].mid[f], sb(P, Q)), seed);
          gs[j].mid[f] = ad(gs[j].up[f], fm(w1, s0[j][f], fm(w2, gc[j][f], -out[j][f])));
          gs[j].up[f] = ad(P, Q);
          gs[j].ck[f] = cn[j][f];
        }
        if (F) {
          const T P = fm(w2, fH[j], fP[j]), Q = fm(w2, fK[j], fR[j]);
          const T dn = sb(P, Q);
          d1[j].S = ad(mid[j].S, dn);
          d1[j].X = fm(w2, sb(Hx[j], Kx[j]), mid[j].X);
          d1[j].Y = fm(w2, sb(Hy[j], Ky[j]), mid[j].Y);
          d1[j].Z = sb(mid[j].Z, dn);
          mid[j].S = ad(up[j].S, fm(w1, f0[j], fm(w2, fD[j], f00[j])));
          mid[j].X = ad(up[j].X, fm(w1, Dx[j], ml(w2, dX[j])));
          mid[j].Y = ad(up[j].Y, fm(w1, Dy[j], ml(w2, dY[j])));
          mid[j].Z = up[j].S;
          up[j].S = ad(P, Q);
          up[j].X = ml(w2, ad(Hx[j], Kx[j]));
          up[j].Y = ml(w2, ad(Hy[j], Ky[j]));
        }
      }
    }
  };

  // stencil: of the node of plane p (the last C plane read): c, partial lap and
  // in-plane gradient, T and the in-plane differences; T and c of plane p - 1
  struct Sten {
    T c, L, X, Y, T_, X1, Y1, Tm, cm;
  };
  Sten st[RY][NF];
#pragma unroll
  for (int j = 0; j < RY; j++)
#pragma unroll
    for (int f = 0; f < NF; f++) st[j][f] = Sten{0, 0, 0, 0, 0, 0, 0, 0, 0};
  Duo<T> solv[RY];
  unsigned near[RY];  // as loaded: tested one plane later
#pragma unroll
  for (int j = 0; j < RY; j++) {
    solv[j].v[0] = solv[j].v[1] = T(0);
    near[j] = 0;
  }
  int nc = z0 * plane + nx * y + x;  // the (first) node that collides next

  issue(0);
  cp_async_commit();
  issue(SM::slot);
  cp_async_commit();
  unsigned s_cur = 0, s_next = 2 * SM::slot;  // slots of plane q and of plane q + 2
  unsigned cw = SM::cring;                    // C slot that plane q - 1 goes to
  int q = z0 - 2;
  auto body = [&](auto steady) {
    constexpr bool S = decltype(steady)::value;
    cp_async_wait<1>();
    __syncthreads();
    if (q + 2 <= z1 + 1) issue(s_next);
    cp_async_commit();
    const unsigned cr_ = cw == SM::cring ? SM::cring + NF * SM::cplane : SM::cring;
    // ---- stencil share of C plane q - 2, collision of plane q - 3
    if (S || q >= z0 + 1) {
      T lap[RY][NF], gr[RY][NF][3], Cz[RY][NF];
#pragma unroll
      for (int f = 0; f < NF; f++) {
        const T *c = reinterpret_cast<const T *>(sm + cr_ + f * SM::cplane) + c0i;
        T v[RY + 2][3];
#pragma unroll
        for (int r = 0; r < RY + 2; r++)
#pragma unroll
          for (int e = 0; e < 3; e++) v[r][e] = c[(r - 1) * M3_CX + e - 1];
#pragma unroll
        for (int j = 0; j < RY; j++) {
          Sten &s = st[j][f];
          const T cc = v[j + 1][1];
          const T xp = v[j + 1][2], xm = v[j + 1][0], yp = v[j + 2][1], ym = v[j][1];
          const T pp = v[j + 2][2], mm = v[j][0], pm = v[j][2], mp = v[j + 2][0];
          const T cr = ad(ad(sb(xp, cc), sb(xm, cc)), ad(sb(yp, cc), sb(ym, cc)));
          const T co = ad(ad(sb(pp, cc), sb(mm, cc)), ad(sb(pm, cc), sb(mp, cc)));
          const T t = ml(w2, cr);
          const T x1 = sb(xp, xm), y1 = sb(yp, ym);
          const T da = sb(pp, mm), db = sb(pm, mp);
          const T dz = sb(cc, s.c);  // C(z + 1) - C(z)
          // the node of plane q - 3 complete
          Cz[j][f] = s.c;
          lap[j][f] = ml(T(6), fm(T(1.0 / 6.0), dz, ad(s.L, t)));
          gr[j][f][0] = ml(T(3), fm(w2, x1, s.X));
          gr[j][f][1] = ml(T(3), fm(w2, y1, s.Y));
          gr[j][f][2] = ml(T(3), fm(T(1.0 / 6.0), sb(cc, s.cm), sb(t, s.Tm)));
          // and this plane's node: from its own plane and the one below
          s.L = fm(T(-1.0 / 6.0), dz, ad(fm(w1, cr, ml(w2, co)), s.T_));
          s.X = fm(w2, s.X1, fm(w1, x1, ml(w2, ad(da, db))));
          s.Y = fm(w2, s.Y1, fm(w1, y1, ml(w2, sb(da, db))));
          s.Tm = s.T_;
          s.cm = s.c;
          s.T_ = t;
          s.X1 = x1;
          s.Y1 = y1;
          s.c = cc;
        }
      }
      if (S || q >= z0 + 3) {
#pragma unroll
        for (int j = 0; j < RY; j++) {
          if (x < nx && y + j < ny) {
            const int n = chk(a.err, nc + j * nx, a.N);
            T Sv = d2[j].S, M[3] = {d2[j].X, d2[j].Y, d2[j].Z};
            if (near[j]) {
              const Quad<T> w = reinterpret_cast<const Quad<T> *>(a.wall)[n];
              Sv = ad(Sv, w.v[0]);
              M[0] = ad(M[0], w.v[1]);
              M[1] = ad(M[1], w.v[2]);
              M[2] = ad(M[2], w.v[3]);
            }
            const MomOut<T, NF> o = mom_collide<3, T, NF>(a, solv[j].v[0], solv[j].v[1], Cz[j],
                                                          lap[j], gr[j], Sv, M);
            Quad<T> r;
            r.v[0] = o.A[0];
            r.v[1] = Cz[j][0];
            r.v[2] = o.u[0];
            r.v[3] = o.u[1];
            reinterpret_cast<Quad<T> *>(a.out.q1)[n] = r;
            r.v[0] = o.dP;
            r.v[1] = o.G[0];
            r.v[2] = o.G[1];
            r.v[3] = o.G[2];
            reinterpret_cast<Quad<T> *>(a.out.q2)[n] = r;
            a.out.w[n] = o.u[2];
#pragma unroll
            for (int e = 1; e < NF; e++) {
              Duo<T> p;
              p.v[0] = o.A[e];
              p.v[1] = Cz[j][e];
              reinterpret_cast<Duo<T> *>(a.out.pe)[(e - 1) * a.N + n] = p;
            }
          }
        }
        nc += plane;
      }
#pragma unroll
      for (int j = 0; j < RY; j++) {
        d2[j] = d1[j];
        // the solid's data of the node that collides next
        if (x < nx && y + j < ny && (S || (q >= z0 + 2 && q < z1 + 2))) {
          const int n = chk(a.err, nc + j * nx, a.N);
          solv[j] = reinterpret_cast<const Duo<T> *>(a.sol)[n];
          near[j] = a.near[n];
        }
      }
    }
    if (!S && q > z1 + 1) return;
    // ---- links of plane q
    T Cd[RY][NF];
    typedef std::integral_constant<int, RY> Rows;
    typedef std::integral_constant<int, 1> One;
    if (S || (q >= z0 - 1 && q <= z1)) links(s_cur, k0, g, Cd, std::true_type(), Rows());
    else links(s_cur, k0, g, Cd, std::false_type(), Rows());
    if (S || q >= z0) {
#pragma unroll
      for (int f = 0; f < NF; f++)
#pragma unroll
        for (int j = 0; j < RY; j++)
          reinterpret_cast<T *>(sm + cw + f * SM::cplane)[c0i + j * M3_CX] = Cd[j][f];
    }
    if (extra) {
      T Ce[1][NF];
      links(s_cur, ke, ge, Ce, std::false_type(), One());
      if (S || q >= z0) {
#pragma unroll
        for (int f = 0; f < NF; f++)
          reinterpret_cast<T *>(sm + cw + f * SM::cplane)[cei] = Ce[0][f];
      }
    }
    if (S || q >= z0) cw = cr_;
    s_cur = s_cur == (M3_RING - 1) * SM::slot ? 0 : s_cur + SM::slot;
    s_next = s_next == (M3_RING - 1) * SM::slot ? 0 : s_next + SM::slot;
  };
  for (; q <= z1 + 2; q++) {
    if (q >= z0 + 3 && q <= z1) body(std::true_type());
    else body(std::false_type());
  }
  cp_async_wait<0>();  // no copy outlives the run
}

template <class T, int NF, int TY, int RY, int BPS>
__global__ void __launch_bounds__(M3_X *TY / RY, sizeof(T) == 8 ? 1 : BPS)
    mom_step3_kernel(const __grid_constant__ MomArgs<T> a, int zrun) {
  const int z0 = blockIdx.z * zrun;
  pdl_wait();
  mom_run3<T, NF, TY, RY>(a, blockIdx.x * M3_X, blockIdx.y * TY, z0, min(z0 + zrun, a.nz),
                              a.seed, zsm);
  pdl_next();
}

// ---------------------------------------------------------------------------
// 2D step (D2Q9).  A block stages a TX x TY tile with a two-node halo, sums
// this step's C on the tile and a one-node halo and the streamed f on the
// tile, and collides.  One launch and 65 B per node in FP32 where the two passes
// over populations took two and 128: 4096^2 0.427 -> 0.283 ms per step, 128 x 64
// in FP64 (bound by the FP64 pipe and the launch) 24.6 -> 10.4 us.  32 x 16 tiles:
// 0.375 ms.  STAGE 1 is the relaxation of the solid itself (C is C1; rho = tau =
// tau_g = 1).  Beyond a mirror face the halo holds the image
// nodes with the normal components of u and G reversed, which gives both the
// streaming's specular reflection and the stencils' zero normal gradient.
// ---------------------------------------------------------------------------
template <class T>
struct Mom1 {                  // stage 1
  const unsigned char *mask;   // solid region S
  T beta2, omega2;
  int mirror[2];               // x, y: mirror faces on both sides
};

template <class T, int TX, int TY>
struct M2Smem {
  static constexpr int HX = TX + 4, HY = TY + 4, CX = TX + 2, CY = TY + 2;
  static constexpr int NS = HX * HY, NC = CX * CY;
  static constexpr unsigned o2 = 4 * sizeof(T) * NS;           // (G_x, G_y)
  static constexpr unsigned oc = 6 * sizeof(T) * NS;           // dP
  static constexpr unsigned on = (7 * sizeof(T) * NS + 15) / 16 * 16;  // this step's C
  static constexpr unsigned total = on + sizeof(T) * NC;
};

template <class T, int TX, int TY, int STAGE>
__device__ __forceinline__ void mom_tile2(const MomArgs<T> &a, const Mom1<T> &m1, int x0, int y0,
                                          unsigned seed, unsigned char *sm) {
  using SM = M2Smem<T, TX, TY>;
  using L = Lat<0>;
  constexpr int NT = TX * TY, PER = (SM::NS + NT - 1) / NT, HX = SM::HX;
  constexpr T w0 = T(4.0 / 9.0), w1 = T(1.0 / 9.0), w2 = T(1.0 / 36.0);
  const int tid = threadIdx.x + TX * threadIdx.y;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int nx = a.nx, ny = a.ny;
  const unsigned sbase = (unsigned)__cvta_generic_to_shared(sm);
  // coordinate c of an axis of n nodes as staged; fl: -1 beyond a mirror
  auto map = [](int c, int n, int mirror, int &fl) {
    fl = 1;
    if (mirror) {
      if (c < 0) {
        c = -1 - c;
        fl = -1;
      } else if (c >= n) {
        c = 2 * n - 1 - c;
        fl = -1;
      }
      return c < 0 ? 0 : c;
    }
    if (c < 0) c += n;
    if (c >= n) c -= n;
    if (c < 0 || c >= n) {
      c %= n;
      if (c < 0) c += n;
    }
    return c;
  };
  // a tile whose halo lies within the lattice needs no map (4096^2 291 -> 283 us per
  // step; the relaxation, whose tiles are lighter, is 5 % faster with it: 13.1 us
  // against 13.7 at 1750 x 450)
  const bool inner = STAGE == 2 && x0 >= 2 && y0 >= 2 && x0 + TX + 2 <= nx && y0 + TY + 2 <= ny;
  int flip[PER];
#pragma unroll
  for (int r = 0; r < PER; r++) {
    const int k = tid + r * NT;
    flip[r] = 0;
    if ((r + 1) * NT <= SM::NS || k < SM::NS) {
      int gx = x0 - 2 + k % HX, gy = y0 - 2 + k / HX;
      if (!inner) {
        int fx, fy;
        gx = map(gx, nx, STAGE == 1 ? m1.mirror[0] : 0, fx);
        gy = map(gy, ny, STAGE == 1 ? m1.mirror[1] : 0, fy);
        flip[r] = (fx < 0 ? 1 : 0) | (fy < 0 ? 2 : 0);
      }
      const long long n = chk(a.err, gx + (long long)nx * gy, a.N);
      cp_async_bytes<4 * sizeof(T)>(sbase + k * (4 * sizeof(T)), a.in.q1 + 4 * n);
      cp_async_bytes<2 * sizeof(T)>(sbase + SM::o2 + k * (2 * sizeof(T)), a.in.q2 + 2 * n);
      cp_async_bytes<sizeof(T)>(sbase + SM::oc + k * sizeof(T), a.in.w + n);
    }
  }
  cp_async_commit();
  const int x = x0 + tx, y = y0 + ty;
  const bool inside = x < nx && y < ny;
  const long long n = x + (long long)nx * y;
  Duo<T> solv;
  solv.v[0] = solv.v[1] = T(0);
  unsigned lkv = 0;
  bool inS = false;
  if (inside) {
    if (STAGE == 2) {
      solv = reinterpret_cast<const Duo<T> *>(a.sol)[n];
      lkv = a.lk[n];
    } else {
      inS = m1.mask[n] != 0;
    }
  }
  cp_async_wait<0>();
  if (STAGE == 1 && !inner) {
#pragma unroll
    for (int r = 0; r < PER; r++) {
      if (flip[r]) {
        const int k = tid + r * NT;
        T *q1 = reinterpret_cast<T *>(sm) + 4 * k;
        T *q2 = reinterpret_cast<T *>(sm + SM::o2) + 2 * k;
        if (flip[r] & 1) {
          q1[2] = -q1[2];
          q2[0] = -q2[0];
        }
        if (flip[r] & 2) {
          q1[3] = -q1[3];
          q2[1] = -q2[1];
        }
      }
    }
  }
  __syncthreads();
  auto Q1 = [&](int k) { return *reinterpret_cast<const Quad<T> *>(sm + k * (4 * sizeof(T))); };
  auto Q2 = [&](int k) {
    return *reinterpret_cast<const Duo<T> *>(sm + SM::o2 + k * (2 * sizeof(T)));
  };
  auto DP = [&](int k) { return *reinterpret_cast<const T *>(sm + SM::oc + k * sizeof(T)); };
  T *cn = reinterpret_cast<T *>(sm + SM::on);
  T S, M[3] = {T(0), T(0), T(0)}, C;
  const int k0 = (ty + 2) * HX + tx + 2, c0i = (ty + 1) * SM::CX + tx + 1;
  {
    const Quad<T> p = Q1(k0);
    const T c = p.v[1];
    const T uu = fm(p.v[3], p.v[3], ml(p.v[2], p.v[2]));
    const T out = ml(ml(T(1.5), c), uu);
    T ga, gb, fS, fX, fY;
    {
      const Quad<T> m = Q1(k0 - 1), q = Q1(k0 + 1);
      const T bm = mom_b(m.v[2]), bp = mom_bn(q.v[2]);
      ga = ad(fm(m.v[1], bm, m.v[0]), fm(q.v[1], bp, q.v[0]));
      const T fa = fm(a.rho, bm, ad(DP(k0 - 1), Q2(k0 - 1).v[0]));
      const T fb = fm(a.rho, bp, sb(DP(k0 + 1), Q2(k0 + 1).v[0]));
      fS = ad(fa, fb);
      fX = sb(fa, fb);
    }
    {
      const Quad<T> m = Q1(k0 - HX), q = Q1(k0 + HX);
      const T bm = mom_b(m.v[3]), bp = mom_bn(q.v[3]);
      ga = ad(ga, ad(fm(m.v[1], bm, m.v[0]), fm(q.v[1], bp, q.v[0])));
      const T fa = fm(a.rho, bm, ad(DP(k0 - HX), Q2(k0 - HX).v[1]));
      const T fb = fm(a.rho, bp, sb(DP(k0 + HX), Q2(k0 + HX).v[1]));
      fS = ad(fS, ad(fa, fb));
      fY = sb(fa, fb);
    }
    T da, sa;
    {
      const Quad<T> m = Q1(k0 - 1 - HX), q = Q1(k0 + 1 + HX);
      const Duo<T> gm = Q2(k0 - 1 - HX), gq = Q2(k0 + 1 + HX);
      const T bm = mom_b(ad(m.v[2], m.v[3])), bp = mom_bn(ad(q.v[2], q.v[3]));
      gb = ad(fm(m.v[1], bm, m.v[0]), fm(q.v[1], bp, q.v[0]));
      const T fa = fm(a.rho, bm, ad(DP(k0 - 1 - HX), ad(gm.v[0], gm.v[1])));
      const T fb = fm(a.rho, bp, sb(DP(k0 + 1 + HX), ad(gq.v[0], gq.v[1])));
      sa = ad(fa, fb);
      da = sb(fa, fb);
    }
    {
      const Quad<T> m = Q1(k0 - 1 + HX), q = Q1(k0 + 1 - HX);
      const Duo<T> gm = Q2(k0 - 1 + HX), gq = Q2(k0 + 1 - HX);
      const T bm = mom_b(sb(m.v[2], m.v[3])), bp = mom_bn(sb(q.v[2], q.v[3]));
      gb = ad(gb, ad(fm(m.v[1], bm, m.v[0]), fm(q.v[1], bp, q.v[0])));
      gb = fm(T(-mom_out<L>()), p.v[0], gb);
      const T fa = fm(a.rho, bm, ad(DP(k0 - 1 + HX), sb(gm.v[0], gm.v[1])));
      const T fb = fm(a.rho, bp, sb(DP(k0 + 1 - HX), sb(gq.v[0], gq.v[1])));
      sa = ad(sa, ad(fa, fb));
      const T db = sb(fa, fb);
      M[0] = fm(w1, fX, ml(w2, ad(da, db)));
      M[1] = fm(w1, fY, ml(w2, sb(da, db)));
    }
    S = fm(w1, fS, fm(w2, sa, ml(w0, DP(k0))));
    C = mom_add(c, fm(w1, ga, fm(w2, gb, -out)), seed);
    cn[c0i] = C;
  }
  constexpr int NE = SM::NC - NT;
  if (tid < NE) {  // a halo node's C
    int ci, cj;
    if (tid < 2 * SM::CX) {
      ci = tid % SM::CX;
      cj = tid < SM::CX ? 0 : SM::CY - 1;
    } else {
      const int t = tid - 2 * SM::CX;
      ci = t < TY ? 0 : SM::CX - 1;
      cj = 1 + (t < TY ? t : t - TY);
    }
    const int k = (cj + 1) * HX + ci + 1;
    const Quad<T> p = Q1(k);
    const T c = p.v[1];
    const T uu = fm(p.v[3], p.v[3], ml(p.v[2], p.v[2]));
    const T out = ml(ml(T(1.5), c), uu);
    Quad<T> m = Q1(k - 1), q = Q1(k + 1);
    T ga = ad(fm(m.v[1], mom_b(m.v[2]), m.v[0]), fm(q.v[1], mom_bn(q.v[2]), q.v[0]));
    m = Q1(k - HX);
    q = Q1(k + HX);
    ga = ad(ga, ad(fm(m.v[1], mom_b(m.v[3]), m.v[0]), fm(q.v[1], mom_bn(q.v[3]), q.v[0])));
    m = Q1(k - 1 - HX);
    q = Q1(k + 1 + HX);
    T gb = ad(fm(m.v[1], mom_b(ad(m.v[2], m.v[3])), m.v[0]),
              fm(q.v[1], mom_bn(ad(q.v[2], q.v[3])), q.v[0]));
    m = Q1(k - 1 + HX);
    q = Q1(k + 1 - HX);
    gb = ad(gb, ad(fm(m.v[1], mom_b(sb(m.v[2], m.v[3])), m.v[0]),
                   fm(q.v[1], mom_bn(sb(q.v[2], q.v[3])), q.v[0])));
    gb = fm(T(-mom_out<L>()), p.v[0], gb);
    cn[cj * SM::CX + ci] = mom_add(c, fm(w1, ga, fm(w2, gb, -out)), seed);
  }
  __syncthreads();
  if (!inside) return;
  T g[1][3], lap[1], Cv[1] = {C};
  {
    const T *c = cn + c0i;
    constexpr int CX = SM::CX;
    const T xp = c[1], xm = c[-1], yp = c[CX], ym = c[-CX];
    const T pp = c[CX + 1], mm = c[-CX - 1], pm = c[-CX + 1], mp = c[CX - 1];
    const T cr = ad(ad(sb(xp, C), sb(xm, C)), ad(sb(yp, C), sb(ym, C)));
    const T co = ad(ad(sb(pp, C), sb(mm, C)), ad(sb(pm, C), sb(mp, C)));
    const T da = sb(pp, mm), db = sb(pm, mp);
    lap[0] = ml(T(6), fm(w1, cr, ml(w2, co)));
    g[0][0] = ml(T(3), fm(w1, sb(xp, xm), ml(w2, ad(da, db))));
    g[0][1] = ml(T(3), fm(w1, sb(yp, ym), ml(w2, sb(da, db))));
    g[0][2] = T(0);
  }
  T A, dP, u[2], G[2];
  if (STAGE == 2) {
    if (lkv)  // every node it needs is staged
      mom_walls<L>(
          a, lkv, n,
          [&](int j) {
            const int k = k0 + L::cx(j) + HX * L::cy(j);
            const Quad<T> p = Q1(k);
            const Duo<T> d = Q2(k);
            MomNode<T> m;
            m.dP = DP(k);
            m.u[0] = p.v[2];
            m.u[1] = p.v[3];
            m.G[0] = d.v[0];
            m.G[1] = d.v[1];
            m.u[2] = m.G[2] = T(0);
            return m;
          },
          S, M);
    const MomOut<T, 1> o = mom_collide<2, T, 1>(a, solv.v[0], solv.v[1], Cv, lap, g, S, M);
    A = o.A[0];
    dP = o.dP;
    u[0] = o.u[0];
    u[1] = o.u[1];
    G[0] = o.G[0];
    G[1] = o.G[1];
  } else {
    // k[0], ak[0]: kappa_1 + kappa_3 and its alpha^2 multiple
    T mu = fm(a.k[0], mom_well(C), ml(-a.ak[0], lap[0]));
    if (inS ? C < T(0.5) : C > T(0.5)) mu = fm(m1.beta2, sb(C, T(0.5)), mu);
    if (C < T(0)) mu = fm(m1.omega2, C, mu);
    if (C > T(1)) mu = fm(-m1.omega2, sb(T(1), C), mu);
    T uu = T(0), bad = mu;
#pragma unroll
    for (int e = 0; e < 2; e++) {
      const T F = ml(mu, g[0][e]);
      u[e] = fm(T(0.5), F, M[e]);
      G[e] = ml(T(1.5), F);
      uu = fm(u[e], u[e], uu);
      bad = ad(bad, u[e]);
    }
    const T h = ml(T(-1.5), uu);
    dP = ad(S, h);
    A = fm(C, h, mu);
    if (!isfinite(ad(bad, dP))) atomicOr(a.err, ERR_NONFINITE);
  }
  const long long m = chk(a.err, n, a.N);
  Quad<T> r;
  r.v[0] = A;
  r.v[1] = C;
  r.v[2] = u[0];
  r.v[3] = u[1];
  reinterpret_cast<Quad<T> *>(a.out.q1)[m] = r;
  Duo<T> d;
  d.v[0] = G[0];
  d.v[1] = G[1];
  reinterpret_cast<Duo<T> *>(a.out.q2)[m] = d;
  a.out.w[m] = dP;
}

template <class T, int TX, int TY, int STAGE>
__global__ void __launch_bounds__(TX *TY)
    mom_step2_kernel(const __grid_constant__ MomArgs<T> a, const __grid_constant__ Mom1<T> m1) {
  pdl_next();
  pdl_wait();
  mom_tile2<T, TX, TY, STAGE>(a, m1, blockIdx.x * TX, blockIdx.y * TY, a.seed, zsm);
}

// ---------------------------------------------------------------------------
// Around the step: the frozen solid's data, the rest state, conversion from and
// to the canonical state (f, A, u, C), populations.
// ---------------------------------------------------------------------------

// sol, lk and qpl from C1 (a.sol, a.lk, a.qpl are written here)
template <int K, class T>
__global__ void __launch_bounds__(256) mom_solid_kernel(const __grid_constant__ MomArgs<T> a) {
  using L = Lat<K>;
  constexpr int Q = L::Q;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z * blockDim.z + threadIdx.z;
  if (x >= a.nx || y >= a.ny || z >= a.nz) return;
  Hood h;
  h.init(x, y, z, a.nx, a.ny, a.nz);
  h.guard(a.err);
  const int n = h.g(h.ox[1] + h.oy[1] + h.oz[1]);
  const T c1 = a.c1[n];
  T lap = T(0), g[3] = {T(0), T(0), T(0)};
  unsigned lk = 0;
#pragma unroll
  for (int i = 1; i < Q; i++) {
    const T v = a.c1[h.plus<L>(i)], w = T(L::w(i));
    lap += w * (v - c1);
    if (L::cx(i)) g[0] += w * T(L::cx(i)) * v;
    if (L::cy(i)) g[1] += w * T(L::cy(i)) * v;
    if (L::cz(i)) g[2] += w * T(L::cz(i)) * v;
    lk |= (v >= T(0.5) ? 1u : 0u) << i;
  }
  if (c1 >= T(0.5)) lk = 0;
  Duo<T> s;
  s.v[0] = c1;
  s.v[1] = T(6) * lap;
  reinterpret_cast<Duo<T> *>(const_cast<T *>(a.sol))[n] = s;
  if (K == 0) const_cast<unsigned *>(a.lk)[n] = lk;
  else const_cast<unsigned char *>(a.near)[n] = lk != 0;
  if (!lk) return;
  int k = n;
  if (K == 1) {
    k = chk(a.err, atomicAdd(a.count, 1), a.N);
    a.list[k] = n;
    const_cast<unsigned *>(a.lk)[k] = lk;
  }
#pragma unroll
  for (int d = 0; d < 3; d++) g[d] *= T(3);
  const T cc = c1 < T(1e-9) ? T(1e-9) : c1;
  const T xs = T(2) * a.alpha_s * atanh(T(2) * cc - T(1));
  const T gn = sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
#pragma unroll
  for (int j = 1; j < Q; j++) {
    const int i = L::opp(j);
    const bool link = (lk >> i) & 1u;
    if (link || K == 1)
      const_cast<T *>(a.qpl)[(long long)(j - 1) * a.pitch + k] =
          link ? link_fraction<L, T>(xs, gn, g[0], g[1], g[2], i) : T(0.5);
  }
}

// stores one node of a buffer
template <int K, class T>
__device__ __forceinline__ void mom_store(const MomBuf<T> &b, long long n, T A, T dP, T ux, T uy,
                                          T uz, T C, T Gx, T Gy, T Gz) {
  Quad<T> r;
  r.v[0] = A;
  r.v[1] = C;
  r.v[2] = ux;
  r.v[3] = uy;
  reinterpret_cast<Quad<T> *>(b.q1)[n] = r;
  if (K == 1) {
    r.v[0] = dP;
    r.v[1] = Gx;
    r.v[2] = Gy;
    r.v[3] = Gz;
    reinterpret_cast<Quad<T> *>(b.q2)[n] = r;
    b.w[n] = uz;
  } else {
    Duo<T> d;
    d.v[0] = Gx;
    d.v[1] = Gy;
    reinterpret_cast<Duo<T> *>(b.q2)[n] = d;
    b.w[n] = dP;
  }
}

// C of the next step at one node, from its neighbours' (A, C, u)
template <int K, class T, int NF>
__global__ void __launch_bounds__(256)
    mom_c_kernel(const __grid_constant__ MomArgs<T> a, T *out, long long ostride) {
  using L = Lat<K>;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z * blockDim.z + threadIdx.z;
  if (x >= a.nx || y >= a.ny || z >= a.nz) return;
  Hood h;
  h.init(x, y, z, a.nx, a.ny, a.nz);
  h.guard(a.err);
  const int n = h.g(h.ox[1] + h.oy[1] + h.oz[1]);
  T sa[NF], sd[NF], out0[NF], ak[NF], ck[NF];
#pragma unroll
  for (int i = 0; i < L::Q; i++) {
    const int m = i == 0 ? n : h.minus<L>(i);
    const Quad<T> q = reinterpret_cast<const Quad<T> *>(a.in.q1)[m];
    const T u[3] = {q.v[2], q.v[3], L::D == 3 && (i == 0 || L::cz(i)) ? a.in.w[m] : T(0)};
    const T b = i == 0 ? T(0) : mom_b(mom_dot<L>(i, u));
    const T uu = i == 0 ? fm(u[2], u[2], fm(u[1], u[1], ml(u[0], u[0]))) : T(0);
#pragma unroll
    for (int f = 0; f < NF; f++) {
      T A = q.v[0], C = q.v[1];
      if (f > 0) {
        const Duo<T> d = reinterpret_cast<const Duo<T> *>(a.in.pe)[(f - 1) * a.N + m];
        A = d.v[0];
        C = d.v[1];
      }
      if (i == 0) {
        ck[f] = C;
        out0[f] = ml(ml(T(1.5), C), uu);
        ak[f] = A;
        sa[f] = sd[f] = T(0);
      } else if (L::w(i) == L::w(1)) {
        sa[f] = ad(sa[f], fm(C, b, A));
      } else {
        sd[f] = ad(sd[f], fm(C, b, A));
      }
    }
  }
#pragma unroll
  for (int f = 0; f < NF; f++) {
    sd[f] = fm(T(-mom_out<L>()), ak[f], sd[f]);
    const T d = fm(T(L::w(1)), sa[f], fm(T(L::w(L::Q - 1)), sd[f], -out0[f]));
    out[f * ostride + n] = mom_add(ck[f], d, a.seed);
  }
}

// The rest of the step at one node, from this step's C (planes cn, cstride
// apart): the second of two passes (MODE_STEP), one field (MODE_FIELDS) or the
// observables (MODE_OBS).
template <int K, class T, int NF, int MODE>
__global__ void __launch_bounds__(256)
    mom_node_kernel(const __grid_constant__ MomArgs<T> a, const T *cn, long long cstride, T *fields,
                    int field, int index, double *partials) {
  using L = Lat<K>;
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  int z = blockIdx.z * blockDim.z + threadIdx.z;
  const bool valid = x < a.nx && y < a.ny && z < a.nz;
  if (MODE != MODE_OBS && !valid) return;
  if (!valid) x = y = z = 0;
  Hood h;
  h.init(x, y, z, a.nx, a.ny, a.nz);
  h.guard(a.err);
  const int n = h.g(h.ox[1] + h.oy[1] + h.oz[1]);
  const Duo<T> s = reinterpret_cast<const Duo<T> *>(a.sol)[n];
  T C[NF], lap[NF], g[NF][3];
#pragma unroll
  for (int f = 0; f < NF; f++) {
    const T *c = cn + f * cstride;
    C[f] = c[n];
    T la = T(0), ld = T(0), ga[3] = {T(0), T(0), T(0)}, gd[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int i = 1; i < L::Q; i += 2) {  // opposite neighbours
      const T p = c[h.plus<L>(i)], m = c[h.plus<L>(i + 1)];
      const T l = ad(sb(p, C[f]), sb(m, C[f])), d = sb(p, m);
      const bool axis = L::w(i) == L::w(1);
      if (axis) la = ad(la, l);
      else ld = ad(ld, l);
#pragma unroll
      for (int e = 0; e < 3; e++) {
        const int ce = e == 0 ? L::cx(i) : (e == 1 ? L::cy(i) : L::cz(i));
        if (ce == 0) continue;
        T &t = axis ? ga[e] : gd[e];
        t = ce > 0 ? ad(t, d) : sb(t, d);
      }
    }
    lap[f] = ml(T(6), fm(T(L::w(1)), la, ml(T(L::w(L::Q - 1)), ld)));
#pragma unroll
    for (int e = 0; e < 3; e++)
      g[f][e] = ml(T(3), fm(T(L::w(1)), ga[e], ml(T(L::w(L::Q - 1)), gd[e])));
  }
  T Sa = T(0), Sd = T(0), Ma[3] = {T(0), T(0), T(0)}, Md[3] = {T(0), T(0), T(0)};
  T S = T(0);
#pragma unroll
  for (int j = 0; j < L::Q; j++) {
    const T v = mom_phi<L>(mom_load<L>(a.in, j == 0 ? n : h.minus<L>(j)), j, a.rho);
    if (j == 0) {
      S = ml(T(L::w(0)), v);
      continue;
    }
    const bool axis = L::w(j) == L::w(1);
    if (axis) Sa = ad(Sa, v);
    else Sd = ad(Sd, v);
#pragma unroll
    for (int e = 0; e < 3; e++) {
      const int ce = e == 0 ? L::cx(j) : (e == 1 ? L::cy(j) : L::cz(j));
      if (ce == 0) continue;
      T &t = axis ? Ma[e] : Md[e];
      t = ce > 0 ? ad(t, v) : sb(t, v);
    }
  }
  S = fm(T(L::w(1)), Sa, fm(T(L::w(L::Q - 1)), Sd, S));
  T M[3];
#pragma unroll
  for (int e = 0; e < 3; e++) M[e] = fm(T(L::w(1)), Ma[e], ml(T(L::w(L::Q - 1)), Md[e]));
  if constexpr (K == 1) {  // summed ahead (mom_wall_nodes)
    if (a.near[n]) {
      const Quad<T> w = reinterpret_cast<const Quad<T> *>(a.wall)[n];
      S = ad(S, w.v[0]);
#pragma unroll
      for (int e = 0; e < 3; e++) M[e] = ad(M[e], w.v[1 + e]);
    }
  } else {
    const unsigned lk = a.lk[n];
    if (lk)
      mom_walls<L>(
          a, lk, n, [&](int j) { return mom_load<L>(a.in, j == 0 ? n : h.plus<L>(j)); }, S, M);
  }
  const MomOut<T, NF> o = mom_collide<L::D, T, NF>(a, s.v[0], s.v[1], C, lap, g, S, M);
  const bool solid = s.v[0] >= T(0.5);
  if constexpr (MODE == MODE_STEP) {
    mom_store<K, T>(a.out, n, o.A[0], o.dP, o.u[0], o.u[1], o.u[2], C[0], o.G[0], o.G[1], o.G[2]);
#pragma unroll
    for (int e = 1; e < NF; e++) {
      Duo<T> d;
      d.v[0] = o.A[e];
      d.v[1] = C[e];
      reinterpret_cast<Duo<T> *>(a.out.pe)[(e - 1) * a.N + n] = d;
    }
  } else if constexpr (MODE == MODE_FIELDS) {
    T v, last = sb(T(1), s.v[0]);
#pragma unroll
    for (int f = 0; f < NF; f++) last = sb(last, C[f]);
    switch (field) {
      case DSM_FIELD_C1: v = s.v[0]; break;
      case DSM_FIELD_C2:
        v = last;
#pragma unroll
        for (int f = 0; f < NF; f++)
          if (index == f) v = C[f];
        break;
      case DSM_FIELD_C3: v = last; break;
      case DSM_FIELD_MU:
        v = o.mu[0];
#pragma unroll
        for (int f = 1; f < NF; f++)
          if (index == f) v = o.mu[f];
        break;
      case DSM_FIELD_UX: v = o.u[0]; break;
      case DSM_FIELD_UY: v = o.u[1]; break;
      case DSM_FIELD_UZ: v = o.u[2]; break;
      case DSM_FIELD_PT: v = solid ? T(1) : ad(T(1), S); break;
      case DSM_FIELD_RHO: v = a.rho; break;
      default: v = T(1); break;
    }
    fields[n] = v;
  } else {
    const bool bad = (!solid && !isfinite(S)) || !isfinite(C[0]);
    const long long b = blockIdx.x + (long long)gridDim.x * (blockIdx.y + (long long)gridDim.y * blockIdx.z);
    if constexpr (sizeof(T) == 4) {
      const float vals[OBS_K] = {valid ? float(C[0]) : 0.f, valid ? float(s.v[0]) : 0.f,
                                 valid ? 0.5f * float(a.rho) * float(o.uu) : 0.f,
                                 valid ? sqrtf(float(o.uu)) : 0.f, (valid && bad) ? 1.f : 0.f};
      const int is_max[OBS_K] = {0, 0, 0, 1, 1};
      block_reduce_ff<OBS_K>(vals, is_max, partials + b * OBS_K);
    } else {
      const double vals[OBS_K] = {valid ? double(C[0]) : 0.0, valid ? double(s.v[0]) : 0.0,
                                  valid ? 0.5 * double(a.rho) * double(o.uu) : 0.0,
                                  valid ? sqrt(double(o.uu)) : 0.0, (valid && bad) ? 1.0 : 0.0};
      block_reduce_obs(vals, partials + b * OBS_K);
    }
  }
}

// 3D, two fluids: a field (MODE_FIELDS) or the observables (MODE_OBS) of the state
// whose next step is in a.in.  That step's moments hold C and u themselves, and
// pt = 1 + dP + 3/2 rho u.u and mu = A + 3/2 C u.u.  The step stages its points once,
// where mom_node_kernel gathers 19 neighbours' nine reals through L1: C2 and then pt
// of 384 x 384 x 256 2.48 -> 1.79 ms, the step's 0.98 among them.
template <class T, int MODE>
__global__ void __launch_bounds__(256)
    mom_peek_kernel(const __grid_constant__ MomArgs<T> a, T *fields, int field, double *partials) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z * blockDim.z + threadIdx.z;
  const bool valid = x < a.nx && y < a.ny && z < a.nz;
  if (MODE != MODE_OBS && !valid) return;
  const long long n = valid ? chk(a.err, x + (long long)a.nx * (y + (long long)a.ny * z), a.N) : 0;
  const Quad<T> q = reinterpret_cast<const Quad<T> *>(a.in.q1)[n];
  if constexpr (MODE == MODE_FIELDS) {
    const T uz = a.in.w[n];
    const T uu = fm(uz, uz, fm(q.v[3], q.v[3], ml(q.v[2], q.v[2])));
    const T h = ml(T(-1.5), uu);
    T v;
    switch (field) {
      case DSM_FIELD_C2: v = q.v[1]; break;
      case DSM_FIELD_C3:
        v = sb(sb(T(1), reinterpret_cast<const Duo<T> *>(a.sol)[n].v[0]), q.v[1]);
        break;
      case DSM_FIELD_MU: v = fm(-q.v[1], h, q.v[0]); break;
      case DSM_FIELD_UX: v = q.v[2]; break;
      case DSM_FIELD_UY: v = q.v[3]; break;
      case DSM_FIELD_UZ: v = uz; break;
      // (a solid node holds dP = u = 0)
      case DSM_FIELD_PT: v = ad(T(1), fm(-a.rho, h, a.in.q2[4 * n])); break;
      case DSM_FIELD_RHO: v = a.rho; break;
      default: v = T(1); break;
    }
    fields[n] = v;
  } else {
    const T c1 = reinterpret_cast<const Duo<T> *>(a.sol)[n].v[0], uz = a.in.w[n];
    const T uu = fm(uz, uz, fm(q.v[3], q.v[3], ml(q.v[2], q.v[2])));
    const bool bad = !isfinite(a.in.q2[4 * n]) || !isfinite(q.v[1]);
    const long long b = blockIdx.x + (long long)gridDim.x * (blockIdx.y + (long long)gridDim.y * blockIdx.z);
    if constexpr (sizeof(T) == 4) {
      const float vals[OBS_K] = {valid ? float(q.v[1]) : 0.f, valid ? float(c1) : 0.f,
                                 valid ? 0.5f * float(a.rho) * float(uu) : 0.f,
                                 valid ? sqrtf(float(uu)) : 0.f, (valid && bad) ? 1.f : 0.f};
      const int is_max[OBS_K] = {0, 0, 0, 1, 1};
      block_reduce_ff<OBS_K>(vals, is_max, partials + b * OBS_K);
    } else {
      const double vals[OBS_K] = {valid ? double(q.v[1]) : 0.0, valid ? double(c1) : 0.0,
                                  valid ? 0.5 * double(a.rho) * double(uu) : 0.0,
                                  valid ? sqrt(double(uu)) : 0.0, (valid && bad) ? 1.0 : 0.0};
      block_reduce_obs(vals, partials + b * OBS_K);
    }
  }
}

// the state at rest of C (N reals per free fluid, cstride apart) into a.out:
// f_i = w_i, g_i = g_eq_i(C, mu(C), 0), i.e. A = mu and dP = u = G = 0
template <int K, class T, int NF>
__global__ void __launch_bounds__(256)
    mom_init_kernel(const __grid_constant__ MomArgs<T> a, const T *cf, long long cstride) {
  using L = Lat<K>;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z * blockDim.z + threadIdx.z;
  if (x >= a.nx || y >= a.ny || z >= a.nz) return;
  Hood h;
  h.init(x, y, z, a.nx, a.ny, a.nz);
  h.guard(a.err);
  const int n = h.g(h.ox[1] + h.oy[1] + h.oz[1]);
  const Duo<T> s = reinterpret_cast<const Duo<T> *>(a.sol)[n];
  T c[NF], lap[NF], sum = s.v[0], sl = s.v[1];
#pragma unroll
  for (int f = 0; f < NF; f++) {
    c[f] = cf[f * cstride + n];
    lap[f] = T(0);
#pragma unroll
    for (int i = 1; i < L::Q; i++)
      lap[f] += T(L::w(i)) * (cf[f * cstride + h.plus<L>(i)] - c[f]);
    lap[f] *= T(6);
    sum += c[f];
    sl += lap[f];
  }
  const T dl = a.kl * mom_well(sum) - a.akl * sl;
#pragma unroll
  for (int f = 0; f < NF; f++) {
    const T mu = a.k[f] * mom_well(c[f]) - a.ak[f] * lap[f] + dl;
    if (f == 0) {
      mom_store<K, T>(a.out, n, mu, T(0), T(0), T(0), T(0), c[0], T(0), T(0), T(0));
    } else {
      Duo<T> d;
      d.v[0] = mu;
      d.v[1] = c[f];
      reinterpret_cast<Duo<T> *>(a.out.pe)[(f - 1) * a.N + n] = d;
    }
  }
}

// Stage 1: the state at rest of C1 (cf) into a.out, and the C1 the next step
// would see.  Beyond a mirror the neighbour is the edge node, its velocity
// reversed along the normal.
template <class T>
__global__ void __launch_bounds__(256)
    mom_relax_init_kernel(const __grid_constant__ MomArgs<T> a, const __grid_constant__ Mom1<T> m1,
                          const T *cf) {
  using L = Lat<0>;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= a.nx || y >= a.ny) return;
  const int face[6] = {m1.mirror[0], m1.mirror[0], m1.mirror[1], m1.mirror[1], 0, 0};
  Hood h;
  h.init_faces(x, y, 0, a.nx, a.ny, 1, face);
  h.guard(a.err);
  const int n = h.g(h.ox[1] + h.oy[1]);
  const T C = cf[n];
  T lap = T(0);
#pragma unroll
  for (int i = 1; i < L::Q; i++) lap += T(L::w(i)) * (cf[h.plus<L>(i)] - C);
  T mu = a.k[0] * mom_well(C) - a.ak[0] * (T(6) * lap);
  if (m1.mask[n] != 0 ? C < T(0.5) : C > T(0.5)) mu += m1.beta2 * (C - T(0.5));
  if (C < T(0)) mu += m1.omega2 * C;
  if (C > T(1)) mu -= m1.omega2 * (T(1) - C);
  mom_store<0, T>(a.out, n, mu, T(0), T(0), T(0), T(0), C, T(0), T(0), T(0));
}
template <class T>
__global__ void __launch_bounds__(256)
    mom_relax_c_kernel(const __grid_constant__ MomArgs<T> a, const __grid_constant__ Mom1<T> m1,
                       T *out) {
  using L = Lat<0>;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= a.nx || y >= a.ny) return;
  const int face[6] = {m1.mirror[0], m1.mirror[0], m1.mirror[1], m1.mirror[1], 0, 0};
  Hood h;
  h.init_faces(x, y, 0, a.nx, a.ny, 1, face);
  h.guard(a.err);
  const int n = h.g(h.ox[1] + h.oy[1]);
  const Quad<T> q = reinterpret_cast<const Quad<T> *>(a.in.q1)[n];
  const T uu = fm(q.v[3], q.v[3], ml(q.v[2], q.v[2]));
  T sa = T(0), sd = T(0);
#pragma unroll
  for (int i = 1; i < L::Q; i++) {
    const Quad<T> p = reinterpret_cast<const Quad<T> *>(a.in.q1)[h.minus<L>(i)];
    const bool rx = m1.mirror[0] && x - L::cx(i) != (x - L::cx(i) + a.nx) % a.nx;
    const bool ry = m1.mirror[1] && y - L::cy(i) != (y - L::cy(i) + a.ny) % a.ny;
    const T u[3] = {rx ? -p.v[2] : p.v[2], ry ? -p.v[3] : p.v[3], T(0)};
    const T g = fm(p.v[1], mom_b(mom_dot<L>(i, u)), p.v[0]);
    if (L::w(i) == L::w(1)) sa = ad(sa, g);
    else sd = ad(sd, g);
  }
  sd = fm(T(-mom_out<L>()), q.v[0], sd);
  const T d = fm(T(L::w(1)), sa, fm(T(L::w(L::Q - 1)), sd, -ml(ml(T(1.5), q.v[1]), uu)));
  out[n] = mom_add(q.v[1], d, a.seed);
}

// canonical state planes: f (Q, storage type S), u (D), and A and C of each free
// fluid
template <class T, class S = T>
struct MomCanon {
  S *f;
  T *A, *U, *C;  // planes pitch apart
};
// f_i - w_i of a stored population, and the way back from phi_i
template <class T, class S>
__device__ __forceinline__ T mom_f_dev(S v, double w) {
  if constexpr (Store<S>::k16) return T(Store<S>::dec(v));
  else return T(v) - T(w);
}
template <class T, class S>
__device__ __forceinline__ S mom_f_of(T phi, double w) {
  if constexpr (Store<S>::k16) return Store<S>::enc(float(ml(T(w), phi)));
  else return fm(T(w), phi, T(w));
}

// canonical state whose last step had every relaxation time 1 -> a.out:
// the moments of f_i - w_i fix dP and G (sum_i w_i phi_i = dP + 3/2 rho u.u,
// sum_i c_i w_i phi_i = rho u + G/3)
template <int K, class T, int NF, class S>
__global__ void __launch_bounds__(256)
    mom_enter_kernel(const __grid_constant__ MomArgs<T> a, MomCanon<T, S> s) {
  using L = Lat<K>;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < a.N;
       n += (long long)gridDim.x * blockDim.x) {
    T m0 = mom_f_dev<T>(s.f[n], L::w(0)), m[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int j = 1; j < L::Q; j += 2) {
      const S va = s.f[(long long)j * a.pitch + n], vb = s.f[(long long)(j + 1) * a.pitch + n];
      const T fa = mom_f_dev<T>(va, L::w(j)), fb = mom_f_dev<T>(vb, L::w(j));
      m0 += fa + fb;
      const T d = Store<S>::k16 ? fa - fb : T(Store<S>::dec(va)) - T(Store<S>::dec(vb));
      if (L::cx(j)) m[0] += T(L::cx(j)) * d;
      if (L::cy(j)) m[1] += T(L::cy(j)) * d;
      if (L::cz(j)) m[2] += T(L::cz(j)) * d;
    }
    T u[3] = {s.U[n], s.U[a.pitch + n], L::D == 3 ? s.U[2 * a.pitch + n] : T(0)}, G[3];
    const T uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
#pragma unroll
    for (int e = 0; e < 3; e++) G[e] = T(3) * (m[e] - a.rho * u[e]);
    mom_store<K, T>(a.out, n, s.A[n], m0 - T(1.5) * a.rho * uu, u[0], u[1], u[2], s.C[n], G[0],
                    G[1], G[2]);
#pragma unroll
    for (int e = 1; e < NF; e++) {
      Duo<T> d;
      d.v[0] = s.A[e * a.pitch + n];
      d.v[1] = s.C[e * a.pitch + n];
      reinterpret_cast<Duo<T> *>(a.out.pe)[(e - 1) * a.N + n] = d;
    }
  }
}

// a.in -> the canonical state (for reads and other step forms; what = 1), or
// the populations f and g, planes N apart (what = 2; null: not written)
template <int K, class T, int NF, class S>
__global__ void __launch_bounds__(256)
    mom_expand_kernel(const __grid_constant__ MomArgs<T> a, MomCanon<T, S> s, int what) {
  using L = Lat<K>;
  const long long stride = what == 1 ? a.pitch : a.N;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < a.N;
       n += (long long)gridDim.x * blockDim.x) {
    const MomNode<T> m = mom_load<L>(a.in, n);
    T A[NF], C[NF];
    A[0] = a.in.q1[4 * n];
    C[0] = a.in.q1[4 * n + 1];
#pragma unroll
    for (int e = 1; e < NF; e++) {
      const Duo<T> d = reinterpret_cast<const Duo<T> *>(a.in.pe)[(e - 1) * a.N + n];
      A[e] = d.v[0];
      C[e] = d.v[1];
    }
    if (s.f) {
#pragma unroll
      for (int i = 0; i < L::Q; i++)
        s.f[i * stride + n] = mom_f_of<T, S>(mom_phi<L>(m, i, a.rho), L::w(i));
    }
    if (what == 1) {
#pragma unroll
      for (int f = 0; f < NF; f++) {
        s.A[f * stride + n] = A[f];
        s.C[f * stride + n] = C[f];
      }
#pragma unroll
      for (int e = 0; e < L::D; e++) s.U[e * stride + n] = m.u[e];
    } else if (s.C) {
      const T uu = m.u[0] * m.u[0] + m.u[1] * m.u[1] + m.u[2] * m.u[2];
#pragma unroll
      for (int f = 0; f < NF; f++) {
        T *g = s.C + (long long)f * L::Q * stride;
        g[n] = C[f] - (T(1.0 - L::w(0)) * A[f] + T(1.5) * C[f] * uu);
#pragma unroll
        for (int i = 1; i < L::Q; i++)
          g[i * stride + n] = T(L::w(i)) * geq_core(A[f], C[f], cdot<L>(i, m.u[0], m.u[1], m.u[2]));
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Batched launch: one cooperative launch advances many lattices.  Every lattice
// owns a share of the resident blocks in proportion to its work; its blocks
// walk its tiles (3D: tiles and runs of planes) and meet at a barrier of their
// own after each step, so lattices do not wait for one another.  Every wait is
// bounded as in the population form's batch (grid_barrier).
// ---------------------------------------------------------------------------
template <class T>
struct MomItem {
  MomArgs<T> a[2];  // a[p]: reads buffer p
  int block0, blocks, tx, ty, runs, zrun, nsteps, cur0;
  unsigned bar[2];  // arrivals, generation
};

template <class T>
__device__ __forceinline__ bool mom_barrier(MomItem<T> *items, int nitems, MomItem<T> *it,
                                            unsigned long long limit) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    ok = 1;
    volatile unsigned *gen = it->bar + 1;
    const unsigned g = *gen;
    __threadfence();
    if (atomicAdd(it->bar, 1u) == (unsigned)it->blocks - 1) {
      atomicExch(it->bar, 0u);
      __threadfence();
      atomicAdd(it->bar + 1, 1u);
    } else {
      unsigned long long spins = 0;
      while (*gen == g) {
        if (++spins > limit) {
          for (int i = 0; i < nitems; i++) atomicOr(items[i].a[0].err, ERR_TIMEOUT);
          ok = 0;
          break;
        }
        __nanosleep(40);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

template <int K>
constexpr int mom_batch_threads() {
  return K == 1 ? 128 : 256;
}
template <int K, class T>
__global__ void __launch_bounds__(mom_batch_threads<K>(), sizeof(T) == 8 ? 1 : 4)
    mom_batch_kernel(MomItem<T> *items, int nitems, const int *owner,
                     unsigned long long spin_limit) {
  __shared__ MomArgs<T> sa[2];
  __shared__ int meta[8];
  MomItem<T> *it = items + owner[blockIdx.x];
  const int tid = threadIdx.x + 32 * threadIdx.y;
  constexpr int NT = mom_batch_threads<K>();
  for (int w = tid; w < (int)(sizeof(sa) / sizeof(int)); w += NT)
    ((int *)sa)[w] = ((const int *)it->a)[w];
  if (tid < 8) meta[tid] = (&it->block0)[tid];
  __syncthreads();
  const int tiles = meta[2] * meta[3] * meta[4];
  for (int t = 0; t < meta[6]; t++) {
    const MomArgs<T> &a = sa[(meta[7] + t) & 1];
    if constexpr (K == 1) {
      mom_wall_nodes(a, (blockIdx.x - meta[0]) * NT + tid, meta[1] * NT);
      if (!mom_barrier(items, nitems, it, spin_limit)) return;
    }
    for (int b = blockIdx.x - meta[0]; b < tiles; b += meta[1]) {
      const int bx = b % meta[2], by = (b / meta[2]) % meta[3];
      if constexpr (K == 1) {
        const int z0 = b / (meta[2] * meta[3]) * meta[5];
        mom_run3<T, 1, 8, 2>(a, bx * M3_X, by * 8, z0, min(z0 + meta[5], a.nz),
                             a.seed + MOM_SEED * (unsigned)t, zsm);
      } else {
        mom_tile2<T, 32, 8, 2>(a, Mom1<T>{}, bx * 32, by * 8, a.seed + MOM_SEED * (unsigned)t, zsm);
      }
      __syncthreads();  // the tile's shared memory is free
    }
    if (!mom_barrier(items, nitems, it, spin_limit)) return;
  }
}

// ---- host side -----------------------------------------------------------------
template <class T>
MomArgs<T> mom_typed(const MomRaw &r) {
  MomArgs<T> a;
  a.nx = r.nx;
  a.ny = r.ny;
  a.nz = r.nz;
  a.N = r.N;
  a.pitch = r.pitch;
  a.in = {(T *)r.in[0], (T *)r.in[1], (T *)r.in[2], (T *)r.in[3]};
  a.out = {(T *)r.out[0], (T *)r.out[1], (T *)r.out[2], (T *)r.out[3]};
  a.sol = (const T *)r.sol;
  a.lk = (const unsigned *)r.lk;
  a.qpl = (const T *)r.qpl;
  a.near = (const unsigned char *)r.near;
  a.list = (unsigned *)r.list;
  a.count = r.count;
  a.wall = (T *)r.wall;
  a.c1 = (const T *)r.c1;
  a.err = r.err;
  for (int f = 0; f < MOM_NF; f++) {
    a.k[f] = T(r.k[f]);
    a.ak[f] = T(r.ak[f]);
    a.body[f] = T(r.body[f]);
  }
  a.kl = T(r.kl);
  a.akl = T(r.akl);
  a.rho = T(r.rho);
  a.irho = T(1.0 / r.rho);
  a.alpha_s = T(r.alpha_s);
  a.seed = MOM_SEED * r.step;
  return a;
}

// Several translation units include this file, and each has kernels of its own
// of the same name and template arguments: what follows is local to the unit,
// so that an attribute set once is set on the unit's own kernel.
namespace {

inline int mom_sms() {
  static const int sms = [] {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 152;
  }();
  return sms;
}
// Opts a kernel in to its dynamic shared memory, once on each device (the attribute is
// the device's; done: bit d for device d, devices beyond 63 every time).
template <class... P>
bool mom_opt_in(void (*kernel)(P...), int bytes, std::atomic<unsigned long long> &done) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
  if (done.load(std::memory_order_relaxed) & bit) return true;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess)
    return false;
  done.fetch_or(bit, std::memory_order_relaxed);
  return true;
}
// Dynamic shared memory of a launch of FP64 blocks no more than the SMs: so much that
// no two share an SM (and its FP64 pipe) while others idle (48^3: 283 -> 157 us).
template <class T>
constexpr unsigned mom_spread(unsigned smem, long long blocks, int sms) {
  return sizeof(T) == 8 && blocks <= sms && smem < 116u * 1024u ? 116u * 1024u : smem;
}

// The 3D step's launches for one set of template arguments.
template <class T, int NF, int TY, int RY, int BPS>
struct Mom3 {
  static constexpr auto kernel() { return mom_step3_kernel<T, NF, TY, RY, BPS>; }
  static constexpr unsigned smem = M3Smem<T, NF, TY>::total;
  static bool prepare() {
    static std::atomic<unsigned long long> done{0};
    return mom_opt_in(kernel(), (int)mom_spread<T>(smem, 0, 1), done);
  }
  static int resident() {
    int b = 0;
    if (!prepare() || cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                          &b, kernel(), M3_X * TY / RY, M3Smem<T, NF, TY>::total) != cudaSuccess)
      return 0;
    return b;
  }
  static cudaError_t step(const MomRaw &r, int zrun, cudaStream_t st) {
    if (!prepare() || zrun < 1) return cudaErrorInvalidValue;
    if (zrun > r.nz) zrun = r.nz;
    const MomArgs<T> a = mom_typed<T>(r);
    // Each lets the next launch in when its blocks are done (pdl_next at their end):
    // 101^3 46.3 -> 42.1 us per step, 256 x 256 x 192 279 -> 275.  Let in at their
    // start, the next launch's blocks took SM space from those still to run (51.1).
    const cudaError_t e = launch_pdl(mom_wall_kernel<T>, dim3(152 * 8), dim3(128), 0, st, a);
    if (e != cudaSuccess) return e;
    const dim3 g((r.nx + M3_X - 1) / M3_X, (r.ny + TY - 1) / TY, (r.nz + zrun - 1) / zrun);
    return launch_pdl(kernel(), g, dim3(M3_X, TY / RY),
                      mom_spread<T>(smem, (long long)g.x * g.y * g.z, mom_sms()), st, a, zrun);
  }
};

// Planes per block of the 3D step: runs of zr planes give tiles * ceil(nz / zr)
// blocks in waves of the resident ones; a run costs about three planes more
// than it advances (two of halo on each side, partly summed, and the first
// copies).  The blocks of an SM share its issue slots, in FP64 its FP64 pipe: a single
// wave of k blocks per SM takes a + (1 - a) k / per_sm of a full one (FP64 0.54 and 1;
// FP32, with the copies' latency, 0.55, 0.7, 0.85 and 1), so that a small lattice is
// faster in few longer runs than in many short ones: 48^3 17.7 -> 15.3 us per step,
// 64^3 20.5 -> 19.1; FP64 33 x 32 x 33 160 -> 115, 40^3 201 -> 136, 64^3 284 -> 245.
// 101^3: 41.1 us with the 10 planes this gives, 45.2 / 44.7 / 45.9 with 6 / 12 / 16;
// 256 x 256 x 192: 241 with 28, 251 with 20 or 32, 266 with 96 (without the wall pass).
inline int mom_zrun(int nx, int ny, int nz, int sms, int per_sm, bool f64) {
  if (per_sm < 1) per_sm = 1;
  const long long resident = (long long)sms * per_sm;
  const long long tiles = (long long)((nx + M3_X - 1) / M3_X) * ((ny + 7) / 8);
  const double a = f64 ? 0.08 : 0.4;
  double best = 1e300;
  int run = 1;
  for (int zr = 1; zr <= nz; zr++) {
    const long long blocks = tiles * ((nz + zr - 1) / zr), full = (blocks - 1) / resident;
    const long long k = (blocks - full * resident + sms - 1) / sms;
    const double cost = (full ? full + 1.0 : a + (1.0 - a) * k / per_sm) * (zr + 3.0);
    if (cost < best - 1e-9) {
      best = cost;
      run = zr;
    }
  }
  return run;
}

inline int mom_blocks(long long n) {
  const long long b = (n + 255) / 256;
  return (int)(b < 152 * 16 ? (b > 0 ? b : 1) : 152 * 16);
}

// S: storage type of the canonical state's populations f
template <int K, class T, int NF = 1, class S = T>
struct MomOps {
  // 3D: 32 x 8 tiles, two nodes per thread; blocks per SM by what the sums of
  // NF fluids leave of the registers (128, 168, 255 per thread)
  using Step3 = Mom3<T, NF, 8, 2, (NF == 1 ? 4 : NF == 2 ? 3 : 2)>;
  static cudaError_t step(const MomRaw &r, int zrun, cudaStream_t st) {
    if constexpr (K == 1) {
      return Step3::step(r, zrun, st);
    } else {
      Mom1<T> m1 = {};
      // small lattices: 64-thread tiles, so that the work spreads over the SMs
      if ((long long)r.nx * r.ny < 2ll * 152 * 256)
        return launch_pdl(mom_step2_kernel<T, 16, 4, 2>, dim3((r.nx + 15) / 16, (r.ny + 3) / 4),
                          dim3(16, 4), M2Smem<T, 16, 4>::total, st, mom_typed<T>(r), m1);
      return launch_pdl(mom_step2_kernel<T, 32, 8, 2>, dim3((r.nx + 31) / 32, (r.ny + 7) / 8),
                        dim3(32, 8), M2Smem<T, 32, 8>::total, st, mom_typed<T>(r), m1);
    }
  }
  static int resident() {
    if constexpr (K == 1) return Step3::resident();
    else return 0;
  }
  static cudaError_t solid(const MomRaw &r, cudaStream_t st) {
    if (K == 1) {
      const cudaError_t e = cudaMemsetAsync(r.count, 0, sizeof(int), st);
      if (e != cudaSuccess) return e;
    }
    mom_solid_kernel<K, T><<<lb_grid(K, r.nx, r.ny, r.nz), lb_block(K, r.nx, r.ny, r.nz), 0, st>>>(
        mom_typed<T>(r));
    return cudaGetLastError();
  }
  // (c, cn, out: planes cstride apart, one per free fluid)
  static cudaError_t init(const MomRaw &r, const void *c, long long cstride, cudaStream_t st) {
    mom_init_kernel<K, T, NF><<<lb_grid(K, r.nx, r.ny, r.nz), lb_block(K, r.nx, r.ny, r.nz), 0,
                               st>>>(mom_typed<T>(r), (const T *)c, cstride);
    return cudaGetLastError();
  }
  static cudaError_t enter(const MomRaw &r, const MomPlanes &p, cudaStream_t st) {
    mom_enter_kernel<K, T, NF, S><<<mom_blocks(r.N), 256, 0, st>>>(
        mom_typed<T>(r), MomCanon<T, S>{(S *)p.f, (T *)p.A, (T *)p.U, (T *)p.C});
    return cudaGetLastError();
  }
  static cudaError_t c_pass(const MomRaw &r, void *out, long long cstride, cudaStream_t st) {
    mom_c_kernel<K, T, NF><<<lb_grid(K, r.nx, r.ny, r.nz), lb_block(K, r.nx, r.ny, r.nz), 0, st>>>(
        mom_typed<T>(r), (T *)out, cstride);
    return cudaGetLastError();
  }
  static cudaError_t node(const MomRaw &r, const void *cn, long long cstride, int mode, int field,
                          int index, void *fields, double *partials, cudaStream_t st) {
    const dim3 g = lb_grid(K, r.nx, r.ny, r.nz), b = lb_block(K, r.nx, r.ny, r.nz);
    const MomArgs<T> a = mom_typed<T>(r);
    const T *c = (const T *)cn;
    T *o = (T *)fields;
    if (K == 1) mom_wall_kernel<T><<<152 * 8, 128, 0, st>>>(a);
    if (mode == MODE_STEP)
      mom_node_kernel<K, T, NF, MODE_STEP><<<g, b, 0, st>>>(a, c, cstride, o, field, index, partials);
    else if (mode == MODE_FIELDS)
      mom_node_kernel<K, T, NF, MODE_FIELDS><<<g, b, 0, st>>>(a, c, cstride, o, field, index, partials);
    else if constexpr (NF == 1)
      mom_node_kernel<K, T, NF, MODE_OBS><<<g, b, 0, st>>>(a, c, cstride, o, field, index, partials);
    return cudaGetLastError();
  }
  static cudaError_t peek(const MomRaw &r, int mode, int field, void *fields, double *partials,
                          cudaStream_t st) {
    if constexpr (K != 1 || NF != 1) {
      return cudaErrorNotSupported;
    } else {
      const dim3 g = lb_grid(K, r.nx, r.ny, r.nz), b = lb_block(K, r.nx, r.ny, r.nz);
      if (mode == MODE_FIELDS)
        mom_peek_kernel<T, MODE_FIELDS><<<g, b, 0, st>>>(mom_typed<T>(r), (T *)fields, field, partials);
      else
        mom_peek_kernel<T, MODE_OBS><<<g, b, 0, st>>>(mom_typed<T>(r), (T *)fields, field, partials);
      return cudaGetLastError();
    }
  }
  static cudaError_t expand(const MomRaw &r, const MomPlanes &p, int what, cudaStream_t st) {
    if (what == 1)
      mom_expand_kernel<K, T, NF, S><<<mom_blocks(r.N), 256, 0, st>>>(
          mom_typed<T>(r), MomCanon<T, S>{(S *)p.f, (T *)p.A, (T *)p.U, (T *)p.C}, what);
    else  // (a user's arrays of reals)
      mom_expand_kernel<K, T, NF, T><<<mom_blocks(r.N), 256, 0, st>>>(
          mom_typed<T>(r), MomCanon<T>{(T *)p.f, (T *)p.A, (T *)p.U, (T *)p.C}, what);
    return cudaGetLastError();
  }
  static Mom1<T> relax_typed(const MomRelax &m) {
    Mom1<T> m1;
    m1.mask = m.mask;
    m1.beta2 = T(m.beta2);
    m1.omega2 = T(m.omega2);
    m1.mirror[0] = m.mirror[0];
    m1.mirror[1] = m.mirror[1];
    return m1;
  }
  // stage 1 (2D): what 0, the state at rest of c; 1, one step; 2, C into c
  static cudaError_t relax(const MomRaw &r, const MomRelax &m, int what, void *c, cudaStream_t st) {
    if constexpr (K != 0) {
      return cudaErrorNotSupported;
    } else {
      const dim3 g = lb_grid(K, r.nx, r.ny, 1), b = lb_block(K, r.nx, r.ny, 1);
      const MomArgs<T> a = mom_typed<T>(r);
      const Mom1<T> m1 = relax_typed(m);
      if (what == 0) {
        mom_relax_init_kernel<T><<<g, b, 0, st>>>(a, m1, (const T *)c);
      } else if (what == 2) {
        mom_relax_c_kernel<T><<<g, b, 0, st>>>(a, m1, (T *)c);
      } else if ((long long)r.nx * r.ny < 2ll * 152 * 256) {
        return launch_pdl(mom_step2_kernel<T, 16, 4, 1>, dim3((r.nx + 15) / 16, (r.ny + 3) / 4),
                          dim3(16, 4), M2Smem<T, 16, 4>::total, st, a, m1);
      } else {
        return launch_pdl(mom_step2_kernel<T, 32, 8, 1>, dim3((r.nx + 31) / 32, (r.ny + 7) / 8),
                          dim3(32, 8), M2Smem<T, 32, 8>::total, st, a, m1);
      }
      return cudaGetLastError();
    }
  }
  static constexpr size_t batch_smem() {
    return K == 1 ? (size_t)M3Smem<T, 1, 8>::total : (size_t)M2Smem<T, 32, 8>::total;
  }
  static constexpr int kMaxBlocks = 4096;  // of one launch, for the owner table
  static size_t batch_bytes(int n) {
    return (size_t)round_up((long long)n * sizeof(MomItem<T>), 256) + kMaxBlocks * sizeof(int);
  }
  static cudaError_t batch(const MomBatchRaw *items, int n, void *scratch, size_t bytes,
                           unsigned long long spins, cudaStream_t st) {
    if (bytes < batch_bytes(n)) return cudaErrorInvalidValue;
    static std::atomic<unsigned long long> done{0};
    const bool ok = mom_opt_in(mom_batch_kernel<K, T>, (int)mom_spread<T>(batch_smem(), 0, 1), done);
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (!ok || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mom_batch_kernel<K, T>,
                                                             mom_batch_threads<K>(), batch_smem()) != cudaSuccess ||
        per_sm < 1)
      return cudaErrorInvalidValue;
    const int resident = sms * per_sm < kMaxBlocks ? sms * per_sm : kMaxBlocks;
    char *base = (char *)scratch;
    MomItem<T> *d_items = (MomItem<T> *)base;
    int *d_owner = (int *)(base + round_up((long long)n * sizeof(MomItem<T>), 256));
    // at most `resident` lattices per launch, so that each has a block
    for (int i0 = 0; i0 < n; i0 += resident) {
      const int m = n - i0 < resident ? n - i0 : resident;
      std::vector<MomItem<T>> hi(m);
      std::vector<int> owner;
      double work = 0.0;
      for (int i = 0; i < m; i++) {
        const MomBatchRaw &b = items[i0 + i];
        MomItem<T> &h = hi[i];
        memset((void *)&h, 0, sizeof(h));
        h.a[0] = mom_typed<T>(b.r[0]);
        h.a[1] = mom_typed<T>(b.r[1]);
        h.tx = (b.r[0].nx + 31) / 32;
        h.ty = (b.r[0].ny + 7) / 8;
        h.runs = 1;
        h.zrun = b.r[0].nz;
        h.nsteps = (int)b.nsteps;
        h.cur0 = b.cur0;
        work += (double)h.tx * h.ty * b.r[0].nz * (double)h.nsteps;
      }
      if (work == 0.0) continue;
      for (int i = 0; i < m; i++) {
        MomItem<T> &h = hi[i];
        const double share = (double)h.tx * h.ty * h.zrun * h.nsteps / work;
        // (rounded down, at least one: the sum stays within the resident blocks)
        int nb = 1 + (int)((resident - m) * share);
        if (K == 1) {  // runs of planes so that the tiles fill the blocks once
          const int tiles = h.tx * h.ty, nz = h.zrun;
          int runs = (nb + tiles - 1) / tiles;
          if (runs * tiles > nb && runs > 1) runs--;
          if (runs > nz) runs = nz;
          h.zrun = (nz + runs - 1) / runs;
          if (m == 1 && sizeof(T) == 8)
            h.zrun = mom_zrun(h.a[0].nx, h.a[0].ny, nz, sms, per_sm, true);
          h.runs = (nz + h.zrun - 1) / h.zrun;
        }
        const int tiles = h.tx * h.ty * h.runs;
        h.blocks = nb < tiles ? nb : tiles;
        h.block0 = (int)owner.size();
        owner.insert(owner.end(), (size_t)h.blocks, i);
      }
      cudaError_t e = cudaMemcpyAsync(d_items, hi.data(), m * sizeof(MomItem<T>),
                                      cudaMemcpyHostToDevice, st);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(d_owner, owner.data(), owner.size() * sizeof(int),
                            cudaMemcpyHostToDevice, st);
      // the copies read pageable host memory: finish them before it goes
      if (e == cudaSuccess) e = cudaStreamSynchronize(st);
      if (e != cudaSuccess) return e;
      MomItem<T> *pi = d_items;
      const int *po = d_owner;
      int cnt = m;
      unsigned long long lim = spins ? spins : kBarrierSpins;
      void *args[] = {(void *)&pi, (void *)&cnt, (void *)&po, (void *)&lim};
      e = cudaLaunchCooperativeKernel((const void *)mom_batch_kernel<K, T>,
                                      dim3((unsigned)owner.size()),
                                      dim3(32, mom_batch_threads<K>() / 32), args,
                                      K == 1 ? mom_spread<T>(batch_smem(), (long long)owner.size(), sms)
                                             : batch_smem(),
                                      st);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  static void table(LBTable &t) {
    t.mom_relax = &relax;
    t.mom_step = &step;
    t.mom_resident = &resident;
    t.mom_solid = &solid;
    t.mom_init = &init;
    t.mom_enter = &enter;
    t.mom_expand = &expand;
    t.mom_c = &c_pass;
    t.mom_node = &node;
    t.mom_peek = &peek;
    t.mom_batch = &batch;
    t.mom_batch_bytes = &batch_bytes;
  }
};

}  // namespace

}  // namespace dsm
