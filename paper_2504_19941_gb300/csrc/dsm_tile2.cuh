// dsm_tile2.cuh -- the whole stage-2 lattice Boltzmann step (Sec. II.B) of a
// D2Q9 lattice in one pass over the populations f, for lattices whose g
// collision gives g_eq (tau_g = 1) and whose faces are periodic or mirrors.
// Lattices that the step on moments takes (dsm_mom.cuh) do not come here: this
// is the step with viscosities or densities that differ between the fluids.
// Included by dsm_lb_impl.cuh after the fused pass (node_body), whose per-node
// arithmetic it shares.
//
// State: f as ever, and one quad (A, C, u_x, u_y) per node, which fixes g_eq
// (A = mu - 3/2 C u.u).  A block stages the quads of its tile and a two-node
// halo, sums this step's C on the tile and a one-node halo, and collides; the
// populations are pulled into registers while the staging copies are in
// flight.  Beyond a mirror the halo holds the image nodes, the normal component
// of u reversed: the links from there are the specularly reflected ones.
//
// Per node and step f and the quad in and out and C1 in: 108 B in FP32.  The two
// passes this replaces moved 172 with periodic faces and, as mirror lattices
// kept g as populations, 188 with mirrors, in two launches.
#pragma once

namespace dsm {

// The fused pass's view of the neighbourhood: this step's C and C1 in shared
// memory (beyond a mirror the edge node), the pulled f in registers.
template <class T, bool RC>
struct TileIO {
  static constexpr bool kUnrollWall = true;
  static constexpr bool kSolidFirst = false;
  static constexpr bool kFetched = true;
  static constexpr bool kRho = RC;
  const T *c, *c1, *r;
  int ox[3], oy[3];
  T f[9];
  template <class L, class T_, class S>
  __device__ __forceinline__ T C(const LBArgs<T_, S> &, const Hood &, int i) const {
    return c[ox[L::cx(i) + 1] + oy[L::cy(i) + 1]];
  }
  template <class L, class T_, class S>
  __device__ __forceinline__ T C1(const LBArgs<T_, S> &, const Hood &, int i) const {
    return c1[ox[L::cx(i) + 1] + oy[L::cy(i) + 1]];
  }
  template <class L>
  __device__ __forceinline__ T rho(int i) const {
    return r[ox[L::cx(i) + 1] + oy[L::cy(i) + 1]];
  }
  template <class L, class S>
  __device__ __forceinline__ void put_eq(const LBArgs<T, S> &a, int n, T c, T A, T ux, T uy,
                                         T) const {
    Quad<T> m;
    m.v[0] = A;
    m.v[1] = c;
    m.v[2] = ux;
    m.v[3] = uy;
    reinterpret_cast<Quad<T> *>(a.Qz)[chk(a.err, n, a.N)] = m;
  }
};

// Quads in qin -> a.Qz, f in a.fin -> a.fout.  mirror: x, y axis.
template <class T, class S, int TX, int TY, bool RC, bool FC>
__global__ void __launch_bounds__(TX *TY)
    tile2_kernel(const __grid_constant__ LBArgs<T, S> a, const T *qin, int mirror_x,
                 int mirror_y) {
  pdl_next();
  pdl_wait();
  using L = Lat<0>;
  constexpr int HX = TX + 4, NS = HX * (TY + 4);  // staged quads
  constexpr int CX = TX + 2, NC = CX * (TY + 2);  // this step's C, and C1
  constexpr int NT = TX * TY;
  __shared__ Quad<T> sq[NS];
  __shared__ T sc[NC], s1[NC], sr[RC ? NC : 1];
  const int tx = threadIdx.x, ty = threadIdx.y, tid = tx + TX * ty;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
  // node of staged coordinate c of an axis of n nodes; flip: beyond a mirror
  auto map = [](int c, int n, int mirror, bool &flip) {
    flip = false;
    if (mirror) {
      flip = c < 0 || c >= n;
      c = c < 0 ? -1 - c : c >= n ? 2 * n - 1 - c : c;
      return c < 0 ? 0 : c;  // (beyond what a ragged tile uses)
    }
    if (c < 0) c += n;
    if (c >= n) c -= n;
    if (c < 0 || c >= n) {
      c %= n;
      if (c < 0) c += n;
    }
    return c;
  };
  // a tile whose halo lies within the lattice needs no map (1750 x 450: 24.0 -> 22.7
  // us per step)
  const bool inner = x0 >= 2 && y0 >= 2 && x0 + TX + 2 <= a.nx && y0 + TY + 2 <= a.ny;
  constexpr int PER = (NS + NT - 1) / NT;
  int flip[PER];
#pragma unroll
  for (int r = 0; r < PER; r++) {
    const int k = tid + r * NT;
    flip[r] = 0;
    if (k < NS) {
      int gx = x0 - 2 + k % HX, gy = y0 - 2 + k / HX;
      if (!inner) {
        bool fx, fy;
        gx = map(gx, a.nx, FC ? mirror_x : 0, fx);
        gy = map(gy, a.ny, FC ? mirror_y : 0, fy);
        flip[r] = (fx ? 1 : 0) | (fy ? 2 : 0);
      }
      cp_async_bytes<4 * sizeof(T)>((unsigned)__cvta_generic_to_shared(sq + k),
                                    qin + 4ll * chk(a.err, gx + a.nx * gy, a.N));
    }
  }
  for (int k = tid; k < NC; k += NT) {
    int gx = x0 - 1 + k % CX, gy = y0 - 1 + k / CX;
    if (!inner) {
      bool fx, fy;
      gx = map(gx, a.nx, FC ? mirror_x : 0, fx);
      gy = map(gy, a.ny, FC ? mirror_y : 0, fy);
    }
    cp_async_bytes<sizeof(T)>((unsigned)__cvta_generic_to_shared(s1 + k),
                              a.C1 + chk(a.err, gx + a.nx * gy, a.N));
  }
  cp_async_commit();
  const int x = x0 + tx, y = y0 + ty;
  const bool inside = x < a.nx && y < a.ny;
  TileIO<T, RC> io;
#pragma unroll
  for (int j = 0; j < L::Q; j++) io.f[j] = T(0);
  if (inside) {
    Hood h;
    if constexpr (FC) h.init_faces(x, y, 0, a.nx, a.ny, 1, a.p.face);
    else h.init(x, y, 0, a.nx, a.ny, 1);
    h.guard(a.err);
#pragma unroll
    for (int j = 0; j < L::Q; j++)
      io.f[j] = load_f<T, S>(a.fin[j], h.minus<L>(j), j, L::w(j));
  }
  cp_async_wait<0>();
  if (FC && !inner) {
#pragma unroll
    for (int r = 0; r < PER; r++) {
      if (flip[r] & 1) sq[tid + r * NT].v[2] = -sq[tid + r * NT].v[2];
      if (flip[r] & 2) sq[tid + r * NT].v[3] = -sq[tid + r * NT].v[3];
    }
  }
  __syncthreads();
  for (int k = tid; k < NC; k += NT) {
    const int k0 = (k / CX + 1) * HX + k % CX + 1;
    T Ay[L::Q], Cy[L::Q], uy[L::Q][3];
#pragma unroll
    for (int i = 0; i < L::Q; i++) {
      const Quad<T> m = sq[k0 - (L::cx(i) + HX * L::cy(i))];  // x - c_i
      Ay[i] = m.v[0];
      Cy[i] = m.v[1];
      uy[i][0] = (i == 0 || L::cx(i)) ? m.v[2] : T(0);
      uy[i][1] = (i == 0 || L::cy(i)) ? m.v[3] : T(0);
      uy[i][2] = T(0);
    }
    const T C = moments_eq_node<L, T>(Ay, Cy, uy);
    sc[k] = C;
    if (RC) sr[k] = rho_map(a.c, C, s1[k]);
  }
  __syncthreads();
  if (!inside) return;
  io.c = sc;
  io.c1 = s1;
  io.r = sr;
#pragma unroll
  for (int e = 0; e < 3; e++) {
    io.ox[e] = tx + e;
    io.oy[e] = (ty + e) * CX;
  }
  if constexpr (FC) {
    if (mirror_x && x == 0) io.ox[0] = io.ox[1];
    if (mirror_x && x == a.nx - 1) io.ox[2] = io.ox[1];
    if (mirror_y && y == 0) io.oy[0] = io.oy[1];
    if (mirror_y && y == a.ny - 1) io.oy[2] = io.oy[1];
  }
  node_body<0, T, S, 2, MODE_STEP, RC, true, FC, TileIO<T, RC>>(a, x, y, 0, true, 0, io);
}

// quads q <-> the canonical g_eq planes (A, u_x, u_y in M, C): pack != 0 into q
template <class T>
__global__ void __launch_bounds__(256)
    tile2_pack_kernel(long long N, long long pitch, T *M, T *C, T *q, int pack) {
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    Quad<T> *p = reinterpret_cast<Quad<T> *>(q) + n;
    if (pack) {
      Quad<T> m;
      m.v[0] = M[n];
      m.v[1] = C[n];
      m.v[2] = M[pitch + n];
      m.v[3] = M[2 * pitch + n];
      *p = m;
    } else {
      const Quad<T> m = *p;
      M[n] = m.v[0];
      C[n] = m.v[1];
      M[pitch + n] = m.v[2];
      M[2 * pitch + n] = m.v[3];
    }
  }
}

}  // namespace dsm
