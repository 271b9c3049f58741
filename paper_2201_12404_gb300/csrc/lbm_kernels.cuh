// Kernels of one time step and of the field I/O, templated on the lattice
// dimension D, the population storage type S and the arithmetic type R.
//
//  moments_eos_kernel    (pass 1)  gather f, form rho and j, evaluate the
//                                  Peng-Robinson pseudo-potential; writes (rho, psi) and
//                                  j to the padded auxiliary fields, ghosts included.
//  qflux_tile_kernel     (pass 1b) F from the (rho, psi) halo tile (Eq. Kforce_final)
//                                  and q = rho v^3, v = (j + F/2)/rho the fluid
//                                  velocity; q to the node and the ghosts imaging it,
//                                  F over the node's j.
//  collide_stream_kernel (pass 2)  gather f, the node's F from pass 1b, Phi from the
//                                  staged q boxes (Eq. correction), f^eq and
//                                  f* (Eqs. LBMeq, LBMstar), k/s/h split (Appendix A),
//                                  gamma (Sec. 2.4), relaxation (Eq. LBGK), A-A write.
#pragma once

#include <type_traits>

#include "lbm_device.cuh"

namespace lbm {

// ---------------------------------------------------------------------------
// Pass 1: one thread per interior node; the node also writes the ghost nodes
// that image it (periodic wrap or mirror across a half-way wall).
// ---------------------------------------------------------------------------
// Interior coordinate that padded coordinate cp (ghost layers of 2) images along
// an axis of n nodes: periodic wrap, or the mirror across a half-way wall (which
// sets *flip).
__device__ __forceinline__ int ghost_image(int cp, int n, int wlo, int whi, bool* flip) {
  int t = cp - 2;
  if (t < 0) { if (wlo) { t = -1 - t; *flip = true; } else t += n; }
  else if (t >= n) { if (whi) { t = 2 * n - 1 - t; *flip = true; } else t -= n; }
  return t;
}

// Pass 1 at interior node (x, y, z): rho and j from the gathered populations, psi
// from the Peng-Robinson pressure.  The (rho, psi) pair goes to the node's padded
// position and to every ghost node imaging it (each combination of its own or its
// ghost coordinate on the axes that have one), so that the later passes index
// their stencils without wrap logic; j goes to the node alone (pass 1b reads it
// there).  A warp is one aligned x row of 32 interior nodes, so each of its 27
// population loads is one 128-byte line.
template <int D, int P, typename S, typename R, typename A, bool kFace>
__device__ __forceinline__ void moments_eos_node(const DevDomain& d, int x, int y, int z) {
  constexpr int Q = Lattice<D>::Q;
  if (x >= d.nx || y >= d.ny || z >= d.nz) return;
  R f[Q];
  gather<D, P, S, R, kFace>(d, x, y, z, f);
  NodeMoments<R> m;
  row_moments<D, R>(f, m);
  const R rho = m.rho, j[3] = {m.jx, m.jy, m.jz};
  if (!(rho > (R)0) || !(rho < (R)INFINITY)) atomicOr(d.flags, 1u);

  A* aux = (A*)d.aux;
  Two<A>* a2 = (Two<A>*)d.aux;
  const long long pn = bc_pnode(d, pnode_of<D>(d, x, y, z));
  const Two<A> pair = two<A>((A)rho, (A)psi_of<R>(d, rho));
  a2[pn] = pair;
#pragma unroll
  for (int a = 0; a < D; ++a) aux[(2 + D + a) * d.PN + pn] = (A)j[a];
  // a ghost images only nodes within one of a face
  if ((unsigned)(x - 2) < (unsigned)(d.nx - 4) && (unsigned)(y - 2) < (unsigned)(d.ny - 4) &&
      (D == 2 || (unsigned)(z - 2) < (unsigned)(d.nz - 4)))
    return;
  bool wall = false;
  const int gx = ghost_of(x, d.nx, d.wall_lo[0], d.wall_hi[0], &wall);
  const int gy = ghost_of(y, d.ny, d.wall_lo[1], d.wall_hi[1], &wall);
  const int gz = D == 3 ? ghost_of(z, d.nz, d.wall_lo[2], d.wall_hi[2], &wall) : -1;
  if (gx < 0 && gy < 0 && gz < 0) return;
#pragma unroll 1
  for (int k = 1; k < (1 << D); ++k) {
    if (((k & 1) && gx < 0) || ((k & 2) && gy < 0) || ((k & 4) && gz < 0)) continue;
    const int cx = (k & 1) ? gx : x + 2, cy = (k & 2) ? gy : y + 2, cz = D == 3 ? ((k & 4) ? gz : z + 2) : 0;
    a2[bc_pnode(d, (long long)cx + (long long)d.px * ((long long)cy + (long long)d.py * cz))] = pair;
  }
}

// Pass 1 on the tile of EX x EY x EZ nodes at (x0, y0, z0), one per thread of the block.
template <int D, int P, typename S, typename R, typename A>
__device__ __forceinline__ void moments_eos_tile(const DevDomain& d, int x0, int y0, int z0, int EX, int EY, int EZ) {
  const int x = x0 + threadIdx.x, y = y0 + threadIdx.y, z = z0 + (D == 3 ? threadIdx.z : 0);
  if ((P == 1 || DevStorage<S>::value) && tile_on_face<D>(d, x0, y0, z0, EX, EY, EZ)) moments_eos_node<D, P, S, R, A, true>(d, x, y, z);
  else moments_eos_node<D, P, S, R, A, false>(d, x, y, z);
}

// The (rho, psi) pairs of every padded node straight from a density field
// (device, float64, N values), ghosts included: what pass 1 writes for a state
// whose density is that field, without forming populations first.  q is left
// alone (the next pass 1 writes it).
template <int D, typename R, typename A>
__global__ void __launch_bounds__(256) aux_density_kernel(DevDomain d, const double* rho_in) {
  const int xp = blockIdx.x * blockDim.x + threadIdx.x, yp = blockIdx.y * blockDim.y + threadIdx.y;
  const int zp = blockIdx.z * blockDim.z + threadIdx.z;
  if (xp >= d.nx + 4 || yp >= d.py || zp >= d.pz) return;
  bool flip = false;
  const int x = ghost_image(xp, d.nx, d.wall_lo[0], d.wall_hi[0], &flip);
  const int y = ghost_image(yp, d.ny, d.wall_lo[1], d.wall_hi[1], &flip);
  const int z = D == 3 ? ghost_image(zp, d.nz, d.wall_lo[2], d.wall_hi[2], &flip) : 0;
  const R rho = (R)rho_in[node_of(d, x, y, z)];
  if (!(rho > (R)0) || !(rho < (R)INFINITY)) atomicOr(d.flags, 1u);
  const long long pn = (long long)xp + (long long)d.px * ((long long)yp + (long long)d.py * (long long)zp);
  ((Two<A>*)d.aux)[pn] = two<A>((A)rho, (A)psi_of<R>(d, rho));
}

// Resident 64-thread blocks per SM asked of the register allocator in 3-D float32
// arithmetic: 20 (48 registers) for float32 storage, passes 1 + 1b on 512x512x256 1.82 ms,
// 1.85 at 16; 16 (64) for float16 deviations, on 256x256x128 271 us against 285 at 14.  2-D:
// 16 128-thread blocks (32 registers) for float32 storage, 2048x1024 40.5 us, 40.8 with 37.
#ifndef LBM_K1_MINBLOCKS_F32
#define LBM_K1_MINBLOCKS_F32 20
#endif
#ifndef LBM_K1_MINBLOCKS_F16
#define LBM_K1_MINBLOCKS_F16 16
#endif
#ifndef LBM_K1_MINBLOCKS_F32_2D
#define LBM_K1_MINBLOCKS_F32_2D 16
#endif
template <int D, int P, typename S, typename R, typename A>
__global__ void __launch_bounds__(Blocks<D, R>::bx * Blocks<D, R>::by * Blocks<D, R>::bz,
                                  sizeof(R) == 8   ? 1
                                  : D == 2         ? (sizeof(S) == 2 ? 1 : LBM_K1_MINBLOCKS_F32_2D)
                                  : sizeof(S) == 2 ? LBM_K1_MINBLOCKS_F16
                                                   : LBM_K1_MINBLOCKS_F32)
moments_eos_kernel(DevDomain d) {
  using B = Blocks<D, R>;
  moments_eos_tile<D, P, S, R, A>(d, blockIdx.x * B::bx, tile_y<D>() * B::by, D == 3 ? blockIdx.z * B::bz : 0, B::bx, B::by,
                                  B::bz);
}

// Pass 1 of a 3-D domain over consecutive nodes of a layer (FlatNode).
template <int P, typename S, typename R, typename A>
__global__ void __launch_bounds__(kFlatThreads, sizeof(R) == 8 ? 1 : (sizeof(S) == 2 ? LBM_K1_MINBLOCKS_F16 : LBM_K1_MINBLOCKS_F32))
moments_eos_flat_kernel(DevDomain d) {
  const FlatNode f(d);
  if ((P == 1 || DevStorage<S>::value) && f.on_face) moments_eos_node<3, P, S, R, A, true>(d, f.x, f.y, f.z);
  else moments_eos_node<3, P, S, R, A, false>(d, f.x, f.y, f.z);
}

}  // namespace lbm

#include "lbm_collide.cuh"

namespace lbm {

// ---------------------------------------------------------------------------
// f := f^eq(rho, u) at every node (natural layout, parity 0).
// ---------------------------------------------------------------------------
template <int D, typename S, typename R>
__global__ void init_equilibrium_kernel(DevDomain d, const double* rho, const double* ux,
                                        const double* uy, const double* uz) {
  constexpr int Q = Lattice<D>::Q;
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= d.N) return;
  const R r = (R)rho[n];
  const R u[3] = {(R)ux[n], (R)uy[n], D == 3 ? (R)uz[n] : (R)0};
  R X[3][3];
  for (int a = 0; a < 3; ++a) {
    const R u2 = u[a] * u[a];
    X[a][1] = a < D ? (R)1 - (R)(1.0 / 3.0) - u2 : (R)1;
    X[a][2] = a < D ? (R)0.5 * ((R)(1.0 / 3.0) + u2 + u[a]) : (R)0;
    X[a][0] = a < D ? (R)0.5 * ((R)(1.0 / 3.0) + u2 - u[a]) : (R)0;
  }
  S* F = (S*)d.f;
  if constexpr (DevStorage<S>::value) {
    // each slot is encoded against the density of its upstream (writer) node; the
    // next step (even parity) decodes with rho_w[0] of that node
    const int x = (int)(n % d.nx), y = (int)((n / d.nx) % d.ny), z = (int)(n / ((long long)d.nx * d.ny));
    const FaceLinks<D> fl(d, x, y, z);
    d.rho_w[0][n] = (float)r;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const R rw = (R)(float)rho[upstream_node<D>(d, fl, n, i)];
      const R feq = r * X[0][cxi(i) + 1] * X[1][cyi(i) + 1] * X[2][D == 3 ? czi(i) + 1 : 1];
      F[(long long)i * d.N + n] = __float2half_rn((float)(feq / ((R)wq<D>(i) * rw) - (R)1));
    }
  } else {
#pragma unroll
    for (int i = 0; i < Q; ++i)
      st_pop<S, R>(F + (long long)i * d.N + n, r * X[0][cxi(i) + 1] * X[1][cyi(i) + 1] * X[2][D == 3 ? czi(i) + 1 : 1]);
  }
}

// ---------------------------------------------------------------------------
// Canonical (post-stream, pre-collision) populations <-> float64 buffer.
// ---------------------------------------------------------------------------
template <int D, typename S>
__global__ void canonical_read_kernel(DevDomain d, int parity, double* out) {
  constexpr int Q = Lattice<D>::Q;
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= d.N) return;
  const int x = (int)(n % d.nx), y = (int)((n / d.nx) % d.ny), z = (int)(n / ((long long)d.nx * d.ny));
  double f[Q];
  gather<D, S, double>(d, parity, x, y, z, f);
  for (int i = 0; i < Q; ++i) out[(long long)i * d.N + n] = f[i];
}

// The same for the nodes of a box: window node (i, j, k) is domain node
// ((ox + i) mod nx, (oy + j) mod ny, (oz + k) mod nz); the host checks 0 <= o < n
// and 1 <= e <= n per axis, so o + i < 2n never overflows.
template <int D, typename S>
__global__ void canonical_window_kernel(DevDomain d, int parity, int ox, int oy, int oz, int ex, int ey, int ez,
                                        double* out) {
  constexpr int Q = Lattice<D>::Q;
  const long long m = (long long)ex * ey * ez;
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= m) return;
  const int i = (int)(k % ex), j = (int)((k / ex) % ey), l = (int)(k / ((long long)ex * ey));
  int x = ox + i, y = oy + j, z = oz + l;
  if (x >= d.nx) x -= d.nx;
  if (y >= d.ny) y -= d.ny;
  if (z >= d.nz) z -= d.nz;
  double f[Q];
  gather<D, S, double>(d, parity, x, y, z, f);
  for (int q = 0; q < Q; ++q) out[(long long)q * m + k] = f[q];
}

template <int D, typename S>
__global__ void canonical_write_kernel(DevDomain d, const double* in) {
  constexpr int Q = Lattice<D>::Q;
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= d.N) return;
  S* F = (S*)d.f;
  if constexpr (DevStorage<S>::value) {
    // rho_w[0] holds every node's density (canonical_density_kernel, launched before)
    const int x = (int)(n % d.nx), y = (int)((n / d.nx) % d.ny), z = (int)(n / ((long long)d.nx * d.ny));
    const FaceLinks<D> fl(d, x, y, z);
    for (int i = 0; i < Q; ++i) {
      const double rw = (double)d.rho_w[0][upstream_node<D>(d, fl, n, i)];
      F[(long long)i * d.N + n] = __float2half_rn((float)(in[(long long)i * d.N + n] / (wq<D>(i) * rw) - 1.0));
    }
  } else {
    for (int i = 0; i < Q; ++i) st_pop<S, double>(F + (long long)i * d.N + n, in[(long long)i * d.N + n]);
  }
}

// float16-deviation storage: density of every node of a canonical state into rho_w[0].
template <int D>
__global__ void canonical_density_kernel(DevDomain d, const double* in) {
  constexpr int Q = Lattice<D>::Q;
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= d.N) return;
  double r = 0.0;
  for (int i = 0; i < Q; ++i) r += in[(long long)i * d.N + n];
  d.rho_w[0][n] = (float)r;
}

// ---------------------------------------------------------------------------
// Force density F at node (x, y, z) from the auxiliary fields of the current
// state (Eq. Kforce_final with the sign of reading R1), rho the node's density:
// the link-by-link form of the stencil pass 2 evaluates row by row.
// ---------------------------------------------------------------------------
template <int D, typename R, typename A>
__device__ __forceinline__ void aux_force(const DevDomain& d, int x, int y, int z, R rho, R* F) {
  constexpr int Q = Lattice<D>::Q;
  const Two<A>* a2 = (const Two<A>*)d.aux;  // (rho, psi)
  const long long pc = pnode_of<D>(d, x, y, z);
  const long long sy = d.px, sz = (long long)d.px * d.py;
  R g4[3] = {0, 0, 0}, g3[3] = {0, 0, 0};
  for (int i = 0; i < Q; ++i) {
    if (i == Lattice<D>::REST) continue;
    const long long o = cxi(i) + sy * cyi(i) + (D == 3 ? sz * czi(i) : 0);
    const R t4 = (R)(4.0 / 3.0) * (R)a2[pc + o].y - (R)(1.0 / 6.0) * (R)a2[pc + 2 * o].y;
    const R t3 = (R)2 * (R)a2[pc + o].x - (R)a2[pc + 2 * o].x;
    const R W = (R)(3.0 * wq<D>(i));
    for (int a = 0; a < D; ++a) {
      const int c = cq<D>(i, a);
      g4[a] += W * (R)c * t4;
      g3[a] += W * (R)c * t3;
    }
  }
  const R spsi_c = psi_sign<R>(phys<R>(d), (R)a2[pc].x) * (R)a2[pc].y;
  for (int a = 0; a < 3; ++a)
    F[a] = a < D ? -((R)2 * spsi_c * g4[a] + phys<R>(d).kappa * rho * g3[a]) + rho * phys<R>(d).g[a] : (R)0;
}

// ---------------------------------------------------------------------------
// Drop-on-film initial fields (float64, natural layout): see lbm_init_drop_on_film.
// The white noise draws from SplitMix64 (Steele, Lea & Flood 2014) keyed by
// (seed, node, component), two uniforms per value, normal by Box-Muller.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__device__ __forceinline__ double unit_open(unsigned long long z) {  // (0, 1]
  return ((double)(z >> 11) + 1.0) * (1.0 / 9007199254740992.0);
}

template <int D>
__global__ void drop_on_film_kernel(DevDomain d, double R, double film, double gap, double U, double W, double noise,
                                    unsigned long long seed, double rho_l, double rho_v, double* rho, double* u) {
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= d.N) return;
  const int x = (int)(n % d.nx), y = (int)((n / d.nx) % d.ny), z = (int)(n / ((long long)d.nx * d.ny));
  const double vert = D == 3 ? (double)z : (double)y;
  const double cv = film + R + gap;
  const double dx = x - 0.5 * (d.nx - 1);
  const double dy = D == 3 ? y - 0.5 * (d.ny - 1) : vert - cv;
  const double dz = D == 3 ? vert - cv : 0.0;
  const double d_drop = sqrt(dx * dx + dy * dy + dz * dz) - R;
  const double d_film = film > 0 ? vert - (film - 0.5) : INFINITY;
  const double dist = fmin(d_drop, d_film);
  rho[n] = 0.5 * (rho_l + rho_v) - 0.5 * (rho_l - rho_v) * tanh(2.0 * dist / W);
  const double liq = 0.5 - 0.5 * tanh(2.0 * d_drop / W);
  for (int a = 0; a < D; ++a) {
    double v = a == D - 1 ? -U * liq : 0.0;
    if (noise > 0) {
      const unsigned long long key = seed ^ ((unsigned long long)n * (unsigned long long)(2 * D) + 2ull * a) * 0xD1B54A32D192ED03ull;
      const double u1 = unit_open(splitmix64(key)), u2 = unit_open(splitmix64(key + 1));
      v += noise * U * liq * sqrt(-2.0 * log(u1)) * cos(6.283185307179586 * u2);
    }
    u[a * d.N + n] = v;
  }
}

// ---------------------------------------------------------------------------
// Largest |grad rho| of the auxiliary density (second-order central differences;
// the ghost layer supplies the wrapped or mirrored neighbours): kDiagBlocks blocks at
// most, each over every gridDim-th tile of 32 x 8 nodes, one partial maximum per block.
// Float64 is 58 times slower than float32, so a warp differences in float64 only the
// nodes whose float32 gradient is not clearly below the largest it has met (1e-35 off the
// bound on its square: squares below the normal numbers have lost their relative precision).
// ---------------------------------------------------------------------------
constexpr int kDiagBlocks = 152 * 6;

template <int D, typename A>
__global__ void __launch_bounds__(256) grad_partial_kernel(DevDomain d, int ntx, int nty, int ntiles, double* partial) {
  const Two<A>* a2 = (const Two<A>*)d.aux;
  const long long e[3] = {1, d.px, (long long)d.px * d.py};
  float top = 0.0f;
  double best = 0;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int x = (t % ntx) * 32 + threadIdx.x, y = ((t / ntx) % nty) * 8 + threadIdx.y, z = t / (ntx * nty);
    const bool in = x < d.nx && y < d.ny;
    A r[2 * D];
    float g2f = 0.0f;
    if (in) {
      const long long pc = pnode_of<D>(d, x, y, z);
#pragma unroll
      for (int a = 0; a < D; ++a) {
        r[2 * a] = a2[bc_pnode(d, pc - e[a])].x;
        r[2 * a + 1] = a2[bc_pnode(d, pc + e[a])].x;
        const float g = (float)(r[2 * a + 1] - r[2 * a]);
        g2f = fmaf(g, g, g2f);
      }
    }
    // non-negative floats order as their bits; a NaN is above them all
    top = fmaxf(top, __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(g2f))));
    if (in && !(g2f < fmaf(0.99f, top, -1e-35f))) {
      double g2 = 0;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const double ga = 0.5 * ((double)r[2 * a + 1] - (double)r[2 * a]);
        g2 += ga * ga;
      }
      best = fmax(best, g2);  // a NaN is passed over
    }
  }
  block_max_store<256>(threadIdx.x + 32 * threadIdx.y, sqrt(best), partial, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Crown radius: over the nodes of one layer (index `layer` along the last axis),
// the largest distance from the vertical axis through the domain centre of a
// node whose auxiliary density exceeds rho_mid; one partial maximum per block
// (0 where no node qualifies).
// ---------------------------------------------------------------------------
template <int D, typename A>
__global__ void __launch_bounds__(256) crown_partial_kernel(DevDomain d, int layer, double rho_mid, double* partial) {
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nl = D == 3 ? (long long)d.nx * d.ny : d.nx;
  double rm = 0;
  if (k < nl) {
    const int x = (int)(k % d.nx);
    const int y = D == 3 ? (int)(k / d.nx) : layer;
    const int z = D == 3 ? layer : 0;
    const Two<A>* a2 = (const Two<A>*)d.aux;
    if ((double)a2[pnode_of<D>(d, x, y, z)].x > rho_mid) {
      const double dx = x - 0.5 * (d.nx - 1), dy = D == 3 ? y - 0.5 * (d.ny - 1) : 0.0;
      rm = sqrt(dx * dx + dy * dy);
    }
  }
  block_max_store<256>(threadIdx.x, rm, partial, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Bare velocity of a state at rest in the reported sense: u -= F dt/(2 rho) in
// place, F from the auxiliary fields of the current (equilibrium) state.
// ---------------------------------------------------------------------------
template <int D, typename R, typename A>
__global__ void bare_velocity_kernel(DevDomain d, const double* rho_in, double* u) {
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= d.N) return;
  const int x = (int)(n % d.nx), y = (int)((n / d.nx) % d.ny), z = (int)(n / ((long long)d.nx * d.ny));
  const R rho = (R)((const Two<A>*)d.aux)[pnode_of<D>(d, x, y, z)].x;
  R F[3];
  aux_force<D, R, A>(d, x, y, z, rho, F);
  for (int a = 0; a < D; ++a) u[a * d.N + n] -= (double)F[a] / (2.0 * rho_in[n]);
}

// ---------------------------------------------------------------------------
// Deterministic totals: kDiagBlocks blocks, each over every kDiagBlocks-th tile of
// 32 x 8 nodes, then one block (diag_final_kernel) over their sums in a fixed order.
// partial layout: [block][5] = mass, jx, jy, jz, max|u|.
//
// Bound by the float64 pipe.  The totals are linear in the populations, so a thread sums
// each of its Q slots over all of its nodes (one addition per population, 388 us of the pipe
// on 256x256x128) and forms the moments once at the end; max|u| needs the moments of
// every node, which float32 storage forms in float32 first and in float64 only where the
// node may be the fastest: slower_than_top is right whatever the order in which the blocks
// meet their nodes (lbm_read_diag there 576 us; 695 with each warp's own largest).
// ---------------------------------------------------------------------------

// Whether a node is slower than one met before, from float32 speeds squared: u2f of this
// node, top the largest so far.  Both nodes have populations >= 0, so a momentum of five
// additions deep is within 5 2^-24 rho of the exact one (the vector within 5.2e-7 rho) and
// rho within 6 2^-24 of itself; with the roundings of the quotient a float32 speed is within
// 6e-7 + 1e-6 |u| of the exact one.  A relative margin alone, as wide as 0.999 of the
// square, would pass over the fastest node below speeds of 1e-3.
__device__ __forceinline__ bool slower_than_top(float u2f, float top) {
  const float least = fmaf(sqrtf(top), 0.9999f, -2e-6f);
  return least > 0.0f && u2f < least * least;
}

// g = (double)f, exactly.  For float32 by moving the fields of the bits where all Q values
// are normal numbers: the float64 pipe, which also runs the conversion instruction, sets
// the pace.
template <int Q>
__device__ __forceinline__ void widen(const float (&f)[Q], double (&g)[Q]) {
  bool normal = true;
#pragma unroll
  for (int i = 0; i < Q; ++i) normal = normal && (__float_as_uint(f[i]) & 0x7fffffffu) - 0x00800000u < 0x7f000000u;
  if (normal) {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const unsigned b = __float_as_uint(f[i]);
      g[i] = __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
    }
  } else {
#pragma unroll
    for (int i = 0; i < Q; ++i) g[i] = (double)f[i];
  }
}
template <int Q>
__device__ __forceinline__ void widen(const double (&f)[Q], double (&g)[Q]) {
#pragma unroll
  for (int i = 0; i < Q; ++i) g[i] = f[i];
}

template <int D, typename S>
__global__ void __launch_bounds__(256, 2) diag_partial_kernel(DevDomain d, int parity, int ntx, int nty, int ntiles,
                                                              double* partial) {
  constexpr int Q = Lattice<D>::Q;
  using L = typename std::conditional<sizeof(S) == 4, float, double>::type;  // populations as loaded
  __shared__ double sh[5][8];
  const int tid = threadIdx.x + 32 * threadIdx.y;
  double acc[Q], u2max = 0;
  float top = 0.0f;  // largest float32 speed squared that this warp knows of
  // shared by the grid: the bits of the largest so far, after the partials
  volatile unsigned* top_all = (unsigned*)(partial + 5 * (long long)gridDim.x);
#pragma unroll
  for (int i = 0; i < Q; ++i) acc[i] = 0;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int x = (t % ntx) * 32 + threadIdx.x, y = ((t / ntx) % nty) * 8 + threadIdx.y, z = t / (ntx * nty);
    bool in = x < d.nx && y < d.ny;
    L f[Q];
    double g[Q];
    float u2f = 0.0f;
    bool known_speed = false;  // u2f holds to within the bound of slower_than_top
    unsigned known = 0;
    if constexpr (sizeof(L) == 4) known = *top_all;
    if (in) {
      gather<D, S, L>(d, parity, x, y, z, f);
      if constexpr (sizeof(L) == 4) {
        NodeMoments<float> m;
        row_moments<D, float>(f, m);
        unsigned signs = 0;
#pragma unroll
        for (int i = 0; i < Q; ++i) signs |= __float_as_uint(f[i]);
        known_speed = (int)signs >= 0 && m.rho > 1e-15f && m.rho < 1e15f;  // (a NaN is not)
        if (known_speed) u2f = (m.jx * m.jx + m.jy * m.jy + m.jz * m.jz) / (m.rho * m.rho);
      }
      widen<Q>(f, g);
#pragma unroll
      for (int i = 0; i < Q; ++i) acc[i] += g[i];
    }
    if constexpr (sizeof(L) == 4) {
      // non-negative floats order as their bits
      const float others = __uint_as_float(known);
      top = fmaxf(fmaxf(top, others), __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(u2f))));
      if (top > others && threadIdx.x == 0) atomicMax((unsigned*)top_all, __float_as_uint(top));
      in = in && !(known_speed && slower_than_top(u2f, top));
    }
    if (in) {
      NodeMoments<double> m;
      row_moments<D, double>(g, m);
      const double u2 = (m.jx * m.jx + m.jy * m.jy + m.jz * m.jz) / (m.rho * m.rho);
      u2max = fmax(u2max, u2);  // a NaN is passed over
    }
  }
  NodeMoments<double> m;
  row_moments<D, double>(acc, m);
  double v[5] = {m.rho, m.jx, m.jy, m.jz, sqrt(u2max)};
#pragma unroll
  for (int k = 0; k < 5; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double w = __shfl_xor_sync(0xffffffffu, v[k], o);
      v[k] = k < 4 ? v[k] + w : fmax(v[k], w);
    }
    if (threadIdx.x == 0) sh[k][threadIdx.y] = v[k];
  }
  __syncthreads();
  if (tid < 5) {
    double s = sh[tid][0];
    for (int w = 1; w < 8; ++w) s = tid < 4 ? s + sh[tid][w] : fmax(s, sh[tid][w]);
    partial[blockIdx.x * 5 + tid] = s;
  }
}

// Sums (fields 0-3) and maximum (field 4) of the partials by one block of 32 x 5 threads:
// warp k takes field k, every lane every 32nd block.  (One thread over all of them, with
// one partial per 256 nodes, took 7.9 ms on 8.4 million nodes.)
static __global__ void diag_final_kernel(const double* partial, int nblocks, double* out) {
  const int k = threadIdx.y;
  double v = 0;
  for (int b = threadIdx.x; b < nblocks; b += 32) v = k < 4 ? v + partial[b * 5 + k] : fmax(v, partial[b * 5 + k]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double w = __shfl_xor_sync(0xffffffffu, v, o);
    v = k < 4 ? v + w : fmax(v, w);
  }
  if (threadIdx.x == 0) out[k] = v;
}

// Largest of n partial maxima, by one block of 1024 threads, to out[0]; the domain's error word
// to out[1], so that one copy tells the host whether a block gave up its wait.
static __global__ void __launch_bounds__(1024) max_final_kernel(const double* partial, long long n, const unsigned* flags,
                                                                double* out) {
  double v = 0;
  for (long long b = threadIdx.x; b < n; b += 1024) v = fmax(v, partial[b]);
  block_max_store<1024>(threadIdx.x, v, out, 0);
  if (threadIdx.x == 0) out[1] = (double)*flags;
}

}  // namespace lbm
