// Instantiates the launch table for one lattice dimension (included once per
// lattice translation unit so that the two lattices compile in parallel).
#pragma once

#include "lbm_kernels.cuh"
#include "lbm_ops.h"

namespace lbm {

// Once per device, outside any capture: the dynamic shared memory limit of kernel K.
template <auto K>
inline void configure(size_t smem) {
  constexpr int kMaxDev = 64;
  static bool done[kMaxDev] = {};
  if (smem <= 48 * 1024) return;
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < kMaxDev && done[dev]) return;
  cudaFuncSetAttribute((const void*)K, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (dev >= 0 && dev < kMaxDev) done[dev] = true;
}

template <int D, typename S, typename R, typename A>
struct Launch {
  using B = Blocks<D, R>;
  static dim3 block() { return dim3(B::bx, B::by, B::bz); }
  static dim3 tile_grid(const DevDomain& d) {
    const unsigned ty = (d.ny + B::by - 1) / B::by;
    const unsigned gx = (d.nx + B::bx - 1) / B::bx;
    if (D == 2) {  // tile_y
      const unsigned gz = (ty + 65534) / 65535;
      return dim3(gx, (ty + gz - 1) / gz, gz);
    }
    return dim3(gx, ty, (d.nz + B::bz - 1) / B::bz);
  }
  // Whether passes 1 and 2 take consecutive nodes of a layer instead of tiles: where the tiles
  // have over 8% more lanes than the layer has nodes.  Without tiles pass 2 reads q from global
  // memory, which costs more than it gives where few lanes idle (pass 2 of 512x512x256
  // in float32: 2.69 ms against 2.58, of 128^3 90.0 us against 87.6) and less elsewhere
  // (67^3, 45% more: 16.4 us against 19.4; 107^3, 21%: 54.5, 57.5; 85^3, 14%: 26.6, 28.5;
  // 203x187x149, 11%: 239.8, 239.5 and in float16 deviations 233, 255).  Pass 1 gains
  // up to 2.5 us of 26 and never lost more than 1%.
  static bool flat(const DevDomain& d) {
    if (D == 2 || (long long)d.nx * d.ny >= 1 << 30 || (d.ny + B::by - 1) / B::by > 65535 || d.nz > 65535) return false;
    const long long lanes = (long long)((d.nx + B::bx - 1) / B::bx * B::bx) * ((d.ny + B::by - 1) / B::by * B::by);
    return 100 * lanes > 108 * ((long long)d.nx * d.ny);
  }
  static dim3 flat_grid(const DevDomain& d) { return dim3((d.nx * d.ny + kFlatThreads - 1) / kFlatThreads, d.nz); }
  template <int P>
  static void moments_eos_parity(const DevDomain& d, cudaStream_t s) {
    if constexpr (D == 3) {
      if (flat(d)) {
        constexpr auto k = moments_eos_flat_kernel<P, S, R, A>;
        k<<<flat_grid(d), kFlatThreads, 0, s>>>(d);
        return;
      }
    }
    constexpr auto k = moments_eos_kernel<D, P, S, R, A>;
    k<<<tile_grid(d), block(), 0, s>>>(d);
  }
  static void moments_eos(const DevDomain& d, int parity, cudaStream_t s) {
    if (parity == 0) moments_eos_parity<0>(d, s);
    else moments_eos_parity<1>(d, s);
  }
  template <bool kSmall> using QT = QTile<D, 2 * sizeof(A), kSmall>;
  template <int kMode, bool kSmall>
  static void qflux_tiles(const DevDomain& d, const TileMaps& maps, double* out0, double* out1, cudaStream_t s) {
    using T = QT<kSmall>;
    constexpr size_t smem = qflux_dyn_smem<D, T, A>();
    constexpr auto k = qflux_tile_kernel<D, R, A, T, kMode>;
    configure<k>(smem);
    const dim3 g((d.nx + T::EX - 1) / T::EX, (d.ny + T::EY - 1) / T::EY, (d.nz + T::EZ - 1) / T::EZ);
    k<<<g, dim3(T::TX, T::TY), smem, s>>>(d, maps, out0, out1);
  }
  template <int kMode>
  static void qflux_launch(const DevDomain& d, const TileMaps& maps, double* out0, double* out1, cudaStream_t s) {
    if (maps.qtile_small) qflux_tiles<kMode, true>(d, maps, out0, out1, s);
    else qflux_tiles<kMode, false>(d, maps, out0, out1, s);
  }
  static void qflux(const DevDomain& d, const TileMaps& maps, cudaStream_t s) {
    qflux_launch<kQfluxStep>(d, maps, nullptr, nullptr, s);
  }
  template <int P>
  static void collide_stream_parity(const DevDomain& d, const TileMaps& maps, cudaStream_t s) {
    if constexpr (D == 3) {
      if (flat(d)) {
        constexpr size_t smem = collide_dyn_smem<D, R>(kFlatThreads);
        constexpr auto k = collide_stream_flat_kernel<P, S, R, A>;
        configure<k>(smem);
        k<<<flat_grid(d), kFlatThreads, smem, s>>>(d);
        return;
      }
    }
    constexpr size_t smem = collide_dyn_smem<D, R>(B::bx * B::by * B::bz);
    constexpr auto k = collide_stream_kernel<D, P, S, R, A>;
    configure<k>(smem);
    k<<<tile_grid(d), block(), smem, s>>>(d, maps);
  }
  static void collide_stream(const DevDomain& d, const TileMaps& maps, int parity, cudaStream_t s) {
    if (parity == 0) collide_stream_parity<0>(d, maps, s);
    else collide_stream_parity<1>(d, maps, s);
  }
  static unsigned blocks1d(const DevDomain& d) { return (unsigned)((d.N + 255) / 256); }
  static void init_equilibrium(const DevDomain& d, const double* rho, const double* ux, const double* uy,
                               const double* uz, cudaStream_t s) {
    init_equilibrium_kernel<D, S, R><<<blocks1d(d), 256, 0, s>>>(d, rho, ux, uy, uz);
  }
  static void aux_density(const DevDomain& d, const double* rho, cudaStream_t s) {
    dim3 blk(32, D == 3 ? 2 : 4, 1);
    dim3 grd((d.px + blk.x - 1) / blk.x, (d.py + blk.y - 1) / blk.y, (d.pz + blk.z - 1) / blk.z);
    aux_density_kernel<D, R, A><<<grd, blk, 0, s>>>(d, rho);
  }
  static void canonical_read(const DevDomain& d, int parity, double* out, cudaStream_t s) {
    canonical_read_kernel<D, S><<<blocks1d(d), 256, 0, s>>>(d, parity, out);
  }
  static void canonical_window(const DevDomain& d, int parity, const int o[3], const int e[3], double* out,
                               cudaStream_t s) {
    const long long m = (long long)e[0] * e[1] * e[2];
    canonical_window_kernel<D, S><<<(unsigned)((m + 255) / 256), 256, 0, s>>>(d, parity, o[0], o[1], o[2], e[0], e[1],
                                                                              e[2], out);
  }
  static void canonical_write(const DevDomain& d, const double* in, cudaStream_t s) {
    if constexpr (DevStorage<S>::value) canonical_density_kernel<D><<<blocks1d(d), 256, 0, s>>>(d, in);
    canonical_write_kernel<D, S><<<blocks1d(d), 256, 0, s>>>(d, in);
  }
  static void macroscopic(const DevDomain& d, const TileMaps& maps, double* rho, double* u, cudaStream_t s) {
    qflux_launch<kQfluxFields>(d, maps, rho, u, s);
  }
  static void bare_velocity(const DevDomain& d, const double* rho, double* u, cudaStream_t s) {
    bare_velocity_kernel<D, R, A><<<blocks1d(d), 256, 0, s>>>(d, rho, u);
  }
  // Tiles of 32 x 8 nodes for the grid-stride readings, and the blocks that walk them.
  struct Tiles {
    int x, y, n, blocks;
    explicit Tiles(const DevDomain& d) : x((d.nx + 31) / 32), y((d.ny + 7) / 8), n(x * y * d.nz), blocks(n < kDiagBlocks ? n : kDiagBlocks) {}
  };
  static int diag_partial(const DevDomain& d, int parity, double* partial, cudaStream_t s) {
    const Tiles t(d);
    cudaMemsetAsync(partial + 5 * t.blocks, 0, sizeof(double), s);
    diag_partial_kernel<D, S><<<t.blocks, dim3(32, 8), 0, s>>>(d, parity, t.x, t.y, t.n, partial);
    return t.blocks;
  }
  static long long speed_partial(const DevDomain& d, const TileMaps& maps, double* partial, cudaStream_t s) {
    const long long n = maps.qtile_small ? tiles_of<QT<true>>(d) : tiles_of<QT<false>>(d);
    if (partial) {  // the word after the maxima, where their maximum goes in the end, starts the blocks at 0
      cudaMemsetAsync(partial + n, 0, sizeof(double), s);
      qflux_launch<kQfluxSpeed>(d, maps, partial, partial + n, s);
    }
    return n;
  }
  static void drop_on_film(const DevDomain& d, const lbm_drop_on_film& g, double rho_l, double rho_v, double* rho,
                           double* u, cudaStream_t s) {
    drop_on_film_kernel<D><<<blocks1d(d), 256, 0, s>>>(d, g.radius, g.film, g.gap, g.speed, g.width, g.noise,
                                                       (unsigned long long)g.seed, rho_l, rho_v, rho, u);
  }
  static long long grad_partial(const DevDomain& d, double* partial, cudaStream_t s) {
    const Tiles t(d);
    if (partial) grad_partial_kernel<D, A><<<t.blocks, dim3(32, 8), 0, s>>>(d, t.x, t.y, t.n, partial);
    return t.blocks;
  }
  static long long crown_partial(const DevDomain& d, int layer, double rho_mid, double* partial, cudaStream_t s) {
    const long long nl = D == 3 ? (long long)d.nx * d.ny : d.nx;
    const unsigned nb = (unsigned)((nl + 255) / 256);
    if (partial) crown_partial_kernel<D, A><<<nb, 256, 0, s>>>(d, layer, rho_mid, partial);
    return (long long)nb;
  }
  static Ops table() {
    return Ops{D, Lattice<D>::Q, sizeof(S), sizeof(A), &moments_eos, &qflux, &collide_stream, &init_equilibrium, &aux_density,
               &canonical_read, &canonical_write, &canonical_window, &macroscopic, &bare_velocity, &diag_partial,
               &speed_partial, &drop_on_film, &grad_partial, &crown_partial};
  }
};

}  // namespace lbm
