// Launchers of the step kernels, instantiated once per storage format.
#pragma once
#include "step_impl.cuh"

namespace lbcg {

inline int sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

// CTAs of a kernel that fit on one SM at once (computed once per kernel).
template <typename K>
inline int resident_ctas(K kern, int threads, size_t smem) {
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, threads, smem) != cudaSuccess || b < 1) {
    cudaGetLastError();
    b = 1;
  }
  return b;
}

// 32-bit byte offsets within a z plane of nx x ny nodes (moment storage: 16-byte records)
template <int ST>
inline bool fits_idx32(const Geo& g) {
  return (unsigned long long)Lay<ST>::plane(g) * (Store<ST>::MOMENT ? 16 : sizeof(typename Store<ST>::E)) < (1ull << 32);
}

// Calls f with the staging halo (1, 4, 6 or 7) as a compile-time constant.
template <typename F>
inline cudaError_t with_stage_halo(int halo, F&& f) {
  switch (halo) {
    case 1: return f(std::integral_constant<int, 1>{});
    case 4: return f(std::integral_constant<int, 4>{});
    case 6: return f(std::integral_constant<int, 6>{});
    case 7: return f(std::integral_constant<int, 7>{});
  }
  return cudaErrorInvalidValue;
}

// Launch with programmatic stream serialisation (see launch_dependents).
template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

template <int ST>
cudaError_t launch_phi_acc_t(const Geo& g, const StateBuf& in, unsigned long long* acc, cudaStream_t st) {
  static const int occ = resident_ctas(k_phi_acc<ST>, 256, 0);
  const long long need = (g.N + 255) / 256;
  const long long cap = (long long)sm_count() * occ;
  const int blocks = (int)(need < cap ? need : cap);
  auto kern = k_phi_acc<ST>;
  trace_kernel("k_phi_acc", kern, dim3(blocks), dim3(256), 0);
  kern<<<blocks, 256, 0, st>>>(view<ST>(in), g, acc);
  return cudaGetLastError();
}

// k_phi into the padded array; zero: accumulator to clear, or null.
template <int ST>
inline cudaError_t launch_phi(const Geo& g, const Phys& p, const InitBuf& init, PhiSrc src, void* phi, const PadGeo& pg,
                              unsigned long long* zero, cudaStream_t st) {
  using R = typename Store<ST>::R;
  const long long groups = ((long long)g.ny * g.nz + 7) / 8;
  const long long cap = (long long)sm_count() * 8;
  const int blocks = (int)(groups < cap ? groups : cap);
  auto run = [&](auto kern) {
    trace_kernel("k_phi", kern, dim3(blocks), dim3(32, 8), 0);
    return launch_pdl(kern, dim3(blocks), dim3(32, 8), 0, st, src, init, g, pg, R(p.psi0), reinterpret_cast<R*>(phi), zero);
  };
  if constexpr (Store<ST>::TWOSET) {
    if (p.model == 1) return run(k_phi<R, true>);
  }
  return run(k_phi<R, false>);
}

template <int ST, int LOADER, bool WS, bool WF, int TX, int TY, int TZ, int H, bool IDX32, int MINB, bool SC>
inline cudaError_t launch_step_t(const Geo& g, const Phys& p, const StateBuf& in, const InitBuf& init, PhiSrc src,
                                 AccBufs ab, StateBuf out, const void* phi, const PadGeo& pg, const FieldOut& fields,
                                 unsigned* status, cudaStream_t st) {
  using R = typename Store<ST>::R;
  const size_t smem = Layout<R, TX, TY, TZ, H, SC ? (WF ? 3 : 2) : 1>::bytes;
  auto kern = k_step<ST, LOADER, WS, WF, TX, TY, TZ, H, IDX32, MINB, SC>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  dim3 grid((g.nx + TX - 1) / TX, (g.ny + TY - 1) / TY, (g.nz + TZ - 1) / TZ);
  dim3 block(TX, TY, 1);
  trace_kernel("k_step", kern, grid, block, smem);
  return launch_pdl(kern, grid, block, smem, st, view<ST>(in), view<ST>(out), init, src.acc, ab.out,
                    reinterpret_cast<const R*>(phi), pg, g, phys_as<R>(p), fields, status);
}

// Tile shapes of the hot variant (pull, write state): kTiles and kShallow;
// Shan-Chen takes 32x8x4 and the shallow ones (48^3, walls in x and y: 32x8x4 24.4 us a
// step, 32x8x2 15.5).  Other variants, the wide halos (6, 7), FP64 and planes that
// need 64-bit offsets use 32x8x4.
template <int ST, int LOADER, bool WS, bool WF, bool SC>
inline cudaError_t launch_step_tiles(int tile, const Geo& g, const Phys& p, const StateBuf& in, const InitBuf& init,
                                     PhiSrc src, AccBufs ab, StateBuf out, void* phi, int halo, const FieldOut& fields,
                                     unsigned* status, cudaStream_t st) {
  const PadGeo pg = pad_geo(g, halo);
  cudaError_t e = launch_phi<ST>(g, p, init, src, phi, pg, WS ? ab.zero : nullptr, st);
  if (e != cudaSuccess) return e;
  const bool i32 = fits_idx32<ST>(g);
  auto go = [&](auto hc) -> cudaError_t {
    constexpr int H = decltype(hc)::value;
#define LBCG_TILE(TY, TZ, I32, MB) \
  launch_step_t<ST, LOADER, WS, WF, 32, TY, TZ, H, I32, MB, SC>(g, p, in, init, src, ab, out, phi, pg, fields, status, st)
    if constexpr (LOADER == LOAD_PULL && WS && !WF && ST != 3 && H < 6) {
      if (i32) {
        switch (tile) {
          case 1:
          case 5:
            if constexpr (!SC) return LBCG_TILE(8, 8, true, 2);
            break;
          case 4:
            if constexpr (!SC) return LBCG_TILE(4, 4, true, 4);
            break;
          case 6: return LBCG_TILE(8, 2, true, 2);
          case 7: return LBCG_TILE(8, 1, true, 2);
          default: break;
        }
      }
    }
    return i32 ? LBCG_TILE(8, 4, true, 2) : LBCG_TILE(8, 4, false, 2);
#undef LBCG_TILE
  };
  if constexpr (SC) return go(std::integral_constant<int, 1>{});
  else return with_stage_halo(halo, go);
}

// phi of the current level into the padded array, nothing else
template <int ST>
cudaError_t launch_phi_s(const Geo& g, const Phys& p, const InitBuf& init, PhiSrc src, void* phi, int halo, cudaStream_t st) {
  return launch_phi<ST>(g, p, init, src, phi, pad_geo(g, halo), nullptr, st);
}

// the density test of the current level alone
template <int ST>
cudaError_t launch_density_t(int loader, const Geo& g, const Phys& p, const StateBuf& in, const InitBuf& init,
                             const unsigned long long* accin, unsigned* status, cudaStream_t st) {
  auto run = [&](auto kern) {
    const long long need = ((long long)g.ny * g.nz + 7) / 8, cap = (long long)sm_count() * 8;
    const int blocks = (int)(need < cap ? need : cap);
    trace_kernel("k_density", kern, dim3(blocks), dim3(32, 8), 0);
    kern<<<blocks, dim3(32, 8), 0, st>>>(view<ST>(in), init, accin, g, phys_as<typename Store<ST>::R>(p), status);
    return cudaGetLastError();
  };
  return loader == LOAD_PULL ? run(k_density<ST, LOAD_PULL>) : run(k_density<ST, LOAD_FIELDS>);
}

template <int ST>
cudaError_t launch_step_s(int loader, bool ws, bool wf, int tile, const Geo& g, const Phys& p, const StateBuf& in,
                          const InitBuf& init, PhiSrc src, AccBufs ab, StateBuf out, void* phi, int halo, const FieldOut& fields,
                          unsigned* status, cudaStream_t st) {
  auto go = [&](auto sc) -> cudaError_t {
    constexpr bool SC = decltype(sc)::value;
#define LBCG_GO(LD, WS, WF, T) \
  launch_step_tiles<ST, LD, WS, WF, SC>(T, g, p, in, init, src, ab, out, phi, halo, fields, status, st)
    if (loader == LOAD_PULL) {
      if (ws && !wf) return LBCG_GO(LOAD_PULL, true, false, tile);
      if (!ws && wf) return LBCG_GO(LOAD_PULL, false, true, 0);
    } else {
      if (ws && !wf) return LBCG_GO(LOAD_FIELDS, true, false, 0);
      if (!ws && wf) return LBCG_GO(LOAD_FIELDS, false, true, 0);
    }
    return cudaErrorInvalidValue;
#undef LBCG_GO
  };
  if (p.model == 1) {
    if constexpr (Store<ST>::TWOSET) return go(std::true_type{});
    else return cudaErrorInvalidValue;
  }
  return go(std::false_type{});
}

template <int ST>
cudaError_t launch_export_t(int loader, const Geo& g, const Phys& p, const StateBuf& in, const InitBuf& init,
                                   int x0, int y0, int z0, int bx, int by, int bz, double* outA, double* outB,
                                   cudaStream_t st) {
  const long long M = (long long)bx * by * bz;
  const long long need = (M + 127) / 128;
  const int blocks = (int)(need < 4096 ? need : 4096);
  if (loader == LOAD_PULL)
    k_export<ST, LOAD_PULL><<<blocks, 128, 0, st>>>(view<ST>(in), init, g, phys_as<typename Store<ST>::R>(p), x0, y0, z0, bx, by, bz, outA, outB);
  else
    k_export<ST, LOAD_FIELDS><<<blocks, 128, 0, st>>>(view<ST>(in), init, g, phys_as<typename Store<ST>::R>(p), x0, y0, z0, bx, by, bz, outA, outB);
  return cudaGetLastError();
}

template <int ST, int TX, int TY, int TZ, int H, bool IDX32, int MINB>
inline cudaError_t launch_batched_step_t(const RunDesc* d_runs, const int* run_of, long long ntiles, int parity, int k,
                                         int blocks, unsigned* status, cudaStream_t st) {
  using R = typename Store<ST>::R;
  const size_t smem = Layout<R, TX, TY, TZ, H>::bytes;
  auto kern = k_step_batched<ST, TX, TY, TZ, H, IDX32, MINB>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  trace_kernel("k_step_batched", kern, dim3(blocks), dim3(TX, TY), smem);
  return launch_pdl(kern, dim3(blocks), dim3(TX, TY), smem, st, d_runs, run_of, ntiles, parity, k, status);
}

template <int ST>
cudaError_t launch_batched_t(const RunDesc* d_runs, const int* run_of, long long ntiles, long long ngroups, int tile, int halo,
                             long long max_blocks, int parity, int k, int blocks_per_sm, unsigned* status,
                             cudaStream_t st) {
  const long long cap = (long long)sm_count() * 8;
  const int pblocks = (int)(ngroups < cap ? ngroups : cap);
  trace_kernel("k_phi_batched", k_phi_batched<float>, dim3(pblocks), dim3(32, 8), 0);
  cudaError_t e = launch_pdl(k_phi_batched<float>, dim3(pblocks), dim3(32, 8), 0, st, d_runs, run_of + ntiles, ngroups, k);
  if (e != cudaSuccess) return e;
  const int blocks = sm_count() * (blocks_per_sm > 0 ? blocks_per_sm : 2);
  Geo wide{};  // a plane with as many blocks as the largest of the runs
  wide.nx = BLK;
  wide.ny = (int)max_blocks;
  const bool i32 = fits_idx32<ST>(wide);
  return with_stage_halo(halo, [&](auto hc) -> cudaError_t {
    constexpr int H = decltype(hc)::value;
#define LBCG_TILE(TY, TZ, I32, MB) \
  launch_batched_step_t<ST, 32, TY, TZ, H, I32, MB>(d_runs, run_of, ntiles, parity, k, blocks, status, st)
    if constexpr (H < 6) {
      if (i32) {
        switch (tile) {
          case 1:
          case 3:
          case 5: return LBCG_TILE(8, 8, true, 2);
          case 4: return LBCG_TILE(4, 4, true, 4);
          default: break;
        }
      }
    }
    return i32 ? LBCG_TILE(8, 4, true, 2) : LBCG_TILE(8, 4, false, 2);
#undef LBCG_TILE
  });
}

}  // namespace lbcg
