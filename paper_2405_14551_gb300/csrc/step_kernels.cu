// Storage-format dispatch of the step launchers.
#include "internal.h"
#include "lattice.cuh"

namespace lbcg {

const Tile kTiles[NUM_TILES] = {{32, 8, 4}, {32, 8, 8}, {32, 8, 4}, {32, 8, 8}, {32, 4, 4}, {32, 8, 8}};
const Tile kShallow[NUM_SHAPES - NUM_TILES] = {{32, 8, 2}, {32, 8, 1}};

template <int ST>
cudaError_t launch_phi_acc_t(const Geo& g, const StateBuf& in, unsigned long long* acc, cudaStream_t st);
template <int ST>
cudaError_t launch_step_s(int loader, bool ws, bool wf, int tile, const Geo& g, const Phys& p, const StateBuf& in,
                          const InitBuf& init, PhiSrc src, AccBufs ab, StateBuf out, void* phi, int halo, const FieldOut& fields, unsigned* status,
                          cudaStream_t st);
template <int ST>
cudaError_t launch_phi_s(const Geo& g, const Phys& p, const InitBuf& init, PhiSrc src, void* phi, int halo, cudaStream_t st);
template <int ST>
cudaError_t launch_density_t(int loader, const Geo& g, const Phys& p, const StateBuf& in, const InitBuf& init,
                             const unsigned long long* accin, unsigned* status, cudaStream_t st);
template <int ST>
cudaError_t launch_batched_t(const RunDesc* d_runs, const int* run_of, long long ntiles, long long ngroups, int tile, int halo,
                             long long max_blocks, int parity, int k, int blocks_per_sm, unsigned* status,
                             cudaStream_t st);
template <int ST>
cudaError_t launch_export_t(int loader, const Geo& g, const Phys& p, const StateBuf& in, const InitBuf& init, int x0,
                            int y0, int z0, int bx, int by, int bz, double* outA, double* outB, cudaStream_t st);

cudaError_t launch_phi_acc(int storage, const Geo& g, const StateBuf& in, unsigned long long* acc, cudaStream_t st) {
  switch (storage) {
    case 0: return launch_phi_acc_t<0>(g, in, acc, st);
    case 1: return launch_phi_acc_t<1>(g, in, acc, st);
    case 2: return launch_phi_acc_t<2>(g, in, acc, st);
    case 3: return launch_phi_acc_t<3>(g, in, acc, st);
    case 4: return launch_phi_acc_t<4>(g, in, acc, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_step(int storage, int loader, bool write_state, bool write_fields, int tile, const Geo& g,
                        const Phys& p, const StateBuf& in, const InitBuf& init, PhiSrc src, AccBufs ab, StateBuf out, void* phi, int halo, const FieldOut& fields, unsigned* status, cudaStream_t st) {
  switch (storage) {
    case 0: return launch_step_s<0>(loader, write_state, write_fields, tile, g, p, in, init, src, ab, out, phi, halo, fields, status, st);
    case 1: return launch_step_s<1>(loader, write_state, write_fields, tile, g, p, in, init, src, ab, out, phi, halo, fields, status, st);
    case 2: return launch_step_s<2>(loader, write_state, write_fields, tile, g, p, in, init, src, ab, out, phi, halo, fields, status, st);
    case 3: return launch_step_s<3>(loader, write_state, write_fields, tile, g, p, in, init, src, ab, out, phi, halo, fields, status, st);
    case 4: return launch_step_s<4>(loader, write_state, write_fields, tile, g, p, in, init, src, ab, out, phi, halo, fields, status, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_phi_only(int storage, const Geo& g, const Phys& p, const InitBuf& init, PhiSrc src, void* phi, int halo,
                            cudaStream_t st) {
  switch (storage) {
    case 0: return launch_phi_s<0>(g, p, init, src, phi, halo, st);
    case 1: return launch_phi_s<1>(g, p, init, src, phi, halo, st);
    case 2: return launch_phi_s<2>(g, p, init, src, phi, halo, st);
    case 3: return launch_phi_s<3>(g, p, init, src, phi, halo, st);
    case 4: return launch_phi_s<4>(g, p, init, src, phi, halo, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_density(int storage, int loader, const Geo& g, const Phys& p, const StateBuf& in, const InitBuf& init,
                           const unsigned long long* accin, unsigned* status, cudaStream_t st) {
  switch (storage) {
    case 0: return launch_density_t<0>(loader, g, p, in, init, accin, status, st);
    case 1: return launch_density_t<1>(loader, g, p, in, init, accin, status, st);
    case 2: return launch_density_t<2>(loader, g, p, in, init, accin, status, st);
    case 3: return launch_density_t<3>(loader, g, p, in, init, accin, status, st);
    case 4: return launch_density_t<4>(loader, g, p, in, init, accin, status, st);
  }
  return cudaErrorInvalidValue;
}

template <typename R>
__global__ void __launch_bounds__(256) k_phi_fill(size_t n, R* __restrict__ phi) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) phi[i] = R(PHI_SOLID);
}
cudaError_t launch_phi_fill(int storage, const PadGeo& pg, int fields, void* phi, cudaStream_t st) {
  const size_t n = (size_t)pg.px * pg.py * pg.pz * (size_t)fields;
  const unsigned blocks = (unsigned)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
  if (storage == 3) k_phi_fill<<<blocks, 256, 0, st>>>(n, (double*)phi);
  else k_phi_fill<<<blocks, 256, 0, st>>>(n, (float*)phi);
  return cudaGetLastError();
}

template <typename R>
__global__ void __launch_bounds__(256) k_phi_plain(Geo g, PadGeo pg, const R* __restrict__ phi, R* __restrict__ plain) {
  const long long rows = (long long)g.ny * g.nz;
  for (long long row = (long long)blockIdx.x * 8 + threadIdx.y; row < rows; row += (long long)gridDim.x * 8) {
    const long long y = row % g.ny, z = row / g.ny;
    const R* src = phi + pg.hx + (long long)pg.px * (pg.h + y + (long long)pg.py * (pg.h + z));
    const bool solid_row = (g.wy && (y == 0 || y == g.ny - 1)) || (g.wz && (z == 0 || z == g.nz - 1));
    for (int x = threadIdx.x; x < g.nx; x += 32)  // by place, not by the marker: phi itself may be as large
      plain[row * g.nx + x] = solid_row || (g.wx && (x == 0 || x == g.nx - 1)) ? R(0) : src[x];
  }
}
cudaError_t launch_phi_plain(int storage, const Geo& g, const PadGeo& pg, const void* phi, void* plain, cudaStream_t st) {
  const long long groups = ((long long)g.ny * g.nz + 7) / 8;
  const unsigned blocks = (unsigned)(groups < 8192 ? groups : 8192);
  if (storage == 3) k_phi_plain<<<blocks, dim3(32, 8), 0, st>>>(g, pg, (const double*)phi, (double*)plain);
  else k_phi_plain<<<blocks, dim3(32, 8), 0, st>>>(g, pg, (const float*)phi, (float*)plain);
  return cudaGetLastError();
}

cudaError_t launch_export(int storage, int loader, const Geo& g, const Phys& p, const StateBuf& in,
                          const InitBuf& init, int x0, int y0, int z0, int bx, int by, int bz, double* outA,
                          double* outB, cudaStream_t st) {
  switch (storage) {
    case 0: return launch_export_t<0>(loader, g, p, in, init, x0, y0, z0, bx, by, bz, outA, outB, st);
    case 1: return launch_export_t<1>(loader, g, p, in, init, x0, y0, z0, bx, by, bz, outA, outB, st);
    case 2: return launch_export_t<2>(loader, g, p, in, init, x0, y0, z0, bx, by, bz, outA, outB, st);
    case 3: return launch_export_t<3>(loader, g, p, in, init, x0, y0, z0, bx, by, bz, outA, outB, st);
    case 4: return launch_export_t<4>(loader, g, p, in, init, x0, y0, z0, bx, by, bz, outA, outB, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_batched(int storage, const RunDesc* d_runs, const int* run_of, long long ntiles, long long ngroups, int tile,
                           int halo, long long max_blocks, int parity, int k, int blocks_per_sm, unsigned* status,
                           cudaStream_t st) {
  switch (storage) {
    case 0: return launch_batched_t<0>(d_runs, run_of, ntiles, ngroups, tile, halo, max_blocks, parity, k, blocks_per_sm, status, st);
    case 1: return launch_batched_t<1>(d_runs, run_of, ntiles, ngroups, tile, halo, max_blocks, parity, k, blocks_per_sm, status, st);
    case 2: return launch_batched_t<2>(d_runs, run_of, ntiles, ngroups, tile, halo, max_blocks, parity, k, blocks_per_sm, status, st);
  }
  return cudaErrorInvalidValue;  // no batched FP64 or moment instantiation
}

int batched_tile(int storage, int tile, int halo, long long max_blocks) {
  const unsigned long long plane = (unsigned long long)max_blocks * BLK * (unsigned long long)state_arrays(storage) * elem_bytes(storage);
  return halo >= 6 || plane >= (1ull << 32) ? 0 : tile;
}

int sm_count_host() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

template <typename E>
__global__ void __launch_bounds__(256) k_direction(Geo g, E* __restrict__ f, int nd, int dir, E* __restrict__ plain, bool gather) {
  const long long nb = (long long)plane_blocks(g);
  const int pitch = row_pitch(g.nx);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < g.N; i += (long long)gridDim.x * blockDim.x) {
    const long long row = i / g.nx, z = row / g.ny, n = (row - z * g.ny) * pitch + (i - row * g.nx);
    E& v = f[((z * nb + n / BLK) * nd + dir) * BLK + n % BLK];
    if (gather) plain[i] = v;
    else v = plain[i];
  }
}

cudaError_t launch_direction(int storage, const Geo& g, void* f, int dir, void* plain, bool gather, cudaStream_t st) {
  const long long need = (g.N + 255) / 256;
  const int blocks = (int)(need < 8192 ? need : 8192), nd = state_arrays(storage);
  switch (elem_bytes(storage)) {
    case 2: k_direction<<<blocks, 256, 0, st>>>(g, (uint16_t*)f, nd, dir, (uint16_t*)plain, gather); break;
    case 4: k_direction<<<blocks, 256, 0, st>>>(g, (uint32_t*)f, nd, dir, (uint32_t*)plain, gather); break;
    default: k_direction<<<blocks, 256, 0, st>>>(g, (uint64_t*)f, nd, dir, (uint64_t*)plain, gather); break;
  }
  return cudaGetLastError();
}

size_t elem_bytes(int storage) { return storage == 3 ? 8 : (storage == 2 ? 2 : 4); }
int state_arrays(int storage) { return storage == 4 ? MOMENT_COEFS : (storage == 0 || storage == 3 ? 2 * Q : Q); }
size_t state_elems(int storage, const Geo& g) {
  if (storage == 4) return (size_t)MOMENT_COEFS * (size_t)g.N;
  return plane_blocks(g) * BLK * (size_t)g.nz * (size_t)state_arrays(storage);
}
bool storage_is_twoset(int storage) { return storage == 0 || storage == 3; }
bool storage_is_f64(int storage) { return storage == 3; }

}  // namespace lbcg
