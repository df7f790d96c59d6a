// Internal interface between the C-ABI runtime and the kernel translation units.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <string>

namespace lbcg {

// Box geometry; w* = 1 makes layers 0 and n-1 of that axis solid.
struct Geo {
  int nx, ny, nz;
  int wx, wy, wz;
  long long N;
};

// Model parameters as seen by the kernels (converted to the compute type in
// the kernel prologue).
struct Phys {
  double tau_a, tau_b;
  int equal_tau;
  double A2;  // (A_a + A_b) / 2
  double beta;
  double A_h, h_min, h_max;
  int K;      // floor(h_max): scan length
  double phi_I;
  double g[3];
  int g_mode;
  int collision;  // 0 BGK, 1 regularised
  int model;      // 0 colour gradient, 1 Shan-Chen
  double G;       // Shan-Chen coupling
  double psi0;    // Shan-Chen pseudo-potential scale rho_0
};

// Nodes from one row of the population blocks to the next: rows start on whole
// 32-byte sectors where that costs at most a sixteenth of the memory, so that the
// stores of neighbouring tiles share no sector (two-set FP32, 153x217x170, 32x8x8: 460 us
// a step against 544 with rows of exactly nx), else they are exactly nx.
__host__ __device__ constexpr int row_pitch(int nx) {
  const int pad = (8 - nx % 8) % 8;
  return 16 * pad <= nx ? nx + pad : nx;
}
// Blocks of 32 nodes in a z plane.
__host__ __device__ constexpr size_t plane_blocks(const Geo& g) {
  return ((size_t)row_pitch(g.nx) * (size_t)g.ny + 31) / 32;
}

// Device pointers of one population lattice.  Two-set storage: f holds f^A
// and f^B in blocks of 32 nodes of a z plane, [z][(x + pitch y) / 32][54 directions][32]
// (the last block of a plane is padded).  Reduced storage: f holds f* (FP32 or
// FP16 deviations) in blocks of 27 directions and sv holds the colour scalars
// (s, vx, vy, vz) of each node as one float4, [z][y][x].
struct StateBuf {
  void* f;
  float4* sv;
};

// Initial fields (device, float): phi[N], rho[N] or null, u[3][N] or null.
struct InitBuf {
  const float* phi;
  const float* rho;
  const float* u;
  int regularised;
};

enum Loader { LOAD_PULL = 0, LOAD_FIELDS = 1 };

// The same parameters in the compute type of the kernels.
template <typename R>
struct PhysR {
  R tau_a, tau_b, A2, beta, A_h, h_min, h_max, phi_I, G, psi0;
  R g[3];
  int equal_tau, K, g_mode, collision;
};
template <typename R>
inline PhysR<R> phys_as(const Phys& p) {
  return PhysR<R>{R(p.tau_a), R(p.tau_b), R(p.A2),    R(p.beta), R(p.A_h), R(p.h_min), R(p.h_max), R(p.phi_I), R(p.G), R(p.psi0),
                  {R(p.g[0]), R(p.g[1]), R(p.g[2])}, p.equal_tau, p.K, p.g_mode, p.collision};
}

// The padded array of phi (Shan-Chen: phi, psi_A, psi_B) that k_phi writes
// every step: nodes -hx..., -h... of the lattice first, rows a multiple of 32
// bytes, extents that cover the halo of every tile (tiles are at most 32 x 8 x
// 8 nodes).
constexpr int pad_hx(int h) { return h > 4 ? 8 : 4; }
struct PadGeo {
  int px, py, pz, hx, h;
};
inline PadGeo pad_geo(const Geo& g, int halo) {
  PadGeo p;
  p.hx = pad_hx(halo);
  p.h = halo;
  p.px = (g.nx + 31) / 32 * 32 + 2 * p.hx;
  p.py = g.ny + 7 + 2 * halo;
  p.pz = g.nz + 7 + 2 * halo;
  return p;
}

// Where k_phi reads the phase field: the accumulator of the previous step, or
// the initial phi.  Exactly one is non-null.
struct PhiSrc {
  const float* phi;
  const unsigned long long* acc;
};

// Where the fields kernel writes: field k at p + slot[k] N, or nowhere (-1).
struct FieldOut {
  void* p = nullptr;
  signed char slot[16] = {-1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1};
};
// the fields of mask, each at its own index (packed: in increasing order)
inline FieldOut field_out(void* p, uint32_t mask, bool packed) {
  FieldOut o;
  o.p = p;
  int n = 0;
  for (int k = 0; k < 14; ++k)
    if ((mask >> k) & 1u) o.slot[k] = (signed char)(packed ? n++ : k);
  return o;
}

// Accumulators written by a step: out receives the component densities of
// the next time level (all zero before the step); the step zeroes its own
// nodes of zero (read by the step before, written by the step after).
struct AccBufs {
  unsigned long long* out;
  unsigned long long* zero;
};

// 64-bit words of one node's accumulator: 1 (FP32 storages, both component
// sums packed), 2 (FP64).
inline int acc_words(int storage) { return storage == 3 ? 2 : 1; }

// One run of a batch, as seen by the batched persistent kernel.
struct RunDesc {
  Geo g;
  PhysR<float> p;
  StateBuf S[2];
  unsigned long long* acc[3];  // accumulator rotation (see AccBufs)
  float* phi;                  // padded phase field
  PadGeo pg;
  long long tile_begin;        // first work items of this run: tiles and
  long long row_begin;         // groups of eight rows
};

// Tile shapes of the fused step kernel (x, y extent of the thread block and z
// nodes per thread).
struct Tile {
  int tx, ty, tz;
};
constexpr int NUM_TILES = 6;   // what lb_set_tile takes
constexpr int NUM_SHAPES = 8;  // and two shallow shapes that only the choice by size takes
extern const Tile kTiles[NUM_TILES];
extern const Tile kShallow[NUM_SHAPES - NUM_TILES];
inline const Tile& tile_shape(int shape) { return shape < NUM_TILES ? kTiles[shape] : kShallow[shape - NUM_TILES]; }

size_t elem_bytes(int storage);
// population-like arrays of a state: 2 x 27 (two sets), 27 (single set) or
// the 10 quadratic-form coefficients of the moment storage
int state_arrays(int storage);
// elements of f as the device holds it (padded planes)
size_t state_elems(int storage, const Geo& g);
bool storage_is_twoset(int storage);
bool storage_is_f64(int storage);

// --- step_kernels.cu -------------------------------------------------------
// halo of the phi tile a step stages: 1 without near contact, else 4 (scan
// length K <= 3), 6 (K <= 5) or 7 (K = 6).  The wide halos have one tile, 32x8x4:
// deeper ones stage fewer values a node but leave one CTA an SM less to hide the
// scan behind (K = 5 on 150x93x203, us/step: 314 with 32x8x4, 336 with 32x8x8;
// two-set 339 against 430).  6 instead of 7 for K <= 5: 315 -> 303 us a step
// of the reduced storage there.
inline int stage_halo(const Phys& p) { return p.A_h == 0.0 ? 1 : (p.K <= 3 ? 4 : p.K <= 5 ? 6 : 7); }
// one direction of a state (not the moment storage) from its blocks to a plain
// [z][y][x] array (gather) or back
cudaError_t launch_direction(int storage, const Geo& g, void* f, int dir, void* plain, bool gather, cudaStream_t st);
// rebuild the accumulator of the current time level from the populations of in
cudaError_t launch_phi_acc(int storage, const Geo& g, const StateBuf& in, unsigned long long* acc, cudaStream_t st);
// one step (write_state) or the fields of the current level (write_fields): two
// launches, k_phi into the padded array phi (for a halo of `halo` nodes), then
// the tiles; tile indexes kTiles (only tile 0 for the variants that are not hot)
cudaError_t launch_step(int storage, int loader, bool write_state, bool write_fields, int tile, const Geo& g,
                        const Phys& p, const StateBuf& in, const InitBuf& init, PhiSrc src, AccBufs ab, StateBuf out,
                        void* phi, int halo, const FieldOut& fields, unsigned* status, cudaStream_t st);
// the density test of the current level alone (status bit 1; accin: its accumulator, null with LOAD_FIELDS)
cudaError_t launch_density(int storage, int loader, const Geo& g, const Phys& p, const StateBuf& in, const InitBuf& init,
                           const unsigned long long* accin, unsigned* status, cudaStream_t st);
// phi of the current level into the padded array, nothing else
cudaError_t launch_phi_only(int storage, const Geo& g, const Phys& p, const InitBuf& init, PhiSrc src, void* phi, int halo,
                            cudaStream_t st);
// PHI_SOLID into the whole padded array of `fields` fields (once, at its creation)
cudaError_t launch_phi_fill(int storage, const PadGeo& pg, int fields, void* phi, cudaStream_t st);
// the padded phi as a plain [z][y][x] array, 0 at solid nodes
cudaError_t launch_phi_plain(int storage, const Geo& g, const PadGeo& pg, const void* phi, void* plain, cudaStream_t st);
// export pre-collision populations of a box, canonical order, as double
cudaError_t launch_export(int storage, int loader, const Geo& g, const Phys& p, const StateBuf& in,
                          const InitBuf& init, int x0, int y0, int z0, int bx, int by, int bz, double* outA,
                          double* outB, cudaStream_t st);

// batched step (run_of: the run of every tile, then of every row group): k_phi_batched over ngroups groups of eight
// rows, then one persistent launch of blocks_per_sm x SMs CTAs over the
// tiles; parity selects S[parity] as input, k the accumulator phase (runs read
// acc[k], add into acc[(k+1)%3], clear acc[(k+2)%3]); halo is the staging halo
// that every run of the batch was created with, max_blocks the most population blocks in a z plane of a run
cudaError_t launch_batched(int storage, const RunDesc* d_runs, const int* run_of, long long ntiles, long long ngroups, int tile,
                           int halo, long long max_blocks, int parity, int k, int blocks_per_sm, unsigned* status,
                           cudaStream_t st);
// the tile shape that launch_batched takes for tile: the wide halos and planes
// beyond 32-bit byte offsets have one shape only
int batched_tile(int storage, int tile, int halo, long long max_blocks);
int sm_count_host();

// --- aux_kernels.cu ----------------------------------------------------------
cudaError_t launch_init_droplets(const Geo& g, int n, const double* d_centres, const double* d_radii, double width,
                                 float* phi0, float* rho0, float* u0, cudaStream_t st);
// deterministic FP64 sums of the fields buffer; partials needs nblocks*8 doubles
int reduce_blocks(long long N);
cudaError_t launch_reduce(int storage, const Geo& g, const void* fields, double* partials, double* out8,
                          cudaStream_t st);
cudaError_t launch_laplace(int storage, const Geo& g, const void* fields, double cut, double* partials,
                           double* out4, cudaStream_t st);
// droplet count of the padded phi
cudaError_t launch_cc(int storage, const Geo& g, const void* padded, const PadGeo& pg, int* labels, int* count,
                      unsigned* status, cudaStream_t st);
// droplet count and dispersed volume of a float phase-field array [N]
cudaError_t launch_phi_monitor(const Geo& g, const float* phi, int* labels, int* count, double* partials,
                               double* volume, unsigned* status, cudaStream_t st);

// --- surrogate_rt.cu ---------------------------------------------------------
struct SurrogateState;
void destroy_surrogate(SurrogateState* s);

// --- runtime.cu --------------------------------------------------------------
// record code + message as the calling thread's last error; returns code
int report_error(int code, const std::string& msg);
}  // namespace lbcg
struct lb_handle;
namespace lbcg {
// handle internals for the surrogate runtime
cudaStream_t handle_stream(lb_handle* h);
void handle_dims(const lb_handle* h, int* nx, int* ny, int* nz, uint32_t* walls);
void* handle_alloc(lb_handle* h, size_t bytes);  // owned (freed) by the handle
SurrogateState*& handle_surrogate(lb_handle* h);
// add n to the library's kernel launch counter
void count_launches(int n);

}  // namespace lbcg
