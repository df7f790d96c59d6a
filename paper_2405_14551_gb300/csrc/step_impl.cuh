#pragma once
// Device code of the time step of the two-component colour-gradient LB scheme on D3Q27
// (arXiv 2405.14551, Sec. III.B-III.D) for sm_103a.
//
// A step is two kernels.  k_phi decodes the phase field of the current level
// from the component densities that the step before accumulated (item 3), once
// per node, into an array padded by the staging halo, and zeroes the
// accumulator two steps ahead.  k_step works on CTA tiles of TX x TY x TZ nodes
// (TX x TY threads, TZ nodes per thread):
//   1. stage phi(t) of the tile plus a halo of H nodes in shared memory
//      (16-byte asynchronous copies from k_phi's array);
//   2. every thread walks its column of nodes.  Per node it issues the loads of
//      the 27 (x2) populations (periodic wrap, halfway bounce-back at solid
//      neighbours, Sec. III.D), takes the colour gradient from the staged tile
//      and, at an interface node with near contact (A_h != 0, halo H > K), scans
//      along its outward normal (Eqs. stress_jump, near_cont_force) while the
//      loads are in flight; then the moments, the repulsion from the distance h,
//      the Guo-shifted velocity, the relaxation of the total populations (BGK),
//      the perturbation Omega^(2) and the forcing source, the recolouring (Eqs.
//      ome3_1/2), and the post-collision state is stored once;
//   3. each post-collision component population f*^k_i(x) is also what the
//      node x + c_i pulls at the next step (x itself, as direction opp(i),
//      when x + c_i is solid), so it is x's contribution to rho_k there.  The
//      CTA sums the contributions over its tile plus a one-node ring in
//      shared memory as fixed-point integers and adds the sums to a global
//      accumulator with 64-bit integer atomics.  Integer sums are exact, so
//      phi(t+1) does not depend on the order of the additions (tile shape,
//      CTA schedule, batching), and it equals what a pull of the stored
//      populations gives (k_phi_acc rebuilds it that way after a load).
// The accumulators rotate over three buffers: a step reads phi(t) from one,
// adds phi(t+1) into the next (zeroed by the step before) and zeroes the third
// (read by the step before and not read again).  The populations are read and
// written once per step; the accumulators and the phase field add 8 B read,
// 16 B atomically updated, 8 B zeroed and 4 B written and read per node (FP32
// storages).
// Populations lie in blocks of 32 nodes of a z plane, [z][(x + pitch y) / 32][dir][32]
// (Lay<ST>): for a fixed direction a warp reads 32 consecutive nodes of one or two
// blocks, and all directions of a node are a constant offset apart.
#include <cstdio>
#include <cstdlib>
#include <type_traits>

#include "internal.h"
#include "lattice.cuh"

namespace lbcg {

// LBCG_TRACE=1 prints every launch of this file with the kernel's attributes.
inline bool trace_on() {
  static int on = -1;
  if (on < 0) {
    const char* v = std::getenv("LBCG_TRACE");
    on = (v && v[0] == '1') ? 1 : 0;
  }
  return on == 1;
}

template <typename K>
inline void trace_kernel(const char* what, K kern, dim3 grid, dim3 block, size_t smem) {
  if (!trace_on()) return;
  cudaFuncAttributes a{};
  cudaError_t e = cudaFuncGetAttributes(&a, kern);
  std::fprintf(stderr, "[lbcg] %s grid=(%u,%u,%u) block=(%u,%u,%u) smem=%zu attr=%s regs=%d maxthreads=%d local=%zu\n",
               what, grid.x, grid.y, grid.z, block.x, block.y, block.z, smem, cudaGetErrorString(e), a.numRegs,
               a.maxThreadsPerBlock, (size_t)a.localSizeBytes);
  std::fflush(stderr);
}


// ---------------------------------------------------------------------------
// storage traits
// ---------------------------------------------------------------------------
template <int ST>
struct Store;
template <>
struct Store<0> {  // LB_STORAGE_TWOSET_F32
  using R = float;
  using E = float;
  static constexpr bool TWOSET = true;
  static constexpr bool MOMENT = false;
};
template <>
struct Store<1> {  // LB_STORAGE_REDUCED_F32
  using R = float;
  using E = float;
  static constexpr bool TWOSET = false;
  static constexpr bool MOMENT = false;
};
template <>
struct Store<2> {  // LB_STORAGE_REDUCED_F16
  using R = float;
  using E = __half;
  static constexpr bool TWOSET = false;
  static constexpr bool MOMENT = false;
};
template <>
struct Store<3> {  // LB_STORAGE_TWOSET_F64
  using R = double;
  using E = double;
  static constexpr bool TWOSET = true;
  static constexpr bool MOMENT = false;
};
// LB_STORAGE_MOMENT_F32: the coefficients of f*_i = w_i (alpha + beta.c_i +
// c_i.Gamma.c_i) in three arrays of 16- and 8-byte records, so that a
// direction reads at most three vectors: qa[N] = (alpha, beta_x, beta_y,
// beta_z), qb[N] = (Gamma_xx, Gamma_yy, Gamma_zz, 2 Gamma_xy) from float 4N
// on, qc[N] = (2 Gamma_xz, 2 Gamma_yz) from float 8N on; the colour scalars
// as in the reduced storage.
template <>
struct Store<4> {
  using R = float;
  using E = float;
  static constexpr bool TWOSET = false;
  static constexpr bool MOMENT = true;
};

template <int ST>
__device__ __forceinline__ typename Store<ST>::R decode(typename Store<ST>::E v, int i) {
  if constexpr (ST == 2) {
    return wgt<float>(i) + __half2float(v) * F16_INV_SCALE;
  } else {
    return v;
  }
}
template <int ST>
__device__ __forceinline__ typename Store<ST>::E encode(typename Store<ST>::R v, int i) {
  if constexpr (ST == 2) {
    return __float2half_rn((v - wgt<float>(i)) * F16_SCALE);
  } else {
    return v;
  }
}

// Rounded products without contraction: the sending and the pulling node
// must form the same component populations bit for bit (see colour_split).
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// Moment storage (Sec. IV.C, Eq. eq:llb-pull): f*_i = w_i (alpha + beta.c +
// c.Gamma.c) of a node's coefficients at c = c_i, or at c = -c_i when bb
// (bounce-back from the node itself, dir = opp(i)).  Only the coefficients
// that c_i touches enter; the products with c components are exact (+-1).
template <typename R>
__device__ __forceinline__ R eval_moment(const float4& qa, const float4& qb, const float2& qc, int i, bool bb) {
  R lin = R(0), quad = R(0);
  if (cx(i)) lin += R(cx(i)) * qa.y;
  if (cy(i)) lin += R(cy(i)) * qa.z;
  if (cz(i)) lin += R(cz(i)) * qa.w;
  if (cx(i)) quad += qb.x;
  if (cy(i)) quad += qb.y;
  if (cz(i)) quad += qb.z;
  if (cx(i) && cy(i)) quad += R(cx(i) * cy(i)) * qb.w;
  if (cx(i) && cz(i)) quad += R(cx(i) * cz(i)) * qc.x;
  if (cy(i) && cz(i)) quad += R(cy(i) * cz(i)) * qc.y;
  return mul_rn(wgt<R>(i), qa.x + quad + (bb ? -lin : lin));
}

// Stored post-collision total population f*_dir of node src (single set
// storages).  Reduced: the stored value.  Moment storage: the node's
// quadratic form (eval_moment); only the records that c_i touches are read.
template <int ST, typename I>
__device__ __forceinline__ typename Store<ST>::R load_fs(const typename Store<ST>::E* __restrict__ f, size_t N, int dir,
                                                         I src, int i, bool bb) {
  using R = typename Store<ST>::R;
  if constexpr (Store<ST>::MOMENT) {
    const float4 qa = reinterpret_cast<const float4*>(f)[src];
    float4 qb = make_float4(0.f, 0.f, 0.f, 0.f);
    float2 qc = make_float2(0.f, 0.f);
    if (cx(i) || cy(i) || cz(i)) qb = reinterpret_cast<const float4*>(f + 4 * N)[src];
    if ((cx(i) && cz(i)) || (cy(i) && cz(i))) qc = reinterpret_cast<const float2*>(f + 8 * N)[src];
    return eval_moment<R>(qa, qb, qc, i, bb);
  } else {
    return decode<ST>(f[src + dir * BLK], i);  // src: Lay::at of the node
  }
}

__device__ __forceinline__ float sqrt_(float v) { return sqrtf(v); }
__device__ __forceinline__ double sqrt_(double v) { return sqrt(v); }
__device__ __forceinline__ float round_(float v) { return roundf(v); }  // half away from zero
__device__ __forceinline__ double round_(double v) { return round(v); }
__device__ __forceinline__ bool finite_(float v) { return isfinite(v); }
__device__ __forceinline__ bool finite_(double v) { return isfinite(v); }

// The output of a Shan-Chen collision apart from the relaxed populations, as a
// quadratic form in the lattice velocity: w_i (alpha + beta.c_i +
// c_i.Gamma.c_i).  The equilibrium and the Guo source are of this shape, so a
// node forms these ten coefficients once per component and each opposite pair
// (p, 26 - p) takes its even part w (alpha + c.Gamma.c) and its odd part
// w beta.c with one or two additions from sums that the pairs share, in place
// of scalar products and their products per direction.  128x128x256: 441 ->
// 408 us per step when it came in.  xy, xz, yz hold 2 Gamma.  The roundings are
// explicit, so every instantiation of the step forms the same values.  (The
// colour-gradient collision keeps its products per pair: the same change there
// gained 3 to 6 %, but near contact turns a last-bit difference into other
// scan decisions within tens of steps.)
template <typename R>
struct QForm {
  R a, bx, by, bz, xx, yy, zz, xy, xz, yz;
};

// The form's parts for the directions of one speed (CLS = |c|^2: 1 faces, 2
// edges, 3 corners), scaled by that class's weight.
template <typename R, int CLS>
struct QClass {
  R lx, ly, lz;     // w beta
  R d0, d1, d2;     // w (alpha + diagonal): faces x, y, z; edges xy, xz, yz; corners d0 only
  R kxy, kxz, kyz;  // w 2 Gamma_ab (edges, corners)
  __device__ __forceinline__ explicit QClass(const QForm<R>& q) {
    constexpr R W = CLS == 1 ? R(2) / R(27) : CLS == 2 ? R(1) / R(54) : R(1) / R(216);
    lx = mul_rn(W, q.bx);
    ly = mul_rn(W, q.by);
    lz = mul_rn(W, q.bz);
    const R ax = q.a + q.xx, ay = q.a + q.yy, az = q.a + q.zz;
    if constexpr (CLS == 1) {
      d0 = mul_rn(W, ax);
      d1 = mul_rn(W, ay);
      d2 = mul_rn(W, az);
    } else {
      kxy = mul_rn(W, q.xy);
      kxz = mul_rn(W, q.xz);
      kyz = mul_rn(W, q.yz);
      if constexpr (CLS == 2) {
        d0 = mul_rn(W, ax + q.yy);
        d1 = mul_rn(W, ax + q.zz);
        d2 = mul_rn(W, ay + q.zz);
      } else {
        d0 = mul_rn(W, (ax + q.yy) + q.zz);
      }
    }
  }
  // w c_p.Gamma.c_p + w alpha
  __device__ __forceinline__ R even(int p) const {
    if constexpr (CLS == 1) return cx(p) ? d0 : cy(p) ? d1 : d2;
    else if constexpr (CLS == 2)
      return cz(p) == 0   ? (cx(p) * cy(p) > 0 ? d0 + kxy : d0 - kxy)
             : cy(p) == 0 ? (cx(p) * cz(p) > 0 ? d1 + kxz : d1 - kxz)
                          : (cy(p) * cz(p) > 0 ? d2 + kyz : d2 - kyz);
    else
      return (cx(p) * cy(p) > 0 ? d0 + kxy : d0 - kxy) +
             (cx(p) * cz(p) > 0 ? (cy(p) * cz(p) > 0 ? kxz + kyz : kxz - kyz)
                                : (cy(p) * cz(p) > 0 ? kyz - kxz : -(kxz + kyz)));
  }
  // w beta.c_p
  __device__ __forceinline__ R odd(int p) const { return along(p, lx, ly, lz); }
  // c_p.(x, y, z)
  __device__ __forceinline__ static R along(int p, R x, R y, R z) {
    if constexpr (CLS == 1) {
      const R v = cx(p) ? x : cy(p) ? y : z;
      return cx(p) + cy(p) + cz(p) > 0 ? v : -v;
    } else if constexpr (CLS == 2) {
      const R u = cx(p) ? x : y, v = cz(p) ? z : y;
      const int su = cx(p) ? cx(p) : cy(p), sv = cz(p) ? cz(p) : cy(p);
      const R r = su * sv > 0 ? u + v : u - v;
      return su > 0 ? r : -r;
    } else {
      const R u = cx(p) * cy(p) > 0 ? x + y : x - y;
      const R r = cx(p) * cz(p) > 0 ? u + z : u - z;
      return cx(p) > 0 ? r : -r;
    }
  }
};

// Wrapped neighbour coordinates of a node: c[d+1] = coordinate + d on periodic
// axes (mod n); raw on wall axes.  solid[d+1] marks a solid layer.
struct Nbr {
  int xs[3], ys[3], zs[3];
  bool sx[3], sy[3], sz[3];
};

__device__ __forceinline__ void make_nbr(const Geo& g, int x, int y, int z, Nbr& n) {
#pragma unroll
  for (int d = -1; d <= 1; ++d) {
    int a = x + d, b = y + d, c = z + d;
    if (!g.wx) a = a < 0 ? a + g.nx : (a >= g.nx ? a - g.nx : a);
    if (!g.wy) b = b < 0 ? b + g.ny : (b >= g.ny ? b - g.ny : b);
    if (!g.wz) c = c < 0 ? c + g.nz : (c >= g.nz ? c - g.nz : c);
    n.xs[d + 1] = a;
    n.ys[d + 1] = b;
    n.zs[d + 1] = c;
    n.sx[d + 1] = g.wx && (a <= 0 || a >= g.nx - 1);
    n.sy[d + 1] = g.wy && (b <= 0 || b >= g.ny - 1);
    n.sz[d + 1] = g.wz && (c <= 0 || c >= g.nz - 1);
  }
}

__device__ __forceinline__ bool is_solid(const Geo& g, int x, int y, int z) {
  return (g.wx && (x == 0 || x == g.nx - 1)) || (g.wy && (y == 0 || y == g.ny - 1)) ||
         (g.wz && (z == 0 || z == g.nz - 1));
}

__device__ __forceinline__ bool near_wall(const Geo& g, int x, int y, int z) {
  return (g.wx && (x <= 1 || x >= g.nx - 2)) || (g.wy && (y <= 1 || y >= g.ny - 2)) ||
         (g.wz && (z <= 1 || z >= g.nz - 2));
}

// Directions whose source x - c_i is solid, as bit i of a word: the x and y part of
// a fluid node's column, and the z part of the node.  One bit test a direction
// replaces three flags and their union, for the pull and (bit opp(i): x + c_i) for
// the sends.
__host__ __device__ constexpr unsigned dirs_along(int axis, int sign) {
  unsigned m = 0;
  for (int i = 0; i < Q; ++i)
    if ((axis == 0 ? cx(i) : axis == 1 ? cy(i) : cz(i)) == sign) m |= 1u << i;
  return m;
}
__device__ __forceinline__ unsigned axis_bits(int wall, int v, int n, unsigned lower, unsigned upper) {
  return wall ? (v <= 1 ? lower : 0u) | (v >= n - 2 ? upper : 0u) : 0u;
}
__device__ __forceinline__ unsigned column_bits(const Geo& g, int x, int y) {
  return axis_bits(g.wx, x, g.nx, dirs_along(0, 1), dirs_along(0, -1)) | axis_bits(g.wy, y, g.ny, dirs_along(1, 1), dirs_along(1, -1));
}
__device__ __forceinline__ unsigned node_bits(const Geo& g, int z) {
  return axis_bits(g.wz, z, g.nz, dirs_along(2, 1), dirs_along(2, -1));
}

// Whether the box [x0 - d, x0 + TX - 1 + d] x ... (a tile and its halo of d
// nodes) holds a solid layer or leaves the box on a walled axis.
__device__ __forceinline__ bool region_walled(const Geo& g, int x0, int y0, int z0, int tx, int ty, int tz, int d) {
  return (g.wx && (x0 - d <= 0 || x0 + tx - 1 + d >= g.nx - 1)) ||
         (g.wy && (y0 - d <= 0 || y0 + ty - 1 + d >= g.ny - 1)) ||
         (g.wz && (z0 - d <= 0 || z0 + tz - 1 + d >= g.nz - 1));
}

// Populations of a state (all storages but the moment records) are stored in
// blocks of 32 nodes: the nodes of a z plane are counted x + pitch y, and block k
// of the plane holds the ND directions of its 32 nodes one after the other, 32
// values each.  A node's 27 (54) values then sit at constant offsets from one
// address, and so do the values that one neighbour row contributes, so that the
// pulls and stores of a node take their direction from the instruction's immediate
// offset; with nx a multiple of 32 a warp's store of a whole node row is 32 x ND
// consecutive values.  With one array per direction ([dir][z][y][x]) every access
// carried its own 64-bit address, some fifty registers of them: 2.84 -> 2.57 ms per
// step of the 256x256x512 emulsion, 385 -> 358 us of Shan-Chen 128x128x256.  Rows
// that each began a block of their own cost nx = 33 1.94 times the memory, nx = 1 32
// times, and their holes cost L2: 36x184x35, walls in y, 46.0 us a step against 38.7.
template <int ST>
struct Lay {
  using E = typename Store<ST>::E;
  static constexpr bool MOMENT = Store<ST>::MOMENT;
  static constexpr int ND = Store<ST>::TWOSET ? 2 * Q : Q;
  static constexpr int DS = MOMENT ? 1 : BLK;         // stride of the directions
  // nodes from one row to the next; elements of one z plane; the element of node n
  // of a plane at direction 0 (moment storage: the node itself)
  __host__ __device__ __forceinline__ static int pitch(const Geo& g) { return MOMENT ? g.nx : row_pitch(g.nx); }
  __host__ __device__ __forceinline__ static size_t plane(const Geo& g) {
    if constexpr (MOMENT) return (size_t)g.nx * (size_t)g.ny;
    else return plane_blocks(g) * (ND * BLK);
  }
  template <typename I>
  __host__ __device__ __forceinline__ static I in_plane(I n) {
    return MOMENT ? n : n / BLK * (I)(ND * BLK) + n % BLK;
  }
  __host__ __device__ __forceinline__ static size_t at(const Geo& g, int x, int y, int z) {
    return plane(g) * (size_t)z + in_plane((size_t)x + (size_t)pitch(g) * (size_t)y);
  }
};

template <int ST>
struct View {
  using E = typename Store<ST>::E;
  E* f;
  float4* sv;
};

template <int ST>
__host__ __device__ __forceinline__ View<ST> view(const StateBuf& b) {
  View<ST> v;
  v.f = reinterpret_cast<typename Store<ST>::E*>(b.f);
  v.sv = b.sv;
  return v;
}

// Component split of a single-set population as the pulling node rebuilds it
// (recolouring, Eq. ome3_1, evaluated one step later): f^A_i = s f*_i +
// w_i c_i.v/|c_i|, f^B_i = f*_i - f^A_i, with (s, v) the colour scalars of the
// node that stored f*_i.  bb: bounce-back, the node's own f*_opp(i) pulled as
// direction i, whose segregation term is the negative of direction i's.  The
// rounding is explicit, so the sender of a value (step_nodes) and its puller
// form the same f^A_i, f^B_i bit for bit.
template <typename R, bool MAYBB>
__device__ __forceinline__ void colour_split(R fs, const float4& sv, int i, bool bb, R& va, R& vb) {
  R cv = R(0);
  if (cx(i)) cv += R(cx(i)) * R(sv.y);
  if (cy(i)) cv += R(cy(i)) * R(sv.z);
  if (cz(i)) cv += R(cz(i)) * R(sv.w);
  const R k = wgt<R>(i) * inv_norm<R>(i);  // folded to one constant per direction
  R seg = mul_rn(k, cv);
  if constexpr (MAYBB) seg = bb ? -seg : seg;
  va = fma_rn(R(sv.x), fs, seg);
  vb = fs - va;
}

// Pull the pre-collision populations of node `self` (streaming, Eq. eq:lbm):
// f_i(x) = f*_i(x - c_i), or f*_{opp(i)}(x) when x - c_i is solid (halfway
// bounce-back).  Returns the totals f_i and the component densities.  With
// per-component output (fa, fb non-null) also the component populations.
template <int ST, bool COMP>
__device__ __forceinline__ void pull_node(const View<ST>& S, const Geo& g, const Nbr& n, long long self,
                                          typename Store<ST>::R f[Q], typename Store<ST>::R& rA,
                                          typename Store<ST>::R& rB, typename Store<ST>::R* fa,
                                          typename Store<ST>::R* fb) {
  using R = typename Store<ST>::R;
  const size_t N = (size_t)g.N;
  rA = R(0);
  rB = R(0);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int a = 1 - cx(i), b = 1 - cy(i), c = 1 - cz(i);
    const bool bb = n.sx[a] | n.sy[b] | n.sz[c];
    const int sx = bb ? n.xs[1] : n.xs[a], sy = bb ? n.ys[1] : n.ys[b], sz = bb ? n.zs[1] : n.zs[c];
    const size_t src = Lay<ST>::at(g, sx, sy, sz);
    const int dir = bb ? opp(i) : i;
    R va, vb;
    if constexpr (Store<ST>::TWOSET) {
      va = decode<ST>(S.f[src + (size_t)dir * BLK], i);
      vb = decode<ST>(S.f[src + (size_t)(Q + dir) * BLK], i);
      f[i] = va + vb;
    } else {
      const R fs = load_fs<ST>(S.f, N, dir, src, i, bb);
      colour_split<R, true>(fs, S.sv[(size_t)sx + (size_t)g.nx * ((size_t)sy + (size_t)g.ny * sz)], i, bb, va, vb);
      f[i] = fs;
    }
    rA += va;
    rB += vb;
    if constexpr (COMP) {
      fa[i] = va;
      fb[i] = vb;
    }
  }
}

// Pre-collision populations from fields (initial state or reconstruction):
// f_i = f^eq_i(rho, u) (Eq. disteq) [+ w_i/(2 cs^4) Q_i:Pi^neq], f^A = (rhoA/rho) f.
template <typename R, bool COMP>
__device__ __forceinline__ void fields_node(const InitBuf& I, const Geo& g, const PhysR<R>& P, const Nbr& n,
                                            long long self, R f[Q], R& rA, R& rB, R* fa, R* fb) {
  const R ph = I.phi[self];
  const R rho = I.rho ? R(I.rho[self]) : R(1);
  R u[3] = {R(0), R(0), R(0)};
  if (I.u) {
    u[0] = I.u[self];
    u[1] = I.u[(size_t)g.N + self];
    u[2] = I.u[2 * (size_t)g.N + self];
  }
  rA = rho * (R(1) + ph) * R(0.5);
  rB = rho * (R(1) - ph) * R(0.5);
  R Pi[6] = {R(0), R(0), R(0), R(0), R(0), R(0)};  // xx yy zz xy xz yz
  if (I.regularised && I.u) {
    // isotropic stencil gradient du[b][a] = d_a u_b; solid neighbour -> own value
    R du[3][3] = {{R(0), R(0), R(0)}, {R(0), R(0), R(0)}, {R(0), R(0), R(0)}};
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      if (i == REST) continue;
      const int a = 1 + cx(i), b = 1 + cy(i), c = 1 + cz(i);
      const bool sol = n.sx[a] | n.sy[b] | n.sz[c];
      const long long m =
          sol ? self : (long long)n.xs[a] + (long long)g.nx * ((long long)n.ys[b] + (long long)g.ny * n.zs[c]);
      const R w3 = R(3) * wgt<R>(i);
#pragma unroll
      for (int bcomp = 0; bcomp < 3; ++bcomp) {
        const R ub = I.u[(size_t)bcomp * g.N + m];
        du[bcomp][0] += w3 * R(cx(i)) * ub;
        du[bcomp][1] += w3 * R(cy(i)) * ub;
        du[bcomp][2] += w3 * R(cz(i)) * ub;
      }
    }
    R tau;
    if (P.equal_tau) {
      tau = R(P.tau_a);
    } else {
      const R nu_a = (R(P.tau_a) - R(0.5)) / R(3), nu_b = (R(P.tau_b) - R(0.5)) / R(3);
      const R nu = R(1) / ((rA / rho) / nu_a + (rB / rho) / nu_b);
      tau = R(3) * nu + R(0.5);
    }
    const R pref = -rho * tau / R(3);  // Pi^neq = -rho cs2 tau (grad u + grad u^T)
    Pi[0] = pref * R(2) * du[0][0];
    Pi[1] = pref * R(2) * du[1][1];
    Pi[2] = pref * R(2) * du[2][2];
    Pi[3] = pref * (du[0][1] + du[1][0]);
    Pi[4] = pref * (du[0][2] + du[2][0]);
    Pi[5] = pref * (du[1][2] + du[2][1]);
  }
  const R uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const R trPi = Pi[0] + Pi[1] + Pi[2];
  const R sA = rA / rho;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const R cu = R(cx(i)) * u[0] + R(cy(i)) * u[1] + R(cz(i)) * u[2];
    R fi = wgt<R>(i) * rho * (R(1) + R(3) * cu + R(4.5) * cu * cu - R(1.5) * uu);
    // (c c - cs2 I):Pi with symmetric Pi
    const R qpi = R(cx(i) * cx(i)) * Pi[0] + R(cy(i) * cy(i)) * Pi[1] + R(cz(i) * cz(i)) * Pi[2] +
                  R(2 * cx(i) * cy(i)) * Pi[3] + R(2 * cx(i) * cz(i)) * Pi[4] + R(2 * cy(i) * cz(i)) * Pi[5] -
                  trPi / R(3);
    fi += wgt<R>(i) * R(4.5) * qpi;
    f[i] = fi;
    if constexpr (COMP) {
      fa[i] = sA * fi;
      fb[i] = fi - sA * fi;
    }
  }
}

// A value that is the same in every lane, in a form the compiler knows to be
// uniform (a warp reduction's result), so that base addresses made from it
// take the uniform path as kernel parameters do.
__device__ __forceinline__ int uniform(int v) { return (int)__reduce_or_sync(0xffffffffu, (unsigned)v); }
__device__ __forceinline__ float uniform(float v) { return __int_as_float(uniform(__float_as_int(v))); }
template <typename T>
__device__ __forceinline__ T* uniform(T* p) {
  const unsigned long long v = reinterpret_cast<unsigned long long>(p);
  const unsigned lo = __reduce_or_sync(0xffffffffu, (unsigned)v), hi = __reduce_or_sync(0xffffffffu, (unsigned)(v >> 32));
  return reinterpret_cast<T*>(((unsigned long long)hi << 32) | lo);
}
// Where a node reads its neighbours' values.  The z plane of a source is the
// same for the whole CTA, so a thread keeps nine offsets within a plane (3 x 3
// neighbours in x and y, wrapped; a fluid node of a walled axis never wraps)
// for all its nodes; 27 addresses serve all pulls.  IDX32: the byte offsets
// within one z plane fit in 32 bits.
template <int ST, bool IDX32>
struct PlaneIdx {
  using I = typename std::conditional<IDX32, unsigned, size_t>::type;
  I o[3][3];  // [y + 1][x + 1] element offset within a plane (moment storage: node offset)
  __device__ __forceinline__ static I at(const Geo& g, int x, int y) { return Lay<ST>::in_plane((I)x + (I)Lay<ST>::pitch(g) * (I)y); }
  __device__ __forceinline__ void init(const Geo& g, int x, int y) {
    int xs[3], ys[3];
#pragma unroll
    for (int d = -1; d <= 1; ++d) {
      int a = x + d, b = y + d;
      xs[d + 1] = a < 0 ? a + g.nx : (a >= g.nx ? a - g.nx : a);
      ys[d + 1] = b < 0 ? b + g.ny : (b >= g.ny ? b - g.ny : b);
    }
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
      for (int a = 0; a < 3; ++a) o[b][a] = at(g, xs[a], ys[b]);
  }
};
// value at element offset o of a plane whose first element is base
template <typename T, typename I>
__device__ __forceinline__ T plane_ld(const T* __restrict__ base, I o) {
  return *reinterpret_cast<const T*>(reinterpret_cast<const char*>(base) + (I)(o * (I)sizeof(T)));
}
// The raw stored values a node pulls (both sets, or the single set's totals),
// loaded before anything is decoded so that independent work (gradient, scan)
// runs while they are in flight.  Not WALLFREE: where wall has the direction's
// bit, the opposite direction of the node itself (halfway bounce-back), as one
// predicated load each way (selecting the address: 3 % slower at walls in x, single set).
template <int ST, bool IDX32, bool WALLFREE>
__device__ __forceinline__ void pull_plane(const View<ST>& S, const Geo& g, const PlaneIdx<ST, IDX32>& ix, const int zs[3],
                                           unsigned wall, typename Store<ST>::E ra[Q], typename Store<ST>::E rb[Q]) {
  using E = typename Store<ST>::E;
  const size_t plane = Lay<ST>::plane(g);
  const E* zp[3] = {S.f + (size_t)zs[0] * plane, S.f + (size_t)zs[1] * plane, S.f + (size_t)zs[2] * plane};
  auto at = [](const E* z, auto o) { return reinterpret_cast<const E*>(reinterpret_cast<const char*>(z) + o * (unsigned)sizeof(E)); };
  const E* self = at(zp[1], ix.o[1][1]);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int a = 1 - cx(i), b = 1 - cy(i), c = 1 - cz(i);
    const E* p = at(zp[c], ix.o[b][a]);
    if (!WALLFREE && (wall >> i & 1u)) {
      ra[i] = self[opp(i) * BLK];
      if constexpr (Store<ST>::TWOSET) rb[i] = self[(Q + opp(i)) * BLK];
    } else {
      ra[i] = p[i * BLK];
      if constexpr (Store<ST>::TWOSET) rb[i] = p[(Q + i) * BLK];
    }
  }
}
// moment storage: the quadratic forms of the neighbours, evaluated
template <int ST, bool IDX32>
__device__ __forceinline__ void pull_plane_moment(const View<ST>& S, size_t N, size_t plane, const PlaneIdx<ST, IDX32>& ix,
                                                  const int zs[3], typename Store<ST>::R f[Q]) {
  using R = typename Store<ST>::R;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const size_t zp = (size_t)zs[1 - cz(i)] * plane;
    const auto o = ix.o[1 - cy(i)][1 - cx(i)];
    const float4 qa = plane_ld(reinterpret_cast<const float4*>(S.f) + zp, o);
    float4 qb = make_float4(0.f, 0.f, 0.f, 0.f);
    float2 qc = make_float2(0.f, 0.f);
    if (i != REST) qb = plane_ld(reinterpret_cast<const float4*>(S.f + 4 * N) + zp, o);
    if ((cx(i) && cz(i)) || (cy(i) && cz(i))) qc = plane_ld(reinterpret_cast<const float2*>(S.f + 8 * N) + zp, o);
    f[i] = eval_moment<R>(qa, qb, qc, i, false);
  }
}
// The same with solid neighbours in reach, by node index (a lattice has fewer
// than 2^31 nodes).
template <int ST>
__device__ __forceinline__ void pull_walled_moment(const View<ST>& S, const Geo& g, const Nbr& n, unsigned wall, int self,
                                                   typename Store<ST>::R f[Q]) {
  int row[3][3];
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int c = 0; c < 3; ++c) row[b][c] = g.nx * (n.ys[b] + g.ny * n.zs[c]);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int a = 1 - cx(i), b = 1 - cy(i), c = 1 - cz(i);
    const bool bb = wall >> i & 1u;
    f[i] = load_fs<ST>(S.f, (size_t)g.N, i, (unsigned)(bb ? self : n.xs[a] + row[b][c]), i, bb);
  }
}
// The same loads of any node (self: its Lay::at element), at any offset width,
// outside the step.
template <int ST>
__device__ __forceinline__ void pull_walled(const View<ST>& S, const Geo& g, const Nbr& n, size_t self,
                                            typename Store<ST>::E ra[Q], typename Store<ST>::E rb[Q],
                                            typename Store<ST>::R f[Q]) {
  const size_t N = (size_t)g.N;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int a = 1 - cx(i), b = 1 - cy(i), c = 1 - cz(i);
    const bool bb = n.sx[a] | n.sy[b] | n.sz[c];
    const size_t src = bb ? self : Lay<ST>::at(g, n.xs[a], n.ys[b], n.zs[c]);
    const int dir = bb ? opp(i) : i;
    if constexpr (Store<ST>::MOMENT) {
      f[i] = load_fs<ST>(S.f, N, dir, src, i, bb);
    } else {
      ra[i] = S.f[src + dir * BLK];
      if constexpr (Store<ST>::TWOSET) rb[i] = S.f[src + (Q + dir) * BLK];
    }
  }
}
// Decode the raw values: totals f_i and, for two sets, the component densities.
template <int ST>
__device__ __forceinline__ void pull_finish(const typename Store<ST>::E ra[Q], const typename Store<ST>::E rb[Q],
                                            typename Store<ST>::R f[Q], typename Store<ST>::R& rA,
                                            typename Store<ST>::R& rB) {
  using R = typename Store<ST>::R;
  rA = R(0);
  rB = R(0);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    if constexpr (Store<ST>::TWOSET) {
      const R va = decode<ST>(ra[i], i), vb = decode<ST>(rb[i], i);
      f[i] = va + vb;
      rA += va;
      rB += vb;
    } else {
      f[i] = decode<ST>(ra[i], i);
    }
  }
}

// ---------------------------------------------------------------------------
// write-side accumulation of the next time level's component densities
// ---------------------------------------------------------------------------
// Each contribution f*^k_i is rounded to a multiple of 2^-SHIFT and summed as
// an integer.  FP32 storages: SHIFT = 28 (component sums within +-8, step
// 3.7e-9, below the FP32 rounding of a density near 1), the two sums of a
// node packed in one 64-bit word (rhoA in the high half, rhoB in the low
// half, two's complement), so one atomic adds both.  FP64: SHIFT = 56 (sums
// within +-128, step 1.4e-17), two 64-bit words per node.  RHO_MAX bounds the
// density that the status check accepts, so that no sum leaves its range.
// The accumulator words are read, zeroed and updated by every step while the
// population state streams through L2; their stores and reductions carry an
// evict-last L2 policy, so that more of them are still in L2 when the next
// access comes (256x256x512 emulsion, 3.24 -> 3.17 ms per step when it came in,
// before k_phi).
__device__ __forceinline__ unsigned long long acc_policy() {
  unsigned long long pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void acc_red(unsigned long long* p, unsigned long long v) {
  asm volatile("red.global.add.L2::cache_hint.u64 [%0], %1, %2;" ::"l"(__cvta_generic_to_global(p)), "l"(v),
               "l"(acc_policy())
               : "memory");
}
__device__ __forceinline__ void acc_st(unsigned long long* p, unsigned long long v) {
  asm volatile("st.global.L2::cache_hint.u64 [%0], %1, %2;" ::"l"(__cvta_generic_to_global(p)), "l"(v),
               "l"(acc_policy())
               : "memory");
}
template <typename R>
struct Acc;
template <>
struct Acc<float> {
  static constexpr int W = 1;  // 64-bit words per node, in global and in shared memory
  using S = int;               // sum of one component
  static constexpr float RHO_MAX = 4.0f;
  static constexpr float SCALE = 268435456.0f;
  __device__ static __forceinline__ S q(float v) { return __float2int_rn(v * SCALE); }
  // the same for values that are already multiplied by SCALE (exact: a power of two)
  __device__ static __forceinline__ void send_shared_scaled(unsigned long long* sw, int E, int e, float a, float b) {
    int* p = reinterpret_cast<int*>(sw);
    atomicAdd(p + e, __float2int_rn(a));
    atomicAdd(p + E + e, __float2int_rn(b));
  }
  // add one node's contributions (a, b) to the shared partial sums of node e:
  // two planes of E 32-bit words (rhoA, then rhoB) in the E 64-bit words of
  // sw; 32-bit shared atomics (one packed 64-bit shared atomic per direction
  // measured slower)
  __device__ static __forceinline__ void send_shared(unsigned long long* sw, int E, int e, float a, float b) {
    int* p = reinterpret_cast<int*>(sw);
    atomicAdd(p + e, q(a));
    atomicAdd(p + E + e, q(b));
  }
  __device__ static __forceinline__ void flush_shared(unsigned long long* acc, size_t node,
                                                      const unsigned long long* sw, int E, int e) {
    const int* p = reinterpret_cast<const int*>(sw);
    const unsigned long long w = pack(p[e], p[E + e]);
    if (w) acc_red(acc + node, w);
  }
  __device__ static __forceinline__ bool shared_zero(const unsigned long long* sw, int E, int e) {
    const int* p = reinterpret_cast<const int*>(sw);
    return (p[e] | p[E + e]) == 0;
  }
  __device__ static __forceinline__ unsigned long long pack(S a, S b) {
    return ((unsigned long long)(unsigned)a << 32) + (unsigned long long)(long long)b;
  }
  __device__ static __forceinline__ void store(unsigned long long* acc, size_t node, S a, S b) {
    acc[node] = pack(a, b);
  }
  __device__ static __forceinline__ void zero(unsigned long long* acc, size_t node) { acc_st(acc + node, 0ull); }
  // phi = (rhoA - rhoB)/(rhoA + rhoB) of one packed word.  The halves are
  // rhoA and rhoB in units of 2^-28; with densities below RHO_MAX (< 2^30
  // units) the difference and the sum are exact 32-bit integers, each rounded
  // once to FP32, and the quotient is taken with the fast reciprocal (about 2
  // ulp; every stage of phi uses this one function, so results are
  // reproducible).  phi feeds the colour gradient and the near-contact scan
  // only; the component densities come from the sums themselves (densities).
  __device__ static __forceinline__ float phi_word(unsigned long long w) {
    const int lo = (int)(unsigned)w;
    const int hi = (int)(unsigned)(w >> 32) + (int)((unsigned)lo >> 31);  // undo the borrow of a negative low half
    return __fdividef((float)(hi - lo), (float)(hi + lo));
  }
  __device__ static __forceinline__ float phi(const unsigned long long* acc, size_t node) {
    return phi_word(acc[node]);
  }
  // rhoA and rhoB of a node, each rounded once
  __device__ static __forceinline__ void densities(const unsigned long long* acc, size_t node, float& a, float& b) {
    const unsigned long long w = acc[node];
    const int lo = (int)(unsigned)w;
    const int hi = (int)(unsigned)(w >> 32) + (int)((unsigned)lo >> 31);
    a = (float)hi * (1.0f / 268435456.0f);
    b = (float)lo * (1.0f / 268435456.0f);
  }
};
template <>
struct Acc<double> {
  static constexpr int W = 2;
  using S = long long;
  static constexpr double RHO_MAX = 64.0;
  __device__ static __forceinline__ S q(double v) { return __double2ll_rn(v * 72057594037927936.0); }
  // two planes of E shared words: rhoA at sw[e], rhoB at sw[E + e]
  __device__ static __forceinline__ void send_shared(unsigned long long* sw, int E, int e, double a, double b) {
    atomicAdd(sw + e, (unsigned long long)q(a));
    atomicAdd(sw + E + e, (unsigned long long)q(b));
  }
  __device__ static __forceinline__ void flush_shared(unsigned long long* acc, size_t node,
                                                      const unsigned long long* sw, int E, int e) {
    if (sw[e]) acc_red(acc + 2 * node, sw[e]);
    if (sw[E + e]) acc_red(acc + 2 * node + 1, sw[E + e]);
  }
  __device__ static __forceinline__ bool shared_zero(const unsigned long long* sw, int E, int e) {
    return (sw[e] | sw[E + e]) == 0ull;
  }
  __device__ static __forceinline__ void store(unsigned long long* acc, size_t node, S a, S b) {
    acc[2 * node] = (unsigned long long)a;
    acc[2 * node + 1] = (unsigned long long)b;
  }
  __device__ static __forceinline__ void zero(unsigned long long* acc, size_t node) {
    acc_st(acc + 2 * node, 0ull);
    acc_st(acc + 2 * node + 1, 0ull);
  }
  __device__ static __forceinline__ double phi_words(unsigned long long wa, unsigned long long wb) {
    const long long a = (long long)wa, b = (long long)wb;
    return (double)(a - b) / (double)(a + b);
  }
  __device__ static __forceinline__ double phi(const unsigned long long* acc, size_t node) {
    return phi_words(acc[2 * node], acc[2 * node + 1]);
  }
  __device__ static __forceinline__ void densities(const unsigned long long* acc, size_t node, double& a, double& b) {
    a = (double)(long long)acc[2 * node] * (1.0 / 72057594037927936.0);
    b = (double)(long long)acc[2 * node + 1] * (1.0 / 72057594037927936.0);
  }
};

// The integer sums of the component populations a node pulls (the same
// values, hence the same sums, as the senders accumulated).
template <int ST, bool WALLFREE>
__device__ __forceinline__ void pull_acc(const View<ST>& S, const Geo& g, const Nbr& n,
                                         typename Acc<typename Store<ST>::R>::S& sa,
                                         typename Acc<typename Store<ST>::R>::S& sb) {
  using R = typename Store<ST>::R;
  using A = Acc<R>;
  const size_t N = (size_t)g.N;
  sa = 0;
  sb = 0;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int a = 1 - cx(i), b = 1 - cy(i), c = 1 - cz(i);
    const bool bb = WALLFREE ? false : (n.sx[a] | n.sy[b] | n.sz[c]);
    const int sx = bb ? n.xs[1] : n.xs[a], sy = bb ? n.ys[1] : n.ys[b], sz = bb ? n.zs[1] : n.zs[c];
    const size_t src = Lay<ST>::at(g, sx, sy, sz);
    const int dir = bb ? opp(i) : i;
    R va, vb;
    if constexpr (Store<ST>::TWOSET) {
      va = decode<ST>(S.f[src + dir * BLK], i);
      vb = decode<ST>(S.f[src + (Q + dir) * BLK], i);
    } else {
      const R fs = load_fs<ST>(S.f, N, dir, src, i, bb);
      colour_split<R, !WALLFREE>(fs, S.sv[(size_t)sx + (size_t)g.nx * ((size_t)sy + (size_t)g.ny * sz)], i, bb, va, vb);
    }
    sa += A::q(va);
    sb += A::q(vb);
  }
}

// Rebuild the accumulator of the current time level from stored populations
// (after a checkpoint load or a state copy): one node per thread.
template <int ST>
__global__ void __launch_bounds__(256) k_phi_acc(View<ST> S, Geo g, unsigned long long* __restrict__ acc) {
  using A = Acc<typename Store<ST>::R>;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < g.N; idx += stride) {
    const int x = (int)(idx % g.nx);
    const long long yz = idx / g.nx;
    const int y = (int)(yz % g.ny);
    const int z = (int)(yz / g.ny);
    if (is_solid(g, x, y, z)) {
      A::zero(acc, (size_t)idx);
      continue;
    }
    Nbr n;
    make_nbr(g, x, y, z, n);
    typename A::S sa, sb;
    if (near_wall(g, x, y, z))
      pull_acc<ST, false>(S, g, n, sa, sb);
    else
      pull_acc<ST, true>(S, g, n, sa, sb);
    A::store(acc, (size_t)idx, sa, sb);
  }
}

// ---------------------------------------------------------------------------
// phase field of the current level
// ---------------------------------------------------------------------------
// k_phi decodes the staged scalars of the whole lattice once per step into a
// padded array (PadGeo), so that a tile stages its halo with plain 16-byte
// asynchronous copies: no wrap, no solid test and no decoding in the tile.
// The decoding of one value (two integer-to-float conversions and a
// reciprocal) used to be repeated for every tile that holds the node in its
// halo, 5 times per node for a 32x8x8 tile with near contact.
// Fields: phi, or (Shan-Chen) phi, psi_A, psi_B.  A warp takes a row of nodes,
// reads each word once and stores it to every padded position that wraps onto
// it; positions beyond a wall and solid layers hold PHI_SOLID from the array's
// creation (k_phi_fill) on.  It also zeroes the accumulator two steps ahead
// (AccBufs::zero, or null).
// Bound: bytes (8 B read, 4 B written, 8 B zeroed per node).
template <typename R>
__device__ __forceinline__ R sc_psi(R r, R psi0) {
  if constexpr (sizeof(R) == 4) return psi0 * (1.0f - expf(-r / psi0));
  else return psi0 * (1.0 - exp(-r / psi0));
}

// The launches of a step (k_phi, k_step, k_phi of the next, ...) follow one
// another with programmatic dependent launch: a kernel lets its successor
// start filling free SMs once all its own CTAs run, and touches global memory
// only after its predecessor has completed.  That hides the launch latency,
// the larger part of a step on small lattices.  Together with k_phi reading each
// word once: 58.1 -> 54.5 us per step at 64x64x128 (an event after every step; 44.7
// when 12 steps replay from a graph), 2.57 -> 2.50 ms at 256x256x512.
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_primary() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Source coordinate of padded coordinate c - h on an axis of n nodes; -1
// where the position is solid or beyond a wall.
__device__ __forceinline__ int pad_source(int c, int h, int n, int wall) {
  int v = c - h;
  if (wall) return v <= 0 || v >= n - 1 ? -1 : v;
  if ((unsigned)v < (unsigned)n) return v;
  v += v < 0 ? n : -n;
  if ((unsigned)v < (unsigned)n) return v;
  return ((v % n) + n) % n;
}

template <typename R, bool SC>
__device__ __forceinline__ void phi_row(const PhiSrc& src, const InitBuf& init, const Geo& g, const PadGeo& pg, R psi0,
                                        R* __restrict__ out, unsigned long long* __restrict__ zero, int y, int z) {
  if ((g.wy && (y == 0 || y == g.ny - 1)) || (g.wz && (z == 0 || z == g.nz - 1))) return;
  const int lane = threadIdx.x;
  const size_t fld = (size_t)pg.px * pg.py * pg.pz;
  const size_t base = (size_t)g.nx * ((size_t)y + (size_t)g.ny * z);
  const int xa = g.wx ? 1 : 0, xb = g.wx ? g.nx - 1 : g.nx;  // fluid nodes of the row
  // padded coordinates that wrap onto the row: its own first
  const int ey = g.wy ? 0 : g.ny, ez = g.wz ? 0 : g.nz, limy = g.ny + 2 * pg.h, limz = g.nz + 2 * pg.h;
  int cy0 = y + pg.h, cz0 = z + pg.h;
  while (ey && cy0 >= ey) cy0 -= ey;
  while (ez && cz0 >= ez) cz0 -= ez;
  for (int x0 = xa; x0 < xb; x0 += 128) {
    R v[4][SC ? 3 : 1];
    // four positions a lane, 32 apart: their loads are in flight together
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int x = x0 + 32 * j + lane;
      if (x >= xb) continue;
      if constexpr (SC) {
        R ra, rb;
        if (src.acc) {
          Acc<R>::densities(src.acc, base + x, ra, rb);
        } else {
          const R ph = R(src.phi[base + x]);
          const R rho = init.rho ? R(init.rho[base + x]) : R(1);
          ra = rho * (R(1) + ph) * R(0.5);
          rb = rho * (R(1) - ph) * R(0.5);
        }
        v[j][0] = (ra - rb) / (ra + rb);
        v[j][1] = sc_psi(ra, psi0);
        v[j][2] = sc_psi(rb, psi0);
      } else {
        v[j][0] = src.acc ? Acc<R>::phi(src.acc, base + x) : R(src.phi[base + x]);
      }
    }
    if (zero) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (x0 + 32 * j + lane < xb) Acc<R>::zero(zero, base + x0 + 32 * j + lane);
    }
    for (int cz = cz0; cz < limz; cz += ez ? ez : limz) {
      for (int cy = cy0; cy < limy; cy += ey ? ey : limy) {
        R* row = out + (size_t)pg.px * ((size_t)cy + (size_t)pg.py * cz);
        auto put = [&](int c, const R* w) {
          row[c] = w[0];
          if constexpr (SC) {
            row[fld + c] = w[1];
            row[2 * fld + c] = w[2];
          }
        };
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int x = x0 + 32 * j + lane;
          if (x >= xb) continue;
          const int c = x + pg.hx;
          put(c, v[j]);
          if (!g.wx) {
            for (int d = c - g.nx; d >= 0; d -= g.nx) put(d, v[j]);
            for (int d = c + g.nx; d < g.nx + 2 * pg.hx; d += g.nx) put(d, v[j]);
          }
        }
      }
    }
  }
}

template <typename R, bool SC>
__global__ void __launch_bounds__(256) k_phi(PhiSrc src, InitBuf init, Geo g, PadGeo pg, R psi0, R* __restrict__ out,
                                             unsigned long long* __restrict__ zero) {
  launch_dependents();
  wait_primary();
  const long long rows = (long long)g.ny * g.nz;
  for (long long row = (long long)blockIdx.x * 8 + threadIdx.y; row < rows; row += (long long)gridDim.x * 8)
    phi_row<R, SC>(src, init, g, pg, psi0, out, zero, (int)(row % g.ny), (int)(row / g.ny));
}

// The density test of the step and of the field pass (rho within (0, RHO_MAX),
// or the run is marked unstable) by itself, for readouts of phi alone: k_phi's
// sums are integers that a population which is not a number does not enter, so
// the populations are pulled and summed as the step does it.  Initial fields
// (LOAD_FIELDS) need phi and rho only, since fields_node's densities do not
// depend on its populations.  A warp takes a row; bound by the population bytes
// (half a step's), or 4 to 8 bytes a node: two-set FP32, 128x128x256, 151 us pulled
// (133 at the copy rate), 13 us of initial fields (about 100 with a thread per node
// and its two 64-bit divisions).
template <int ST, int LOADER>
__global__ void __launch_bounds__(256) k_density(View<ST> S, InitBuf init, const unsigned long long* __restrict__ accin, Geo g,
                                                 PhysR<typename Store<ST>::R> P, unsigned* __restrict__ status) {
  using R = typename Store<ST>::R;
  using E = typename Store<ST>::E;
  bool bad = false;
  const long long rows = (long long)g.ny * g.nz;
  for (long long row = (long long)blockIdx.x * 8 + threadIdx.y; row < rows; row += (long long)gridDim.x * 8) {
    const int z = (int)((unsigned)row / (unsigned)g.ny), y = (int)row - z * g.ny;  // rows <= nodes < 2^31
    for (int x = threadIdx.x; x < g.nx; x += 32) {
      if (is_solid(g, x, y, z)) continue;
      const long long idx = row * g.nx + x;
      Nbr n;
      make_nbr(g, x, y, z, n);
      R f[Q], rA, rB;
      if constexpr (LOADER == LOAD_PULL) {
        E ra[Q], rb[Q];
        pull_walled<ST>(S, g, n, Lay<ST>::at(g, x, y, z), ra, rb, f);
        if constexpr (!Store<ST>::MOMENT) pull_finish<ST>(ra, rb, f, rA, rB);
        if constexpr (!Store<ST>::TWOSET) {
          R rt = R(0);
#pragma unroll
          for (int i = 0; i < Q; ++i) rt += f[i];
          Acc<R>::densities(accin, (size_t)idx, rA, rB);
          rB = rt - rA;
        }
      } else {
        fields_node<R, false>(init, g, P, n, idx, f, rA, rB, nullptr, nullptr);
      }
      const R rho = rA + rB;
      bad |= !(rho > R(0) && rho < R(Acc<R>::RHO_MAX));
    }
  }
  if (bad) atomicOr(status, 1u);
}

// ---------------------------------------------------------------------------
// shared-memory layout of a tile
// ---------------------------------------------------------------------------
// The staged scalar fields (NPH of them) of the tile plus a halo of H nodes
// (pad_hx(H) along x, so that rows are whole 16-byte pieces of the padded
// array) and the component partial sums over the tile plus a one-node ring.
constexpr size_t align16(size_t b) { return (b + 15) / 16 * 16; }

template <typename R, int TX, int TY, int TZ, int H, int NPH = 1>
struct Layout {
  static constexpr int HX = pad_hx(H);
  static constexpr int SX = TX + 2 * HX, SY = TY + 2 * H, SZ = TZ + 2 * H, SXY = SX * SY, NS = SXY * SZ;
  static constexpr int EX = TX + 2, EY = TY + 2, EZ = TZ + 2, EXY = EX * EY, E = EXY * EZ;
  static constexpr size_t off_acc = align16(sizeof(R) * (size_t)NS * NPH);
  static constexpr size_t bytes = off_acc + align16(8 * (size_t)Acc<R>::W * (size_t)E);
};

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Issue the copies of the tile's staged fields (the caller waits for them
// with cp_async_wait_all and a barrier).
template <typename R, int TX, int TY, int TZ, int H, int NPH>
__device__ __forceinline__ void stage_tile(const R* __restrict__ phi, const PadGeo& pg, R* sp, int x0, int y0, int z0) {
  using L = Layout<R, TX, TY, TZ, H, NPH>;
  constexpr int V = 16 / (int)sizeof(R), QR = L::SX / V, ROWS = L::SY * L::SZ, NT = TX * TY;
  const size_t fld = (size_t)pg.px * pg.py * pg.pz;
  const R* base = phi + (size_t)x0 + (size_t)pg.px * ((size_t)y0 + (size_t)pg.py * z0);
  const int tid = threadIdx.y * TX + threadIdx.x;
#pragma unroll
  for (int k = 0; k < (QR * ROWS + NT - 1) / NT; ++k) {
    const int q = tid + k * NT;
    if (q >= QR * ROWS) break;
    const int row = q / QR, c = (q - row * QR) * V;
    const int lz = row / L::SY, ly = row - lz * L::SY;
    const size_t o = (size_t)pg.px * ((size_t)ly + (size_t)pg.py * lz) + c;
#pragma unroll
    for (int f = 0; f < NPH; ++f) cp_async16(sp + f * L::NS + row * L::SX + c, base + f * fld + o);
  }
}

// ---------------------------------------------------------------------------
// colour gradient and near-contact scan on the staged tile
// ---------------------------------------------------------------------------
// Colour gradient grad phi(p) = (1/cs2) sum_i w_i c_i phi(p + c_i) on the
// shared tile; a solid neighbour contributes phi(p) (neutral wetting).  The
// D3Q27 weights factor: for c_a = +-1, w(c) = v(c_b) v(c_c) / 216 with v(0) =
// 4, v(+-1) = 1 on the two other axes, so each component is the central
// difference along its axis smoothed by (1, 4, 1) x (1, 4, 1) across the
// others, times 3/216 = 1/72.  One z plane of the 3x3x3 block contributes its
// smoothed x and y differences and its smoothed sum (GradPlane).
template <typename R>
struct GradPlane {
  R ex, ey, sm;
};
template <typename R, bool WALLFREE, bool CENTRE>
__device__ __forceinline__ GradPlane<R> grad_plane(const R* sp, int c, int SX, R p0) {
  R p[3][3];
#pragma unroll
  for (int dy = -1; dy <= 1; ++dy) {
#pragma unroll
    for (int dx = -1; dx <= 1; ++dx) {
      R v = sp[c + dx + SX * dy];
      if constexpr (!WALLFREE) v = (v > R(0.5) * R(PHI_SOLID)) ? p0 : v;
      p[dy + 1][dx + 1] = v;
    }
  }
  GradPlane<R> o;
  o.ex = fma_rn(R(4), p[1][2] - p[1][0], (p[0][2] - p[0][0]) + (p[2][2] - p[2][0]));
  o.ey = fma_rn(R(4), p[2][1] - p[0][1], (p[2][0] - p[0][0]) + (p[2][2] - p[0][2]));
  // the plane smoothed over x and y enters the z difference
  o.sm = R(0);
  if constexpr (CENTRE)
    o.sm = fma_rn(R(4), fma_rn(R(4), p[1][1], p[1][0] + p[1][2]),
                  fma_rn(R(4), p[0][1], p[0][0] + p[0][2]) + fma_rn(R(4), p[2][1], p[2][0] + p[2][2]));
  return o;
}
template <typename R>
__device__ __forceinline__ void grad_from(const GradPlane<R>& lo, const GradPlane<R>& mid, const GradPlane<R>& hi,
                                          R gr[3]) {
  constexpr R k72 = R(1) / R(72);
  gr[0] = mul_rn(fma_rn(R(4), mid.ex, lo.ex) + hi.ex, k72);
  gr[1] = mul_rn(fma_rn(R(4), mid.ey, lo.ey) + hi.ey, k72);
  gr[2] = mul_rn(hi.sm - lo.sm, k72);
}
template <typename R, bool WALLFREE>
__device__ __forceinline__ void tile_grad(const R* sp, int c, int SX, int SXY, R gr[3]) {
  const R p0 = sp[c];
  const GradPlane<R> lo = grad_plane<R, WALLFREE, true>(sp, c - SXY, SX, p0);
  const GradPlane<R> mid = grad_plane<R, WALLFREE, false>(sp, c, SX, p0);
  const GradPlane<R> hi = grad_plane<R, WALLFREE, true>(sp, c + SXY, SX, p0);
  grad_from(lo, mid, hi, gr);
}

// round(v) to an int, half away from zero: v + 0.5 sign(v) towards zero, then
// truncated (the sum rounded towards zero keeps its integer part).  Not
// finite: 0.
__device__ __forceinline__ int iround(float v) { return __float2int_rz(__fadd_rz(v, copysignf(0.5f, v))); }
__device__ __forceinline__ int iround(double v) { return __double2int_rz(__dadd_rz(v, copysign(0.5, v))); }

// Near-contact scan of one interface node (Eqs. stress_jump, near_cont_force):
// step along the outward normal n_out = -grad phi/|grad phi| by round(k n_out),
// k = 1..K; the first target that is an interface node (|phi| < phi_I,
// |grad phi| >= NC_GRAD_MIN) with a normal antiparallel to the node's own
// gives h = k; 0 when there is none.  The scan stops at a wall layer.  sp is
// the phi tile with a halo of at least K + 1, c the node's tile index, gr and
// gg = |gr| its gradient.
template <typename R, bool WALLFREE>
__device__ __forceinline__ int nc_scan(const R* sp, int c, int SX, int SXY, int K, int x, int y, int z, const Geo& g,
                                       R phi_I, const R gr[3], R gg) {
  const R inv = R(-1) / gg;
  // components within [-1, 1] (the clamp also maps a normal that is not a
  // number into it), so a target lies at most k <= K nodes away on each axis
  const R no0 = fmax(R(-1), fmin(R(1), gr[0] * inv)), no1 = fmax(R(-1), fmin(R(1), gr[1] * inv)),
          no2 = fmax(R(-1), fmin(R(1), gr[2] * inv));
#pragma unroll 1
  for (int k = 1; k <= K; ++k) {
    const int dx = iround(R(k) * no0), dy = iround(R(k) * no1), dz = iround(R(k) * no2);
    if constexpr (!WALLFREE) {
      if (g.wx && (x + dx <= 0 || x + dx >= g.nx - 1)) break;
      if (g.wy && (y + dy <= 0 || y + dy >= g.ny - 1)) break;
      if (g.wz && (z + dz <= 0 || z + dz >= g.nz - 1)) break;
    }
    const int ct = c + dx + SX * dy + SXY * dz;
    if (!(fabs(sp[ct]) < phi_I)) continue;
    R gt[3];
    tile_grad<R, WALLFREE>(sp, ct, SX, SXY, gt);
    const R gm2 = gt[0] * gt[0] + gt[1] * gt[1] + gt[2] * gt[2];
    if (gm2 < R(NC_GRAD_MIN) * R(NC_GRAD_MIN)) continue;
    const R dot = gr[0] * gt[0] + gr[1] * gt[1] + gr[2] * gt[2];
    if (dot < -R(NC_COS_TOL) * gg * sqrt_(gm2)) return k;
  }
  return 0;
}

// ---------------------------------------------------------------------------
// the nodes of one tile
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ void put_field(const FieldOut& o, int k, size_t N, size_t self, R v) {
  if (o.slot[k] >= 0) reinterpret_cast<R*>(o.p)[(size_t)o.slot[k] * N + self] = v;
}

// Send the component populations (a, b) of direction i of the node at
// accumulator index e0 to the node that pulls them: x + c_i, or the node
// itself when x + c_i is solid (halfway bounce-back).
template <bool WALLFREE, int EX, int EXY>
__device__ __forceinline__ int send_to(int e0, unsigned wall, int i) {
  int e = e0 + cx(i) + EX * cy(i) + EXY * cz(i);
  if constexpr (!WALLFREE) {
    if (wall >> opp(i) & 1u) e = e0;
  }
  return e;
}
template <typename R, bool WALLFREE, int EX, int EXY, int E>
__device__ __forceinline__ void send(unsigned long long* sw, int e0, unsigned wall, int i, R a, R b) {
  Acc<R>::send_shared(sw, E, send_to<WALLFREE, EX, EXY>(e0, wall, i), a, b);
}

// Single-set storages: what colour_split gives the puller of the stored total
// fs (with the colour scalars sv), formed from fs already multiplied by the
// fixed-point scale.  A power of two passes through every rounding, so these
// are the bits of colour_split's values times the scale, and the two
// multiplications a direction fall away (bound by issue; FP16 storage at
// 128x128x256: 329 -> 322 us a step).
template <bool WALLFREE, typename L>
__device__ __forceinline__ void send_split(unsigned long long* sw, int e0, unsigned wall, int i, float fs, const float4& sv,
                                           float seg) {
  const float va = fma_rn(sv.x, fs, seg);
  Acc<float>::send_shared_scaled(sw, L::E, send_to<WALLFREE, L::EX, L::EXY>(e0, wall, i), va, fs - va);
}
// the scaled segregation term w_i c_i.v/|c_i| of colour_split
__device__ __forceinline__ float split_seg(const float4& sv, int i) {
  float cv = 0.f;
  if (cx(i)) cv += (float)cx(i) * sv.y;
  if (cy(i)) cv += (float)cy(i) * sv.z;
  if (cz(i)) cv += (float)cz(i) * sv.w;
  return mul_rn(wgt<float>(i) * inv_norm<float>(i) * Acc<float>::SCALE, cv);
}
template <int ST>
__device__ __forceinline__ float decode_scaled(typename Store<ST>::E v, int i) {
  if constexpr (ST == 2) return fma_rn(__half2float(v), F16_INV_SCALE * Acc<float>::SCALE, wgt<float>(i) * Acc<float>::SCALE);
  else return mul_rn((float)v, Acc<float>::SCALE);
}

// Pull, collide, recolour and store every node of the tile; with WS also
// send the post-collision component populations to the tile's partial sums.
// sp holds phi of the tile and its halo (Layout), accin the accumulator of the
// current level (null: the densities come from phi).  The near-contact scan of
// an interface node runs between the loads and the sums of its pull, while
// the loads are in flight (EARLY), or before the loads where the registers cannot
// hold a node's raw values through it: two-set batches, whose run parameters are
// loaded (12 runs of 48^3 to 96^3, near contact: 502 us a step early, 484 late).
template <int ST, int LOADER, bool WS, bool WF, int TX, int TY, int TZ, int H, bool WALLFREE, bool IDX32, bool REG, bool EARLY>
__device__ __forceinline__ void step_nodes(const View<ST>& S, const View<ST>& O, const InitBuf& init, const Geo& g,
                                           const PhysR<typename Store<ST>::R>& P,
                                           const FieldOut& fields,
                                           unsigned* __restrict__ status, const typename Store<ST>::R* sp,
                                           unsigned long long* sw, const unsigned long long* __restrict__ accin,
                                           int x0, int y0, int z0) {
  using R = typename Store<ST>::R;
  using L = Layout<R, TX, TY, TZ, H>;
  using E = typename Store<ST>::E;
  const R tau_a = R(P.tau_a), tau_b = R(P.tau_b);
  const R A2 = R(P.A2), beta = R(P.beta), A_h = R(P.A_h), phi_I = R(P.phi_I);
  const size_t N = (size_t)g.N, plane = (size_t)g.nx * (size_t)g.ny;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int x = x0 + tx, y = y0 + ty;
  if (x >= g.nx || y >= g.ny) return;
  using PI = PlaneIdx<ST, IDX32>;
  PI ix;
  ix.init(g, x, y);
  const unsigned wall_xy = WALLFREE ? 0u : column_bits(g, x, y);
  const auto self_o = ix.o[1][1];
  const size_t plane_e = Lay<ST>::plane(g);  // elements of a z plane
  int c = H * L::SXY + (ty + H) * L::SX + (tx + L::HX);
  int e0 = L::EXY + (ty + 1) * L::EX + (tx + 1);
  // gradient planes at z - 1 and z: a wall-free column takes one new plane a node
  GradPlane<R> glo, gmid;
  if constexpr (WALLFREE) {
    glo = grad_plane<R, true, true>(sp, c - L::SXY, L::SX, R(0));
    gmid = grad_plane<R, true, true>(sp, c, L::SX, R(0));
  }
#pragma unroll 1
  for (int lz = 0; lz < TZ; ++lz, c += L::SXY, e0 += L::EXY) {
    const int z = z0 + lz;
    if (z >= g.nz) break;
    const size_t self = (size_t)z * plane + (size_t)g.nx * (size_t)y + (size_t)x;
    if (!WALLFREE && is_solid(g, x, y, z)) {
      if constexpr (WF) {
        for (int k = 0; k < NFIELDS; ++k) put_field<R>(fields, k, N, self, R(0));
      }
      continue;
    }
    Nbr n;
    const unsigned wall = WALLFREE ? 0u : wall_xy | node_bits(g, z);
    if constexpr (LOADER != LOAD_PULL || (Store<ST>::MOMENT && !WALLFREE)) make_nbr(g, x, y, z, n);
    R f[Q], rA, rB;
    E ra[Q], rb[Q];
    auto pull = [&]() {
      const int zs[3] = {z > 0 ? z - 1 : g.nz - 1, z, z + 1 < g.nz ? z + 1 : 0};
      if constexpr (Store<ST>::MOMENT && !WALLFREE) pull_walled_moment<ST>(S, g, n, wall, (int)self, f);
      else if constexpr (Store<ST>::MOMENT) pull_plane_moment<ST, IDX32>(S, N, plane, ix, zs, f);
      else pull_plane<ST, IDX32, WALLFREE>(S, g, ix, zs, wall, ra, rb);
    };
    if constexpr (LOADER == LOAD_PULL && EARLY) pull();
    const R phx = sp[c];
    // colour gradient from the tile; near-contact distance from the scan
    R gr[3];
    if constexpr (WALLFREE) {
      const GradPlane<R> ghi = grad_plane<R, true, true>(sp, c + L::SXY, L::SX, R(0));
      grad_from(glo, gmid, ghi, gr);
      glo = gmid;
      gmid = ghi;
    } else {
      tile_grad<R, false>(sp, c, L::SX, L::SXY, gr);
    }
    const R gg = sqrt_(gr[0] * gr[0] + gr[1] * gr[1] + gr[2] * gr[2]);
    int h = 0;
    if (H > 1 && A_h != R(0) && fabs(phx) < phi_I && gg >= R(NC_GRAD_MIN))
      h = nc_scan<R, WALLFREE>(sp, c, L::SX, L::SXY, P.K, x, y, z, g, phi_I, gr, gg);
    if constexpr (LOADER == LOAD_PULL) {
      if constexpr (!EARLY) pull();
      if constexpr (!Store<ST>::MOMENT) pull_finish<ST>(ra, rb, f, rA, rB);
      if constexpr (!Store<ST>::TWOSET) {
        // single set: rhoA of the node is the sum the senders accumulated
        // (what a pull of the rebuilt f^A_i gives), so the neighbours' colour
        // scalars need not be read
        R rt = R(0);
#pragma unroll
        for (int i = 0; i < Q; ++i) rt += f[i];
        if (accin) {
          Acc<R>::densities(accin, self, rA, rB);
        } else {  // phi given as an array: split the pulled total by it
          rA = R(0.5) * rt * (R(1) + phx);
        }
        rB = rt - rA;  // rho is the sum of the pulled totals, as for the momentum
      }
    } else {
      fields_node<R, false>(init, g, P, n, (long long)self, f, rA, rB, nullptr, nullptr);
    }

    // moments (Sec. III.C.1): rho = rhoA + rhoB, j = sum_i f_i c_i taken over
    // opposite pairs (p, 26-p), p = 0..12
    const R rho = rA + rB;
    R j0 = R(0), j1 = R(0), j2 = R(0);
#pragma unroll
    for (int p = 0; p < REST; ++p) {
      const R d = f[p] - f[opp(p)];
      if (cx(p)) j0 += R(cx(p)) * d;
      if (cy(p)) j1 += R(cy(p)) * d;
      if (cz(p)) j2 += R(cz(p)) * d;
    }
    R Ahh = R(0);
    if (H > 1 && A_h != R(0)) {
      if (h > 0) {
        const R hk = R(h);
        if (hk <= R(P.h_min)) Ahh = A_h;
        else if (hk <= R(P.h_max)) {
          const R q = R(P.h_min) / hk;
          Ahh = A_h * q * q * q;
        }
      }
    }
    // F_rep = -A_h n_out delta_I, delta_I = |grad phi|/2  ->  (A_h/2) grad phi
    const R Fr0 = R(0.5) * Ahh * gr[0], Fr1 = R(0.5) * Ahh * gr[1], Fr2 = R(0.5) * Ahh * gr[2];
    R F0 = Fr0, F1 = Fr1, F2 = Fr2;
    if (P.g_mode == 1) {
      F0 += rho * R(P.g[0]);
      F1 += rho * R(P.g[1]);
      F2 += rho * R(P.g[2]);
    } else if (P.g_mode == 2) {
      const R sg = (z == 0 || 2 * z == g.nz) ? R(0) : (2 * z < g.nz ? R(1) : R(-1));
      F0 += sg * rA * R(P.g[0]);
      F1 += sg * rA * R(P.g[1]);
      F2 += sg * rA * R(P.g[2]);
    }

    // Guo-shifted velocity
    const R irho = R(1) / rho;
    const R u0 = (j0 + R(0.5) * F0) * irho, u1 = (j1 + R(0.5) * F1) * irho, u2 = (j2 + R(0.5) * F2) * irho;
    // a density outside (0, RHO_MAX), or not finite, marks the run unstable
    if (!(rho > R(0) && rho < R(Acc<R>::RHO_MAX))) atomicOr(status, 1u);

    if constexpr (WF) {
      put_field<R>(fields, F_PHI, N, self, phx);
      put_field<R>(fields, F_RHO, N, self, rho);
      put_field<R>(fields, F_UX, N, self, u0);
      put_field<R>(fields, F_UY, N, self, u1);
      put_field<R>(fields, F_UZ, N, self, u2);
      put_field<R>(fields, F_RHOA, N, self, rA);
      put_field<R>(fields, F_RHOB, N, self, rB);
      put_field<R>(fields, F_FRX, N, self, Fr0);
      put_field<R>(fields, F_FRY, N, self, Fr1);
      put_field<R>(fields, F_FRZ, N, self, Fr2);
      put_field<R>(fields, F_H, N, self, R(h));
      put_field<R>(fields, F_GX, N, self, gr[0]);
      put_field<R>(fields, F_GY, N, self, gr[1]);
      put_field<R>(fields, F_GZ, N, self, gr[2]);
    }
    if constexpr (!WS) continue;

    // mixture relaxation time (harmonic nu_bar, Eq. sigmaA)
    R tau;
    if (P.equal_tau) {
      tau = tau_a;
    } else {
      const R nu_a = (tau_a - R(0.5)) / R(3), nu_b = (tau_b - R(0.5)) / R(3);
      const R nu = R(1) / ((rA * irho) / nu_a + (rB * irho) / nu_b);
      tau = R(3) * nu + R(0.5);
    }
    const R omega = R(1) / tau;
    const R keep = R(1) - omega;
    const R guo = R(1) - R(0.5) * omega;
    const R uu = u0 * u0 + u1 * u1 + u2 * u2;
    const R uF = u0 * F0 + u1 * F1 + u2 * F2;
    // perturbation: (A_a+A_b)/2 |g| [w (c.n)^2 - B] = A2 [w (c.grad)^2/|g| - |g| B]
    const bool pert = gg >= R(GRAD_EPS);
    const R A2g = pert ? A2 * gg : R(0);
    const R A2ig = pert ? A2 / gg : R(0);
    // recolouring segregation amplitude beta rhoA rhoB / rho with the normal
    // grad phi / max(|grad phi|, floor)
    const R gn = gg > R(NORMAL_FLOOR) ? gg : R(NORMAL_FLOOR);
    const R segamp = beta * rA * rB * irho / gn;
    const R sA = rA * irho;
    // equilibrium (Eq. disteq) and Guo source split into parts even and odd
    // under c -> -c: feq = w [rho(1 - 1.5 uu) + 4.5 rho (c.u)^2] + 3 w rho (c.u),
    // S = guo w [9 (c.u)(c.F) - 3 u.F] + 3 guo w (c.F)
    const R r0 = rho * (R(1) - R(1.5) * uu);
    const R r45 = R(4.5) * rho;
    const R r3 = R(3) * rho;
    const R g9 = R(9) * guo, g3 = R(3) * guo, gm3uF = -R(3) * guo * uF;
    // BGK relaxes f towards feq: keep f + omega feq.  The regularised
    // collision (collision == 1) keeps feq and relaxes the non-equilibrium
    // part projected on Hermite orders 1 and 2:
    //   feq + keep w [3 c.J + 4.5 (c.Pi.c - tr(Pi)/3)],
    //   J = j - rho u = -F/2,  Pi = sum_i c c f_i - rho (u u + I/3).
    constexpr bool reg = REG;
    const R wf = reg ? R(1) : omega;
    R Pxx = R(0), Pyy = R(0), Pzz = R(0), Pxy = R(0), Pxz = R(0), Pyz = R(0), trP = R(0);
    if constexpr (reg) {
#pragma unroll
      for (int p = 0; p < REST; ++p) {
        const R sp2 = f[p] + f[opp(p)];
        if (cx(p)) Pxx += sp2;
        if (cy(p)) Pyy += sp2;
        if (cz(p)) Pzz += sp2;
        if (cx(p) && cy(p)) Pxy += R(cx(p) * cy(p)) * sp2;
        if (cx(p) && cz(p)) Pxz += R(cx(p) * cz(p)) * sp2;
        if (cy(p) && cz(p)) Pyz += R(cy(p) * cz(p)) * sp2;
      }
      const R r3rd = rho * (R(1) / R(3));
      Pxx -= rho * u0 * u0 + r3rd;
      Pyy -= rho * u1 * u1 + r3rd;
      Pzz -= rho * u2 * u2 + r3rd;
      Pxy -= rho * u0 * u1;
      Pxz -= rho * u0 * u2;
      Pyz -= rho * u1 * u2;
      trP = Pxx + Pyy + Pzz;
    }
    // colour scalars of the single-set storages, as stored
    float4 svo = make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (!Store<ST>::TWOSET) {
      svo = make_float4(sA, segamp * gr[0], segamp * gr[1], segamp * gr[2]);
      O.sv[self] = svo;
    }
    if constexpr (Store<ST>::MOMENT) {
      // f*_i = w_i (alpha + beta.c_i + c_i.Gamma.c_i): the equilibrium, the
      // relaxed Hermite orders 1-2, the perturbation (B_i = w_i (|c_i|^2 - 2/3))
      // and the Guo source below are each w_i times a quadratic form in c_i
      // (Eqs. disteq, distnoneq, LBpostmom; the host admits this storage with
      // the regularised collision only)
      const R kP = keep * R(4.5), hg9 = R(0.5) * g9;
      const R bF = g3 - R(1.5) * keep;  // beta = 3 rho u + (3 guo - 1.5 keep) F
      const float4 qa = make_float4(r0 + gm3uF - R(1.5) * keep * trP + (R(2) / R(3)) * A2g, r3 * u0 + bF * F0,
                                    r3 * u1 + bF * F1, r3 * u2 + bF * F2);
      const float4 qb = make_float4(r45 * u0 * u0 + g9 * u0 * F0 + A2ig * gr[0] * gr[0] - A2g + kP * Pxx,
                                    r45 * u1 * u1 + g9 * u1 * F1 + A2ig * gr[1] * gr[1] - A2g + kP * Pyy,
                                    r45 * u2 * u2 + g9 * u2 * F2 + A2ig * gr[2] * gr[2] - A2g + kP * Pzz,
                                    R(2) * (r45 * u0 * u1 + hg9 * (u0 * F1 + F0 * u1) + A2ig * gr[0] * gr[1] + kP * Pxy));
      const float2 qc =
          make_float2(R(2) * (r45 * u0 * u2 + hg9 * (u0 * F2 + F0 * u2) + A2ig * gr[0] * gr[2] + kP * Pxz),
                      R(2) * (r45 * u1 * u2 + hg9 * (u1 * F2 + F1 * u2) + A2ig * gr[1] * gr[2] + kP * Pyz));
      reinterpret_cast<float4*>(O.f)[self] = qa;
      reinterpret_cast<float4*>(O.f + 4 * N)[self] = qb;
      reinterpret_cast<float2*>(O.f + 8 * N)[self] = qc;
      // what the neighbours will pull: the quadratic form at each c_i
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const float fs = mul_rn(eval_moment<R>(qa, qb, qc, i, false), Acc<float>::SCALE);
        send_split<WALLFREE, L>(sw, e0, wall, i, fs, svo, i == REST ? 0.f : split_seg(svo, i));
      }
      continue;
    }
    E* op = O.f + ((size_t)z * plane_e + self_o);
    {  // rest direction
      const R W = wgt<R>(REST);
      const R rel = reg ? R(-1.5) * W * trP : f[REST];
      const R fs = keep * rel + wf * W * r0 - bweight<R>(REST) * A2g + W * gm3uF;
      if constexpr (Store<ST>::TWOSET) {
        const R fa = sA * fs;
        const R fb = fs - fa;
        op[REST * BLK] = encode<ST>(fa, REST);
        op[(Q + REST) * BLK] = encode<ST>(fb, REST);
        send<R, WALLFREE, L::EX, L::EXY, L::E>(sw, e0, wall, REST, fa, fb);
      } else {
        const typename Store<ST>::E enc = encode<ST>(fs, REST);
        op[REST * BLK] = enc;
        send_split<WALLFREE, L>(sw, e0, wall, REST, decode_scaled<ST>(enc, REST), svo, 0.f);
      }
    }
#pragma unroll
    for (int p = 0; p < REST; ++p) {
      const int q = opp(p);
      const R W = wgt<R>(p);
      R cu = R(0), cF = R(0), cg = R(0);
      if (cx(p)) { cu += R(cx(p)) * u0; cF += R(cx(p)) * F0; cg += R(cx(p)) * gr[0]; }
      if (cy(p)) { cu += R(cy(p)) * u1; cF += R(cy(p)) * F1; cg += R(cy(p)) * gr[1]; }
      if (cz(p)) { cu += R(cz(p)) * u2; cF += R(cz(p)) * F2; cg += R(cz(p)) * gr[2]; }
      R even = W * (wf * (r0 + r45 * cu * cu) + g9 * cu * cF + gm3uF + A2ig * cg * cg) - bweight<R>(p) * A2g;
      R odd = W * (wf * r3 * cu + g3 * cF);
      const R bp = f[p], bq = f[q];
      if constexpr (reg) {
        // c.Pi.c and c.J = -(c.F)/2 for this pair's velocity
        R cpc = R(0);
        if (cx(p)) cpc += Pxx;
        if (cy(p)) cpc += Pyy;
        if (cz(p)) cpc += Pzz;
        if (cx(p) && cy(p)) cpc += R(2 * cx(p) * cy(p)) * Pxy;
        if (cx(p) && cz(p)) cpc += R(2 * cx(p) * cz(p)) * Pxz;
        if (cy(p) && cz(p)) cpc += R(2 * cy(p) * cz(p)) * Pyz;
        even += keep * W * R(4.5) * (cpc - trP * (R(1) / R(3)));
        odd += keep * W * R(-1.5) * cF;
      }
      const R fsp = reg ? even + odd : keep * bp + even + odd;
      const R fsq = reg ? even - odd : keep * bq + even - odd;
      if constexpr (Store<ST>::TWOSET) {
        const R seg = segamp * W * inv_norm<R>(p) * cg;
        const R fap = sA * fsp + seg;
        const R faq = sA * fsq - seg;
        const R fbp = fsp - fap, fbq = fsq - faq;
        op[p * BLK] = encode<ST>(fap, p);
        op[q * BLK] = encode<ST>(faq, q);
        op[(Q + p) * BLK] = encode<ST>(fbp, p);
        op[(Q + q) * BLK] = encode<ST>(fbq, q);
        send<R, WALLFREE, L::EX, L::EXY, L::E>(sw, e0, wall, p, fap, fbp);
        send<R, WALLFREE, L::EX, L::EXY, L::E>(sw, e0, wall, q, faq, fbq);
      } else {
        const typename Store<ST>::E ep = encode<ST>(fsp, p), eq = encode<ST>(fsq, q);
        op[p * BLK] = ep;
        op[q * BLK] = eq;
        // p and its opposite q: c_q.v = -(c_p.v) exactly, so the segregation term
        // is formed once and negated (bit for bit what colour_split gives for q)
        const float seg = split_seg(svo, p);
        send_split<WALLFREE, L>(sw, e0, wall, p, decode_scaled<ST>(ep, p), svo, seg);
        send_split<WALLFREE, L>(sw, e0, wall, q, decode_scaled<ST>(eq, q), svo, -seg);
      }
    }
  }
}

// Add the tile's partial sums (tile plus a one-node ring) to the global
// accumulator; entries beyond a wall are never sent to, periodic axes wrap.
// A warp takes whole rows of the ring (its y and z are then the warp's), the
// two columns past the 32 lanes come last.
template <typename R, int TX, int TY, int TZ, typename L>
__device__ __forceinline__ void flush_partials(const unsigned long long* sw, unsigned long long* __restrict__ acc,
                                               const Geo& g, int x0, int y0, int z0) {
  static_assert(TX == 32, "one lane per column");
  constexpr int ROWS = L::EY * L::EZ;
  // node of ring column ex, or -1 beyond a wall (pad_source also drops the
  // solid layers, whose sums are zero)
  auto row_base = [&](int row) -> long long {
    const int ez = row / L::EY, ey = row - ez * L::EY;
    const int gy = pad_source(y0 + ey, 1, g.ny, g.wy), gz = pad_source(z0 + ez, 1, g.nz, g.wz);
    return gy < 0 || gz < 0 ? -1 : (long long)g.nx * ((long long)gy + (long long)g.ny * gz);
  };
  const int gx = pad_source(x0 + (int)threadIdx.x, 1, g.nx, g.wx);
  for (int row = threadIdx.y; row < ROWS; row += TY) {
    const int e = row * L::EX + (int)threadIdx.x;
    const long long rb = row_base(row);
    if (rb >= 0 && gx >= 0 && !Acc<R>::shared_zero(sw, L::E, e)) Acc<R>::flush_shared(acc, (size_t)(rb + gx), sw, L::E, e);
  }
  for (int k = threadIdx.y * TX + threadIdx.x; k < 2 * ROWS; k += TX * TY) {
    const int row = k >> 1, ex = TX + (k & 1), e = row * L::EX + ex;
    if (Acc<R>::shared_zero(sw, L::E, e)) continue;
    const long long rb = row_base(row);
    const int gt = pad_source(x0 + ex, 1, g.nx, g.wx);
    if (rb >= 0 && gt >= 0) Acc<R>::flush_shared(acc, (size_t)(rb + gt), sw, L::E, e);
  }
}

// ---------------------------------------------------------------------------
// Shan-Chen multicomponent model (Sec. III.C.3, lattice pseudo-potential)
// ---------------------------------------------------------------------------
// The nodes of one tile in the Shan-Chen model: pull both components, the
// pseudo-potential forces F_A = -psi_A G sum_i w_i psi_B(x + c_i) c_i (= -psi_A
// (G/3) times the stencil gradient of psi_B; a solid neighbour contributes the
// node's own psi) and F_B alike, the body force, the common velocity
// u' = sum_k (j_k + F_k/2)/tau_k / sum_k rho_k/tau_k, then per component BGK
// towards f^eq(rho_k, u') with the Guo source of F_k, store and send.
template <int ST, int LOADER, bool WS, bool WF, int TX, int TY, int TZ, bool WALLFREE, bool IDX32>
__device__ __forceinline__ void step_nodes_sc(const View<ST>& S, const View<ST>& O, const InitBuf& init,
                                              const Geo& g, const PhysR<typename Store<ST>::R>& P,
                                              const FieldOut& fields,
                                              unsigned* __restrict__ status, const typename Store<ST>::R* sp,
                                              const typename Store<ST>::R* spa, const typename Store<ST>::R* spb,
                                              unsigned long long* sw, int x0, int y0, int z0) {
  using R = typename Store<ST>::R;
  using L = Layout<R, TX, TY, TZ, 1, WF ? 3 : 2>;
  const size_t N = (size_t)g.N, plane = (size_t)g.nx * (size_t)g.ny;
  const R wa = R(1) / R(P.tau_a), wb = R(1) / R(P.tau_b);
  const R G3 = R(P.G) / R(3);
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int x = x0 + tx, y = y0 + ty;
  if (x >= g.nx || y >= g.ny) return;
  using PI = PlaneIdx<ST, IDX32>;
  PI ix;
  ix.init(g, x, y);
  const unsigned wall_xy = WALLFREE ? 0u : column_bits(g, x, y);
  const auto self_o = ix.o[1][1];
  const size_t plane_e = Lay<ST>::plane(g);  // elements of a z plane
  int c = L::SXY + (ty + 1) * L::SX + (tx + L::HX);
  int e0 = L::EXY + (ty + 1) * L::EX + (tx + 1);
  GradPlane<R> alo, amid, blo, bmid;
  if constexpr (WALLFREE) {
    alo = grad_plane<R, true, true>(spa, c - L::SXY, L::SX, R(0));
    amid = grad_plane<R, true, true>(spa, c, L::SX, R(0));
    blo = grad_plane<R, true, true>(spb, c - L::SXY, L::SX, R(0));
    bmid = grad_plane<R, true, true>(spb, c, L::SX, R(0));
  }
#pragma unroll 1
  for (int lz = 0; lz < TZ; ++lz, c += L::SXY, e0 += L::EXY) {
    const int z = z0 + lz;
    if (z >= g.nz) break;
    const size_t self = (size_t)z * plane + (size_t)g.nx * (size_t)y + (size_t)x;
    if (!WALLFREE && is_solid(g, x, y, z)) {
      if constexpr (WF) {
        for (int k = 0; k < NFIELDS; ++k) put_field<R>(fields, k, N, self, R(0));
      }
      continue;
    }
    Nbr n;
    const unsigned wall = WALLFREE ? 0u : wall_xy | node_bits(g, z);
    if constexpr (LOADER != LOAD_PULL) make_nbr(g, x, y, z, n);
    R fa[Q], fb[Q], rA = R(0), rB = R(0);
    if constexpr (LOADER == LOAD_PULL) {  // two-set storages: the stored values are the populations
      const int zs[3] = {z > 0 ? z - 1 : g.nz - 1, z, z + 1 < g.nz ? z + 1 : 0};
      pull_plane<ST, IDX32, WALLFREE>(S, g, ix, zs, wall, fa, fb);
    }
    R gA[3], gB[3], gphi[3];
    if constexpr (WALLFREE) {
      const GradPlane<R> ahi = grad_plane<R, true, true>(spa, c + L::SXY, L::SX, R(0));
      grad_from(alo, amid, ahi, gA);
      alo = amid;
      amid = ahi;
      const GradPlane<R> bhi = grad_plane<R, true, true>(spb, c + L::SXY, L::SX, R(0));
      grad_from(blo, bmid, bhi, gB);
      blo = bmid;
      bmid = bhi;
    } else {
      tile_grad<R, false>(spa, c, L::SX, L::SXY, gA);
      tile_grad<R, false>(spb, c, L::SX, L::SXY, gB);
    }
    if constexpr (LOADER == LOAD_PULL) {
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        rA += fa[i];
        rB += fb[i];
      }
    } else {
      R f[Q];
      fields_node<R, true>(init, g, P, n, (long long)self, f, rA, rB, fa, fb);
    }
    R jA[3] = {R(0), R(0), R(0)}, jB[3] = {R(0), R(0), R(0)};
#pragma unroll
    for (int i = 0; i < REST; ++i) {  // opposite pairs
      const R da = fa[i] - fa[opp(i)], db = fb[i] - fb[opp(i)];
      if (cx(i)) { jA[0] += R(cx(i)) * da; jB[0] += R(cx(i)) * db; }
      if (cy(i)) { jA[1] += R(cy(i)) * da; jB[1] += R(cy(i)) * db; }
      if (cz(i)) { jA[2] += R(cz(i)) * da; jB[2] += R(cz(i)) * db; }
    }
    R FA[3], FB[3], Fs[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      FA[a] = -spa[c] * G3 * gB[a];
      FB[a] = -spb[c] * G3 * gA[a];
      Fs[a] = FA[a] + FB[a];
    }
    if (P.g_mode == 1) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        FA[a] += rA * R(P.g[a]);
        FB[a] += rB * R(P.g[a]);
      }
    } else if (P.g_mode == 2) {
      const R sg = (z == 0 || 2 * z == g.nz) ? R(0) : (2 * z < g.nz ? R(1) : R(-1));
#pragma unroll
      for (int a = 0; a < 3; ++a) FA[a] += sg * rA * R(P.g[a]);
    }
    const R rho = rA + rB;
    if (!(rho > R(0) && rho < R(Acc<R>::RHO_MAX))) atomicOr(status, 1u);
    const R iw = R(1) / (wa * rA + wb * rB);
    R u[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) u[a] = (wa * (jA[a] + R(0.5) * FA[a]) + wb * (jB[a] + R(0.5) * FB[a])) * iw;
    if constexpr (WF) {
      tile_grad<R, WALLFREE>(sp, c, L::SX, L::SXY, gphi);
      const R irho = R(1) / rho;
      put_field<R>(fields, F_PHI, N, self, sp[c]);
      put_field<R>(fields, F_RHO, N, self, rho);
      put_field<R>(fields, F_UX, N, self, (jA[0] + jB[0] + R(0.5) * (FA[0] + FB[0])) * irho);
      put_field<R>(fields, F_UY, N, self, (jA[1] + jB[1] + R(0.5) * (FA[1] + FB[1])) * irho);
      put_field<R>(fields, F_UZ, N, self, (jA[2] + jB[2] + R(0.5) * (FA[2] + FB[2])) * irho);
      put_field<R>(fields, F_RHOA, N, self, rA);
      put_field<R>(fields, F_RHOB, N, self, rB);
      put_field<R>(fields, F_FRX, N, self, Fs[0]);
      put_field<R>(fields, F_FRY, N, self, Fs[1]);
      put_field<R>(fields, F_FRZ, N, self, Fs[2]);
      put_field<R>(fields, F_H, N, self, R(0));
      put_field<R>(fields, F_GX, N, self, gphi[0]);
      put_field<R>(fields, F_GY, N, self, gphi[1]);
      put_field<R>(fields, F_GZ, N, self, gphi[2]);
    }
    if constexpr (!WS) continue;
    const R uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    // per component: f*_i = (1 - 1/tau_k) f_i + w_i (alpha + beta.c + c.Gamma.c)
    // with feq(rho_k, u') / tau_k and the Guo source (1 - 1/(2 tau_k)) w_i
    // [3 (c_i - u') + 9 (c_i.u') c_i].F_k
    auto form = [&](R w, R r, const R F[3]) {
      const R gk = R(1) - R(0.5) * w, wr = w * r, hg9 = R(4.5) * gk, r45 = R(4.5) * wr, r3 = R(3) * wr;
      const R uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2];
      const R v0 = fma_rn(r45, u[0], mul_rn(hg9, F[0])), v1 = fma_rn(r45, u[1], mul_rn(hg9, F[1])),
              v2 = fma_rn(r45, u[2], mul_rn(hg9, F[2]));
      const R k0 = mul_rn(hg9, u[0]), k1 = mul_rn(hg9, u[1]), k2 = mul_rn(hg9, u[2]);
      QForm<R> q;
      q.a = fma_rn(R(-3) * gk, uF, wr * (R(1) - R(1.5) * uu));
      q.bx = fma_rn(r3, u[0], R(3) * gk * F[0]);
      q.by = fma_rn(r3, u[1], R(3) * gk * F[1]);
      q.bz = fma_rn(r3, u[2], R(3) * gk * F[2]);
      q.xx = fma_rn(v0, u[0], mul_rn(k0, F[0]));
      q.yy = fma_rn(v1, u[1], mul_rn(k1, F[1]));
      q.zz = fma_rn(v2, u[2], mul_rn(k2, F[2]));
      q.xy = R(2) * fma_rn(v0, u[1], mul_rn(k0, F[1]));
      q.xz = R(2) * fma_rn(v0, u[2], mul_rn(k0, F[2]));
      q.yz = R(2) * fma_rn(v1, u[2], mul_rn(k1, F[2]));
      return q;
    };
    const QForm<R> qa = form(wa, rA, FA), qb = form(wb, rB, FB);
    const R ka = R(1) - wa, kb = R(1) - wb;
    auto* op = O.f + ((size_t)z * plane_e + self_o);
    auto put = [&](int i, R oa, R ob) {
      op[i * BLK] = encode<ST>(oa, i);
      op[(Q + i) * BLK] = encode<ST>(ob, i);
      send<R, WALLFREE, L::EX, L::EXY, L::E>(sw, e0, wall, i, oa, ob);
    };
    put(REST, fma_rn(ka, fa[REST], mul_rn(wgt<R>(REST), qa.a)), fma_rn(kb, fb[REST], mul_rn(wgt<R>(REST), qb.a)));
    auto pairs = [&](auto cls) {
      constexpr int CLS = decltype(cls)::value;
      const QClass<R, CLS> ca(qa), cb(qb);
#pragma unroll
      for (int p = 0; p < REST; ++p) {
        if (cnorm2(p) != CLS) continue;
        const int q = opp(p);
        const R ea = ca.even(p), oa = ca.odd(p), eb = cb.even(p), ob = cb.odd(p);
        put(p, fma_rn(ka, fa[p], ea + oa), fma_rn(kb, fb[p], eb + ob));
        put(q, fma_rn(ka, fa[q], ea - oa), fma_rn(kb, fb[q], eb - ob));
      }
    };
    pairs(std::integral_constant<int, 1>{});
    pairs(std::integral_constant<int, 2>{});
    pairs(std::integral_constant<int, 3>{});
  }
}

// A tile of either model: clear the partial sums while the staged fields are
// copied in, step the nodes, flush.  Ends with a barrier when AGAIN (the caller
// reuses the shared memory).
template <int ST, int LOADER, bool WS, bool WF, int TX, int TY, int TZ, int H, bool IDX32, bool SC, bool EARLY, bool AGAIN>
__device__ __forceinline__ void step_tile(const View<ST>& S, const View<ST>& O, const InitBuf& init,
                                          const unsigned long long* __restrict__ accin, unsigned long long* __restrict__ accout,
                                          const typename Store<ST>::R* __restrict__ phi, const PadGeo& pg, const Geo& g,
                                          const PhysR<typename Store<ST>::R>& P,
                                          const FieldOut& fields, unsigned* __restrict__ status,
                                          unsigned char* smem, int x0, int y0, int z0) {
  using R = typename Store<ST>::R;
  constexpr int NPH = SC ? (WF ? 3 : 2) : 1;
  using L = Layout<R, TX, TY, TZ, H, NPH>;
  R* sp = reinterpret_cast<R*>(smem);
  unsigned long long* sw = reinterpret_cast<unsigned long long*>(smem + L::off_acc);
  const int tid = threadIdx.y * TX + threadIdx.x;
  if constexpr (WS && !AGAIN) {
    for (int e = tid; e < Acc<R>::W * L::E; e += TX * TY) sw[e] = 0ull;
    wait_primary();
  }
  // a step of the Shan-Chen model needs psi_A, psi_B only (fields 1 and 2)
  stage_tile<R, TX, TY, TZ, H, NPH>(SC && !WF ? phi + (size_t)pg.px * pg.py * pg.pz : phi, pg, sp, x0, y0, z0);
  if constexpr (WS && AGAIN) {
    for (int e = tid; e < Acc<R>::W * L::E; e += TX * TY) sw[e] = 0ull;
  }
  cp_async_wait_all();
  __syncthreads();
  // A warp (a row of the tile) whose one-node halo (with near contact: the scan's
  // halo of K + 1 nodes) holds no solid node needs no bounce-back or wall tests.
  // Decided per warp: at a wall in y one row of eight takes the walled path.
  const bool wallfree =
      !region_walled(g, x0, uniform(y0 + (int)threadIdx.y), z0, TX, 1, TZ, (H > 1 && P.A_h != R(0)) ? P.K + 1 : 1);
  if constexpr (SC) {
    R* spa = sp + (NPH - 2) * L::NS;
    R* spb = spa + L::NS;
    if (wallfree)
      step_nodes_sc<ST, LOADER, WS, WF, TX, TY, TZ, true, IDX32>(S, O, init, g, P, fields, status, sp, spa, spb, sw, x0,
                                                                 y0, z0);
    else
      step_nodes_sc<ST, LOADER, WS, WF, TX, TY, TZ, false, IDX32>(S, O, init, g, P, fields, status, sp, spa, spb, sw,
                                                                  x0, y0, z0);
  } else {
    auto nodes = [&](auto wf, auto reg) {
      step_nodes<ST, LOADER, WS, WF, TX, TY, TZ, H, decltype(wf)::value, IDX32, decltype(reg)::value, EARLY>(
          S, O, init, g, P, fields, status, sp, sw, accin, x0, y0, z0);
    };
    // (the moment storage holds the regularised collision only; a BGK copy of its
    // loop, which nothing reached, cost it 3 to 5 % in registers)
    if (Store<ST>::MOMENT || P.collision == 1) {  // regularised collision
      if (wallfree) nodes(std::true_type{}, std::true_type{});
      else nodes(std::false_type{}, std::true_type{});
    } else {
      if (wallfree) nodes(std::true_type{}, std::false_type{});
      else nodes(std::false_type{}, std::false_type{});
    }
  }
  if constexpr (WS) {
    __syncthreads();
    flush_partials<R, TX, TY, TZ, L>(sw, accout, g, x0, y0, z0);
  }
  if constexpr (AGAIN) __syncthreads();
}

template <int ST, int LOADER, bool WS, bool WF, int TX, int TY, int TZ, int H, bool IDX32, int MINB, bool SC>
__global__ void __launch_bounds__(TX* TY, (ST == 3) ? 1 : MINB)
    k_step(View<ST> S, View<ST> O, InitBuf init, const unsigned long long* accin, unsigned long long* accout,
           const typename Store<ST>::R* phi, PadGeo pg, Geo g, PhysR<typename Store<ST>::R> P,
           FieldOut fields, unsigned* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  launch_dependents();
  if constexpr (!WS) wait_primary();
  constexpr bool EARLY = ST == 3 || TX * TY * MINB <= 512;  // 128 registers a thread or more
  step_tile<ST, LOADER, WS, WF, TX, TY, TZ, H, IDX32, SC, EARLY, false>(S, O, init, accin, accout, phi, pg, g, P, fields, status,
                                                                 smem_raw, blockIdx.x * TX, blockIdx.y * TY,
                                                                 blockIdx.z * TZ);
}

// ---------------------------------------------------------------------------
// batched persistent kernels: many independent runs of uneven sizes and
// parameters, one k_phi_batched and one k_step_batched launch per step.  Work
// items are (run, row group) and (run, tile); persistent CTAs stride over the
// item list and look the run of an item up in a table (run_of; a binary search
// over the runs' prefix offsets put six dependent loads before every tile).  Every run's accumulators are at the same phase k of their
// rotation.
// ---------------------------------------------------------------------------
__device__ __forceinline__ Geo uniform(const Geo& d) {
  Geo g;
  g.nx = uniform(d.nx);
  g.ny = uniform(d.ny);
  g.nz = uniform(d.nz);
  const int w = uniform(d.wx | d.wy << 1 | d.wz << 2);
  g.wx = w & 1;
  g.wy = w >> 1 & 1;
  g.wz = w >> 2 & 1;
  g.N = (long long)g.nx * g.ny * g.nz;
  return g;
}

template <typename R>
__global__ void __launch_bounds__(256) k_phi_batched(const RunDesc* __restrict__ runs, const int* __restrict__ run_of,
                                                     long long ngroups, int k) {
  launch_dependents();
  wait_primary();
  for (long long t = blockIdx.x; t < ngroups; t += gridDim.x) {
    const RunDesc& d = runs[run_of[t]];
    const PhiSrc src{nullptr, d.acc[k]};
    const InitBuf none{nullptr, nullptr, nullptr, 0};
    // eight rows of the run, one a warp
    const long long row = (t - d.row_begin) * 8 + threadIdx.y;
    if (row < (long long)d.g.ny * d.g.nz)
      phi_row<R, false>(src, none, d.g, d.pg, R(0), d.phi, d.acc[(k + 2) % 3], (int)(row % d.g.ny), (int)(row / d.g.ny));
  }
}

template <int ST, int TX, int TY, int TZ, int H, bool IDX32, int MINB>
__global__ void __launch_bounds__(TX* TY, MINB)
    k_step_batched(const RunDesc* __restrict__ runs, const int* __restrict__ run_of, long long ntiles, int parity, int k,
                   unsigned* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  InitBuf none{nullptr, nullptr, nullptr, 0};
  launch_dependents();
  wait_primary();
  int next = run_of[blockIdx.x < ntiles ? blockIdx.x : 0];
  for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const RunDesc& d = runs[next];
    if (t + gridDim.x < ntiles) next = run_of[t + gridDim.x];  // its load runs through the tile
    const int lt = uniform((int)(t - d.tile_begin));
    const Geo g = uniform(d.g);
    const int tiles_x = (g.nx + TX - 1) / TX, tiles_y = (g.ny + TY - 1) / TY;
    const int bx = lt % tiles_x, by = (lt / tiles_x) % tiles_y, bz = lt / (tiles_x * tiles_y);
    PadGeo pg = d.pg;
    View<ST> S = view<ST>(d.S[parity]), O = view<ST>(d.S[parity ^ 1]);
    S.f = uniform(S.f);
    O.f = uniform(O.f);
    O.sv = uniform(O.sv);
    PhysR<float> P = d.p;
    P.tau_a = uniform(P.tau_a);
    P.tau_b = uniform(P.tau_b);
    P.A2 = uniform(P.A2);
    P.beta = uniform(P.beta);
    P.A_h = uniform(P.A_h);
    P.h_min = uniform(P.h_min);
    P.h_max = uniform(P.h_max);
    P.phi_I = uniform(P.phi_I);
#pragma unroll
    for (int a = 0; a < 3; ++a) P.g[a] = uniform(P.g[a]);
    const int bits = uniform(P.equal_tau | P.K << 1 | P.g_mode << 4 | P.collision << 6);
    P.equal_tau = bits & 1;
    P.K = bits >> 1 & 7;
    P.g_mode = bits >> 4 & 3;
    P.collision = bits >> 6;
    step_tile<ST, LOAD_PULL, true, false, TX, TY, TZ, H, IDX32, false, (TX * TY * MINB <= 512 && !Store<ST>::TWOSET), true>(
        S, O, none, d.acc[k], d.acc[(k + 1) % 3], d.phi, pg, g, P, FieldOut{}, status, smem_raw, bx * TX, by * TY, bz * TZ);
  }
}

// ---------------------------------------------------------------------------
// population export (pre-collision, both components, canonical order, double)
// ---------------------------------------------------------------------------
template <int ST, int LOADER>
__global__ void __launch_bounds__(128) k_export(View<ST> S, InitBuf init, Geo g, PhysR<typename Store<ST>::R> P, int x0, int y0, int z0,
                                                int bx, int by, int bz, double* outA, double* outB) {
  using R = typename Store<ST>::R;
  const long long M = (long long)bx * by * bz;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < M;
       e += (long long)gridDim.x * blockDim.x) {
    const int lx = (int)(e % bx);
    const int ly = (int)((e / bx) % by);
    const int lz = (int)(e / ((long long)bx * by));
    const int x = x0 + lx, y = y0 + ly, z = z0 + lz;
    const long long self = (long long)x + (long long)g.nx * ((long long)y + (long long)g.ny * z);
    if (is_solid(g, x, y, z)) {
      for (int i = 0; i < Q; ++i) {
        outA[(size_t)i * M + e] = 0.0;
        outB[(size_t)i * M + e] = 0.0;
      }
      continue;
    }
    Nbr n;
    make_nbr(g, x, y, z, n);
    R f[Q], fa[Q], fb[Q], rA, rB;
    if constexpr (LOADER == LOAD_PULL) {
      pull_node<ST, true>(S, g, n, self, f, rA, rB, fa, fb);
    } else {
      fields_node<R, true>(init, g, P, n, self, f, rA, rB, fa, fb);
    }
    for (int i = 0; i < Q; ++i) {
      outA[(size_t)i * M + e] = (double)fa[i];
      outB[(size_t)i * M + e] = (double)fb[i];
    }
  }
}

}  // namespace lbcg
