// lbm_device.cuh -- device code of the HMCSC D3Q19 kernels, shared by the
// per-storage translation units (lbm_st_*.cu) that instantiate it.
//
// One time step is two launches:
//   k_density        rho_sigma(x) = sum_i f_i,sigma(x)                (Eq. A.4)
//   k_collide_stream moments, Shan-Chen forces (Eqs. 3-5), equilibrium
//                    velocity (Eq. 6), equilibrium (Eq. A.3), gray collision
//                    with partial bounce-back (Eq. 1) and in-place streaming
//   (or k_collide_pipe, the same arithmetic with the next plane's
//   populations copied into shared memory ahead of use)
// plus, as options, the single-pass sweep (k_sp_bulk + k_sp_seams) and the
// batched kernels that advance many lattices per launch.
//
// Density reservoirs (Sec. 4) reset their layers to the equilibrium at rest
// after every step, velocity boundary cells (Sec. 3.1) to the equilibrium at
// their velocity.  No kernel writes that reset: every reader of a node's
// populations (both passes, the fields pass, the host read-back) takes the
// prescribed equilibrium for a node inside such a layer, which is the state
// the reset defines, and what neighbours streamed into its slots is never
// read.
// StepParams::res holds the reservoirs that were in effect at the end of the
// previous step.
//
// Populations live in 32-node x-tiles (see lbm_internal.cuh) and stream in
// place with the AA pattern:
//   even t: node n reads slot i at n, writes its post-collision f_i to slot
//           opp(i) at n (population i of node n + c_i at t + 1);
//   odd t:  node n reads population i from slot opp(i) at n - c_i, writes
//           its post-collision f_i to slot i at n + c_i.
// Every (slot, node) a thread writes is one it read itself, so the update is
// race-free in place, and after an odd step the layout is natural again.
// One warp is one tile, and both components of a direction travel as one
// pair: on even steps all 19 loads and 19 stores of a thread are one pointer
// plus a constant; on odd steps there is one pointer per neighbour offset,
// shared by the load and the store at that offset.
#pragma once
#include "lbm_internal.cuh"

namespace hmcsc {
namespace {


// threadIdx.y and .z are the same for all lanes of a warp (blocks are 32
// threads wide); read through lane 0 the compiler knows it too and keeps row
// and plane arithmetic in uniform registers.
__device__ __forceinline__ int warp_ty() { return __shfl_sync(0xffffffffu, (int)threadIdx.y, 0); }
__device__ __forceinline__ int warp_tz() { return __shfl_sync(0xffffffffu, (int)threadIdx.z, 0); }

// Periodic neighbourhood of one node: rows are uniform over a warp, the x
// part is the lane's own.
struct Geo {
  int row[3][3];     // first tile of row (y + dy, z + dz): ntx * (y' + ny * z')
  int xw[3];         // x - 1, x, x + 1 (wrapped): the node inside its row
  unsigned xp[3];    // pair offset of slot 0 of that node inside its row
  __device__ __forceinline__ int tile(int dx, int dy, int dz) const {
    return row[dy + 1][dz + 1] + xw[dx + 1] / kTile;
  }
  __device__ __forceinline__ int lane(int dx) const { return xw[dx + 1] % kTile; }
  // tiled node index of x + (dx, dy, dz)
  __device__ __forceinline__ int node(int dx, int dy, int dz) const {
    return row[dy + 1][dz + 1] * kTile + xw[dx + 1];
  }
  // pair offset of slot 0 of node x + (dx, dy, dz) in the population array
  // (fits 32 bits: the host requires ntiles * 1216 < 2^32)
  __device__ __forceinline__ unsigned pop_off(int dx, int dy, int dz) const {
    return (unsigned)row[dy + 1][dz + 1] * (unsigned)kTilePairs + xp[dx + 1];
  }
};

__device__ __forceinline__ Geo make_geo(const StepParams &p, int x, int y,
                                        int z) {
  Geo g;
  g.xw[0] = x == 0 ? p.nx - 1 : x - 1;
  g.xw[1] = x;
  g.xw[2] = x == p.nx - 1 ? 0 : x + 1;
#pragma unroll
  for (int a = 0; a < 3; ++a)
    g.xp[a] = (unsigned)(g.xw[a] / kTile) * (unsigned)kTilePairs + (unsigned)(g.xw[a] % kTile);
  const int yw[3] = {y == 0 ? p.ny - 1 : y - 1, y, y == p.ny - 1 ? 0 : y + 1};
  const int zw[3] = {z == 0 ? p.nz - 1 : z - 1, z, z == p.nz - 1 ? 0 : z + 1};
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) g.row[a][b] = p.ntx * (yw[a] + p.ny * zw[b]);
  return g;
}

// Decode references of population i of node x (both components): w_i times
// the node's own previous density (*_LOCAL) or the constants (*_OFFSET).
// The product is rounded on its own (no contraction) so that the host
// read-back decodes identically.
template <int ST>
__device__ __forceinline__ float2 dec_ref(const StepParams &p, float2 own_prev,
                                          int i) {
  if (storage_local(ST))
    return make_float2(__fmul_rn(wgt(i), own_prev.x), __fmul_rn(wgt(i), own_prev.y));
  return p.ref[wclass(i)];
}

// The 19 populations of both components at the current time step, decoded
// to float32.  MUT: the encoding densities may have been written earlier in
// the same launch, so they are not read through the read-only path.
template <int PARITY, int ST, bool MUT = false>
__device__ __forceinline__ void load_pops(const StepParams &p, const Workspace &w,
                                          const Geo &g, float2 (&v)[kQ]) {
  using C = Codec2<ST>;
  const typename C::T2 *f = static_cast<const typename C::T2 *>(w.f);
  const long long nodes = p.ntiles * kTile, pairs = p.ntiles * kTilePairs;
  int own = g.node(0, 0, 0);
  float2 own_prev = make_float2(0.f, 0.f);
  if (storage_local(ST)) {
    if (kChecked && !in_bounds(w.fault, own, nodes, kFaultRhoLoad)) own = 0;
    own_prev = MUT ? __ldca(&w.rho_enc[own]) : __ldg(&w.rho_enc[own]);
  }
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    // population i of node x: slot i at x (even), slot opp(i) at x - c_i (odd)
    const int slot = PARITY == 0 ? i : opp(i);
    const typename C::T2 *src =
        f + (PARITY == 0 ? g.pop_off(0, 0, 0) : g.pop_off(-cx(i), -cy(i), -cz(i)));
    if (kChecked && !in_bounds(w.fault, (src - f) + slot * kTile, pairs, kFaultPopLoad))
      src = f - slot * kTile;  // reads element 0
    const typename C::T2 raw = src[slot * kTile];
    v[i] = C::dec(raw, dec_ref<ST>(p, own_prev, i));
  }
}

// Zeroth moment of both components, summed in direction order; k_density
// and k_collide_stream share this order so both see bit-identical densities.
__device__ __forceinline__ float2 sum19(const float2 (&v)[kQ]) {
  float2 r = v[0];
#pragma unroll
  for (int i = 1; i < kQ; ++i) r = add2(r, v[i]);
  return r;
}

__device__ __forceinline__ void first_moment(const float2 (&v)[kQ], float2 (&j)[3]) {
  j[0] = j[1] = j[2] = pair_of(0.0f);
#pragma unroll
  for (int i = 1; i < kQ; ++i) {
    if (cx(i)) j[0] = cx(i) > 0 ? add2(j[0], v[i]) : sub2(j[0], v[i]);
    if (cy(i)) j[1] = cy(i) > 0 ? add2(j[1], v[i]) : sub2(j[1], v[i]);
    if (cz(i)) j[2] = cz(i) > 0 ? add2(j[2], v[i]) : sub2(j[2], v[i]);
  }
}

// A read-only load the compiler may neither merge with an earlier load of
// the same address nor hoist: keeps a value that is needed late from
// occupying a register from the start of the kernel.
__device__ __forceinline__ float2 ld_late(const float2 *ptr) {
  float2 v;
  asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(ptr));
  return v;
}

// Where a pass finds the densities of the current step at x + (dx, dy, dz):
// `at` for the force stencil, `late` for the encoding reference of the
// *_LOCAL storages (a load the compiler keeps next to its use).
struct GlobalRho {  // the density array written by the density pass
  const float2 *__restrict__ rho;
  const Geo &g;
  long long nodes;   // tiled nodes (bounds-checked builds)
  unsigned *fault;
  __device__ __forceinline__ int idx(int dx, int dy, int dz) const {
    const int n = g.node(dx, dy, dz);
    return (kChecked && !in_bounds(fault, n, nodes, kFaultRhoLoad)) ? 0 : n;
  }
  __device__ __forceinline__ float2 at(int dx, int dy, int dz) const {
    return __ldg(&rho[idx(dx, dy, dz)]);
  }
  __device__ __forceinline__ float2 late(int dx, int dy, int dz) const {
    return ld_late(&rho[idx(dx, dy, dz)]);
  }
  // adhesion sources a_1 = G_ads,2 n_s,1 and a_2 (per-component fractions)
  const float *__restrict__ ads;
  const float *__restrict__ ads2;
  __device__ __forceinline__ int gidx(int dx, int dy, int dz) const {
    const int n = g.node(dx, dy, dz);
    return (kChecked && !in_bounds(fault, n, nodes, kFaultGeometry)) ? 0 : n;
  }
  __device__ __forceinline__ float a1(int dx, int dy, int dz) const {
    return __ldg(&ads[gidx(dx, dy, dz)]);
  }
  __device__ __forceinline__ float a2(int dx, int dy, int dz) const {
    return __ldg(&ads2[gidx(dx, dy, dz)]);
  }
  template <bool PC>
  __device__ __forceinline__ void adhesion(float2 (&A)[3]) const;
};
__device__ __forceinline__ GlobalRho global_rho(const StepParams &p, const Workspace &w,
                                                const Geo &g) {
  return GlobalRho{w.rho, g, p.ntiles * kTile, w.fault, w.ads, w.ads2};
}

// Total force per unit mass of each component, F_tot,sigma / rho_sigma
// (Eqs. 3-5; rho_sigma cancels against the prefactor of Eqs. 3-4 and the
// density ratio of Eq. 5, so no division by a vanishing component density):
//   g_1 = -G S_2 + A_1 + F_ext / rho,   g_2 = -G S_1 - A_2 + F_ext / rho
// with S_sigma = sum_i w_i rho_sigma(x + c_i) c_i and A_sigma = sum_i w_i
// a_sigma(x + c_i) c_i, a_sigma = G_ads,2 n_s,sigma (G_ads,1 = -G_ads,2,
// Table 1; the indicator of Eq. 4 is the component's own fraction).  With
// one fraction for both (PC = false) A_1 = A_2.  Opposite directions are
// summed as pairs, so a uniform field gives exactly zero.  Every product is
// fused into the sum it enters, written out so that each kernel rounds alike.
// gf[d] = (g_1, g_2) along axis d.
template <bool PC, typename RS>
__device__ __forceinline__ void adhesion_sum(const RS &rs, float2 (&A)[3]) {
#pragma unroll
  for (int d = 0; d < 3; ++d) A[d] = pair_of(0.0f);
#pragma unroll
  for (int i = 1; i <= 9; ++i) {
    const float da1 = __fsub_rn(rs.a1(cx(i), cy(i), cz(i)), rs.a1(-cx(i), -cy(i), -cz(i)));
    float da2 = 0.0f;
    if (PC) da2 = __fsub_rn(rs.a2(cx(i), cy(i), cz(i)), rs.a2(-cx(i), -cy(i), -cz(i)));
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int c = d == 0 ? cx(i) : d == 1 ? cy(i) : cz(i);
      if (c == 0) continue;
      const float w = c > 0 ? wgt(i) : -wgt(i);
      if (PC)
        A[d] = fma2(pair_of(w), make_float2(da1, da2), A[d]);
      else
        A[d].x = __fmaf_rn(w, da1, A[d].x);
    }
  }
  if (!PC)
#pragma unroll
    for (int d = 0; d < 3; ++d) A[d].y = A[d].x;
}
template <bool PC, typename RS>
__device__ __forceinline__ void force_per_mass(const StepParams &p, const RS &rs,
                                               float rho_tot, float2 (&gf)[3]) {
  float2 s[3], A[3];  // (S_1, S_2) and (A_1, A_2)
#pragma unroll
  for (int d = 0; d < 3; ++d) s[d] = pair_of(0.0f);
#pragma unroll
  for (int i = 1; i <= 9; ++i) {
    const float2 dr = sub2(rs.at(cx(i), cy(i), cz(i)), rs.at(-cx(i), -cy(i), -cz(i)));
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int c = d == 0 ? cx(i) : d == 1 ? cy(i) : cz(i);
      if (c != 0) s[d] = fma2(pair_of(c > 0 ? wgt(i) : -wgt(i)), dr, s[d]);
    }
  }
  rs.template adhesion<PC>(A);
  const float inv_rho = 1.0f / rho_tot;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    gf[d].x = __fmaf_rn(p.F[d], inv_rho, __fmaf_rn(-p.G, s[d].y, A[d].x));
    gf[d].y = __fmaf_rn(p.F[d], inv_rho, __fmaf_rn(-p.G, s[d].x, -A[d].y));
  }
}

template <bool PC>
__device__ __forceinline__ void GlobalRho::adhesion(float2 (&A)[3]) const {
  adhesion_sum<PC>(*this, A);
}

// Reservoir face holding node (x, y, z), -1 if none; the higher face wins.
__device__ __forceinline__ int res_face(const StepParams &p, int x, int y,
                                        int z) {
  const int *L = p.res.layers;
  int face = -1;
  if (L[0] && x < L[0]) face = 0;
  if (L[1] && x >= p.nx - L[1]) face = 1;
  if (L[2] && y < L[2]) face = 2;
  if (L[3] && y >= p.ny - L[3]) face = 3;
  if (L[4] && z < L[4]) face = 4;
  if (L[5] && z >= p.nz - L[5]) face = 5;
  return face;
}

// rho_res of component s on face `face` (selects, no indexed parameter load).
__device__ __forceinline__ float res_rho(const StepParams &p, int face, int s) {
  float r = p.res.rho[0][s];
#pragma unroll
  for (int k = 1; k < kFaces; ++k) r = face == k ? p.res.rho[k][s] : r;
  return r;
}

// Does the block's box [xlo,xhi] x [ylo,yhi] x [zlo,zhi] hold a node inside
// a reservoir?  Uniform over the block, known before any load.
__device__ __forceinline__ bool box_in_reservoir(const StepParams &p, int xlo,
                                                 int xhi, int ylo, int yhi,
                                                 int zlo, int zhi) {
  if (!p.res.any) return false;
  const int *L = p.res.layers;
  return (L[0] && xlo < L[0]) || (L[1] && xhi >= p.nx - L[1]) ||
         (L[2] && ylo < L[2]) || (L[3] && yhi >= p.ny - L[3]) ||
         (L[4] && zlo < L[4]) || (L[5] && zhi >= p.nz - L[5]);
}

// Prescribed velocity component d of face `face` (selects).
__device__ __forceinline__ float res_u(const StepParams &p, int face, int d) {
  float u = p.res.u[0][d];
#pragma unroll
  for (int k = 1; k < kFaces; ++k) u = face == k ? p.res.u[k][d] : u;
  return u;
}

// A node inside a reservoir holds the prescribed equilibrium: at rest for a
// density reservoir, at the face's velocity for velocity boundary cells.
// Only blocks whose box meets a reservoir (`maybe`, block-uniform) look.
__device__ __forceinline__ void reservoir_state(const StepParams &p, bool maybe,
                                                int x, int y, int z, float2 (&v)[kQ]) {
  if (!maybe) return;
  const int face = res_face(p, x, y, z);
  if (face >= 0) {
    const float r1 = res_rho(p, face, 0), r2 = res_rho(p, face, 1);
    if (p.res.moving) {
      const float ux = res_u(p, face, 0), uy = res_u(p, face, 1), uz = res_u(p, face, 2);
#pragma unroll
      for (int i = 0; i < kQ; ++i)
        v[i] = make_float2(res_feq(i, r1, ux, uy, uz), res_feq(i, r2, ux, uy, uz));
    } else {
#pragma unroll
      for (int i = 0; i < kQ; ++i) v[i] = make_float2(wgt(i) * r1, wgt(i) * r2);
    }
  }
}

// The stored form of the pair o of direction i, its destination's density
// being dest (used by the *_LOCAL storages).
template <int ST>
__device__ __forceinline__ typename Codec2<ST>::T2 encode(const StepParams &p, int i, float2 o,
                                                          float2 dest) {
  if constexpr (storage_local(ST))
    return Codec2<ST>::enc_local(o, wgt(i), dest);
  else
    return Codec2<ST>::enc(o, p.nref[wclass(i)]);
}

// Store the post-collision pair (both components) of direction i; it
// becomes the pair of direction i of node x + c_i at t + 1.  Encoding
// reference: w_i times the destination's density at this step (*_LOCAL;
// rho_s for the rest population, the density pass's value otherwise), or the
// constants w_i rho0_sigma (*_OFFSET).
template <int PARITY, int ST, typename RS, bool CS = false, typename GE>
__device__ __forceinline__ void put2(const StepParams &p, const Workspace &w,
                                     const GE &g, const RS &rs, int i, float2 o,
                                     float2 rho) {
  using C = Codec2<ST>;
  typename C::T2 *f = static_cast<typename C::T2 *>(w.f);
  float2 dest = rho;  // the destination's density at this step (*_LOCAL)
  if (storage_local(ST) && i != 0) dest = rs.late(cx(i), cy(i), cz(i));
  const typename C::T2 e = encode<ST>(p, i, o, dest);
  const int slot = PARITY == 0 ? opp(i) : i;
  typename C::T2 *dst = f + (PARITY == 0 ? g.pop_off(0, 0, 0) : g.pop_off(cx(i), cy(i), cz(i)));
  if (!kChecked ||
      in_bounds(w.fault, (dst - f) + slot * kTile, p.ntiles * kTilePairs, kFaultPopStore))
  {
    if (CS)
      __stcs(&dst[slot * kTile], e);  // streaming: evict first from the caches
    else
      dst[slot * kTile] = e;
  }
}

// Eq. 1 for both components: (1 - n_s)[f_i - (f_i - f^eq_i)/tau] +
// n_s f_opp(i) with f^eq of Eq. A.3 at (rho_s, u_s), computed for opposite
// pairs at once.  The rest population's equilibrium is taken as rho_s minus
// the other 18 (sum_i f^eq_i = rho_s holds exactly for Eq. A.3 on D3Q19),
// which keeps the rounding of the float weights from leaking mass step after
// step.  The relaxation weight b = (1 - n_s) / tau is folded into the
// equilibrium: B_i = b f^eq_i = (b w_i rho_s)[1 - 1.5 u.u + 4.5 (c_i.u)^2
// +- 3 c_i.u], so each population costs two fused multiply-adds on top of B_i.
// Every value is the pair of both components.  With E_i = 1 - 1.5 u.u + 4.5
// (c_i.u)^2 and q = 3 b w_i rho, the two products of B_i = b w_i rho E_i + q
// c_i.u cannot both be fused: component 1 rounds q c_i.u and component 2
// rounds b w_i rho E_i, the order every result of this library has been
// computed in, so these six operations stay scalar.
struct Relax {
  float2 a, base, br, br18, br36, q18, q36, moving, ns;
  __device__ __forceinline__ Relax(float2 om, float2 ns_s, float2 rho, const float2 (&u)[3]) {
    ns = ns_s;
    const float2 open = sub2(pair_of(1.0f), ns);
    a = mul2(open, sub2(pair_of(1.0f), om));
    base = fma2(pair_of(-1.5f), fma2(u[2], u[2], fma2(u[0], u[0], mul2(u[1], u[1]))),
                pair_of(1.0f));
    br = mul2(mul2(open, om), rho);
    br18 = mul2(br, pair_of(1.0f / 18.0f));
    br36 = mul2(br, pair_of(1.0f / 36.0f));
    q18 = mul2(pair_of(3.0f), br18);
    q36 = mul2(pair_of(3.0f), br36);
    moving = pair_of(0.0f);  // sum of B_i over the 18 moving directions
  }
  // post-collision values of the opposite pair of directions (i, j) from
  // their pre-collision values vi, vj; cu = c_i . u
  __device__ __forceinline__ void pair(bool axis, float2 cu, float2 vi, float2 vj,
                                       float2 &out_i, float2 &out_j) {
    const float2 bw = axis ? br18 : br36, q = axis ? q18 : q36;
    const float2 e = fma2(mul2(pair_of(4.5f), cu), cu, base);
    const float odd1 = __fmul_rn(q.x, cu.x), even2 = __fmul_rn(bw.y, e.y);
    const float2 B_i = make_float2(__fmaf_rn(bw.x, e.x, odd1), __fmaf_rn(q.y, cu.y, even2));
    const float2 B_j = make_float2(__fmaf_rn(bw.x, e.x, -odd1), __fmaf_rn(-q.y, cu.y, even2));
    moving = add2(moving, add2(B_i, B_j));
    out_i = fma2(a, vi, fma2(ns, vj, B_i));
    out_j = fma2(a, vj, fma2(ns, vi, B_j));
  }
  // post-collision rest population: B_0 = b rho_s - sum of the moving B_i
  __device__ __forceinline__ float2 rest(float2 v0) const {
    return fma2(make_float2(__fadd_rn(a.x, ns.x), __fadd_rn(a.y, ns.y)), v0, sub2(br, moving));
  }
};

// Moments, forces, equilibrium velocity and collision of one node from its
// 19 pairs v (decoded, and replaced by the prescribed state inside a
// reservoir), its n_s and where the step's densities are found; emit(i, o,
// rho) takes the post-collision pair of direction i.
template <bool PC, typename RS, typename Emit>
__device__ __forceinline__ void collide_core(const StepParams &p, const RS &rs,
                                             const float2 (&v)[kQ], float2 ns, Emit emit) {
  const float2 rho = sum19(v);
  float2 j[3];
  first_moment(v, j);

  float2 gf[3];
  force_per_mass<PC>(p, rs, __fadd_rn(rho.x, rho.y), gf);

  // Eq. 6: common velocity sum_s j_s/tau_s / sum_s rho_s/tau_s, then the
  // Shan-Chen shift tau_s F_tot,s / rho_s = tau_s g_s.
  const float inv_den = 1.0f / __fmaf_rn(rho.x, p.omega[0], __fmul_rn(rho.y, p.omega[1]));
  float2 u[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float jc = __fmaf_rn(j[d].x, p.omega[0], __fmul_rn(j[d].y, p.omega[1]));
    u[d].x = __fmaf_rn(jc, inv_den, __fmul_rn(p.tau[0], gf[d].x));
    u[d].y = __fmaf_rn(jc, inv_den, __fmul_rn(p.tau[1], gf[d].y));
  }

  Relax c(make_float2(p.omega[0], p.omega[1]), ns, rho, u);
#pragma unroll
  for (int i = 1; i <= 9; ++i) {
    // of the two, j = i + 9 has the positive first nonzero component, so
    // c_j . u starts without a negation
    const int k = i + 9;
    float2 cu = pair_of(0.0f);
    bool first = true;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int e = d == 0 ? cx(k) : d == 1 ? cy(k) : cz(k);
      if (e == 0) continue;
      cu = first ? u[d] : (e > 0 ? add2(cu, u[d]) : sub2(cu, u[d]));
      first = false;
    }
    float2 oi, ok;
    c.pair(wclass(i) == 1, cu, v[k], v[i], ok, oi);
    emit(i, oi, rho);
    emit(k, ok, rho);
  }
  emit(0, c.rest(v[0]), rho);
}

// The same, each pair stored where the AA pattern puts it: g tells where the
// neighbours' slots lie (pop_off).
template <int PARITY, int ST, bool PC, typename RS, bool CS = false, typename GE>
__device__ __forceinline__ void collide_loaded(const StepParams &p, const Workspace &w,
                                               const GE &g, const RS &rs,
                                               const float2 (&v)[kQ], float2 ns) {
  collide_core<PC>(p, rs, v, ns, [&](int i, float2 o, float2 rho) {
    put2<PARITY, ST, RS, CS>(p, w, g, rs, i, o, rho);
  });
}

// n_s,1 and n_s,2 (the same without per-component fractions) of a node.
template <bool PC>
__device__ __forceinline__ float2 node_ns(const StepParams &p, const Workspace &w, const Geo &g) {
  int own = g.node(0, 0, 0);
  if (!in_bounds(w.fault, own, p.ntiles * kTile, kFaultGeometry)) own = 0;
  const float ns1 = w.ns[own];
  return make_float2(ns1, PC ? w.ns2[own] : ns1);
}

template <int PARITY, int ST, bool PC, typename RS>
__device__ __forceinline__ void collide_node(const StepParams &p, const Workspace &w,
                                             const Geo &g, const RS &rs,
                                             bool maybe_res, int x, int y, int z) {
  float2 v[kQ];
  load_pops<PARITY, ST>(p, w, g, v);
  reservoir_state(p, maybe_res, x, y, z, v);
  collide_loaded<PARITY, ST, PC>(p, w, g, rs, v, node_ns<PC>(p, w, g));
}

template <int PARITY, int ST, bool PC, bool CS = false>
__device__ __forceinline__ void collide_body(const StepParams &p,
                                             const Workspace &w, bool maybe_res,
                                             int x, int y, int z) {
  const Geo g = make_geo(p, x, y, z);
  float2 v[kQ];
  load_pops<PARITY, ST>(p, w, g, v);
  reservoir_state(p, maybe_res, x, y, z, v);
  collide_loaded<PARITY, ST, PC, GlobalRho, CS>(p, w, g, global_rho(p, w, g), v,
                                                node_ns<PC>(p, w, g));
}


// Launch shapes of the passes: a block is 32 x by x bz threads (one node
// each) and minb is the number of blocks per SM its register budget is sized
// for.  Shape 0 of each pass is the default; the autotuner picks among the
// others per lattice size and storage.
struct Shape {
  int by, bz, minb;
  bool cs = false;  // populations stored with the streaming (evict-first) policy
};
__host__ __device__ constexpr Shape density_shape(int cfg) {
  return cfg == 1 ? Shape{8, 1, 1} : cfg == 2 ? Shape{4, 1, 1} : Shape{4, 2, 1};
}
// Shapes of the prefetching fused pass (k_collide_pipe): block 32 x by,
// blocks per SM.  On the 256^3 electrode (us, even / odd step; 168 and 176
// bytes a node at the copy rate of 6690 GB/s are 421 and 441): half offsets
// 519/586 in shape 6, 430/520 in shapes 9/8 (in scalar operations with a copy
// per population 606/737); local half offsets 693/728 in shape 6, 455/553 in
// shape 9 (scalar 726/810; without its streaming stores 547 on even steps);
// float32 (320 bytes: 803) 774/885 in shape 6, 816/881 in shape 7 (scalar
// 837/967), 778/985 in shape 9.  Even steps are bound by HBM.  Odd
// ones store rows shifted by a node, which leave part of a sector at either
// end, and keep 18 addresses: they issue 753-788 instructions a node, 61 % of
// the slots, and the local storages take 168 registers.  Staging the stencil
// pays for the 16-bit storages, whose bytes are fewer than their stencil's
// loads can hide behind; float32 is bound by its bytes either way.  More
// blocks per SM spill: at 10 and 9, half offsets run 525/705.
struct PipeCfg {
  int by, minb_even, minb_odd, minb_even_local, minb_odd_local;
  bool ring;  // neighbour densities and adhesion sources also staged in
              // shared memory (a five-plane ring filled by the block)
  bool cs;    // streaming stores
};
__host__ __device__ constexpr PipeCfg pipe_cfg(int cfg) {
  return cfg == 6   ? PipeCfg{8, 2, 2, 2, 2, false, false}
         : cfg == 7 ? PipeCfg{2, 10, 8, 8, 6, false, false}
         : cfg == 8 ? PipeCfg{2, 8, 8, 8, 6, true, false}
         : cfg == 9 ? PipeCfg{2, 8, 8, 8, 6, true, true}
                    : PipeCfg{4, 4, 4, 4, 3, true, true};
}
constexpr int kPipeRingPlanes = 5, kPipeRingCols = kTile + 2;

// Neighbour densities and adhesion sources from the shared-memory ring of a
// prefetching block: row pointers of the node's ring row in planes z - 1,
// z, z + 1 and the node's column.
struct SmemStencil {
  const float2 *rho[3];
  const float *a[3];
  const float *b[3];
  int c;
  __device__ __forceinline__ float2 at(int dx, int dy, int dz) const {
    return rho[dz + 1][dy * kPipeRingCols + c + dx];
  }
  __device__ __forceinline__ float2 late(int dx, int dy, int dz) const {
    return at(dx, dy, dz);
  }
  __device__ __forceinline__ float a1(int dx, int dy, int dz) const {
    return a[dz + 1][dy * kPipeRingCols + c + dx];
  }
  __device__ __forceinline__ float a2(int dx, int dy, int dz) const {
    return b[dz + 1][dy * kPipeRingCols + c + dx];
  }
  template <bool PC>
  __device__ __forceinline__ void adhesion(float2 (&A)[3]) const {
    adhesion_sum<PC>(*this, A);
  }
};
__host__ __device__ constexpr Shape pipe_shape(int parity, bool local, int cfg) {
  return Shape{pipe_cfg(cfg).by, 1,
               parity == 0 ? (local ? pipe_cfg(cfg).minb_even_local : pipe_cfg(cfg).minb_even)
                           : (local ? pipe_cfg(cfg).minb_odd_local : pipe_cfg(cfg).minb_odd),
               pipe_cfg(cfg).cs};
}
// The odd step keeps one address per neighbour offset and the *_LOCAL
// storages also hold the destination densities for encoding: both get more
// registers per thread (the local odd shape 2 trades occupancy for a budget
// of 170 registers, which needs no spill).  Shape 4 stores with the
// streaming policy (float32 odd step 1.05 -> 0.95 ms in the plain kernel).
__host__ __device__ constexpr Shape collide_shape(int parity, bool local, int cfg) {
  return cfg >= kCollidePipeFirst ? pipe_shape(parity, local, cfg)
         : cfg == 4 ? (local ? Shape{4, 1, 3, true} : Shape{4, 2, 2, true})
         : parity == 0
             ? (local ? (cfg == 1 ? Shape{8, 1, 2} : cfg == 2 ? Shape{4, 1, 4}
                         : cfg == 3 ? Shape{2, 4, 2} : Shape{4, 2, 2})
                      : (cfg == 1 ? Shape{8, 1, 3} : cfg == 2 ? Shape{4, 1, 6}
                         : cfg == 3 ? Shape{2, 4, 3} : Shape{4, 2, 3}))
             : (local ? (cfg == 1 ? Shape{4, 2, 2} : cfg == 2 ? Shape{4, 1, 3}
                         : cfg == 3 ? Shape{2, 2, 4} : Shape{4, 1, 4})
                      : (cfg == 1 ? Shape{4, 2, 2} : cfg == 2 ? Shape{8, 1, 2}
                         : cfg == 3 ? Shape{2, 2, 5} : Shape{4, 1, 5}));
}
template <int CFG>
struct DensityShape {
  static constexpr Shape s = density_shape(CFG);
  static constexpr int threads = kTile * s.by * s.bz;
};
template <int PARITY, int ST, int CFG>
struct CollideShape {
  static constexpr Shape s = collide_shape(PARITY, storage_local(ST), CFG);
  static constexpr int threads = kTile * s.by * s.bz;
};
constexpr int kFieldsBY = 4, kFieldsBZ = 2;

// Does the block's box hold a node inside a reservoir?  Block-uniform.
template <int BY, int BZ>
__device__ __forceinline__ bool block_in_reservoir(const StepParams &p) {
  const int xlo = blockIdx.x * kTile, ylo = blockIdx.y * BY, zlo = blockIdx.z * BZ;
  return box_in_reservoir(p, xlo, min(xlo + kTile, p.nx) - 1, ylo,
                          min(ylo + BY, p.ny) - 1, zlo, min(zlo + BZ, p.nz) - 1);
}

template <int BY, int BZ>
__device__ __forceinline__ void block_coords(int &x, int &y, int &z) {
  x = blockIdx.x * kTile + threadIdx.x;
  y = blockIdx.y * BY + (BY > 1 ? warp_ty() : 0);
  z = blockIdx.z * BZ + (BZ > 1 ? warp_tz() : 0);
}

template <int PARITY, int ST, int CFG>
__global__ void __launch_bounds__(DensityShape<CFG>::threads)
    k_density(StepParams p, Workspace w) {
  constexpr Shape S = DensityShape<CFG>::s;
  int x, y, z;
  block_coords<S.by, S.bz>(x, y, z);
  const bool maybe_res = block_in_reservoir<S.by, S.bz>(p);
  if (x >= p.nx || y >= p.ny || z >= p.nz) return;
  const Geo g = make_geo(p, x, y, z);
  float2 v[kQ];
  load_pops<PARITY, ST>(p, w, g, v);
  reservoir_state(p, maybe_res, x, y, z, v);
  const int own = g.node(0, 0, 0);
  if (in_bounds(w.fault, own, p.ntiles * kTile, kFaultRhoStore)) w.rho[own] = sum19(v);
}

// ---- fused pass with prefetch ----
// Shapes kCollidePipeFirst.. of the fused pass: each block owns 32 x by
// nodes of a run of planes and walks the run plane by plane, one warp per
// row; a warp copies the populations of its row in the next plane into
// shared memory (cp.async, two buffers of the warp's own, so no block
// barrier) while it collides the current plane.  The loads of one plane
// overlap the arithmetic of the one before without holding registers; the
// arithmetic is that of k_collide_stream, so the results are bit-identical.
template <typename T>
__device__ __forceinline__ void cp_async(T *smem, const T *gmem) {
  static_assert(sizeof(T) == 4 || sizeof(T) == 8, "cp.async copies 4 or 8 bytes here");
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(s), "l"(gmem),
               "n"((int)sizeof(T))
               : "memory");
}
// 16 bytes, both addresses 16-byte aligned, through L2 only: a population is
// read once per launch, so it leaves L1 to the force stencil.
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Components of direction i for an i known only at run time (0, 1 or 2 for
// -1, 0, 1), two bits each.
__host__ __device__ constexpr unsigned long long packed_dir(int axis) {
  unsigned long long v = 0;
  for (int i = 0; i < kQ; ++i)
    v |= (unsigned long long)((axis == 1 ? cy(i) : cz(i)) + 1) << (2 * i);
  return v;
}
__device__ __forceinline__ int run_cy(int i) { return (int)((packed_dir(1) >> (2 * i)) & 3) - 1; }
__device__ __forceinline__ int run_cz(int i) { return (int)((packed_dir(2) >> (2 * i)) & 3) - 1; }

// The populations of one row of 32 nodes (x-tile bx, row y), plane by plane,
// copied by one warp in 16-byte chunks.  Even steps read the tile itself,
// one contiguous run.  Odd steps read population i from slot opp(i) of the
// tile at (y - c_y, z - c_z), shifted by c_x: the slot's row of 32 is copied
// whole, and the one node beyond its edge that a shifted read needs (lane 0
// for c_x = 1, the last lane for c_x = -1) goes into element 32 of the row.
// A chunk also carries values of nodes other rows own; they are not used, so
// it does not matter that their owners may be replacing them.  Per warp and
// plane this takes 5 (16-bit) or 10 (float32) copy instructions (odd steps:
// one more and two integer operations each) instead of 19 with an address
// each.
template <int PARITY, typename T2>
struct RowCopy {
  static constexpr int kEl = 16 / (int)sizeof(T2);               // pairs per chunk
  static constexpr int kStride = PARITY == 0 ? kTile : kTile + kEl;  // pairs per slot row
  static constexpr int kPairs = kQ * kStride;                    // pairs per buffer
  static constexpr int kChunks = kTilePairs / kEl;               // chunks per tile
  static constexpr int kCopies = (kChunks + kTile - 1) / kTile;  // per lane
  static constexpr int kOff = PARITY == 0 ? 1 : kCopies;
  unsigned off[kOff];  // source (pairs) of this lane's chunks in the next plane
  unsigned halo;       // source of this lane's edge node (lanes 0..9)
  int at[3];           // element of a slot row this lane reads for c_x = -1, 0, 1
  unsigned plane, total;

  __device__ __forceinline__ RowCopy(const StepParams &p, int bx, int y, int z) {
    const int lane = threadIdx.x;
    plane = (unsigned)(p.ny * p.ntx) * (unsigned)kTilePairs;
    total = plane * (unsigned)p.nz;
    at[1] = lane;
    if (PARITY == 0) {
      off[0] = (unsigned)z * plane + (unsigned)(y * p.ntx + bx) * kTilePairs + lane * kEl;
      return;
    }
    const int xlo = bx * kTile, xhi = min(xlo + kTile, p.nx) - 1;
    at[0] = lane == xhi - xlo ? kTile : lane + 1;  // c_x = -1 reads x + 1
    at[2] = lane == 0 ? kTile : lane - 1;
#pragma unroll
    for (int k = 0; k < kOff; ++k) {
      const int c = lane + k * kTile;
      const int i = min(c / (kTile / kEl), kQ - 1);
      off[k] = source(p, i, bx, y, z) + (unsigned)(c % (kTile / kEl)) * kEl;
    }
    const int h = min(lane, 9);
    const int i = h < 5 ? (h == 0 ? 1 : h + 3) : (h == 5 ? 10 : h + 7);
    int x = h < 5 ? xhi + 1 : xlo - 1;
    x = x < 0 ? p.nx - 1 : (x >= p.nx ? 0 : x);
    halo = source(p, i, x / kTile, y, z) + (unsigned)(x % kTile);
  }
  // slot row of population i of row y, plane z, in x-tile xt (odd steps)
  static __device__ __forceinline__ unsigned source(const StepParams &p, int i, int xt, int y,
                                                    int z) {
    int yw = y - run_cy(i), zw = z - run_cz(i);
    yw = yw < 0 ? p.ny - 1 : (yw >= p.ny ? 0 : yw);
    zw = zw < 0 ? p.nz - 1 : (zw >= p.nz ? 0 : zw);
    const int slot = i == 0 ? 0 : (i <= 9 ? i + 9 : i - 9);
    return (unsigned)((zw * p.ny + yw) * p.ntx + xt) * (unsigned)kTilePairs + slot * kTile;
  }
  // start copying the next plane of the run into buf and move on
  __device__ __forceinline__ void next(const Workspace &w, T2 *buf) {
    const T2 *f = static_cast<const T2 *>(w.f);
    const int lane = threadIdx.x;
#pragma unroll
    for (int k = 0; k < kCopies; ++k) {
      const int c = lane + k * kTile;
      if ((k + 1) * kTile > kChunks && c >= kChunks) break;
      unsigned o = PARITY == 0 ? off[0] + k * kTile * kEl : off[k];
      if (kChecked && !in_bounds(w.fault, (long long)o + kEl, (long long)total + 1, kFaultPopLoad))
        o = 0;
      T2 *dst = PARITY == 0 ? buf + c * kEl
                            : buf + (c / (kTile / kEl)) * kStride + (c % (kTile / kEl)) * kEl;
      cp_async16(dst, f + o);
      if (PARITY == 1) off[k] = step(off[k]);
    }
    if (PARITY == 0) {
      off[0] += plane;
    } else {
      if (lane < 10) {
        const int i = lane < 5 ? (lane == 0 ? 1 : lane + 3) : (lane == 5 ? 10 : lane + 7);
        unsigned o = halo;
        if (kChecked && !in_bounds(w.fault, o, total, kFaultPopLoad)) o = 0;
        cp_async(buf + i * kStride + kTile, f + o);
      }
      halo = step(halo);
    }
  }
  // the same place one plane on, periodic
  __device__ __forceinline__ unsigned step(unsigned o) const {
    o += plane;
    return min(o, o - total);
  }
  // population i of this lane's node
  __device__ __forceinline__ T2 get(const T2 *buf, int i) const {
    return buf[i * kStride + (PARITY == 0 ? at[1] : at[cx(i) + 1])];
  }
};

// Where a block that walks along z finds a node's neighbours: the in-plane
// part does not change from plane to plane.
struct MarchGeo {
  unsigned row[3];     // pair offset of row y + dy inside a plane (uniform)
  unsigned xp[3];      // pair offset of slot 0 of x + dx inside a row
  unsigned pz[3];      // pair offset of planes z - 1, z, z + 1 (uniform)
  unsigned plane, total;
  __device__ __forceinline__ MarchGeo(const StepParams &p, int x, int y, int z) {
    plane = (unsigned)(p.ny * p.ntx) * (unsigned)kTilePairs;
    total = plane * (unsigned)p.nz;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      int xw = x + a - 1, yw = y + a - 1;
      xw = xw < 0 ? p.nx - 1 : (xw >= p.nx ? 0 : xw);
      yw = yw < 0 ? p.ny - 1 : (yw >= p.ny ? 0 : yw);
      xp[a] = (unsigned)(xw / kTile) * (unsigned)kTilePairs + (unsigned)(xw % kTile);
      row[a] = (unsigned)(yw * p.ntx) * (unsigned)kTilePairs;
    }
    pz[1] = (unsigned)z * plane;
    pz[0] = z == 0 ? total - plane : pz[1] - plane;
    pz[2] = z == p.nz - 1 ? 0u : pz[1] + plane;
  }
  __device__ __forceinline__ void next() {
    pz[0] = pz[1];
    pz[1] = pz[2];
    const unsigned o = pz[2] + plane;
    pz[2] = min(o, o - total);
  }
  __device__ __forceinline__ unsigned pop_off(int dx, int dy, int dz) const {
    return (pz[dz + 1] + row[dy + 1]) + xp[dx + 1];
  }
};

// Shared memory of a prefetching block: two buffers of its rows'
// populations, n_s and (local storages) encoding densities, and with the
// ring five planes of (by + 2) x 34 density pairs and adhesion sources.
template <int PARITY, int ST, bool PC, int CFG>
struct PipeSmem {
  using T2 = typename Codec2<ST>::T2;
  static constexpr PipeCfg P = pipe_cfg(CFG);
  static constexpr int NT = kTile * P.by, kRing = (P.by + 2) * kPipeRingCols;
  static constexpr bool L = storage_local(ST);
  alignas(16) T2 pop[2][P.by][RowCopy<PARITY, T2>::kPairs];
  float2 enc[L ? 2 : 1][L ? NT : 1];
  float2 ring_rho[P.ring ? kPipeRingPlanes : 1][P.ring ? kRing : 1];
  float ring_a[P.ring ? kPipeRingPlanes : 1][P.ring ? kRing : 1];
  float ring_b[P.ring && PC ? kPipeRingPlanes : 1][P.ring && PC ? kRing : 1];
  float ns[2][NT];
  float ns2[PC ? 2 : 1][PC ? NT : 1];
};

// The fused pass of one block of a prefetching shape: x-tile bx, rows
// [by0 * by, by0 * by + by) and the run of planes [bz * zc, bz * zc + zc)
// of lattice (p, w).
template <int PARITY, int ST, bool PC, int CFG>
__device__ __forceinline__ void pipe_block(const StepParams &p, const Workspace &w, int zc, int bx,
                                           int by0, int bz) {
  using C = Codec2<ST>;
  using T2 = typename C::T2;
  using Copy = RowCopy<PARITY, T2>;
  constexpr Shape S = CollideShape<PARITY, ST, CFG>::s;
  constexpr int NT = kTile * S.by;
  constexpr bool kRing = pipe_cfg(CFG).ring;
  constexpr bool L = storage_local(ST);
  constexpr int R = S.by + 2, RC = kPipeRingCols;
  using Smem = PipeSmem<PARITY, ST, PC, CFG>;
  extern __shared__ __align__(16) unsigned char pipe_smem[];
  Smem &sm = *reinterpret_cast<Smem *>(pipe_smem);
  const int ty = warp_ty(), tid = ty * kTile + threadIdx.x;
  const int x = bx * kTile + threadIdx.x, y = by0 * S.by + ty;
  const int z0 = bz * zc, zend = min(z0 + zc, p.nz);
  const int xlo = bx * kTile, ylo = by0 * S.by;
  const bool maybe_res = box_in_reservoir(p, xlo, min(xlo + kTile, p.nx) - 1, ylo,
                                          min(ylo + S.by, p.ny) - 1, z0, zend - 1);
  const bool row = y < p.ny;            // warp-uniform
  const bool active = row && x < p.nx;
  // Without the ring no warp reads another's shared memory and idle warps
  // may leave; with it every thread fills the ring and meets the per-plane
  // barrier.
  if (z0 >= zend || (!kRing && !row)) return;
  const long long nodes = p.ntiles * kTile;
  const int plane_nodes = p.ny * p.ntx * kTile;
  Copy copy(p, bx, row ? y : 0, z0);
  // this node (padding lanes: their tile's lane, which exists)
  int own = ((z0 * p.ny + (row ? y : 0)) * p.ntx + bx) * kTile + threadIdx.x;
  auto prefetch = [&](int b, int n) {
    if (!row) return;
    copy.next(w, sm.pop[b][ty]);
    if (kChecked && !in_bounds(w.fault, n, nodes, kFaultGeometry)) n = 0;
    cp_async(&sm.ns[b][tid], &w.ns[n]);
    if (PC) cp_async(&sm.ns2[PC ? b : 0][PC ? tid : 0], &w.ns2[n]);
    if (L) cp_async(&sm.enc[L ? b : 0][L ? tid : 0], &w.rho_enc[n]);
  };
  // ring plane of z (z0 - 1 <= z <= zend): rows y0 - 1 .. y0 + by, columns
  // x0 - 1 .. x0 + 32, periodic.  The in-plane nodes a thread copies are the
  // same for every plane, so the wrapping is worked out once per block.
  constexpr int RE = kRing ? (R * RC + NT - 1) / NT : 1;
  int ring_node[RE];
  if constexpr (kRing) {
#pragma unroll
    for (int k = 0; k < RE; ++k) {
      const int e = tid + k * NT, r = e / RC, c = e % RC;
      int xw = xlo + c - 1, yw = ylo + r - 1;
      xw = xw < 0 ? xw + p.nx : (xw >= p.nx ? xw % p.nx : xw);
      yw = yw < 0 ? yw + p.ny : (yw >= p.ny ? yw % p.ny : yw);
      ring_node[k] = (yw * p.ntx + xw / kTile) * kTile + xw % kTile;
    }
  }
  auto fill_ring = [&](int z, int slot) {
    const int zw = z < 0 ? z + p.nz : (z >= p.nz ? z - p.nz : z);
    const long long plane = (long long)zw * plane_nodes;
#pragma unroll
    for (int k = 0; k < RE; ++k) {
      const int e = tid + k * NT;
      if (e >= R * RC) break;
      long long n = plane + ring_node[k];
      if (kChecked && !in_bounds(w.fault, n, nodes, kFaultRhoLoad)) n = 0;
      if constexpr (kRing) {
        cp_async(&sm.ring_rho[slot][e], &w.rho[n]);
        cp_async(&sm.ring_a[slot][e], &w.ads[n]);
        if (PC) cp_async(&sm.ring_b[PC ? slot : 0][PC ? e : 0], &w.ads2[n]);
      }
    }
  };
  prefetch(0, own);
  if constexpr (kRing) {
    fill_ring(z0 - 1, 0);
    fill_ring(z0, 1);
    fill_ring(z0 + 1, 2);
  }
  cp_async_commit();
  MarchGeo mg(p, min(x, p.nx - 1), min(y, p.ny - 1), z0);
  int slot = 0;  // ring slot of plane z - 1
  for (int z = z0; z < zend; ++z) {
    const int b = (z - z0) & 1;
    // next plane's populations and the ring plane after it; the ring slot
    // refilled here was last read two planes ago, before the previous
    // barrier, and the buffer in the previous plane, by this warp alone
    __syncwarp();
    if (z + 1 < zend) prefetch(b ^ 1, own + plane_nodes);
    if (kRing && z + 2 <= zend)
      fill_ring(z + 2, slot + 3 < kPipeRingPlanes ? slot + 3 : slot - 2);
    cp_async_commit();
    cp_async_wait<1>();  // this thread's copies for plane z are complete
    if constexpr (kRing)
      __syncthreads();   // and every thread's
    else
      __syncwarp();      // and every lane's
    if (active) {
      const T2 *buf = sm.pop[b][ty];
      const float2 own_prev = L ? sm.enc[L ? b : 0][L ? tid : 0] : make_float2(0.f, 0.f);
      const float ns1 = sm.ns[b][tid];
      const float2 ns = make_float2(ns1, PC ? sm.ns2[PC ? b : 0][PC ? tid : 0] : ns1);
      float2 v[kQ];
#pragma unroll
      for (int i = 0; i < kQ; ++i) v[i] = C::dec(copy.get(buf, i), dec_ref<ST>(p, own_prev, i));
      reservoir_state(p, maybe_res, x, y, z, v);
      if constexpr (!kRing) {
        const Geo g = make_geo(p, x, y, z);
        collide_loaded<PARITY, ST, PC, GlobalRho, S.cs>(p, w, mg, global_rho(p, w, g), v, ns);
      } else {
        SmemStencil st;
        const int r = ty + 1;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const int sd = slot + d < kPipeRingPlanes ? slot + d : slot + d - kPipeRingPlanes;
          st.rho[d] = sm.ring_rho[sd] + r * RC;
          st.a[d] = sm.ring_a[sd] + r * RC;
          st.b[d] = PC ? sm.ring_b[PC ? sd : 0] + (PC ? r * RC : 0) : nullptr;
        }
        st.c = threadIdx.x + 1;
        collide_loaded<PARITY, ST, PC, SmemStencil, S.cs>(p, w, mg, st, v, ns);
      }
    }
    slot = slot + 1 < kPipeRingPlanes ? slot + 1 : 0;
    own += plane_nodes;
    mg.next();
  }
}

template <int PARITY, int ST, bool PC, int CFG>
__global__ void __launch_bounds__(CollideShape<PARITY, ST, CFG>::threads,
                                  CollideShape<PARITY, ST, CFG>::s.minb)
    k_collide_pipe(StepParams p, Workspace w, int zc) {
  pipe_block<PARITY, ST, PC, CFG>(p, w, zc, blockIdx.x, blockIdx.y, blockIdx.z);
}

template <int PARITY, int ST, int CFG, bool PC>
__global__ void __launch_bounds__(CollideShape<PARITY, ST, CFG>::threads,
                                  CollideShape<PARITY, ST, CFG>::s.minb)
    k_collide_stream(StepParams p, Workspace w) {
  constexpr Shape S = CollideShape<PARITY, ST, CFG>::s;
  int x, y, z;
  block_coords<S.by, S.bz>(x, y, z);
  const bool maybe_res = block_in_reservoir<S.by, S.bz>(p);
  if (x >= p.nx || y >= p.ny || z >= p.nz) return;
  collide_body<PARITY, ST, PC, S.cs>(p, w, maybe_res, x, y, z);
}

// Macroscopic fields of the current state, linear, x fastest: rho_1, rho_2,
// u_macro (Eq. 7) x, y, z, p (Eq. A.6), those that `out` has a place for.
template <int PARITY, int ST, bool PC>
__global__ void __launch_bounds__(kTile * kFieldsBY * kFieldsBZ)
    k_fields(StepParams p, Workspace w, FieldsOut out) {
  int x, y, z;
  block_coords<kFieldsBY, kFieldsBZ>(x, y, z);
  const bool maybe_res = block_in_reservoir<kFieldsBY, kFieldsBZ>(p);
  if (x >= p.nx || y >= p.ny || z >= p.nz) return;
  const Geo g = make_geo(p, x, y, z);
  float2 v[kQ];
  load_pops<PARITY, ST>(p, w, g, v);
  reservoir_state(p, maybe_res, x, y, z, v);
  const float2 r = sum19(v);
  const float r1 = r.x, r2 = r.y;
  float2 j[3], gf[3];
  first_moment(v, j);
  const float rho = r1 + r2;
  force_per_mass<PC>(p, global_rho(p, w, g), rho, gf);
  int own = g.node(0, 0, 0);
  if (!in_bounds(w.fault, own, p.ntiles * kTile, kFaultGeometry)) own = 0;
  const float fluid = 1.0f - w.ns[own];
  const float fluid2 = PC ? 1.0f - w.ns2[own] : fluid;
  const long long n = x + (long long)p.nx * (y + (long long)p.ny * z);
  if (!in_bounds(w.fault, n, p.nlin, kFaultStage)) return;
  if (out.p[0]) out.p[0][n] = r1;
  if (out.p[1]) out.p[1][n] = r2;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if (!out.p[2 + d]) continue;
    if (PC) {
      const float m = fluid * (j[d].x + 0.5f * r1 * gf[d].x) +
                      fluid2 * (j[d].y + 0.5f * r2 * gf[d].y);
      out.p[2 + d][n] = m / rho;
    } else {
      const float m = (j[d].x + 0.5f * r1 * gf[d].x) + (j[d].y + 0.5f * r2 * gf[d].y);
      out.p[2 + d][n] = fluid * m / rho;
    }
  }
  if (out.p[5]) out.p[5][n] = (rho + p.G * r1 * r2) * (1.0f / 3.0f);
}

// Tiled node index of linear node n = x + nx (y + ny z).
__device__ __forceinline__ long long tiled_of_linear(const StepParams &p,
                                                     long long n) {
  const int x = (int)(n % p.nx);
  const long long yz = n / p.nx;
  return (yz * p.ntx + x / kTile) * kTile + x % kTile;
}

// Populations k0 .. k0 + nk - 1 (k = s * 19 + i) of the current state, decoded,
// in the natural layout: out[k - k0][n], n linear, x fastest.  Blocks as
// k_fields.
template <int PARITY, int ST>
__global__ void __launch_bounds__(kTile * kFieldsBY * kFieldsBZ)
    k_populations(StepParams p, Workspace w, float *__restrict__ out, int k0, int nk) {
  int x, y, z;
  block_coords<kFieldsBY, kFieldsBZ>(x, y, z);
  const bool maybe_res = block_in_reservoir<kFieldsBY, kFieldsBZ>(p);
  if (x >= p.nx || y >= p.ny || z >= p.nz) return;
  const Geo g = make_geo(p, x, y, z);
  float2 v[kQ];
  load_pops<PARITY, ST>(p, w, g, v);
  reservoir_state(p, maybe_res, x, y, z, v);
  const long long N = (long long)p.nx * p.ny * p.nz;
  const long long n = x + (long long)p.nx * (y + (long long)p.ny * z);
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    const int k = i - k0, m = kQ + i - k0;
    if (k >= 0 && k < nk) out[k * N + n] = v[i].x;
    if (m >= 0 && m < nk) out[m * N + n] = v[i].y;
  }
}

// f_i = w_i rho_sigma at rest.  *_LOCAL storages take the initial
// densities as the previous densities of time 0.
template <int ST>
__global__ void k_init_equilibrium(StepParams p, Workspace w,
                                   const float *__restrict__ rho1,
                                   const float *__restrict__ rho2) {
  using C = Codec2<ST>;
  const long long N = (long long)p.nx * p.ny * p.nz;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    const long long tn = tiled_of_linear(p, n);
    if (!in_bounds(w.fault, tn, p.ntiles * kTile, kFaultPopStore)) continue;
    typename C::T2 *b = static_cast<typename C::T2 *>(w.f) + (tn / kTile) * kTilePairs + tn % kTile;
    const float r1 = rho1[n], r2 = rho2[n];
    if (storage_local(ST)) w.rho_enc[tn] = make_float2(r1, r2);
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
      const float2 f = make_float2(__fmul_rn(wgt(i), r1), __fmul_rn(wgt(i), r2));
      // (local: the offset from the node's own density is zero)
      b[i * kTile] = C::enc(f, storage_local(ST) ? mul2(f, pair_of(-C::kScale)) : p.nref[wclass(i)]);
    }
  }
}

// ---- wavefront step: both passes in one persistent launch ----
// The lattice is cut into items: tile T (32 x by nodes of one plane) of
// group g, g = 0 .. nz + lag - 1, numbered group-major and taken by the
// blocks in the order of an atomic ticket.  Item (g, T)
//   - copies the populations of plane q = g - lag of T (if q >= 0) and of
//     plane d(g) = (g - 1) mod nz of T (if g < nz) into shared memory,
//   - waits until the densities of planes q - 1 .. q + 1 of T and of its
//     eight in-plane neighbour tiles are published, then collides and
//     streams plane q of T exactly as k_collide_stream does,
//   - sums the populations of plane d(g) into the density array and
//     publishes them: after a block barrier one thread sets the flag of
//     (d(g), T) to the launch's epoch with a release store.
// The densities a collision of plane q needs come from groups q .. q + 2,
// all before g when lag >= 3, so an item waits only on items with smaller
// tickets; those are held by blocks that are already running, so the launch
// cannot deadlock for any number of resident blocks (every wait is bounded
// all the same, and the launch is cooperative, so every block is resident
// anyway).  The populations of plane q were read from DRAM by the density
// part lag - 1 groups earlier (a group is one plane of the lattice, 10 MB at
// 256^2 in float32) and the collision finds them in L2: one step moves its
// populations through DRAM once instead of twice.  In-place AA streaming
// stays race-free: the collision of node n touches only the slots holding
// n's own populations, whose density part has finished reading them before
// n's flag is set.
// One float32 step of 256^3 takes 1,106 us and moves 335 bytes a node, against
// 1,210 us and 476 in two passes (in scalar operations 1,156).  What bounds it is the chain of each item -- copies from DRAM,
// flags, stencil from L2 -- at 16 warps per SM: fewer instructions (divisions
// as multiplications, copies in chunks) did not shorten it, nor did
// publishing before the collision's stores.
struct WaveCfg {
  int by, minb, minb_local;
};
__host__ __device__ constexpr WaveCfg wave_cfg(int cfg) {
  return cfg == 2 ? WaveCfg{2, 8, 6} : cfg == 3 ? WaveCfg{8, 2, 2} : WaveCfg{4, 4, 3};
}
template <int ST, int CFG>
struct WaveShape {
  static constexpr WaveCfg c = wave_cfg(CFG);
  static constexpr int threads = kTile * c.by;
  static constexpr int minb = storage_local(ST) ? c.minb_local : c.minb;
};
struct WaveArgs {
  unsigned items;       // (nz + lag) * tp
  int tp;               // tiles per plane: ntx * ceil(ny / by)
  int lag;
  unsigned spin_limit;  // polls of one flag before a wait gives up (a few
                        // seconds at the default with the back-off); the item
                        // then goes on and the fault word records kFaultWait
  long long hold;       // a flag the launch leaves unpublished, -1: none
                        // (tests of the failure path)
};

// A flag is set by a release store after a block barrier that follows the
// tile's density stores, and polled with acquire loads: what a lane loads after
// its last poll, and what its warp loads after the __syncwarp behind it, sees
// those densities.  An acquire drops the SM's L1, and with it the stencil's
// cached densities and geometry, once per poll; relaxed polls, which keep it
// and which the memory model gives no order to, are 0.3-1 % faster (us a step:
// 256^3 1,104 and 1,100, 128^3 144.4 and 143.0, 150 x 90 x 70 75.5 and 75.0).
// A fence after relaxed polls also waits for the warp's own stores: 1,175 and
// 156.7.
__device__ __forceinline__ unsigned ld_acquire(const unsigned *ptr) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ptr) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(unsigned *ptr, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(ptr), "r"(v) : "memory");
}

// A wavefront wait that ran out: the fault word records it (and the mapped
// host word, when there is one), and wave[3] names the launch, so that the
// launch's other waits give up at once while later launches wait as usual.
__device__ __forceinline__ void wave_fault(const Workspace &w, unsigned epoch) {
  atomicOr(w.fault, kFaultWait);
  *(volatile unsigned *)&w.wave[3] = epoch;
  if (w.fault_host) *(volatile unsigned *)w.fault_host = kFaultWait;
}

// Densities written earlier in the same launch by other blocks, read after
// their flags (see above): ordinary loads, cached in L1 for the stencil, never
// the read-only path.
struct WaveRho : GlobalRho {
  __device__ __forceinline__ float2 at(int dx, int dy, int dz) const {
    return __ldca(&rho[idx(dx, dy, dz)]);
  }
  __device__ __forceinline__ float2 late(int dx, int dy, int dz) const {
    const float2 *ptr = &rho[idx(dx, dy, dz)];
    float2 v;
    asm volatile("ld.global.ca.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(ptr));
    return v;
  }
};

// One wavefront item: ticket k of the launch's lattice (p, w).  buf is the
// block's two population buffers (this thread's own slots: [b][i][tid]),
// epoch the lattice's launch epoch, hold a flag left unpublished (-1: none;
// failure-path tests).  Ends after a block barrier with the tile's densities
// stored and published and the buffers free.
template <int PARITY, int ST, bool PC, int BY>
__device__ __forceinline__ void wave_tile_item(const StepParams &p, const Workspace &w,
                                               unsigned k, const WaveArgs &a, long long hold,
                                               typename Codec2<ST>::T2 (*buf)[kQ][kTile * BY],
                                               unsigned epoch) {
  using C = Codec2<ST>;
  using T2 = typename C::T2;
  const int tid = threadIdx.y * kTile + threadIdx.x;
  unsigned *ctl = w.wave, *flag = w.wave + kWaveCtlWords;
  const T2 *f = static_cast<const T2 *>(w.f);
  const long long pairs = p.ntiles * kTilePairs, nodes = p.ntiles * kTile;
  const long long nflags = (long long)p.nz * a.tp;
  const int nty = a.tp / p.ntx;
  // populations of node (x, y, z) into buffer b (this thread's own slots)
  auto copy = [&](int x, int y, int z, int b) {
    const Geo g = make_geo(p, x, y, z);
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
      const int slot = PARITY == 0 ? i : opp(i);
      const T2 *src = f + (PARITY == 0 ? g.pop_off(0, 0, 0) : g.pop_off(-cx(i), -cy(i), -cz(i)));
      if (kChecked && !in_bounds(w.fault, (src - f) + slot * kTile, pairs, kFaultPopLoad))
        src = f - slot * kTile;
      cp_async(&buf[b][i][tid], src + slot * kTile);
    }
  };
  auto decode = [&](int b, int own, float2 (&v)[kQ]) {
    const float2 own_prev =
        storage_local(ST)
            ? __ldg(&w.rho_enc[(kChecked && !in_bounds(w.fault, own, nodes, kFaultRhoLoad)) ? 0 : own])
            : make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < kQ; ++i) v[i] = C::dec(buf[b][i][tid], dec_ref<ST>(p, own_prev, i));
  };
  const int grp = (int)(k / (unsigned)a.tp), T = (int)(k % (unsigned)a.tp);
  const int tx = T % p.ntx, ty = T / p.ntx;
  const int x = tx * kTile + threadIdx.x, y = ty * BY + threadIdx.y;
  const bool active = x < p.nx && y < p.ny;
  const int q = grp - a.lag;                     // plane collided, if >= 0
  const int zd = grp == 0 ? p.nz - 1 : grp - 1;  // plane summed, if grp < nz
  const bool has_c = q >= 0, has_d = grp < p.nz;
  const int xlo = tx * kTile, xhi = min(xlo + kTile, p.nx) - 1;
  const int ylo = ty * BY, yhi = min(ylo + BY, p.ny) - 1;
  // one commit group per plane: the collision's first
  if (has_c && active) copy(x, y, q, 0);
  cp_async_commit();
  if (has_d && active) copy(x, y, zd, 1);
  cp_async_commit();
  // every warp waits for the 27 tiles' densities itself
  if (has_c && threadIdx.x < 27) {
    const int l = threadIdx.x;
    const int dx = l % 3 - 1, dy = (l / 3) % 3 - 1, dz = l / 9 - 1;
    const int zz = (q + dz + p.nz) % p.nz, yy = (ty + dy + nty) % nty,
              xx = (tx + dx + p.ntx) % p.ntx;
    long long fi = (long long)zz * a.tp + (long long)yy * p.ntx + xx;
    if (kChecked && !in_bounds(w.fault, fi, nflags, kFaultFlag)) fi = 0;
    // after one wait of this launch has run out the others give up at once
    unsigned n = 0;
    while (ld_acquire(&flag[fi]) != epoch) {
      if (++n == a.spin_limit) {
        wave_fault(w, epoch);
        break;
      }
      if ((n & 255u) == 0 && *(volatile unsigned *)&ctl[3] == epoch) break;
      __nanosleep(64);
    }
  }
  __syncwarp();  // the densities this warp's collisions read are published
  if (has_c && active) {
    cp_async_wait<1>();
    const Geo g = make_geo(p, x, y, q);
    float2 v[kQ];
    decode(0, g.node(0, 0, 0), v);
    reservoir_state(p, box_in_reservoir(p, xlo, xhi, ylo, yhi, q, q), x, y, q, v);
    collide_loaded<PARITY, ST, PC, WaveRho>(p, w, g, WaveRho{global_rho(p, w, g)}, v,
                                            node_ns<PC>(p, w, g));
  }
  cp_async_wait<0>();
  if (has_d && active) {
    const long long own = ((long long)(zd * p.ny + y) * p.ntx + tx) * kTile + threadIdx.x;
    float2 v[kQ];
    decode(1, (int)own, v);
    reservoir_state(p, box_in_reservoir(p, xlo, xhi, ylo, yhi, zd, zd), x, y, zd, v);
    if (in_bounds(w.fault, own, nodes, kFaultRhoStore)) w.rho[own] = sum19(v);
  }
  __syncthreads();  // the tile's densities are stored, the buffers free
  if (has_d && tid == 0) {
    long long fi = (long long)zd * a.tp + T;
    if (fi != hold && (!kChecked || in_bounds(w.fault, fi, nflags, kFaultFlag)))
      st_release(&flag[fi], epoch);
  }
}

// The last block out resets the ticket and done counter (in ctl) and
// advances the epoch of each of the launch's n lattices (ctls[l][2]) for
// the next launch.
__device__ __forceinline__ void wave_exit(unsigned *ctl, unsigned *const *ctls, int n) {
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    __threadfence();
    if (atomicAdd(&ctl[1], 1u) == gridDim.x - 1) {
      volatile unsigned *vc = ctl;
      vc[0] = 0u;
      vc[1] = 0u;
      for (int l = 0; l < n; ++l) {
        volatile unsigned *e = ctls[l];
        e[2] = e[2] + 1u;
      }
      __threadfence();
    }
  }
}

template <int PARITY, int ST, bool PC, int CFG>
__global__ void __launch_bounds__(WaveShape<ST, CFG>::threads, WaveShape<ST, CFG>::minb)
    k_wave(StepParams p, Workspace w, WaveArgs a) {
  using T2 = typename Codec2<ST>::T2;
  constexpr int BY = WaveShape<ST, CFG>::c.by, NT = kTile * BY;
  extern __shared__ __align__(16) unsigned char wave_smem[];
  T2(*buf)[kQ][NT] = reinterpret_cast<T2(*)[kQ][NT]>(wave_smem);  // [0] collision, [1] density
  __shared__ unsigned s_ticket[2], s_epoch;
  const int tid = threadIdx.y * kTile + threadIdx.x;
  unsigned *ctl = w.wave;
  if (tid == 0) {
    s_epoch = *(volatile unsigned *)&ctl[2] + 1u;
    s_ticket[0] = atomicAdd(&ctl[0], 1u);
  }
  __syncthreads();
  const unsigned epoch = s_epoch;
  unsigned k = s_ticket[0];
  int it = 0;
  while (k < a.items) {
    it ^= 1;
    if (tid == 0) s_ticket[it] = atomicAdd(&ctl[0], 1u);  // next item, read at the end
    wave_tile_item<PARITY, ST, PC, BY>(p, w, k, a, a.hold, buf, epoch);
    k = s_ticket[it];
  }
  unsigned *ctls[1] = {ctl};
  wave_exit(ctl, ctls, 1);
}

// ---- single-pass step: density and fused pass in one sweep ----
//
// The two-pass step reads every population twice (160 B/node for the
// density pass).  A single sweep must know the densities of a node's
// neighbours before it collides the node, and a block cannot recompute a
// neighbour's density from that neighbour's populations if another block may
// already have updated them in place.  So the lattice is cut into boxes of
// full x-rows: rows [y0, y0 + kSpBY) and nzc runs of planes along z (run c
// covers [c nz / nzc, (c + 1) nz / nzc), so runs differ by one plane at
// most and the grid is nyb x nzc boxes, a number the host can fit to the
// SM count).  The last row
// and the last plane of every box are seams.  One launch (k_sp_bulk) marches
// each box along z; per plane it computes the densities of the next plane --
// its own rows plus the seam row of the box below -- into a shared-memory
// ring of four planes, and collides the plane's bulk rows with the force
// stencil read from the ring.  Every density a box needs belongs to one of
// its own nodes (computed before that node is updated) or to a seam of
// another box (not updated by this launch).  Each box writes the densities of
// its own nodes to the density array; a second launch (k_sp_seams) then
// updates the seam rows and planes with the two-pass code, reading the
// completed array.  In-place AA streaming keeps every write of a node inside
// that node's own (slot, node) set, so no update disturbs another node's
// reads.  Results are bit-identical to the two-pass step (same densities,
// same arithmetic).
constexpr int kSpBY = 8;            // rows per box, the last one a seam
constexpr int kSpMaxThreads = 256;  // one thread per x: nx <= 256
constexpr int kSpRingPlanes = 4;

// First plane of run c of nzc runs along nz planes.
__host__ __device__ __forceinline__ int sp_run_start(int c, int nz, int nzc) {
  return (int)(((long long)c * nz) / nzc);
}

__host__ __device__ constexpr size_t sp_ring_bytes(int ncol) {
  return sizeof(float2) * kSpRingPlanes * (kSpBY + 1) * (size_t)ncol;
}

// Densities of x +- 1, y +- 1, z +- 1 from the ring.
struct RingRho {
  const float2 *row[3];  // ring row of the node's y in planes z - 1, z, z + 1
  int stride;            // one ring row (columns)
  int xm, xc, xp;        // columns of x - 1, x, x + 1 (periodic)
  const float2 *base;    // the ring and its length (bounds-checked builds)
  long long size;
  unsigned *fault;
  const GlobalRho *glob; // adhesion sources come from global memory
  __device__ __forceinline__ float2 at(int dx, int dy, int dz) const {
    const float2 *q = row[dz + 1] + dy * stride + (dx < 0 ? xm : (dx > 0 ? xp : xc));
    if (kChecked && !in_bounds(fault, q - base, size, kFaultShared)) q = base;
    return *q;
  }
  __device__ __forceinline__ float2 late(int dx, int dy, int dz) const {
    return at(dx, dy, dz);
  }
  __device__ __forceinline__ float a1(int dx, int dy, int dz) const {
    return glob->a1(dx, dy, dz);
  }
  __device__ __forceinline__ float a2(int dx, int dy, int dz) const {
    return glob->a2(dx, dy, dz);
  }
  template <bool PC>
  __device__ __forceinline__ void adhesion(float2 (&A)[3]) const {
    adhesion_sum<PC>(*this, A);
  }
};

// Density pair of node (x, y, z) at the current step.
template <int PARITY, int ST>
__device__ __forceinline__ float2 node_density(const StepParams &p, const Workspace &w,
                                               const Geo &g, int x, int y, int z) {
  float2 v[kQ];
  load_pops<PARITY, ST>(p, w, g, v);
  reservoir_state(p, p.res.any != 0, x, y, z, v);
  return sum19(v);
}

template <int PARITY, int ST, bool PC>
__global__ void __launch_bounds__(kSpMaxThreads, 2)
    k_sp_bulk(StepParams p, Workspace w, int nzc) {
  extern __shared__ float2 ring[];  // [kSpRingPlanes][kSpBY + 1][ncol]
  const int ncol = blockDim.x;
  const int x = threadIdx.x;
  const bool active = x < p.nx;
  const int y0 = blockIdx.x * kSpBY, yend = min(y0 + kSpBY, p.ny);
  const int nr = yend - y0;  // own rows; ring row r <-> y0 - 1 + r
  const int z0 = sp_run_start(blockIdx.y, p.nz, nzc);
  const int zend = sp_run_start(blockIdx.y + 1, p.nz, nzc);
  const int plane_stride = (kSpBY + 1) * ncol;

  // densities of relative plane k (z = z0 - 1 + k) into ring slot k % 4;
  // own nodes (rows 1..nr, planes z0..zend-1) also go to the density array
  auto rho_plane = [&](int k) {
    int z = z0 - 1 + k;
    const bool own_plane = k >= 1;
    if (z < 0) z += p.nz;
    float2 *dst = ring + (k & 3) * plane_stride;
    if (!active) return;
#pragma unroll 2
    for (int r = 0; r <= nr; ++r) {
      int y = y0 - 1 + r;
      if (y < 0) y += p.ny;
      const Geo g = make_geo(p, x, y, z);
      const float2 rho = node_density<PARITY, ST>(p, w, g, x, y, z);
      if (in_bounds(w.fault, (dst - ring) + r * ncol + x,
                    (long long)kSpRingPlanes * plane_stride, kFaultShared))
        dst[r * ncol + x] = rho;
      const int own = g.node(0, 0, 0);
      if (own_plane && r >= 1 && in_bounds(w.fault, own, p.ntiles * kTile, kFaultRhoStore))
        w.rho[own] = rho;
    }
  };

  rho_plane(0);
  rho_plane(1);
  const int xm = x == 0 ? p.nx - 1 : x - 1;
  const int xp = x == p.nx - 1 ? 0 : x + 1;
  for (int j = 0; j + 1 < zend - z0; ++j) {
    rho_plane(j + 2);
    __syncthreads();
    if (!active) continue;
    const int z = z0 + j;
    for (int r = 1; r < nr; ++r) {
      const int y = y0 - 1 + r;
      const Geo g = make_geo(p, x, y, z);
      RingRho rr;
      rr.row[0] = ring + (j & 3) * plane_stride + r * ncol;
      rr.row[1] = ring + ((j + 1) & 3) * plane_stride + r * ncol;
      rr.row[2] = ring + ((j + 2) & 3) * plane_stride + r * ncol;
      rr.stride = ncol;
      rr.xm = xm;
      rr.xc = x;
      rr.xp = xp;
      rr.base = ring;
      rr.size = (long long)kSpRingPlanes * plane_stride;
      rr.fault = w.fault;
      const GlobalRho glob = global_rho(p, w, g);
      rr.glob = &glob;
      collide_node<PARITY, ST, PC>(p, w, g, rr, p.res.any != 0, x, y, z);
    }
  }
}

// Seam rows of every box (all planes), then seam planes of every box (the
// rows that are not seam rows): the two-pass fused update with the density
// array the bulk launch completed.  Blocks of 32 x 4 threads.
template <int PARITY, int ST, bool PC>
__global__ void __launch_bounds__(kTile * 4, 4)
    k_sp_seams(StepParams p, Workspace w, int nzc, int part) {
  const int x = blockIdx.x * kTile + threadIdx.x;
  int y, z;
  if (part == 0) {
    y = min(blockIdx.y * kSpBY + kSpBY - 1, p.ny - 1);
    z = blockIdx.z * 4 + threadIdx.y;
    if (z >= p.nz) return;
  } else {
    y = blockIdx.y * 4 + threadIdx.y;
    z = sp_run_start(blockIdx.z + 1, p.nz, nzc) - 1;
    if (y >= p.ny) return;
    const int yseam = min((y / kSpBY) * kSpBY + kSpBY - 1, p.ny - 1);
    if (y == yseam) return;
  }
  if (x >= p.nx) return;
  collide_body<PARITY, ST, PC>(p, w, p.res.any != 0, x, y, z);
}

// ---- batched kernels: several lattices per launch ----

__device__ __forceinline__ int batch_item_of_block(const BatchArgs &a) {
  int lo = 0, hi = a.n - 1;
  const int b = blockIdx.x;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (a.prefix[mid] <= b) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Node coordinates of this thread inside its item; false for padding.
__device__ __forceinline__ bool batch_coords(const BatchArgs &a, int &r, int &x,
                                             int &y, int &z, bool &maybe_res) {
  r = batch_item_of_block(a);
  const BatchItem &it = a.item[r];
  const int lb = blockIdx.x - a.prefix[r];
  const int bx = lb % it.gx, rest = lb / it.gx;
  const int by = rest % it.gy, bz = rest / it.gy;
  x = bx * kTile + threadIdx.x;
  y = by * kBatchBY + threadIdx.y;
  z = bz;
  maybe_res = box_in_reservoir(it.p, bx * kTile, min(bx * kTile + kTile, it.p.nx) - 1,
                               by * kBatchBY, min(by * kBatchBY + kBatchBY, it.p.ny) - 1,
                               z, z);
  return x < it.p.nx && y < it.p.ny;
}

template <int ST>
__global__ void __launch_bounds__(kTile * kBatchBY)
    k_batch_density(const __grid_constant__ BatchArgs a) {
  int r, x, y, z;
  bool maybe_res;
  if (!batch_coords(a, r, x, y, z, maybe_res)) return;
  const BatchItem &it = a.item[r];
  const Geo g = make_geo(it.p, x, y, z);
  float2 v[kQ];
  if (it.parity == 0)
    load_pops<0, ST>(it.p, it.w, g, v);
  else
    load_pops<1, ST>(it.p, it.w, g, v);
  reservoir_state(it.p, maybe_res, x, y, z, v);
  const int own = g.node(0, 0, 0);
  if (in_bounds(it.w.fault, own, it.p.ntiles * kTile, kFaultRhoStore)) it.w.rho[own] = sum19(v);
}

// All items of one launch have per-component fractions (PC) or none do.
template <int ST, bool PC>
__global__ void __launch_bounds__(kTile * kBatchBY, CollideShape<1, ST, 0>::s.minb)
    k_batch_collide(const __grid_constant__ BatchArgs a) {
  int r, x, y, z;
  bool maybe_res;
  if (!batch_coords(a, r, x, y, z, maybe_res)) return;
  const BatchItem &it = a.item[r];
  if (it.parity == 0)
    collide_body<0, ST, PC>(it.p, it.w, maybe_res, x, y, z);
  else
    collide_body<1, ST, PC>(it.p, it.w, maybe_res, x, y, z);
}

// Blocks per SM the batched prefetching pass is compiled for: those of the
// single-lattice kernel, except the local storages' odd step in shape 9,
// which runs faster held to 8 blocks (128 registers, no spill) than at 6:
// 567 against 576 us a step over twelve lattices of 36^3 .. 160^3.
template <int PARITY, int ST, int CFG>
__host__ __device__ constexpr int batch_pipe_minb() {
  return (storage_local(ST) && PARITY == 1 && CFG == 9) ? 8
                                                        : CollideShape<PARITY, ST, CFG>::s.minb;
}

// The prefetching fused pass over a batch of lattices at one AA parity:
// item r's blocks (prefix[r] .. prefix[r + 1]) tile its lattice as
// k_collide_pipe's grid does for shape CFG (gx x-tiles, gy row groups, runs
// of its zc planes), and each block runs that kernel's body on its lattice.
template <int PARITY, int ST, bool PC, int CFG>
__global__ void __launch_bounds__(CollideShape<PARITY, ST, CFG>::threads,
                                  batch_pipe_minb<PARITY, ST, CFG>())
    k_batch_collide_pipe(const __grid_constant__ BatchArgs a) {
  const int r = batch_item_of_block(a);
  const BatchItem &it = a.item[r];
  const int lb = blockIdx.x - a.prefix[r];
  const int rest = lb / it.gx;
  pipe_block<PARITY, ST, PC, CFG>(it.p, it.w, it.zc, lb % it.gx, rest % it.gy, rest / it.gy);
}

}  // namespace
}  // namespace hmcsc
