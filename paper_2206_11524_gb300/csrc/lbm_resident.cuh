// lbm_resident.cuh -- several time steps of a small lattice in one launch.
//
// A small lattice is bound by latency: the two launches of a step take 8 us
// for 500 nodes, whose arithmetic takes well under one.  Here the blocks stay
// for all the steps of the launch: per step a warp sums the densities of its
// x-tiles, meets a barrier of the whole grid, collides and streams them, and
// meets it again.  The sums and collisions are those of the two passes, so
// the results are bit-identical.  (Times: us a step, float32, two passes and
// here.)
//
//   k_cluster   up to kClusterTiles x-tiles: one tile per warp, one cluster,
//               the populations and densities in its shared memory for the
//               whole launch, neighbours read and written across the
//               cluster, the hardware's cluster barrier.  500 x 1 x 1 nodes
//               8.2, 1.3 (state in L2 instead: 4.1), 50 x 50 9.4, 1.8,
//               64 x 64 9.7, 1.8.
//   k_resident  up to kResidentTiles: the state in the workspace (L2), a
//               counter in the workspace as barrier, cooperative.  32 x 16 x
//               16 10.3, 4.4, 32^3 10.3, 5.5, 48^3 14.4, 13.3; beyond that the
//               two passes win (64^3 21.5, 21.8, 80^3 39.5, 47).
//
// k_resident is for one lattice at a time: its blocks of eight warps at 204-254
// registers leave no room for another's on an SM, so lattices of more than some
// 600 tiles on streams of their own take turns, where the passes of several
// overlap (eight lattices, us per lattice step, here and in two passes: 32^3
// 5.6, 2.9, 40^3 10.8, 7.3, 48^3 13.6, 11.4, 200 x 200 x 1 7.4, 3.0).  Held to
// 128 registers two fit (32^3 3.8, 48^3 8.9), but one alone then takes 7 %
// longer in float32 and 15-25 % in the local storages.
#pragma once
#include "lbm_device.cuh"

namespace hmcsc {
namespace {

constexpr int kResidentWarps = 8;  // most warps per block
constexpr int kResidentCtl = 8;    // control words [8] arrivals, [9] blocks done

struct ResidentArgs {
  int parity;           // AA parity of the first step
  int steps;
  unsigned spin_limit;  // polls of the counter before a wait gives up
  int hold;             // 1: block 0 stays away from the first barrier (tests
                        // of the failure path)
};

// Everything before it, in every thread of the grid, comes before everything
// after it; false when the wait ran out.  Arrivals are release adds and one
// thread of each block polls with acquire loads, between block barriers, so
// the loads that follow are ordinary ones -- but never the read-only path:
// densities and populations change during the launch.
__device__ __forceinline__ bool resident_barrier(const Workspace &w, const ResidentArgs &a,
                                                 unsigned &target, bool &ok) {
  __syncthreads();
  target += gridDim.x;
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    unsigned *count = w.wave + kResidentCtl;
    if (!(a.hold && blockIdx.x == 0 && target == gridDim.x))
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    unsigned v, n = 0;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
    } while ((int)(v - target) < 0 && ++n < a.spin_limit);
    ok = (int)(v - target) >= 0;
  }
  __syncthreads();
  return ok;
}

// One step of this warp's tiles.
template <int PARITY, int ST, bool PC>
__device__ __forceinline__ bool resident_step(const StepParams &p, const Workspace &w,
                                              const ResidentArgs &a, unsigned &target, bool &ok) {
  const int first = blockIdx.x * blockDim.y + warp_ty();
  const int stride = gridDim.x * blockDim.y;
  const int tiles = (int)p.ntiles;
  float2 v[kQ];
  int x = 0, y = 0, z = 0;
  bool maybe = false;
  auto place = [&](int t) {
    const int yz = t / p.ntx, xlo = (t - yz * p.ntx) * kTile;
    x = xlo + threadIdx.x;
    z = yz / p.ny;
    y = yz - z * p.ny;
    maybe = box_in_reservoir(p, xlo, min(xlo + kTile, p.nx) - 1, y, y, z, z);
  };
  // the first tile last, so that v holds it at the barrier
  for (int t = first + (tiles - 1 - first) / stride * stride; t >= first; t -= stride) {
    if (first >= tiles) break;
    place(t);
    if (x >= p.nx) continue;
    const Geo g = make_geo(p, x, y, z);
    load_pops<PARITY, ST, true>(p, w, g, v);
    reservoir_state(p, maybe, x, y, z, v);
    const int own = g.node(0, 0, 0);
    if (in_bounds(w.fault, own, p.ntiles * kTile, kFaultRhoStore)) w.rho[own] = sum19(v);
  }
  if (!resident_barrier(w, a, target, ok)) return false;
  for (int t = first; t < tiles; t += stride) {
    place(t);
    if (x >= p.nx) continue;
    const Geo g = make_geo(p, x, y, z);
    if (t != first) {
      load_pops<PARITY, ST, true>(p, w, g, v);
      reservoir_state(p, maybe, x, y, z, v);
    }
    collide_loaded<PARITY, ST, PC, WaveRho>(p, w, g, WaveRho{global_rho(p, w, g)}, v,
                                            node_ns<PC>(p, w, g));
  }
  return true;
}

template <int ST, bool PC>
__global__ void __launch_bounds__(kTile * kResidentWarps, 1)
    k_resident(const __grid_constant__ StepParams p, Workspace w, ResidentArgs a) {
  __shared__ bool s_ok;
  unsigned target = 0;
  bool fine = true;
  for (int s = 0; s < a.steps && fine; ++s) {
    fine = ((a.parity + s) & 1) == 0 ? resident_step<0, ST, PC>(p, w, a, target, s_ok)
                                     : resident_step<1, ST, PC>(p, w, a, target, s_ok);
    if (storage_local(ST)) {  // this step's densities are the next one's references
      float2 *const r = w.rho;
      w.rho = w.rho_enc;
      w.rho_enc = r;
    }
    if (fine && s + 1 < a.steps) fine = resident_barrier(w, a, target, s_ok);
  }
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    if (!fine) {
      atomicOr(w.fault, kFaultWait);
      if (w.fault_host) *(volatile unsigned *)w.fault_host = kFaultWait;
    }
    unsigned *ctl = w.wave + kResidentCtl;
    __threadfence();
    if (atomicAdd(&ctl[1], 1u) == gridDim.x - 1) {  // the last block out: ready for the next launch
      volatile unsigned *c = ctl;
      c[0] = 0u;
      c[1] = 0u;
    }
  }
}


// ---- one tile per warp, the state in the shared memory of one cluster ----
// Up to 8 warps a block: 16 (128 registers, spills) run 2.1 instead of 1.8 us
// a step on 64 x 64, and 256 tiles 4.9, bound by the traffic between blocks.
constexpr int kClusterWarps = 8;    // most warps (tiles) of a block
constexpr int kClusterBlocks = 16;  // most blocks of the cluster
constexpr int kClusterTiles = kClusterWarps * kClusterBlocks;

// A tile of the lattice in shared memory.
template <typename T2>
struct ClusterTile {
  T2 pop[kQ][kTile];
  float2 rho[kTile];
};

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// address of a shared-memory location of this block in block `rank`
__device__ __forceinline__ unsigned cluster_map(unsigned local, unsigned rank) {
  unsigned a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
  return a;
}
template <typename T2>
__device__ __forceinline__ T2 ld_cluster(unsigned addr) {
  T2 v;
  if constexpr (sizeof(T2) == 8) {
    float2 f;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(f.x), "=f"(f.y) : "r"(addr));
    memcpy(&v, &f, 8);
  } else {
    unsigned u;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(u) : "r"(addr));
    memcpy(&v, &u, 4);
  }
  return v;
}
template <typename T2>
__device__ __forceinline__ void st_cluster(unsigned addr, T2 v) {
  if constexpr (sizeof(T2) == 8) {
    float2 f;
    memcpy(&f, &v, 8);
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(f.x), "f"(f.y)
                 : "memory");
  } else {
    unsigned u;
    memcpy(&u, &v, 4);
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(u) : "memory");
  }
}
__device__ __forceinline__ void cluster_barrier(bool one) {
  __syncwarp();
  if (one) {
    __syncthreads();
  } else {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

// Where the neighbours' slots and densities lie in the cluster, and the
// node's own adhesion sums, which never change.
template <typename T2>
struct ClusterNode {
  unsigned addr[3][3][3];  // slot 0 of node x + (dx, dy, dz)
  unsigned to_rho[3];      // from there to the node's density, for dx = -1, 0, 1
  float2 A[3];
  __device__ __forceinline__ float2 at(int dx, int dy, int dz) const {
    return ld_cluster<float2>(addr[dx + 1][dy + 1][dz + 1] + to_rho[dx + 1]);
  }
  template <bool PC>
  __device__ __forceinline__ void adhesion(float2 (&a)[3]) const {
#pragma unroll
    for (int d = 0; d < 3; ++d) a[d] = A[d];
  }
};

template <int PARITY, int ST, bool PC>
__device__ __forceinline__ void cluster_step(const StepParams &p, ClusterTile<typename Codec2<ST>::T2> &tile,
                                             const ClusterNode<typename Codec2<ST>::T2> &nb,
                                             bool active, bool maybe, int x, int y, int z,
                                             float2 ns, float2 &own_rho, bool one) {
  using C = Codec2<ST>;
  using T2 = typename C::T2;
  constexpr unsigned kRow = kTile * sizeof(T2);
  const int lane = threadIdx.x;
  float2 v[kQ];
  if (active) {
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
      const T2 raw = PARITY == 0 || i == 0
                         ? tile.pop[i][lane]
                         : ld_cluster<T2>(nb.addr[1 - cx(i)][1 - cy(i)][1 - cz(i)] + opp(i) * kRow);
      v[i] = C::dec(raw, dec_ref<ST>(p, own_rho, i));
    }
    reservoir_state(p, maybe, x, y, z, v);
    own_rho = sum19(v);
    tile.rho[lane] = own_rho;
  }
  cluster_barrier(one);
  if (active) {
    float2 o[kQ];
    collide_core<PC>(p, nb, v, ns, [&](int i, float2 out, float2) { o[i] = out; });
    // all destination densities before the first store: a load does not pass
    // a store, and each takes a trip through the cluster
    float2 dest[kQ];
#pragma unroll
    for (int i = 0; i < kQ; ++i)
      dest[i] = storage_local(ST) && i != 0 ? nb.at(cx(i), cy(i), cz(i)) : own_rho;
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
      const T2 e = encode<ST>(p, i, o[i], dest[i]);
      if (PARITY == 0 || i == 0)
        tile.pop[opp(i)][lane] = e;
      else
        st_cluster(nb.addr[1 + cx(i)][1 + cy(i)][1 + cz(i)] + i * kRow, e);
    }
  }
  cluster_barrier(one);
}

template <int ST, bool PC>
__global__ void __launch_bounds__(kTile * kClusterWarps, 1)
    k_cluster(const __grid_constant__ StepParams p, const __grid_constant__ Workspace w,
              int parity, int steps) {
  using T2 = typename Codec2<ST>::T2;
  using Tile = ClusterTile<T2>;
  extern __shared__ __align__(16) unsigned char cluster_smem[];
  Tile *tiles = reinterpret_cast<Tile *>(cluster_smem);
  const int W = blockDim.y, lane = threadIdx.x;
  const int t = (int)cluster_rank() * W + threadIdx.y;
  const bool one = gridDim.x == 1;
  const bool row = t < (int)p.ntiles;
  const int yz = t / p.ntx, xlo = (t - yz * p.ntx) * kTile;
  const int x = xlo + lane, z = yz / p.ny, y = yz - z * p.ny;
  const bool active = row && x < p.nx;
  const bool maybe =
      row && box_in_reservoir(p, xlo, min(xlo + kTile, p.nx) - 1, y, y, z, z);
  Tile &tile = tiles[threadIdx.y];
  T2 *f = static_cast<T2 *>(w.f) + (long long)t * kTilePairs + lane;
  const int own = t * kTile + lane;
  ClusterNode<T2> nb;
  float2 ns = pair_of(0.0f), own_rho = pair_of(0.0f);
  if (row)
#pragma unroll
    for (int i = 0; i < kQ; ++i) tile.pop[i][lane] = f[i * kTile];
  if (active) {
    const Geo g = make_geo(p, x, y, z);
    ns = node_ns<PC>(p, w, g);
    if (storage_local(ST)) own_rho = w.rho_enc[own];
    global_rho(p, w, g).template adhesion<PC>(nb.A);
    const unsigned base = (unsigned)__cvta_generic_to_shared(tiles);
#pragma unroll
    for (int d = 0; d < 3; ++d)
      nb.to_rho[d] = (unsigned)(sizeof(T2) * kTilePairs) + g.lane(d - 1) * (unsigned)(8 - sizeof(T2));
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
      int n = g.tile(cx(i), cy(i), cz(i));
      if (!in_bounds(w.fault, n, p.ntiles, kFaultShared)) n = 0;
      nb.addr[1 + cx(i)][1 + cy(i)][1 + cz(i)] =
          cluster_map(base + (unsigned)(n % W) * (unsigned)sizeof(Tile) +
                          g.lane(cx(i)) * (unsigned)sizeof(T2),
                      (unsigned)(n / W));
    }
  }
  cluster_barrier(one);
  for (int s = 0; s < steps; ++s) {
    if (((parity + s) & 1) == 0)
      cluster_step<0, ST, PC>(p, tile, nb, active, maybe, x, y, z, ns, own_rho, one);
    else
      cluster_step<1, ST, PC>(p, tile, nb, active, maybe, x, y, z, ns, own_rho, one);
  }
  if (row)
#pragma unroll
    for (int i = 0; i < kQ; ++i) f[i * kTile] = tile.pop[i][lane];
  // the last step's densities, in the buffer that step would have written
  if (active) (storage_local(ST) && steps % 2 == 0 ? w.rho_enc : w.rho)[own] = own_rho;
}

}  // namespace
}  // namespace hmcsc
