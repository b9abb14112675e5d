// Lattices that stay in shared memory for many time steps.
//
// A small lattice advanced by one launch per step is bound by latency: a 64 x
// 64 step moves 0.9 MB through L2 but takes the launch, the cold start of its
// blocks and the boundary nodes' chain of loads, 5.0 us (1.9 us here; 128 x
// 128 FP32 2.3; 256 batched obstacle cavities of 64 x 64 66 -> 28 us).  Here a cluster of up
// to sixteen thread blocks holds both states of the lattice in shared memory
// (each block a band of rows with a ghost row on either side), takes any
// number of steps with one cluster barrier each, and writes the last two
// states back.  Rows that a neighbouring band reads are stored twice, once
// locally and once into the neighbour's ghost row through distributed shared
// memory, so every load is local.
//
// Nodes are kept whole (ST consecutive values a node, ST chosen so that 32
// consecutive nodes fall into different banks): one address and immediate
// offsets reach all populations of a neighbour, which spares the address
// arithmetic of 28 planes.  Boundary nodes (the list of the plane kernels)
// have warps of their own, so that interior warps stay convergent (128 x 128
// 3.0 -> 2.3 us).  A step is then as long as the chain load - collide - store
// - cluster barrier of one block; arriving at the barrier early and waiting
// late made it longer (2.3 -> 2.65 us), as did fewer threads and more blocks
// a multiprocessor (256 batched obstacle cavities 33 -> 34 .. 47 us).
#pragma once

namespace clbm {

// Values from one node to the next: 15 words of 4 or 8 bytes (odd, so free of
// bank conflicts), 14 or 18 halves (7 or 9 words).
template <typename S, bool VH>
__host__ __device__ constexpr int node_stride() {
  return sizeof(S) == 2 ? (VH ? 18 : 14) : 15;
}

// A boundary node in shared memory: column, local row, plane index, flags, link table entry.
struct ResNode {
  unsigned short x, y;
  int gi;
  uint32_t fl;
  int slot;
};

__host__ __device__ constexpr size_t align16(size_t n) { return (n + 15) / 16 * 16; }

// Shared memory of a block: descriptor, node flags, boundary nodes (at most nb), two states of
// rows + 2 rows.
template <typename S>
__host__ __device__ inline size_t resident_bytes(int nx, int rows, int nb, bool vh) {
  const size_t nodes = (size_t)nx * (rows + 2);
  const size_t st = vh ? node_stride<S, true>() : node_stride<S, false>();
  return align16(sizeof(ResLat)) + align16(nodes) + align16((size_t)nb * sizeof(ResNode)) +
         2 * align16(nodes * st * sizeof(S));
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of the same shared-memory location in block `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const void* p, uint32_t rank) {
  uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
template <typename S>
__device__ __forceinline__ void st_cluster(uint32_t addr, S v) {
  if constexpr (sizeof(S) == 8) {
    asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(addr), "l"(__double_as_longlong(v)) : "memory");
  } else if constexpr (sizeof(S) == 4) {
    asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(addr), "r"(__float_as_uint(v)) : "memory");
  } else {
    unsigned short u;
    memcpy(&u, &v, 2);
    asm volatile("st.shared::cluster.b16 [%0], %1;" ::"r"(addr), "h"(u) : "memory");
  }
}

// A value rounded to storage as st1 rounds it.
template <typename S, typename R>
__device__ __forceinline__ S round1(R v, int stochastic, uint32_t key, int q, int sub) {
  if constexpr (sizeof(S) == 2) {
    if (stochastic) {
      uint32_t r0, r1;
      sr_words(key, q, r0, r1);
      const uint32_t w = (sub & 2) ? r1 : r0;
      const unsigned short u = (sub & 1) ? (unsigned short)(cvt_rs2<S>(0.0f, v, w) >> 16)
                                         : (unsigned short)(cvt_rs2<S>(v, 0.0f, w) & 0xFFFFu);
      S o;
      memcpy(&o, &u, 2);
      return o;
    }
  }
  return from_r<S, R>(v);
}

// Rows of band r of cl.
__host__ __device__ __forceinline__ int band_start(int r, int cl, int ny) { return (int)((long long)r * ny / cl); }

// One cluster of a.cl blocks per lattice, a.steps steps.
template <typename S, bool VH>
__global__ void __launch_bounds__(kMaxResidentThreads, 1) resident_kernel(const __grid_constant__ ResArgs a) {
  using R = typename Traits<S>::R;
  constexpr int ST = node_stride<S, VH>();
  extern __shared__ __align__(16) uint8_t resident_smem[];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int cl = a.cl, rank = (int)cluster_rank();
  const ResLat* from = a.lats ? a.lats + blockIdx.x / cl : &a.one;
  if (a.active && !a.active[from->lat]) return;  // the whole cluster
  ResLat& L = *reinterpret_cast<ResLat*>(resident_smem);
  {
    static_assert(sizeof(ResLat) % 8 == 0, "descriptor is copied in 8-byte words");
    const unsigned long long* f = reinterpret_cast<const unsigned long long*>(from);
    unsigned long long* t = reinterpret_cast<unsigned long long*>(&L);
    for (int k = tid; k < (int)(sizeof(ResLat) / 8); k += nt) t[k] = f[k];
  }
  __syncthreads();
  const int nx = L.L.g.nx, ny = L.L.g.ny, gpitch = L.L.g.pitch, py = L.L.g.py;
  const long long gplane = L.L.g.plane;
  const uint16_t* gflags = L.L.g.flags;
  const bool masked = gflags != nullptr;
  const int row0 = band_start(rank, cl, ny), rows = band_start(rank + 1, cl, ny) - row0;
  const int nb0 = L.bn_off[rank], nb = L.bn_off[rank + 1] - nb0;
  const int32_t* bnodes = L.bnodes + nb0;
  const int cap_nb = L.bn_most;  // same layout in every block
  __syncthreads();
  if (tid == 0) {  // the band as a slab: own rows 1 .. rows between two ghost rows
    DevGeom& g = L.L.g;
    g.ywlo = !py && rank == 0;
    g.ywhi = !py && rank == cl - 1;
    g.ny = rows + 2;
    g.ylo = 1;
    g.yhi = rows + 1;
    g.pitch = nx;
    g.py = 0;
  }
  const int maxrows = (ny + cl - 1) / cl;  // same layout in every block
  const int nodes = nx * (rows + 2), cap = nx * (maxrows + 2);
  uint8_t* kind = resident_smem + align16(sizeof(ResLat));
  ResNode* edge = reinterpret_cast<ResNode*>(kind + align16(cap));
  S* buf0 = reinterpret_cast<S*>(reinterpret_cast<uint8_t*>(edge) + align16((size_t)cap_nb * sizeof(ResNode)));
  S* buf1 = reinterpret_cast<S*>(reinterpret_cast<uint8_t*>(buf0) + align16((size_t)cap * ST * sizeof(S)));
  for (int k = tid; k < nb; k += nt) {
    const int gi = bnodes[k], gy = gi / gpitch;
    const uint32_t fl = masked ? (uint32_t)gflags[gi] : 0u;
    edge[k] = ResNode{(unsigned short)(gi - gy * gpitch), (unsigned short)(gy - row0 + 1), gi, fl,
                      (fl & kFlagLinks) ? L.L.g.slot[gi] : 0};
  }

  // Whether the node across a band's edge (row gy, around the seam) or one beside it has walls: its
  // wall rules may then read the whole node here, not only what streams across.
  auto walls_near = [&](int gy, int x) {
    if (!masked) return false;
    if (py) gy = gy < 0 ? gy + ny : (gy >= ny ? gy - ny : gy);
    if (gy < 0 || gy >= ny) return false;
    bool any = false;
    for (int dx = -1; dx <= 1; ++dx) {
      const int xx = x + dx < 0 ? nx - 1 : (x + dx >= nx ? 0 : x + dx);
      any = any || (gflags[(long long)gy * gpitch + xx] & 0xFFu);
    }
    return any;
  };
  // the current state with its ghost rows, and what each node is: bit 0 solid, bit 1 boundary,
  // bits 2, 3 the band below / above reads all of it
  const S* in = static_cast<const S*>(L.L.buf[a.cur]);
  for (int i = tid; i < nodes; i += nt) {
    const int yl = i / nx, x = i - yl * nx;
    int gy = row0 + yl - 1;
    if (py) gy = gy < 0 ? gy + ny : (gy >= ny ? gy - ny : gy);
    uint8_t kd = 0;
    if (gy >= 0 && gy < ny) {
      const long long gi = (long long)gy * gpitch + x;
      const uint16_t fl = masked ? gflags[gi] : (uint16_t)0;
      if (fl & kFlagSolid) kd = 1;
      if (x == 0 || x == nx - 1 || (!py && (gy == 0 || gy == ny - 1)) || (fl & 0xFFu)) kd |= 2;
      if (yl == 1 && walls_near(gy - 1, x)) kd |= 4;
      if (yl == rows && walls_near(gy + 1, x)) kd |= 8;
      S* o = buf0 + i * ST;
#pragma unroll
      for (int q = 0; q < (VH ? 15 : 14); ++q) o[q] = in[q * gplane + gi];
    }
    kind[i] = kd;
  }
  const Co<R> c = make_co<R>(L.L.c);
  const long long t0 = a.tptr ? *a.tptr : a.t0;

  // neighbours of the band: below it rank - 1, above it rank + 1 (around the seam of a periodic y axis)
  const bool has_lo = py || rank > 0, has_hi = py || rank < cl - 1;
  const int r_lo = rank > 0 ? rank - 1 : cl - 1, r_hi = rank < cl - 1 ? rank + 1 : 0;
  const int rows_lo = band_start(r_lo + 1, cl, ny) - band_start(r_lo, cl, ny);
  const int last = (rows - 1) * nx;
  // The first bt threads update the boundary nodes, the others the interior: a boundary node takes
  // about as long as two interior ones, and each band waits for its slowest warp.
  const int bt = min((nb + 31) & ~31, nt / 2 & ~31), total = rows * nx;

  // Store of local node li in column x: locally, and into the ghost rows of the neighbours if it
  // lies on an edge of the band (what streams across; all of it where the neighbour has walls).
  auto store = [&](S* dst, int li, int x, bool first, bool lastrow, const R(&d)[9], const R(&h)[5], R qv,
                   uint32_t key) {
    S v[15];
#pragma unroll
    for (int q = 0; q < 14; ++q) v[q] = round1<S, R>(q < 9 ? d[q] : h[q - 9], a.stochastic, key, q, x & 3);
    v[14] = from_r<S, R>(qv);
    S* o = dst + li * ST;
#pragma unroll
    for (int q = 0; q < (VH ? 15 : 14); ++q) o[q] = v[q];
    const uint8_t kd = first || lastrow ? kind[li] : (uint8_t)0;
    if (first && has_lo) {
      const uint32_t to = cluster_addr(dst + ((rows_lo + 1) * nx + x) * ST, r_lo);
#pragma unroll
      for (int q = 0; q < (VH ? 15 : 14); ++q)
        if ((kd & 4) || (q < 9 && ey_of(q) < 0) || q == 13) st_cluster<S>(to + q * (uint32_t)sizeof(S), v[q]);
    }
    if (lastrow && has_hi) {
      const uint32_t to = cluster_addr(dst + x * ST, r_hi);
#pragma unroll
      for (int q = 0; q < (VH ? 15 : 14); ++q)
        if ((kd & 8) || (q < 9 && ey_of(q) > 0) || q == 11) st_cluster<S>(to + q * (uint32_t)sizeof(S), v[q]);
    }
  };
  __syncwarp();
  cluster_sync();

  for (int s = 0; s < a.steps; ++s) {
    const S* src = (s & 1) ? buf1 : buf0;
    S* dst = (s & 1) ? buf0 : buf1;
    uint32_t seed = 0;
    if (a.stochastic) {
      const long long t = t0 + s;
      seed = (uint32_t)(t * 0x9E3779B1ull) ^ (uint32_t)(t >> 32);
    }
    if (tid < bt) {
      for (int i = tid; i < nb; i += bt) {
        R d[9], h[5], qv = R(0);
        const ResNode e = edge[i];
        const NodeSrc<S, ST> ns{src};
        if (masked)
          node_update<NodeSrc<S, ST>, true>(L.L.g, c, ns, e.x, e.y, e.fl, e.slot, d, h, qv);
        else
          node_update<NodeSrc<S, ST>, false>(L.L.g, c, ns, e.x, e.y, 0u, 0, d, h, qv);
        store(dst, e.y * nx + e.x, e.x, e.y == 1, e.y == rows, d, h, qv, sr_key(seed, (long long)e.gi - (e.x & 3)));
      }
    } else {
      for (int n = tid - bt; n < total; n += nt - bt) {
        R d[9], h[5], qv = R(0);
        const int li = n + nx;
        if (kind[li] & 3) continue;
        const S* o = src + li * ST;
#pragma unroll
        for (int q = 0; q < 14; ++q) {
          const int dir = q < 9 ? q : q - 9;
          const S* row = ey_of(dir) > 0 ? o - nx * ST : (ey_of(dir) < 0 ? o + nx * ST : o);
          const R val = to_r(row[q - ex_of(dir) * ST]);
          if (q < 9)
            d[q] = val;
          else
            h[q - 9] = val;
        }
        collide<R, VH>(c, d, h, qv);
        const bool first = n < nx, lastrow = n >= last;
        int x = first ? n : n - last;
        uint32_t key = 0;
        if constexpr (sizeof(S) == 2) {
          if (a.stochastic) {
            const int y = n / nx;
            x = n - y * nx;
            key = sr_key(seed, (long long)(row0 + y) * gpitch + (x & ~3));
          }
        }
        store(dst, li, x, first, lastrow, d, h, qv, key);
      }
    }
    __syncwarp();
    cluster_sync();
  }

  // the last two states back to the planes (own fluid nodes)
  const S* now = (a.steps & 1) ? buf1 : buf0;
  const S* before = (a.steps & 1) ? buf0 : buf1;
  S* gnow = static_cast<S*>(L.L.buf[(a.cur + a.steps) & 1]);
  S* gbefore = static_cast<S*>(L.L.buf[(a.cur + a.steps + 1) & 1]);
  for (int n = tid; n < rows * nx; n += nt) {
    const int y = n / nx, li = n + nx;
    if (kind[li] & 1) continue;
    const long long gi = (long long)(row0 + y) * gpitch + (n - y * nx);
#pragma unroll
    for (int q = 0; q < (VH ? 15 : 14); ++q) {
      gnow[q * gplane + gi] = now[li * ST + q];
      gbefore[q * gplane + gi] = before[li * ST + q];
    }
  }
}

}  // namespace clbm
