// k_resident_cluster.cu -- resident sweeps of small bit-sliced lattices split
// over a thread-block cluster.
//
// A colour pass of a small lattice is a launch's latency (about 3 us) when
// launched by itself, and on one block (k_resident_bits) it is the one SM's
// work.  Here a cluster of C blocks holds one (group, temperature slot) in its
// shared memories for many sweeps: block r the contiguous rows [r rows / C,
// (r + 1) rows / C) of the split layout, with the coupling words and neighbour
// addresses of its sites, and the threshold planes.  Neighbours in other
// blocks are read through distributed shared memory; passes are separated by
// the hardware cluster barrier.
//
// Four neighbouring threads share a word.  Thread j draws plane pairs 2j and
// 2j + 1, for the first word of its next pass while it waits at the barrier
// (they do not depend on the spins), and compares its four planes; the four
// partial results (eq: lanes equal so far, lt: lanes decided below) compose
// like (e1, l1)(e2, l2) = (e1 & e2, l1 | e1 & l2), two shuffle steps.  Lanes
// undecided after 16 planes (a word in a thousand) take a second such round.
//
// The update and its random stream are those of the per-lane-plane sweep
// (sweep_planes.cuh), so the trajectory is the same bit for bit.
//
// Bound: latency, about 0.8 us a pass and 0.6 ns a word and SM.  us per sweep,
// heat bath, 64 samples (launched / one block / cluster): 3D L=8, one replica
// 3.9 / 3.7 / 1.9; L=8 x 2 4.6 / 6.3 / 2.1; L=12 x 2 4.8 / 19 / 3.6; L=16 x 2
// 5.1 / 41 / 6.5 (not taken); L=8 x 2 x 32 temperatures 7.3 / 6.3 / 3.5.
#include "lattice.h"
#include "sweep_planes.cuh"

namespace ianus {

namespace {

constexpr uint32_t kClThreads = 1024;
constexpr uint32_t kClRow = kMaxClasses + 1;  // words per plane row: four rows read side by side miss each other's banks
constexpr size_t kClSmemMax = 200u * 1024u;

// One local word of a colour.
struct ClSite {
  uint32_t yp, ym, zp, zm;  // cluster shared-memory addresses of replica 0's words
  uint32_t xp, xm, self;    // local word offsets
  uint32_t site;            // natural index
};

struct ClParams {
  BitsParams b;
  uint32_t nsweeps;
  uint32_t C;      // blocks of a cluster
  uint32_t words;  // most local words of a block (both colours)
};

__device__ __forceinline__ uint32_t cl_map(uint32_t addr, uint32_t rank) {
  uint32_t d;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(addr), "r"(rank));
  return d;
}

__device__ __forceinline__ uint64_t cl_load(uint32_t addr) {
  uint64_t v;
  asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
  return v;
}

__device__ __forceinline__ void cl_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cl_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Lanes equal so far and lanes decided below, of consecutive planes.
struct Prefix {
  uint64_t eq, lt;
};

__device__ __forceinline__ Prefix cl_then(const Prefix& a, const Prefix& b) {
  return Prefix{a.eq & b.eq, a.lt | (a.eq & b.lt)};
}

// The planes of pairs m and m + 1 (blocks x, y) against the slot's rows.
template <int D, int ALGO>
__device__ __forceinline__ Prefix cl_planes(const uint4& x, const uint4& y, uint32_t m, const uint64_t* tpa, uint64_t u0,
                                            uint64_t u1, uint64_t u2) {
  const uint64_t r[4] = {(uint64_t)x.x | ((uint64_t)x.y << 32), (uint64_t)x.z | ((uint64_t)x.w << 32),
                         (uint64_t)y.x | ((uint64_t)y.y << 32), (uint64_t)y.z | ((uint64_t)y.w << 32)};
  Prefix f{~0ull, 0ull};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint64_t t = planes::class_select<D, ALGO>(tpa + (2u * m + (uint32_t)q) * kClRow, u0, u1, u2);
    f.lt |= f.eq & ~r[q] & t;
    f.eq &= ~(r[q] ^ t);
  }
  return f;
}

// The four threads' results, in the order of their planes.
__device__ __forceinline__ Prefix cl_combine(Prefix f, uint32_t sub) {
#pragma unroll
  for (uint32_t step = 1; step < 4u; step *= 2u) {
    Prefix o;
    o.eq = __shfl_xor_sync(0xffffffffu, (unsigned long long)f.eq, (int)step);
    o.lt = __shfl_xor_sync(0xffffffffu, (unsigned long long)f.lt, (int)step);
    f = (sub & step) ? cl_then(o, f) : cl_then(f, o);
  }
  return f;
}

template <int D, int ALGO>
__global__ void __launch_bounds__(kClThreads, 1) k_resident_bits_cluster(const ClParams cp) {
  extern __shared__ __align__(16) uint8_t cl_sm[];
  const BitsParams& p = cp.b;
  const uint32_t R = (uint32_t)p.R, N = p.geom.N, L = (uint32_t)p.geom.L, h = (uint32_t)p.geom.h;
  const uint32_t C = cp.C, cl = blockIdx.x / C, rank = blockIdx.x - cl * C;
  const uint32_t g = cl / (uint32_t)p.K, tslot = cl - g * (uint32_t)p.K;
  const uint32_t rows = N / L, r0 = rank * rows / C, r1 = (rank + 1u) * rows / C, nr = r1 - r0;
  const uint32_t local = nr * L, nh = nr * h;  // words of the block, of one colour
  ClSite* s_site = reinterpret_cast<ClSite*>(cl_sm);                         // [2][nh] by colour
  uint64_t* s_J = reinterpret_cast<uint64_t*>(s_site + cp.words);            // [2][nh][2 D]
  uint64_t* s_sp = s_J + (size_t)cp.words * 2 * D;                           // [R][words]
  uint64_t* s_tp = s_sp + (size_t)R * cp.words;                              // [R][kPlanes][kClRow]
  const uint32_t sp_addr = (uint32_t)__cvta_generic_to_shared(s_sp);
  uint64_t* g_sp = p.spins + ((size_t)g * p.slots + (size_t)tslot * R) * N + (size_t)r0 * L;
  const uint64_t* g_J = p.J + (size_t)g * D * N;
  const uint64_t* g_tp = p.tp + ((size_t)g * p.slots + (size_t)tslot * R) * kPlanes * kMaxClasses;
  for (uint32_t i = threadIdx.x; i < R * local; i += blockDim.x) {
    const uint32_t a = i / local, j = i - a * local;
    s_sp[(size_t)a * cp.words + j] = g_sp[(size_t)a * N + j];
  }
  for (uint32_t i = threadIdx.x; i < R * kPlanes * kMaxClasses; i += blockDim.x)
    s_tp[(i / kMaxClasses) * kClRow + i % kMaxClasses] = g_tp[i];
  for (uint32_t i = threadIdx.x; i < 2u * nh; i += blockDim.x) {
    const uint32_t c = i / nh, q = i - c * nh;
    const Nbr n = split_neighbours(p.geom, (int)c, r0 * h + q);
    auto at = [&](uint32_t j) {  // word j of replica 0 in its owner's shared memory
      const uint32_t row = j / L, o = ((row + 1u) * C - 1u) / rows;
      return cl_map(sp_addr + 8u * (j - (o * rows / C) * L), o);
    };
    ClSite s;
    s.self = n.self - r0 * L;
    s.xp = n.xp - r0 * L;
    s.xm = n.xm - r0 * L;
    s.yp = at(n.yp);
    s.ym = at(n.ym);
    s.zp = D == 3 ? at(n.zp) : 0u;
    s.zm = D == 3 ? at(n.zm) : 0u;
    s.site = n.site;
    s_site[i] = s;
    uint64_t* jw = s_J + (size_t)i * 2 * D;
    jw[0] = __ldg(g_J + n.self);
    jw[1] = __ldg(g_J + n.xm);
    jw[2] = __ldg(g_J + N + n.self);
    jw[3] = __ldg(g_J + N + n.ym);
    if (D == 3) {
      jw[4] = __ldg(g_J + 2u * N + n.self);
      jw[5] = __ldg(g_J + 2u * N + n.zm);
    }
  }
  cl_arrive();
  cl_wait();
  const Tick t0 = sweep_tick(p.t_lo, p.t_hi, p.t_dev);
  const uint64_t t_first = (uint64_t)t0.lo | ((uint64_t)t0.hi << 32);
  const uint32_t sub = threadIdx.x & 3u, items = R * nh, step = blockDim.x >> 2;
  // plane pairs m, m + 1 of item `it` of colour c at sweep t
  auto draw = [&](uint32_t it, uint32_t c, uint64_t t, uint32_t m, uint4& x, uint4& y) {
    const uint32_t i = min(it, items - 1u), a = i / nh, q = i - a * nh;
    const Tick tk{(uint32_t)t, (uint32_t)(t >> 32)};
    const uint32_t c2 = (TAG_SPIN << 28) | ((tslot * R + a) << 12) | g;
    const planes::PlaneSiteKey sk = planes::plane_site_key(s_site[c * nh + q].site, tk, p.keys);
    x = planes::philox10_split(sk, planes::plane_uniform(c2 | (m << 24), tk, p.keys), p.keys);
    y = planes::philox10_split(sk, planes::plane_uniform(c2 | ((m + 1u) << 24), tk, p.keys), p.keys);
  };
  uint4 x, y;
  draw(threadIdx.x >> 2, 0u, t_first, 2u * sub, x, y);
  const uint32_t npass = 2u * cp.nsweeps;
#pragma unroll 1
  for (uint32_t pass = 0; pass < npass; ++pass) {
    const uint32_t c = pass & 1u;
    const uint64_t t = t_first + (pass >> 1);
#pragma unroll 1
    for (uint32_t it0 = 0; it0 < items; it0 += step) {  // uniform across the block
      const uint32_t it = it0 + (threadIdx.x >> 2);
      if (it0 > 0u) draw(it, c, t, 2u * sub, x, y);
      const bool valid = it < items;
      const uint32_t i = min(it, items - 1u), a = i / nh, q = i - a * nh;
      const ClSite s = s_site[c * nh + q];
      const uint64_t* jw = s_J + (size_t)(c * nh + q) * 2 * D;
      const uint64_t* sp = s_sp + (size_t)a * cp.words;
      const uint32_t ra = 8u * a * cp.words;
      const uint64_t b = sp[s.self];
      uint64_t e[2 * D];
      e[0] = b ^ sp[s.xp] ^ jw[0];
      e[1] = b ^ sp[s.xm] ^ jw[1];
      e[2] = b ^ cl_load(s.yp + ra) ^ jw[2];
      e[3] = b ^ cl_load(s.ym + ra) ^ jw[3];
      if (D == 3) {
        e[4] = b ^ cl_load(s.zp + ra) ^ jw[4];
        e[5] = b ^ cl_load(s.zm + ra) ^ jw[5];
      }
      uint64_t u0, u1, u2;
      count_unsat<D>(e, u0, u1, u2);
      const uint64_t* tpa = s_tp + (size_t)a * kPlanes * kClRow;
      const uint64_t always = planes::class_select<D, 1>(tpa + 32 * kClRow, u0, u1, u2);
      const uint64_t need = ALGO == 1 ? ~0ull : D == 3 ? ~u2 & ~(u1 & u0) : ~u2 & ~u1;
      const uint64_t und = ~always & need;
      Prefix f = cl_combine(cl_planes<D, ALGO>(x, y, 2u * sub, tpa, u0, u1, u2), sub);
      if (__any_sync(0xffffffffu, valid && (und & f.eq) != 0ull)) {
        uint4 x2, y2;
        draw(it, c, t, 8u + 2u * sub, x2, y2);
        f = cl_then(f, cl_combine(cl_planes<D, ALGO>(x2, y2, 8u + 2u * sub, tpa, u0, u1, u2), sub));
      }
      const uint64_t lt = always | (und & f.lt);
      const uint64_t flip = ALGO == 0 ? lt : ~lt;
      if (valid && sub == 0u) s_sp[(size_t)a * cp.words + s.self] = b ^ flip;
    }
    cl_arrive();
    if (pass + 1u < npass) draw(threadIdx.x >> 2, c ^ 1u, t + c, 2u * sub, x, y);
    cl_wait();
  }
  for (uint32_t i = threadIdx.x; i < R * local; i += blockDim.x) {
    const uint32_t a = i / local, j = i - a * local;
    g_sp[(size_t)a * N + j] = s_sp[(size_t)a * cp.words + j];
  }
}

uint32_t cl_words(const Lattice& lat, uint32_t C) {
  const uint32_t rows = lat.N / (uint32_t)lat.L;
  return (rows + C - 1u) / C * (uint32_t)lat.L;
}

// Rounds of a block's threads over a colour's words, evenly filled.
uint32_t cl_rounds(const Lattice& lat, uint32_t C) {
  const uint32_t t = 4u * (uint32_t)lat.R * cl_words(lat, C) / 2u;
  return std::max(1u, (t + kClThreads - 1u) / kClThreads);
}

uint32_t cl_threads(const Lattice& lat, uint32_t C) {
  const uint32_t t = 4u * (uint32_t)lat.R * cl_words(lat, C) / 2u, n = cl_rounds(lat, C);
  return std::max(32u, ((t + n - 1u) / n + 31u) & ~31u);
}

size_t cl_smem(const Lattice& lat, uint32_t C) {
  const size_t words = cl_words(lat, C);
  return words * (sizeof(ClSite) + 16u * (size_t)lat.D + 8u * (size_t)lat.R) +
         (size_t)lat.R * kPlanes * kClRow * sizeof(uint64_t);
}

const void* cl_kernel(const Lattice& lat, int algo) {
  if (lat.D == 3) return algo ? (const void*)k_resident_bits_cluster<3, 1> : (const void*)k_resident_bits_cluster<3, 0>;
  return algo ? (const void*)k_resident_bits_cluster<2, 1> : (const void*)k_resident_bits_cluster<2, 0>;
}

void cl_config(const Lattice& lat, uint32_t C, cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr) {
  cfg = {};
  cfg.gridDim = dim3(C * (unsigned)lat.G * (unsigned)lat.K);
  cfg.blockDim = dim3(cl_threads(lat, C));
  cfg.dynamicSmemBytes = cl_smem(lat, C);
  cfg.stream = lat.stream;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
}

// Whether clusters of C blocks can hold the lattice, all of them at once.
bool cl_fits(const Lattice& lat, uint32_t C) {
  const uint64_t blocks = (uint64_t)lat.G * (uint64_t)lat.K * C;
  if (C > lat.N / (uint32_t)lat.L || cl_smem(lat, C) > kClSmemMax || blocks > 2u * 152u ||
      blocks * cl_threads(lat, C) > 152u * kClThreads)
    return false;
  for (int algo = 0; algo < 2; ++algo) {
    const void* k = cl_kernel(lat, algo);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    cl_config(lat, C, cfg, attr);
    cfg.stream = 0;
    int n = 0;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmemMax) != cudaSuccess ||
        cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess ||
        (uint64_t)n * C < blocks) {
      cudaGetLastError();
      return false;
    }
  }
  return true;
}

// Whether the clusters of C blocks find room with one block per SM (a large
// cluster's blocks must share a GPC, so that some SMs stay empty).
bool cl_alone(const Lattice& lat, uint32_t C) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cl_config(lat, C, cfg, attr);
  cfg.stream = 0;
  cfg.dynamicSmemBytes = kClSmemMax;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, cl_kernel(lat, 0), &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return n >= lat.G * lat.K;
}

// Estimated us per sweep with clusters of C blocks, on one block, and launched
// pass by pass (fits of the sweeps above and of up to 32 temperatures; where two
// blocks share an SM both take twice as long: L=14, 8 temperatures 4.7 us, 5
// temperatures of two replicas, twice the words in 5 clusters, 5.2).
double cl_us(const Lattice& lat, uint32_t C) {
  return 1.5 + (lat.D == 3 ? 5.0e-3 : 4.25e-3) * (cl_alone(lat, C) ? 1.0 : 2.0) * cl_rounds(lat, C) *
                   cl_threads(lat, C);
}

double block_us(const Lattice& lat) { return 1.8 + 7.6e-3 * lat.R * lat.geom.half; }

double launched_us(const Lattice& lat) {
  const double words = (double)lat.G * lat.K * lat.R * lat.geom.half;
  if (lat.K == 1 && lat.R <= 2)
    return (lat.R == 1 ? 4.2 : 4.8) + std::min(0.08e-3 * words, 0.5 + 0.02e-3 * words);
  const bool two = lat.R % 2 == 0;  // replicas a thread
  return (lat.D == 3 ? (two ? 7.0 : 5.8) : (two ? 6.2 : 5.2)) + 0.03e-3 * words;
}

// Blocks of a cluster: the fastest of 16, 8, 4 and 2 that fit; 0 if there is
// none or, unless forced, another sweep is faster.
uint32_t cl_choose(const Lattice& lat, bool force) {
  const double other = resident_bits_fits(lat) ? std::min(block_us(lat), launched_us(lat)) : launched_us(lat);
  uint32_t best = 0;
  double best_us = force ? 1e300 : other;
  for (uint32_t C = 16; C >= 2; C /= 2) {
    if (!cl_fits(lat, C)) continue;
    const double us = cl_us(lat, C);
    if (us < best_us) {
      best = C;
      best_us = us;
    }
  }
  return best;
}

}  // namespace

uint32_t resident_cluster_bits(Lattice& lat) {
  if (lat.layout != IANUS_LAYOUT_BITS64 || lat.model != IANUS_EA_PM_J || lat.field || lat.pool ||
      lat.resident_mode == 2)
    return 0;
  const int mode = lat.resident_mode;
  if (lat.bits_cluster_mode != mode) {
    lat.bits_cluster = cl_choose(lat, mode == 3);
    lat.bits_cluster_mode = mode;
  }
  return lat.bits_cluster;
}

cudaError_t launch_resident_cluster_bits(Lattice& lat, int inv, uint64_t t0, uint32_t nsweeps) {
  const uint32_t C = lat.bits_cluster;
  ClParams cp{};
  BitsParams& p = cp.b;
  p.spins = (uint64_t*)lat.spins;
  p.J = (const uint64_t*)lat.J;
  p.tp = lat.tp;
  p.geom = lat.geom;
  p.G = lat.G;
  p.R = lat.R;
  p.K = lat.K;
  p.slots = lat.slots;
  p.t_lo = (uint32_t)t0;
  p.t_hi = (uint32_t)(t0 >> 32);
  p.keys = lat.keys;
  p.t_dev = lat.capturing ? lat.t_dev : nullptr;
  cp.nsweeps = nsweeps;
  cp.C = C;
  cp.words = cl_words(lat, C);
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cl_config(lat, C, cfg, attr);
  void* args[] = {(void*)&cp};
  const cudaError_t e = cudaLaunchKernelExC(&cfg, cl_kernel(lat, inv ? 1 : 0), args);
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

}  // namespace ianus
