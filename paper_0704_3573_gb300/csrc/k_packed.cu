// k_packed.cu -- resident sweeps of small plain (IANUS_LAYOUT_I8) lattices
// with the sites of a configuration packed 32 to a word.
//
// A colour pass of one configuration of a few thousand sites is too little work
// for a launch (3 us), and split over a cluster with a site per thread it is
// bound by the random numbers: a site needs four Philox blocks at least, and a
// warp or two per scheduler cannot hide them (L=16, one sample: 0.55 us of a
// 0.99 us pass, and 0.28 more for the one site in a hundred that needs further
// blocks).  The random numbers do not depend on the spins.  So
//
//   k_packed_masks draws them on the whole GPU for a run of sweeps at once and
//   keeps, for each word of 32 sites of a colour and each class u (number of
//   unsatisfied bonds), the 32 bits "this site flips if its class is u".  The
//   samples of a 64-lane group share their Philox blocks;
//
//   k_packed_sweep holds a configuration in one block, one word of each colour
//   a thread: the neighbours of 32 sites are 11 unaligned 32-bit reads of the
//   other colour's words, their classes a carry-save adder, the flips a
//   multiplexer tree over the masks, which cp.async brings from L2 several
//   passes ahead.  Passes are separated by a barrier of the block's (few)
//   active warps.
//
// Word order: site w = row L/2 + k of a colour (its x is 2k + xpar, the natural
// index 2w + xpar), 32 consecutive w to a word.  All the y and z neighbours of
// w are at w plus or minus L/2 and L/2 L, cyclically, and the x neighbours at w
// and w +- 1, but for the sites at a face, which are chosen by fixed bit masks
// from words read at the wrapped distance.
//
// Bound: the latency of a pass of one or two warps, about 65 instructions and a
// barrier, 0.17 us at L=16 (0.28 with the unaligned reads of any L); with many
// configurations the random numbers, 90 sites/ns.  Per sweep, heat bath, runs
// of 300 sweeps (cluster-resident / one block / launched / packed): L=16, one
// sample 1.57 / 10.2 / 7.0 / 0.43; 64 samples 5.5 / 10.3 / 15 / 3.0; L=24 5.0 /
// 32 / 7.6 / 1.1; L=36 11.3 / 102 / 7.9 / 3.3.  L=16, one sample, Metropolis,
// 1000 sweeps measured at each: 1972 -> 536 us.
#include <algorithm>

#include "lattice.h"
#include "sweep_planes.cuh"

namespace ianus {

namespace {

constexpr uint32_t kRowsKept = 64;      // measurements summed up at a time
constexpr uint32_t kPackedSmem = 190u * 1024u;
constexpr uint32_t kPackedMin = 512;    // threads of a block: they share the loads and stores at the ends

struct PackedParams {
  int8_t* spins;         // [R][S][N]
  const int8_t* J;       // [S][D][N]
  const uint64_t* thr;   // [kMaxClasses]
  uint4* masks;          // [R][S][sweep][colour][2][words]: classes 0..3, 4..7
  int S, R, L, inv;
  uint32_t N, words;     // words of a colour: N / 64
  uint32_t nsweeps, per_warp, parts;  // samples a warp of k_packed_masks does, warps for a group's samples
  uint64_t t0;
  uint32_t measure_every, cap;
  uint64_t row0;         // series rows recorded before this launch
  int64_t* ser_E;        // [cap][S * R]
  int64_t* ser_M;
  uint64_t* ser_sweep;   // [cap]
  PhiloxKeys keys;
};

__device__ __forceinline__ uint32_t parity_of_row(uint32_t row, uint32_t L, int D) {
  return D == 3 ? (row % L + row / L) & 1u : row & 1u;
}

// Warp: one word of one colour, sweep, group and replica, for per_warp samples
// of the group; lane i its site i.
template <int D>
__global__ void __launch_bounds__(256) k_packed_masks(const PackedParams p) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ uint32_t first_s[8];  // the set of the thresholds' first eight planes
  __shared__ uint32_t thr_s[kMaxClasses];
  uint32_t always = 0;
  for (uint32_t u = 0; u <= 2u * D; ++u) always |= (p.thr[u] >= kTwo32 ? 1u : 0u) << u;
  if (threadIdx.x < 8u) first_s[threadIdx.x] = 0u;
  __syncthreads();
  if (threadIdx.x <= 2u * D) {
    const uint32_t T = (uint32_t)p.thr[threadIdx.x];
    thr_s[threadIdx.x] = T;
    if ((always >> threadIdx.x & 1u) == 0u) atomicOr(&first_s[T >> 29], 1u << (T >> 24 & 31u));
  }
  __syncthreads();
  uint32_t thr[2 * D + 1];
#pragma unroll
  for (int u = 0; u <= 2 * D; ++u) thr[u] = thr_s[u];
  const uint32_t lane = threadIdx.x & 31u;
  uint64_t id = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const uint32_t G = (uint32_t)(p.S + 63) >> 6;
  const uint32_t W = (uint32_t)(id % p.words);
  id /= p.words;
  const uint32_t colour = (uint32_t)(id & 1u);
  id >>= 1;
  const uint32_t it = (uint32_t)(id % p.nsweeps);
  id /= p.nsweeps;
  const uint32_t part = (uint32_t)(id % p.parts);
  id /= p.parts;
  const uint32_t g = (uint32_t)(id % G), sigma = (uint32_t)(id / G);
  if (sigma >= (uint32_t)p.R) return;
  const uint32_t s0 = 64u * g + part * p.per_warp;
  const uint32_t s1 = min(min(s0 + p.per_warp, 64u * g + 64u), (uint32_t)p.S);
  const uint32_t w = 32u * W + lane, h = (uint32_t)p.L / 2u, row = w / h;
  const uint32_t site = 2u * w + ((parity_of_row(row, (uint32_t)p.L, D) ^ colour) & 1u);
  const uint64_t t = p.t0 + it;
  const Tick tk{(uint32_t)t, (uint32_t)(t >> 32)};
  const planes::PlaneSiteKey key = planes::plane_site_key(site, tk, p.keys);
  const uint32_t c2 = (TAG_SPIN << 28) | (sigma << 12) | g;
  uint4 x[4];
#pragma unroll
  for (uint32_t m = 0; m < 4u; ++m)
    x[m] = planes::philox10_split(key, planes::plane_uniform(c2 | (m << 24), tk, p.keys), p.keys);
  for (uint32_t s = s0; s < s1; ++s) {
    const uint32_t sl = s & 31u;
    const bool upper = (s & 32u) != 0u;
    uint32_t r = 0;
#pragma unroll
    for (uint32_t m = 0; m < 4u; ++m)
      r |= ((upper ? x[m].y : x[m].x) >> sl & 1u) << (31u - 2u * m) |
           ((upper ? x[m].w : x[m].z) >> sl & 1u) << (30u - 2u * m);
    // planes 8, 9, ... while they can decide a comparison
    bool open = (first_s[r >> 29] >> (r >> 24 & 31u) & 1u) != 0u;
#pragma unroll 1
    for (uint32_t m = 4; m < 16u && __any_sync(0xffffffffu, open); ++m) {
      const uint4 y = planes::philox10_split(key, planes::plane_uniform(c2 | (m << 24), tk, p.keys), p.keys);
      r |= ((upper ? y.y : y.x) >> sl & 1u) << (31u - 2u * m) | ((upper ? y.w : y.z) >> sl & 1u) << (30u - 2u * m);
      open = false;
#pragma unroll
      for (int u = 0; u <= 2 * D; ++u) open |= (always >> u & 1u) == 0u && ((r ^ thr[u]) >> (30u - 2u * m)) == 0u;
    }
    uint32_t mine = 0;  // lane u < 8: the mask of class u
#pragma unroll
    for (int u = 0; u <= 2 * D; ++u) {
      const bool flip = ((always >> u & 1u) != 0u || r < thr[u]) != (p.inv != 0);
      const uint32_t b = __ballot_sync(0xffffffffu, flip);
      if (lane == (uint32_t)u) mine = b;
    }
    if (lane < 8u) {
      uint32_t* out = (uint32_t*)(p.masks + ((((size_t)sigma * p.S + s) * p.nsweeps + it) * 2u + colour) * 2u * p.words);
      out[((lane >> 2) * p.words + W) * 4u + (lane & 3u)] = mine;
    }
  }
}

// sel ? a : b, bit by bit
__device__ __forceinline__ uint32_t pick(uint32_t sel, uint32_t a, uint32_t b) { return (a & sel) | (b & ~sel); }

// 32 bits from bit `start` of a cyclic bit array: word and shift.
struct Bits32 {
  uint32_t at, sh;
};

__device__ __forceinline__ Bits32 bits_at(uint32_t w, uint32_t offset, uint32_t half) {
  const uint32_t b = w + offset < half ? w + offset : w + offset - half;  // offset < half
  return Bits32{b >> 5, b & 31u};
}

// The array's first word is repeated behind its last.
__device__ __forceinline__ uint32_t read32(const uint32_t* a, const Bits32& s) {
  return __funnelshift_r(a[s.at], a[s.at + 1u], s.sh);
}

template <int D>
__device__ __forceinline__ void unsat32(const uint32_t* e, uint32_t& u0, uint32_t& u1, uint32_t& u2) {
  const uint32_t s1 = e[0] ^ e[1] ^ e[2], c1 = (e[0] & e[1]) | (e[2] & (e[0] | e[1]));
  uint32_t s2 = e[3], c2 = 0u;
  if constexpr (D == 3) {
    s2 = e[3] ^ e[4] ^ e[5];
    c2 = (e[3] & e[4]) | (e[5] & (e[3] | e[4]));
  }
  const uint32_t k = s1 & s2;
  u0 = s1 ^ s2;
  u1 = c1 ^ c2 ^ k;
  u2 = D == 3 ? (c1 & c2) | (k & (c1 | c2)) : c1 & k;
}

// Block: one configuration (sigma, s).  Threads below `words` own word
// threadIdx.x of both colours; STAGES passes' masks are under way.  ALIGNED:
// words hold whole rows and planes whole words (32 % (L/2) == 0; 3D also
// L^2/2 % 32 == 0); x neighbours are then shifts of the same word, y neighbours
// a shift over two words, z neighbours words.
template <int D, int STAGES, bool ALIGNED>
__global__ void __launch_bounds__(STAGES == 8 ? 768 : 1024) k_packed_sweep(const PackedParams p) {
  extern __shared__ __align__(16) uint32_t packed_sm[];
  __shared__ int warp_sum[32][2][kRowsKept];
  const uint32_t nW = p.words, L = (uint32_t)p.L, h = L / 2u, half = p.N / 2u, pitch = nW + 1u;
  uint32_t* s_spin = packed_sm;                                       // [2][pitch]
  uint4* s_ring = (uint4*)(packed_sm + ((2u * pitch + 3u) & ~3u));    // [STAGES][2][nW]
  uint32_t* s_J = (uint32_t*)s_ring;                                  // [2][2 D][nW], before the first masks
  const uint32_t cfg = blockIdx.x, sigma = cfg / (uint32_t)p.S, s = cfg - sigma * (uint32_t)p.S;
  int8_t* gsp = p.spins + (size_t)cfg * p.N;
  const int8_t* gJ = p.J + (size_t)s * D * p.N;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, nwarps = blockDim.x >> 5;
  // pack spins and couplings, a word per warp and step (four steps' loads in flight)
#pragma unroll 4
  for (uint32_t i = warp; i < 2u * nW; i += nwarps) {
    const uint32_t c = i >= nW ? 1u : 0u, W = i - c * nW, w = 32u * W + lane;
    const uint32_t row = w / h, k = w - row * h, y = D == 3 ? row % L : row, z = D == 3 ? row / L : 0u;
    const uint32_t xpar = (c ^ y ^ z) & 1u, site = 2u * w + xpar, base = site - (2u * k + xpar);
    const uint32_t xprev = base + (2u * k == 0u ? L - 1u : 2u * k - 1u);  // x - 1 of an even x
    const uint32_t ym = y == 0u ? site + L * (L - 1u) : site - L;
    bool v[2 * D + 1];
    v[0] = __ldcg((const signed char*)gsp + site) < 0;
    v[1] = __ldg(gJ + 2u * w) < 0;                             // the bond within the pair 2w, 2w + 1
    v[2] = __ldg(gJ + (xpar ? site : xprev)) < 0;                // the other x bond
    v[3] = __ldg(gJ + p.N + site) < 0;
    v[4] = __ldg(gJ + p.N + ym) < 0;
    if constexpr (D == 3) {
      const uint32_t zm = z == 0u ? site + L * L * (L - 1u) : site - L * L;
      v[5] = __ldg(gJ + 2u * p.N + site) < 0;
      v[6] = __ldg(gJ + 2u * p.N + zm) < 0;
    }
#pragma unroll
    for (int q = 0; q <= 2 * D; ++q) {
      const uint32_t b = __ballot_sync(0xffffffffu, v[q]);
      if (lane == 0u) {
        if (q > 0) {
          s_J[(c * 2u * D + (uint32_t)q - 1u) * nW + W] = b;
        } else {
          s_spin[c * pitch + W] = b;
          if (W == 0u) s_spin[c * pitch + nW] = b;
        }
      }
    }
  }
  __syncthreads();
  const uint32_t active = (nW + 31u) & ~31u;
  const bool runs = tid < active, own = tid < nW;
  const uint32_t W = min(tid, nW - 1u), w0 = 32u * W;
  uint32_t J[2][2 * D];
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int q = 0; q < 2 * D; ++q) J[c][q] = s_J[((uint32_t)c * 2u * D + (uint32_t)q) * nW + W];
  __syncthreads();  // the ring takes the couplings' place
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the masks
  if (runs) {
    uint32_t odd = 0, last = 0, first = 0, top = 0, bottom = 0;  // odd x of colour 0; k = h-1, 0; y = L-1, 0
    for (uint32_t i = 0; i < 32u; ++i) {
      const uint32_t row = (w0 + i) / h, k = w0 + i - row * h, y = row % L;
      odd |= parity_of_row(row, L, D) << i;
      last |= (k + 1u == h ? 1u : 0u) << i;
      first |= (k == 0u ? 1u : 0u) << i;
      top |= (y + 1u == L ? 1u : 0u) << i;
      bottom |= (y == 0u ? 1u : 0u) << i;
    }
    const uint32_t plane = h * L;  // distance of z neighbours (3D), of a wrapped y neighbour and its unwrapped
    const Bits32 x_up = bits_at(w0, 1u, half), x_up_wrap = bits_at(w0, half + 1u - h, half);
    const Bits32 x_dn = bits_at(w0, half - 1u, half), x_dn_wrap = bits_at(w0, h - 1u, half);
    const Bits32 y_up = bits_at(w0, h, half), y_dn = bits_at(w0, half - h, half);
    const Bits32 y_up_wrap = bits_at(w0, half - (plane - h), half), y_dn_wrap = bits_at(w0, plane - h, half);
    const Bits32 z_up = bits_at(w0, plane % half, half), z_dn = bits_at(w0, half - plane, half);
    // ALIGNED: the words that continue this one's rows at y + 1 and y - 1
    const uint32_t pw = plane / 32u, in_plane = pw ? W % pw : 0u;
    const uint32_t next = in_plane + 1u == pw ? W + 1u - pw : W + 1u, prev = in_plane == 0u ? W + pw - 1u : W - 1u;
    // a colour's unsatisfied bonds of each site, from the other colour's words
    auto classes = [&](uint32_t c, uint32_t b, uint32_t& u0, uint32_t& u1, uint32_t& u2) {
      const uint32_t* o = s_spin + (c ^ 1u) * pitch;
      const uint32_t xodd = c ? ~odd : odd;
      uint32_t e[2 * D];
      e[0] = o[W];
      if constexpr (ALIGNED) {
        const uint32_t a = e[0];
        e[1] = pick(xodd, pick(last, a << (h - 1u), a >> 1), pick(first, a >> (h - 1u), a << 1));
        e[2] = __funnelshift_rc(a, o[next], h);
        e[3] = __funnelshift_lc(o[prev], a, h);
        if constexpr (D == 3) {
          e[4] = o[z_up.at];
          e[5] = o[z_dn.at];
        }
      } else {
        e[1] = pick(xodd, pick(last, read32(o, x_up_wrap), read32(o, x_up)),
                    pick(first, read32(o, x_dn_wrap), read32(o, x_dn)));
        e[2] = read32(o, y_up);
        e[3] = read32(o, y_dn);
        if constexpr (D == 3) {
          e[2] = pick(top, read32(o, y_up_wrap), e[2]);
          e[3] = pick(bottom, read32(o, y_dn_wrap), e[3]);
          e[4] = read32(o, z_up);
          e[5] = read32(o, z_dn);
        }
      }
#pragma unroll
      for (int q = 0; q < 2 * D; ++q) e[q] ^= b ^ J[c][q];
      unsat32<D>(e, u0, u1, u2);
    };
    auto sync = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(active) : "memory"); };
    const uint4* g_mask = p.masks + (size_t)cfg * p.nsweeps * 4u * nW + W;  // + pass * 2 nW
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(s_ring + W);
    const uint32_t npass = 2u * p.nsweeps;
    auto fetch = [&](uint32_t pass) {
      if (pass < npass) {
        const uint4* src = g_mask + (size_t)pass * 2u * nW;
        const uint32_t dst = ring + (pass % STAGES) * 32u * nW;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * nW), "l"(src + nW) : "memory");
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (uint32_t k = 0; k + 1u < STAGES; ++k) fetch(k);
    uint32_t b[2] = {s_spin[W], s_spin[pitch + W]};
    uint32_t kept = 0;                       // measurements in warp_sum
    uint64_t row = p.row0, first_sweep = 0;  // series row and sweep number of the first of them
    auto flush = [&]() {
      sync();
      for (uint32_t i = tid; i < 2u * kept; i += active) {
        const uint32_t k = i >> 1, q = i & 1u;
        if (k + p.cap < kept) continue;  // the ring keeps the last cap rows
        long long v = 0;
        for (uint32_t j = 0; j < active / 32u; ++j) v += warp_sum[j][q][k];
        const size_t rw = (size_t)((row + k) % p.cap);
        (q ? p.ser_M : p.ser_E)[rw * p.S * p.R + (size_t)s * p.R + sigma] = v;  // one temperature
        if (cfg == 0u && q == 0u) p.ser_sweep[rw] = first_sweep + (uint64_t)k * p.measure_every;
      }
      sync();
      row += kept;
      kept = 0;
    };
    // sweeps until the next measured one: sweep t is measured when (t + 1) % every == 0
    uint32_t left = p.measure_every ? (uint32_t)(p.measure_every - p.t0 % p.measure_every) : 0u;
#pragma unroll 1
    for (uint32_t it = 0; it < p.nsweeps; ++it) {
      uint32_t v0 = 0, v1 = 0, v2 = 0;
#pragma unroll
      for (uint32_t c = 0; c < 2u; ++c) {
        const uint32_t pass = 2u * it + c;
        asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
        const uint4* m = s_ring + (size_t)(pass % STAGES) * 2u * nW + W;
        const uint4 f = m[0], f4 = m[nW];
        fetch(pass + STAGES - 1u);  // into the stage read one pass ago
        uint32_t u0, u1, u2;
        classes(c, b[c], u0, u1, u2);
        const uint32_t lower = pick(u1, pick(u0, f.w, f.z), pick(u0, f.y, f.x));
        const uint32_t flip = pick(u2, D == 3 ? pick(u1, f4.z, pick(u0, f4.y, f4.x)) : f4.x, lower);
        b[c] ^= flip;
        if (own) {
          s_spin[c * pitch + W] = b[c];
          if (W == 0u) s_spin[c * pitch + nW] = b[c];
        }
        if (c == 1u) {  // the classes after the flips: 2 D - u of a flipped site, its lowest bit that of u
          v0 = u0;
          v1 = pick(flip, D == 3 ? ~(u1 ^ u0) : u1 ^ u0, u1);
          v2 = pick(flip, D == 3 ? ~(u2 ^ (u1 & u0)) : ~(u0 | u1 | u2), u2);
        }
        sync();
      }
      if (p.measure_every && --left == 0u) {
        left = p.measure_every;
        // every bond has one site of colour 1
        int e = 2 * (__popc(v0) + 2 * __popc(v1) + 4 * __popc(v2)) - 64 * D;
        int m = 64 - 2 * (__popc(b[0]) + __popc(b[1]));
        e = __reduce_add_sync(0xffffffffu, own ? e : 0);
        m = __reduce_add_sync(0xffffffffu, own ? m : 0);
        if (lane == 0u) {
          warp_sum[warp][0][kept] = e;
          warp_sum[warp][1][kept] = m;
        }
        if (kept++ == 0u) first_sweep = p.t0 + it + 1u;
        if (kept == kRowsKept) flush();
      }
    }
    if (kept) flush();
  }
  __syncthreads();
  for (uint32_t i = warp; i < 2u * nW; i += nwarps) {
    const uint32_t c = i >= nW ? 1u : 0u, Wi = i - c * nW, w = 32u * Wi + lane;
    gsp[2u * w + ((parity_of_row(w / h, L, D) ^ c) & 1u)] = (s_spin[c * pitch + Wi] >> lane & 1u) ? -1 : 1;
  }
}

size_t packed_smem(uint32_t words, uint32_t stages) {
  return 4u * ((2u * (words + 1u) + 3u) & ~3u) + (size_t)stages * 32u * words;
}

template <int D, int STAGES, bool ALIGNED>
cudaError_t packed_sweep(const Lattice& lat, const PackedParams& p) {
  const size_t smem = packed_smem(p.words, STAGES);
  cudaError_t e = cudaFuncSetAttribute(k_packed_sweep<D, STAGES, ALIGNED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kPackedSmem);
  if (e != cudaSuccess) return e;
  void* args[] = {(void*)&p};
  return launch_dependent((const void*)k_packed_sweep<D, STAGES, ALIGNED>, dim3((unsigned)(p.S * p.R)),
                          dim3(std::max(kPackedMin, (p.words + 31u) & ~31u)), args, smem, lat.stream);
}

template <int D>
cudaError_t packed_dispatch(const Lattice& lat, const PackedParams& p) {
  const uint32_t h = (uint32_t)lat.L / 2u;
  const bool deep = packed_smem(p.words, 8) <= kPackedSmem && p.words <= 768u;
  const bool aligned = 32u % h == 0u && (D == 2 || (h * (uint32_t)lat.L) % 32u == 0u);
  if (deep) return aligned ? packed_sweep<D, 8, true>(lat, p) : packed_sweep<D, 8, false>(lat, p);
  return aligned ? packed_sweep<D, 4, true>(lat, p) : packed_sweep<D, 4, false>(lat, p);
}

}  // namespace

size_t packed_mask_bytes(uint32_t N, uint64_t configs) {
  const uint64_t sweep = (uint64_t)N * configs;  // a byte a site
  if ((N / 2u) % 32u != 0u || N > 64u * 1024u || 16u * sweep > kPackedBytes) return 0;
  return (size_t)std::min<uint64_t>(kPackedBytes, 1024u * sweep);
}

// Packing and unpacking a configuration costs what a few sweeps of the other
// kernels do (4 sweeps a run, us a sweep, packed / the fastest other: L=20
// 9.5 / 8.2, L=32 17 / 12.7, 256 x 256 19 / 12; L=8, 512 configurations 13.7 /
// 12.0); from 20 sweeps on it is always ahead (6.4 / 7.7 at the least).
bool packed_i8_pays(const Lattice& lat, uint64_t nsweeps) {
  return lat.masks != nullptr && nsweeps >= 2u + lat.N / 4096u + (uint32_t)(lat.S * lat.R) / 64u;
}

cudaError_t launch_packed_i8(Lattice& lat, int inv, uint32_t nsweeps, uint32_t measure_every) {
  PackedParams p{};
  p.spins = (int8_t*)lat.spins;
  p.J = (const int8_t*)lat.J;
  p.thr = lat.thr;
  p.masks = lat.masks;
  p.S = lat.S;
  p.R = lat.R;
  p.L = lat.L;
  p.inv = inv;
  p.N = lat.N;
  p.words = lat.N / 64u;
  p.measure_every = measure_every;
  p.cap = lat.cap;
  p.ser_E = lat.ser_E;
  p.ser_M = lat.ser_M;
  p.ser_sweep = lat.ser_sweep;
  p.keys = lat.keys;
  const uint64_t sweep = (uint64_t)lat.N * lat.S * lat.R;
  const uint32_t most = (uint32_t)std::min<uint64_t>(lat.mask_bytes / sweep, 1u << 16);
  const uint32_t G = (uint32_t)(lat.S + 63) / 64u;
  uint64_t rows = lat.ser_count;
  for (uint32_t done = 0; done < nsweeps;) {
    p.nsweeps = std::min(most, nsweeps - done);
    p.t0 = lat.sweeps + done;
    p.row0 = rows;
    // warps: whole groups where there are enough of them, else fewer samples each
    const uint64_t items = (uint64_t)p.words * 2u * p.nsweeps * G * (uint32_t)lat.R;
    const uint32_t most_samples = (uint32_t)std::min(lat.S, 64);
    p.per_warp = (uint32_t)std::min<uint64_t>(most_samples, 1u + items * most_samples / (152u * 64u));
    p.parts = (most_samples + p.per_warp - 1u) / p.per_warp;
    const uint64_t warps = items * p.parts;
    const dim3 grid((unsigned)((warps + 7u) / 8u));
    if (lat.D == 3) k_packed_masks<3><<<grid, 256, 0, lat.stream>>>(p);
    else k_packed_masks<2><<<grid, 256, 0, lat.stream>>>(p);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = lat.D == 3 ? packed_dispatch<3>(lat, p) : packed_dispatch<2>(lat, p);
    if (e != cudaSuccess) return e;
    if (measure_every) rows += (p.t0 + p.nsweeps) / measure_every - p.t0 / measure_every;
    done += p.nsweeps;
  }
  return cudaSuccess;
}

}  // namespace ianus
