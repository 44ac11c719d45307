// potts_words.cuh -- what the two q = 4 Potts models share (k_potts.cu,
// k_perm.cu): words of 4 samples (byte b = sample 4q+b, state 0..3) in
// checkerboard-split order in 2 to 4 dimensions, the bytes of a word worked
// on together; the threshold rows; the measurement.
#pragma once
#include "lattice.h"
#include "sweep_planes.cuh"

namespace ianus {
namespace potts {

constexpr int kBlock = 256;
constexpr uint32_t kOnes = 0x01010101u;

// prmt.b32: byte i of the result is byte (sel >> 4i) & 7 of {b, a}, or, with
// bit 3 of the selector nibble set, that byte's sign bit eight times
// (__byte_perm clears those selector bits).
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}

struct Grid {
  FastDiv half, h, L;  // words per colour, L/2, L
  uint32_t N;
};

inline Grid make_grid(const Geom& g) {
  return Grid{fast_div(g.half), fast_div((uint32_t)g.h), fast_div((uint32_t)g.L), g.N};
}

template <int D>
struct Nbr {
  uint32_t self, site;
  uint32_t fw[D], bw[D];  // split indices of i + e_d and i - e_d
};

// Colour-c word w -> its split index, natural index and neighbours (all of
// the other colour, with the same x / 2 but along x).
template <int D>
__device__ __forceinline__ Nbr<D> neighbours(const Grid& g, uint32_t c, uint32_t w) {
  const uint32_t h = g.h.d, L = g.L.d;
  const uint32_t row = div_by(w, g.h), k = w - row * h;
  uint32_t co[D], r = row, psum = c;
#pragma unroll
  for (int d = 1; d < D; ++d) {
    if (d + 1 < D) {
      const uint32_t q = div_by(r, g.L);
      co[d] = r - q * L;
      r = q;
    } else {
      co[d] = r;  // the last coordinate is below L already
    }
    psum ^= co[d];
  }
  const uint32_t xpar = psum & 1u;
  Nbr<D> n;
  n.self = w + (row + c) * h;
  n.site = 2u * w + xpar;
  const uint32_t base_o = 2u * (w - k) + (1u - c) * h, ko = base_o + k;
  uint32_t kp = k + xpar, km = k + xpar - 1u;  // (x + 1) / 2 and (x - 1) / 2, mod h
  if (kp == h) kp = 0u;
  if (km == 0xffffffffu) km = h - 1u;
  n.fw[0] = base_o + kp;
  n.bw[0] = base_o + km;
  uint32_t stride = 2u * h;
#pragma unroll
  for (int d = 1; d < D; ++d) {
    const uint32_t back = stride * (L - 1u);
    n.fw[d] = ko + (co[d] == L - 1u ? 0u - back : stride);
    n.bw[d] = ko + (co[d] == 0u ? back : 0u - stride);
    stride *= L;
  }
  return n;
}

// What a block of a sweep works on: `per` colour words of the flattened list
// (replica group, quad, word) of one temperature slot (blockIdx.y).
struct Params {
  uint32_t* spins;         // [slots][Q4][N]
  const uint32_t* J;       // [Q4][D][N]
  const uint4* tab;        // [K][rows]: T0, T1, T2 (2^32 - 1 where the threshold is 2^32), flags of those
  const int32_t* temp_of;  // [S][R][K]
  Grid grid;
  FastDiv quads;           // Q4 words of 4 samples
  int S, R, K, slots;
  uint32_t colour;
  uint32_t t_lo, t_hi;
  uint32_t per;            // words per block, < 2^30
  uint64_t first, end;     // this launch's words of a temperature slot's R / RT * Q4 * half
  PhiloxKeys keys;
  const uint64_t* t_dev;  // non-null in captured graphs
};

// Smallest k with r < T_k, else 3.  Where T_k = 2^32 the row holds 2^32 - 1
// and its flag: only r = 2^32 - 1 needs the flags.
__device__ __forceinline__ uint32_t pick(const uint4& T, uint32_t r) {
  return r >= T.z ? 3u : r >= T.y ? 2u : r >= T.x ? 1u : 0u;
}

__device__ __forceinline__ uint32_t pick_last(const uint4& T) { return 3u - __popc(T.w & 7u); }

// Sweeps the block's words.  Model supplies
//   kRows: rows of a temperature's table;
//   prepare(J, N, n): coupling words of a site;
//   rows(sf, sb, row): table rows of the 4 samples of a word with those
//     couplings, from the neighbours i + e_d and i - e_d in one replica.
// RT replicas of a site are done together (they share the couplings, the
// index arithmetic and the site's part of the first two Philox rounds).  KONE
// (one temperature): its table is in shared memory, staged before the wait
// for the previous colour pass (nothing a pass writes is read); otherwise
// each sample reads the row of its temperature from global memory.
template <class Model, int D, int RT, bool KONE>
__device__ __forceinline__ void sweep_words(const Params& p, uint4* tab) {
  if (KONE)
    for (uint32_t i = threadIdx.x; i < Model::kRows; i += kBlock) tab[i] = __ldg(p.tab + i);
  dependent_launch_entry();
  const Tick tk = sweep_tick(p.t_lo, p.t_hi, p.t_dev);
  const int tslot = blockIdx.y;
  const uint32_t N = p.grid.N;
  const uint64_t w0 = p.first + (uint64_t)blockIdx.x * p.per;
  const uint32_t count = (uint32_t)min((uint64_t)p.per, p.end - w0);
  const uint32_t piece0 = (uint32_t)(w0 / p.grid.half.d);
  const uint32_t off0 = (uint32_t)(w0 - (uint64_t)piece0 * p.grid.half.d);
  if (KONE) __syncthreads();
  for (uint32_t i = threadIdx.x; i < count; i += kBlock) {
    const uint32_t o = off0 + i, dp = div_by(o, p.grid.half);
    const uint32_t piece = piece0 + dp, w = o - dp * p.grid.half.d;
    const uint32_t ag = div_by(piece, p.quads), q = piece - ag * p.quads.d;
    const Nbr<D> n = neighbours<D>(p.grid, p.colour, w);
    const uint32_t sigma0 = (uint32_t)tslot * (uint32_t)p.R + ag * RT;
    uint32_t* sp0 = p.spins + ((size_t)sigma0 * p.quads.d + q) * N;
    const size_t slot = (size_t)p.quads.d * N;
    // every load of the site first; the random words, which need none of
    // them, while they are in flight
    Model m;
    m.prepare(p.J + (size_t)q * D * N, N, n);
    uint32_t sf[RT][D], sb[RT][D];
#pragma unroll
    for (int ra = 0; ra < RT; ++ra)
#pragma unroll
      for (int d = 0; d < D; ++d) {
        sf[ra][d] = sp0[ra * slot + n.fw[d]];
        sb[ra][d] = sp0[ra * slot + n.bw[d]];
      }
    const planes::PlaneSiteKey sk = planes::plane_site_key(n.site, tk, p.keys);
    uint4 x[RT];
#pragma unroll
    for (int ra = 0; ra < RT; ++ra) {
      const uint32_t c2 = (TAG_POTTS << 28) | ((sigma0 + (uint32_t)ra) << 16) | q;
      x[ra] = planes::philox10_split(sk, planes::plane_uniform(c2, tk, p.keys), p.keys);
    }
#pragma unroll
    for (int ra = 0; ra < RT; ++ra) {
      const uint32_t a = ag * RT + (uint32_t)ra;
      uint32_t row[4];
      m.rows(sf[ra], sb[ra], row);
      const uint32_t r[4] = {x[ra].x, x[ra].y, x[ra].z, x[ra].w};
      const uint4* tb[4];
      if (!KONE) {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int s = 4 * (int)q + b;
          const int k = s < p.S ? p.temp_of[((size_t)s * p.R + a) * p.K + tslot] : tslot;
          tb[b] = p.tab + (size_t)k * Model::kRows;
        }
      }
      uint32_t out = 0;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const uint4 T = KONE ? tab[row[b]] : __ldg(tb[b] + row[b]);
        out |= pick(T, r[b]) << (8 * b);
      }
      if (max(max(r[0], r[1]), max(r[2], r[3])) == 0xffffffffu) {
#pragma unroll
        for (int b = 0; b < 4; ++b)
          if (r[b] == 0xffffffffu) {
            const uint4 T = KONE ? tab[row[b]] : __ldg(tb[b] + row[b]);
            out = (out & ~(0xFFu << (8 * b))) | (pick_last(T) << (8 * b));
          }
      }
      sp0[ra * slot + n.self] = out;
    }
  }
}

// One colour pass with kernel k, RT replicas a thread, blocks_per_sm blocks
// per SM at a time, whole warps of words.
inline cudaError_t launch_sweep(Lattice& lat, int colour, uint64_t t, const void* k, int RT, uint32_t blocks_per_sm) {
  Params p;
  p.spins = (uint32_t*)lat.spins;
  p.J = (const uint32_t*)lat.J;
  p.tab = lat.ptab;
  p.temp_of = lat.temp_of;
  p.grid = make_grid(lat.geom);
  p.S = lat.S;
  p.R = lat.R;
  p.K = lat.K;
  p.quads = fast_div((uint32_t)lat.Q4);
  p.slots = lat.slots;
  p.colour = (uint32_t)colour;
  p.t_lo = (uint32_t)(t & 0xffffffffu);
  p.t_hi = (uint32_t)(t >> 32);
  p.keys = lat.keys;
  p.t_dev = lat.capturing ? lat.t_dev : nullptr;
  const uint64_t pieces = (uint64_t)(p.R / RT) * (uint64_t)lat.Q4, total = pieces * p.grid.half.d;
  const uint64_t n = lat.chains > 1 ? (uint64_t)lat.chains : 1u;  // this chain's share, whole pieces
  p.first = pieces * (uint64_t)lat.chain / n * p.grid.half.d;
  p.end = pieces * ((uint64_t)lat.chain + 1u) / n * p.grid.half.d;
  // one wave of blocks; two or four where a thread keeps 5 or 10 words, so that
  // blocks working at the same time are neighbours in memory and the last ones
  // are short (potts_L64 64 x 2: 1695 -> 1658 us for 20 sweeps; L=96, 128 x 2:
  // 2866 -> 2701 us for 5; L=32, 128 x 2, 3.4 words a thread, would lose 8 %)
  const uint64_t wave = 152ull * blocks_per_sm, per_thread = total * p.K / (wave * kBlock);
  const uint64_t waves = per_thread >= 40 ? 4 : per_thread >= 10 ? 2 : 1;
  const uint64_t want = std::max<uint64_t>(1, wave * waves / (uint64_t)p.K);
  const uint64_t per = std::min<uint64_t>(((total + want - 1) / want + 31) / 32 * 32, 1u << 29);
  p.per = (uint32_t)per;
  void* args[] = {(void*)&p};
  return launch_dependent(k, dim3((unsigned)((p.end - p.first + per - 1) / per), (unsigned)p.K), dim3(kBlock), args, 0,
                          lat.stream);
}

// ---- measurement ----
//
// Per sample and configuration: the satisfied forward bonds (what they add to
// -E is the model's, MODEL below) and the state counts, and for two replicas
// the sites where they agree.  Bytes of a word count together: a thread's
// counters are packed bytes over kMeasIters sites (at most 4 kMeasIters
// <= 255), then 16-bit pairs summed over the warp.  J-weighted model, L=32,
// 128 x 2: 18 us with the overlap in the same pass (57 + 24 us in two, sample
// by sample).
constexpr int kMeasIters = 32;

// bytes -> 1 where the two low bits of x are 0, else 0
__device__ __forceinline__ uint32_t zero2(uint32_t x) { return ~(x | (x >> 1)) & kOnes; }

// Sum of the packed byte counter over the warp: v[b] = byte b's total.
__device__ __forceinline__ void warp_bytes(uint32_t c, int* v) {
  const uint32_t e = __reduce_add_sync(0xffffffffu, c & 0x00ff00ffu);
  const uint32_t o = __reduce_add_sync(0xffffffffu, (c >> 8) & 0x00ff00ffu);
  v[0] = (int)(e & 0xffffu);
  v[1] = (int)(o & 0xffffu);
  v[2] = (int)(e >> 16);
  v[3] = (int)(o >> 16);
}

struct MeasParams {
  const uint32_t* spins;
  const uint32_t* J;
  int64_t* acc;
  Grid grid;
  int S, Q4, slots;
  uint32_t iters;  // sites per thread, at most kMeasIters
};

// Grid (chunks, slots / RT * Q4): RT replicas of one quad together (RT = 2
// only with one temperature, replicas 0 and 1), their overlap too.
template <class Model, int D, int RT>
__global__ void __launch_bounds__(kBlock) k_measure(const MeasParams p) {
  const uint32_t sg = blockIdx.y / (uint32_t)p.Q4, q = blockIdx.y - sg * (uint32_t)p.Q4;
  const uint32_t N = p.grid.N, half = p.grid.half.d;
  const uint32_t* Jq = p.J + (size_t)q * D * N;
  uint32_t good[RT], bad[RT], lo[RT], hi[RT], both[RT], same = 0, sites = 0;
#pragma unroll
  for (int a = 0; a < RT; ++a) good[a] = bad[a] = lo[a] = hi[a] = both[a] = 0;
  const uint32_t base = blockIdx.x * (kBlock * p.iters);
  for (uint32_t it = 0; it < p.iters; ++it) {
    const uint32_t j = base + it * kBlock + threadIdx.x;
    if (j >= N) break;
    const uint32_t c = j >= half ? 1u : 0u;
    const Nbr<D> n = neighbours<D>(p.grid, c, j - c * half);
    uint32_t jw[D], s0 = 0;
#pragma unroll
    for (int d = 0; d < D; ++d) jw[d] = __ldg(Jq + (size_t)d * N + n.self);
#pragma unroll
    for (int a = 0; a < RT; ++a) {
      const uint32_t* sp = p.spins + ((size_t)(sg * RT + a) * p.Q4 + q) * N;
      const uint32_t s = sp[n.self];
#pragma unroll
      for (int d = 0; d < D; ++d) Model::count_bond(s, sp[n.fw[d]], jw[d], good[a], bad[a]);
      lo[a] += s & kOnes;
      hi[a] += (s >> 1) & kOnes;
      both[a] += s & (s >> 1) & kOnes;
      if (a == 0) s0 = s;
      else same += zero2(s0 ^ s);
    }
    ++sites;
  }
  // per warp and sample: sites, overlap, then good, bad, lo, hi, both of each
  // replica; the block's sums by one thread per (replica, sample) and value
  constexpr int NV = 2 + 5 * RT;
  __shared__ __align__(16) int red[kBlock / 32][NV][4];
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
  {
    int v[NV][4];
    const int tot = (int)__reduce_add_sync(0xffffffffu, sites);
    v[0][0] = v[0][1] = v[0][2] = v[0][3] = tot;
    warp_bytes(same, v[1]);
#pragma unroll
    for (int a = 0; a < RT; ++a) {
      warp_bytes(good[a], v[2 + 5 * a]);
      warp_bytes(bad[a], v[3 + 5 * a]);
      warp_bytes(lo[a], v[4 + 5 * a]);
      warp_bytes(hi[a], v[5 + 5 * a]);
      warp_bytes(both[a], v[6 + 5 * a]);
    }
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < NV; ++i) *(int4*)red[warp][i] = make_int4(v[i][0], v[i][1], v[i][2], v[i][3]);
    }
  }
  __syncthreads();
  // thread (a, b): replica a's sample b
  if (threadIdx.x < 4u * RT) {
    const int a = (int)(threadIdx.x >> 2), b = (int)(threadIdx.x & 3u), s = 4 * (int)q + b;
    if (s < p.S) {
      int t[7] = {0, 0, 0, 0, 0, 0, 0};
#pragma unroll
      for (int w = 0; w < kBlock / 32; ++w) {
        t[0] += red[w][0][b];
        t[1] += red[w][1][b];
#pragma unroll
        for (int i = 0; i < 5; ++i) t[2 + i] += red[w][2 + 5 * a + i][b];
      }
      int64_t* ac = p.acc + ((size_t)s * p.slots + sg * RT + a) * kAccStride;
      const long long v[5] = {(long long)(t[3] - t[2]), (long long)(t[0] - t[4] - t[5] + t[6]),
                              (long long)(t[4] - t[6]), (long long)(t[5] - t[6]), (long long)t[6]};
      atomicAdd((unsigned long long*)&ac[0], (unsigned long long)v[0]);
#pragma unroll
      for (int f = 0; f < 4; ++f) atomicAdd((unsigned long long*)&ac[2 + f], (unsigned long long)v[1 + f]);
      if (RT == 2 && a == 0) atomicAdd((unsigned long long*)&ac[6], (unsigned long long)t[1]);
    }
  }
}

// E, the state counts and (want_q) the overlap of every configuration; k1 and
// k2 take one and two replicas a thread.
template <class Kernel>
inline cudaError_t launch_measure(Lattice& lat, int want_q, Kernel k1, Kernel k2) {
  cudaError_t e = cudaMemsetAsync(lat.acc, 0, (size_t)lat.S * lat.slots * kAccStride * sizeof(int64_t), lat.stream);
  if (e != cudaSuccess) return e;
  const bool two = lat.K == 1 && lat.R == 2;
  MeasParams p;
  p.spins = (const uint32_t*)lat.spins;
  p.J = (const uint32_t*)lat.J;
  p.acc = lat.acc;
  p.grid = make_grid(lat.geom);
  p.S = lat.S;
  p.Q4 = lat.Q4;
  p.slots = lat.slots;
  // about 8 blocks per SM, at most kMeasIters sites a thread
  const uint64_t ys = (uint64_t)(two ? 1 : lat.slots) * (uint64_t)lat.Q4;
  const uint64_t want = std::max<uint64_t>(1, 152ull * 8 / ys);
  p.iters = (uint32_t)std::min<uint64_t>(kMeasIters, std::max<uint64_t>(1, (lat.N + want * kBlock - 1) / (want * kBlock)));
  const uint32_t per = (uint32_t)kBlock * p.iters;
  (two ? k2 : k1)<<<dim3((lat.N + per - 1) / per, (unsigned)ys), kBlock, 0, lat.stream>>>(p);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return want_q && lat.R >= 2 && !two ? launch_overlap_potts(lat) : cudaSuccess;
}

}  // namespace potts
}  // namespace ianus
