// k_msc.cu -- the bit-sliced multispin layout (IANUS_LAYOUT_BITS64).
//
// A 64-bit word holds one site of 64 independent disorder samples (lane l =
// sample mod 64), the multi-sample idea of Sec. 4.1.1 carried to a GPU word,
// with an independent random stream per sample.  Words of one colour are
// stored next to each other (checkerboard-split order, Sec. 3.1), so the own
// word, the 2D neighbour words and the coupling words of a warp are
// contiguous loads.
//
// Update cell (Sec. 3.2) in bit-sliced form, per word:
//   e_j = b_i ^ b_j ^ c_ij                    unsatisfied-bond bits (2D words)
//   (u2,u1,u0) = carry-save adder tree of the e_j  (u = 0..2D per lane)
//   m_u = lanes whose count is u              (class masks)
//   threshold bit-plane p: t_p = OR_u (m_u & TP[u][p])
//   lazy compare from the most significant plane: lanes stay undecided while
//   their random bit equals the threshold bit; lt collects r < T.
//   flip = lt ^ inv (Metropolis: inv = 0; heat bath: inv = ~0)
// TP[u][p] are 64-bit lane masks, so every lane can carry its own threshold
// (parallel tempering moves temperatures per sample).
#include <algorithm>
#include <cmath>

#include "lattice.h"
#include "sweep_planes.cuh"

namespace ianus {

namespace {

constexpr int kBlock = 256;

using planes::bits_sweep_smem;
using planes::class_select;

// The per-lane-plane sweep, precompiled (sweep_planes.cuh).
template <int D, int ALGO, int RT, bool P2, bool Q = (ALGO == 1)>
__global__ void __launch_bounds__(kBlock, Q ? 3 : 4) k_sweep_bits(const BitsParams p) {
  planes::sweep_planes_body<D, ALGO, RT, P2, Q>(p, p.geom);
}

// Random-field model (Eq. 2 with h_i = +-|h|, x_i = 1): the class of a lane
// is (u, f) with f = [s_i h_i > 0] = ~(b_i ^ hb_i), hb_i = lane bit set
// where h_i < 0.  TP[p][8 f + u] are per-lane threshold planes as above; a
// lane with T = 2^32 is decided without a random number, every other lane
// compares (T = 0 lanes end at the first set bit of r).
template <int D, int ALGO, bool P2>
__global__ void __launch_bounds__(kBlock) k_sweep_bits_field(const BitsParams p, const uint64_t* __restrict__ hbits) {
  constexpr int NF = kFieldPlaneClasses;
  extern __shared__ uint64_t sm_tp[];  // [R][kPlanes][NF]
  const int R = p.R;
  const int gt = blockIdx.y;
  const int g = gt / p.K, tslot = gt - g * p.K;
  {
    const uint64_t* src = p.tp + ((size_t)g * p.slots + (size_t)tslot * R) * kPlanes * NF;
    for (int k = threadIdx.x; k < R * kPlanes * NF; k += kBlock) sm_tp[k] = src[k];
  }
  __syncthreads();
  const Geom geom = p.geom;
  const uint32_t N = geom.N;
  const uint64_t* Jg = p.J + (size_t)g * D * N;
  const uint64_t* Hg = hbits + (size_t)g * N;
  const Tick tk = sweep_tick(p.t_lo, p.t_hi, p.t_dev);
  const uint32_t w_begin = blockIdx.x * p.words_per_block;
  const uint32_t w_end = min(w_begin + p.words_per_block, geom.half);
  for (uint32_t w = w_begin + threadIdx.x; w < w_end; w += kBlock) {
    const Nbr n = split_neighbours_t<P2>(geom, p.colour, w);
    uint64_t jw[2 * D];
    jw[0] = __ldg(Jg + n.self);
    jw[1] = __ldg(Jg + n.xm);
    jw[2] = __ldg(Jg + N + n.self);
    jw[3] = __ldg(Jg + N + n.ym);
    if (D == 3) {
      jw[4] = __ldg(Jg + 2u * N + n.self);
      jw[5] = __ldg(Jg + 2u * N + n.zm);
    }
    const uint64_t hb = __ldg(Hg + n.self);
#pragma unroll 1
    for (int a = 0; a < R; ++a) {
      const int sigma = tslot * R + a;
      uint64_t* sp = p.spins + ((size_t)g * p.slots + sigma) * N;
      const uint64_t b = sp[n.self];
      uint64_t e[2 * D];
      e[0] = b ^ sp[n.xp] ^ jw[0];
      e[1] = b ^ sp[n.xm] ^ jw[1];
      e[2] = b ^ sp[n.yp] ^ jw[2];
      e[3] = b ^ sp[n.ym] ^ jw[3];
      if (D == 3) {
        e[4] = b ^ sp[n.zp] ^ jw[4];
        e[5] = b ^ sp[n.zm] ^ jw[5];
      }
      uint64_t u0, u1, u2;
      count_unsat<D>(e, u0, u1, u2);
      const uint64_t f = ~(b ^ hb);
      uint64_t mc[2][2 * D + 1];
#pragma unroll
      for (int u = 0; u <= 2 * D; ++u) {
        const uint64_t m = ((u & 4) ? u2 : ~u2) & ((u & 2) ? u1 : ~u1) & ((u & 1) ? u0 : ~u0);
        mc[0][u] = m & ~f;
        mc[1][u] = m & f;
      }
      const uint64_t* tpa = sm_tp + (size_t)a * kPlanes * NF;
      uint64_t always = 0;
#pragma unroll
      for (int u = 0; u <= 2 * D; ++u)
        always |= (mc[0][u] & tpa[32 * NF + u]) | (mc[1][u] & tpa[32 * NF + 8 + u]);
      uint64_t lt = always;
      uint64_t und = ~always;
      const uint32_t c2 = (TAG_SPIN << 28) | ((uint32_t)sigma << 12) | (uint32_t)g;
#pragma unroll 1
      for (uint32_t mm = 0; mm < 16u && und != 0ull; ++mm) {
        const uint4 x = philox10(n.site, tk.lo, c2 | (mm << 24), tk.hi, p.keys);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const uint64_t r = q == 0 ? ((uint64_t)x.x | ((uint64_t)x.y << 32))
                                    : ((uint64_t)x.z | ((uint64_t)x.w << 32));
          const uint64_t* row = tpa + (2u * mm + (uint32_t)q) * NF;
          uint64_t tb = 0;
#pragma unroll
          for (int u = 0; u <= 2 * D; ++u) tb |= (mc[0][u] & row[u]) | (mc[1][u] & row[8 + u]);
          lt |= und & ~r & tb;
          und &= ~(r ^ tb);
        }
      }
      const uint64_t flip = (ALGO == 0) ? lt : ~lt;
      if (flip) sp[n.self] = b ^ flip;
    }
  }
}

// Diluted model (DAFF; Eq. 2 with x_i in {0,1}), generic per-lane planes.
// Per neighbour j the bond contributes c_j = x_j (1 - 2 e_j) to v (e_j the
// unsatisfied bit); c_j + 1 in {0, 1, 2} is 2 hi_j + lo_j with hi_j = x_j &
// ~e_j and lo_j = ~x_j, so t = v + 2D = 2 sum(hi) + sum(lo), 4 bit-planes.
// The plane class is 16 f + t.  Empty sites are never updated.
template <int D, int ALGO, bool P2>
__global__ void __launch_bounds__(kBlock) k_sweep_bits_dilute(const BitsParams p, const uint64_t* __restrict__ hbits,
                                                              const uint64_t* __restrict__ xbits) {
  constexpr int NF = kDiluteClasses;
  constexpr int NT = 4 * D + 1;  // t = 0..4D
  extern __shared__ uint64_t sm_tp[];  // [R][kPlanes][NF]
  const int R = p.R;
  const int gt = blockIdx.y;
  const int g = gt / p.K, tslot = gt - g * p.K;
  {
    const uint64_t* src = p.tp + ((size_t)g * p.slots + (size_t)tslot * R) * kPlanes * NF;
    for (int k = threadIdx.x; k < R * kPlanes * NF; k += kBlock) sm_tp[k] = src[k];
  }
  __syncthreads();
  const Geom geom = p.geom;
  const uint32_t N = geom.N;
  const uint64_t* Jg = p.J + (size_t)g * D * N;
  const uint64_t* Hg = hbits + (size_t)g * N;
  const uint64_t* Xg = xbits + (size_t)g * N;
  const Tick tk = sweep_tick(p.t_lo, p.t_hi, p.t_dev);
  const uint32_t w_begin = blockIdx.x * p.words_per_block;
  const uint32_t w_end = min(w_begin + p.words_per_block, geom.half);
  for (uint32_t w = w_begin + threadIdx.x; w < w_end; w += kBlock) {
    const Nbr n = split_neighbours_t<P2>(geom, p.colour, w);
    uint64_t jw[2 * D], xw[2 * D];
    jw[0] = __ldg(Jg + n.self);
    jw[1] = __ldg(Jg + n.xm);
    jw[2] = __ldg(Jg + N + n.self);
    jw[3] = __ldg(Jg + N + n.ym);
    xw[0] = __ldg(Xg + n.xp);
    xw[1] = __ldg(Xg + n.xm);
    xw[2] = __ldg(Xg + n.yp);
    xw[3] = __ldg(Xg + n.ym);
    if (D == 3) {
      jw[4] = __ldg(Jg + 2u * N + n.self);
      jw[5] = __ldg(Jg + 2u * N + n.zm);
      xw[4] = __ldg(Xg + n.zp);
      xw[5] = __ldg(Xg + n.zm);
    }
    const uint64_t hb = __ldg(Hg + n.self), xs = __ldg(Xg + n.self);
    uint64_t lo[2 * D];
#pragma unroll
    for (int j = 0; j < 2 * D; ++j) lo[j] = ~xw[j];
    uint64_t l0, l1, l2;
    count_unsat<D>(lo, l0, l1, l2);  // sum of lo_j
#pragma unroll 1
    for (int a = 0; a < R; ++a) {
      const int sigma = tslot * R + a;
      uint64_t* sp = p.spins + ((size_t)g * p.slots + sigma) * N;
      const uint64_t b = sp[n.self];
      uint64_t hi[2 * D];
      hi[0] = xw[0] & ~(b ^ sp[n.xp] ^ jw[0]);
      hi[1] = xw[1] & ~(b ^ sp[n.xm] ^ jw[1]);
      hi[2] = xw[2] & ~(b ^ sp[n.yp] ^ jw[2]);
      hi[3] = xw[3] & ~(b ^ sp[n.ym] ^ jw[3]);
      if (D == 3) {
        hi[4] = xw[4] & ~(b ^ sp[n.zp] ^ jw[4]);
        hi[5] = xw[5] & ~(b ^ sp[n.zm] ^ jw[5]);
      }
      uint64_t h0, h1, h2;
      count_unsat<D>(hi, h0, h1, h2);
      // t = 2 (h2 h1 h0) + (l2 l1 l0) <= 4D < 16
      const uint64_t t0 = l0, t1 = h0 ^ l1, k1 = h0 & l1;
      const uint64_t t2 = h1 ^ l2 ^ k1, k2 = (h1 & l2) | (h1 & k1) | (l2 & k1);
      const uint64_t t3 = h2 ^ k2;
      const uint64_t f = ~(b ^ hb);
      uint64_t mc[2][NT];
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        const uint64_t m = ((t & 8) ? t3 : ~t3) & ((t & 4) ? t2 : ~t2) & ((t & 2) ? t1 : ~t1) & ((t & 1) ? t0 : ~t0);
        mc[0][t] = m & ~f;
        mc[1][t] = m & f;
      }
      const uint64_t* tpa = sm_tp + (size_t)a * kPlanes * NF;
      uint64_t always = 0;
#pragma unroll
      for (int t = 0; t < NT; ++t) always |= (mc[0][t] & tpa[32 * NF + t]) | (mc[1][t] & tpa[32 * NF + 16 + t]);
      always &= xs;
      uint64_t lt = always;
      uint64_t und = ~always & xs;
      const uint32_t c2 = (TAG_SPIN << 28) | ((uint32_t)sigma << 12) | (uint32_t)g;
#pragma unroll 1
      for (uint32_t mm = 0; mm < 16u && und != 0ull; ++mm) {
        const uint4 x = philox10(n.site, tk.lo, c2 | (mm << 24), tk.hi, p.keys);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const uint64_t r = q == 0 ? ((uint64_t)x.x | ((uint64_t)x.y << 32))
                                    : ((uint64_t)x.z | ((uint64_t)x.w << 32));
          const uint64_t* row = tpa + (2u * mm + (uint32_t)q) * NF;
          uint64_t tb = 0;
#pragma unroll
          for (int t = 0; t < NT; ++t) tb |= (mc[0][t] & row[t]) | (mc[1][t] & row[16 + t]);
          lt |= und & ~r & tb;
          und &= ~(r ^ tb);
        }
      }
      const uint64_t flip = ((ALGO == 0) ? lt : ~lt) & xs;
      if (flip) sp[n.self] = b ^ flip;
    }
  }
}

// Site disorder of the bit-sliced field models, lane bit l of word (g, i)
// for sample 64 g + l: hbits = [h_i < 0] (RFIM: the H stream; DAFF: 0),
// xbits = [x_i = 1] (RFIM: all; DAFF: r_x < T_occ, r_x from the 32 planes of
// the X stream compared from the most significant plane down).
__global__ void k_init_sites_bits(uint64_t* hbits, uint64_t* xbits, Geom geom, int G, int rfim, int daff,
                                  uint64_t T_occ, PhiloxKeys keys) {
  const uint64_t total = (uint64_t)G * geom.N;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t g = (uint32_t)(idx / geom.N), i = (uint32_t)(idx - (uint64_t)g * geom.N);
    const uint32_t L = (uint32_t)geom.L;
    const int x = (int)(i % L), y = (int)((i / L) % L), z = geom.D == 3 ? (int)(i / (L * L)) : 0;
    const size_t j = (size_t)g * geom.N + split_index(geom, x, y, z);
    uint64_t hw = 0, xw = ~0ull;
    if (rfim) {
      const uint4 r = philox10(i, 0u, (TAG_H << 28) | g, 0u, keys);
      hw = (uint64_t)r.x | ((uint64_t)r.y << 32);
    }
    if (daff) {
      if (T_occ >= kTwo32) {
        xw = ~0ull;
      } else {
        uint64_t lt = 0, und = ~0ull;
        for (uint32_t m = 0; m < 16u && und != 0ull; ++m) {
          const uint4 r = philox10(i, 0u, (TAG_X << 28) | (m << 24) | g, 0u, keys);
          for (int q = 0; q < 2; ++q) {
            const uint64_t w = q == 0 ? ((uint64_t)r.x | ((uint64_t)r.y << 32)) : ((uint64_t)r.z | ((uint64_t)r.w << 32));
            const uint64_t tb = ((T_occ >> (31u - (2u * m + (uint32_t)q))) & 1ull) ? ~0ull : 0ull;
            lt |= und & ~w & tb;
            und &= ~(w ^ tb);
          }
        }
        xw = lt;
      }
    }
    hbits[j] = hw;
    xbits[j] = xw;
  }
}

__global__ void k_get_sites_bits(const uint64_t* hbits, const uint64_t* xbits, int8_t* out_hs, int8_t* out_occ,
                                 Geom geom, int S) {
  const uint64_t total = (uint64_t)S * geom.N;
  const uint32_t L = (uint32_t)geom.L;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t i = (uint32_t)(idx % geom.N);
    const int s = (int)(idx / geom.N);
    const int x = (int)(i % L), y = (int)((i / L) % L), z = geom.D == 3 ? (int)(i / (L * L)) : 0;
    const size_t j = (size_t)(s >> 6) * geom.N + split_index(geom, x, y, z);
    out_hs[idx] = ((hbits[j] >> (s & 63)) & 1ull) ? -1 : 1;
    out_occ[idx] = (int8_t)((xbits[j] >> (s & 63)) & 1ull);
  }
}

__global__ void k_set_sites_bits(uint64_t* hbits, uint64_t* xbits, const int8_t* in_hs, const int8_t* in_occ,
                                 Geom geom, int S, int G) {
  const uint64_t total = (uint64_t)G * geom.N;
  const uint32_t L = (uint32_t)geom.L;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t i = (uint32_t)(idx % geom.N);
    const int g = (int)(idx / geom.N);
    const int x = (int)(i % L), y = (int)((i / L) % L), z = geom.D == 3 ? (int)(i / (L * L)) : 0;
    const size_t j = (size_t)g * geom.N + split_index(geom, x, y, z);
    uint64_t hw = hbits[j], xw = xbits[j];
    for (int l = 0; l < 64; ++l) {
      const int s = 64 * g + l;
      if (s >= S) break;
      const uint64_t hbit = in_hs[(size_t)s * geom.N + i] < 0 ? 1ull : 0ull;
      const uint64_t xbit = in_occ[(size_t)s * geom.N + i] ? 1ull : 0ull;
      hw = (hw & ~(1ull << l)) | (hbit << l);
      xw = (xw & ~(1ull << l)) | (xbit << l);
    }
    hbits[j] = hw;
    xbits[j] = xw;
  }
}

// ---- fused serving: several jobs in the lanes of one group ----
//
// One block per (word range, group).  The block stages the group's per-lane
// threshold planes, its segment table and, per running segment and plane
// pair, the part of Philox rounds 0 and 1 that its sites share
// (plane_uniform).  Per plane pair every segment that still has undecided
// lanes draws one Philox block from its own stream (key of the job's seed,
// counter of the job's sweep) and contributes its bits 0..n-1 shifted to its
// lanes.  Heat-bath lanes flip on "not less" (inv lanes), Metropolis lanes on
// "less"; lanes of no live segment never flip.
//
// T neighbouring threads share a word: thread j of them draws pairs m + j of
// all segments, the T pairs' random words then pass through shuffles and every
// thread does the compare.  A word's blocks are otherwise a serial chain (four
// pairs times its segments): with few words T = 4 is the faster, with many the
// repeated compare costs more than it hides.  L=16, 4 groups, 9 jobs: 6.5 us
// per colour pass and a launch per sweep to advance the counters -> 3.6 us.
constexpr int kFusedBlock = 128;

struct FusedParams {
  BitsParams b;          // t_lo: sweeps since the segments' counters were advanced
  const Segment* segs;
  const uint32_t* nseg;
  int early;             // the tables were last written before the previous kernel started
};

struct FusedShared {
  uint64_t tpa[kPlanes * kMaxClasses];
  uint4 u[kMaxSegs * 16];              // shared part of rounds 0 and 1 per (segment, pair)
  uint64_t mask[kMaxSegs];
  uint32_t klo[kMaxSegs], khi[kMaxSegs], lane0[kMaxSegs], thi[kMaxSegs];
  uint64_t live, inv;
  int n;
};

__device__ __forceinline__ void stage_fused(FusedShared& sh, const FusedParams& fp, int g) {
  const BitsParams& p = fp.b;
  for (int k = threadIdx.x; k < kPlanes * kMaxClasses; k += kFusedBlock)
    sh.tpa[k] = p.tp[(size_t)g * kPlanes * kMaxClasses + k];
  if (threadIdx.x < 32u) {  // one warp packs the running segments, two candidates a thread
    const uint32_t lane = threadIdx.x, ns = min(fp.nseg[g], (uint32_t)kMaxSegs);
    uint64_t live = 0, inv = 0;
    int n = 0;
    for (uint32_t j0 = 0; j0 < ns; j0 += 32u) {
      const uint32_t j = j0 + lane;
      Segment sg{};
      if (j < ns) sg = fp.segs[(size_t)g * kMaxSegs + j];
      const uint64_t t = sg.t + p.t_lo;
      const bool run = j < ns && sg.mask != 0ull && t < sg.t_end;
      const uint32_t bal = __ballot_sync(0xffffffffu, run);
      if (run) {
        const int i = n + __popc(bal & ((1u << lane) - 1u));
        sh.mask[i] = sg.mask;
        sh.klo[i] = sg.key_lo;
        sh.khi[i] = sg.key_hi;
        sh.lane0[i] = sg.lane0;
        sh.thi[i] = (uint32_t)(t >> 32) ^ sg.key_hi;
        // plane_uniform of every pair: counter word c2 = slot 0 of the job's own group
#pragma unroll
        for (uint32_t m = 0; m < 16u; ++m) {
          const uint64_t p1 = (uint64_t)0xCD9E8D57u * ((TAG_SPIN << 28) | (m << 24) | sg.jgroup);
          const uint32_t c0 = (uint32_t)(p1 >> 32) ^ (uint32_t)t ^ sg.key_lo;
          const uint64_t p0 = (uint64_t)0xD2511F53u * c0;
          sh.u[i * 16 + (int)m] = make_uint4((uint32_t)p1 ^ (sg.key_lo + 0x9E3779B9u),
                                             (uint32_t)(p0 >> 32) ^ (sg.key_hi + 0xBB67AE85u), (uint32_t)p0, 0u);
        }
        live |= sg.mask;
        if (sg.inv) inv |= sg.mask;
      }
      n += __popc(bal);
    }
    const uint32_t ll = __reduce_or_sync(0xffffffffu, (uint32_t)live);
    const uint32_t lh = __reduce_or_sync(0xffffffffu, (uint32_t)(live >> 32));
    const uint32_t il = __reduce_or_sync(0xffffffffu, (uint32_t)inv);
    const uint32_t ih = __reduce_or_sync(0xffffffffu, (uint32_t)(inv >> 32));
    if (lane == 0) {
      sh.n = n;
      sh.live = (uint64_t)ll | ((uint64_t)lh << 32);
      sh.inv = (uint64_t)il | ((uint64_t)ih << 32);
    }
  }
  __syncthreads();
}

// Segment i's Philox block of plane pair m for a site: rounds 0 and 1 from
// their parts, rounds 2..9 with the job's bumped key.
__device__ __forceinline__ uint4 fused_block(const FusedShared& sh, int i, uint32_t m, uint32_t site) {
  const uint64_t q0 = (uint64_t)0xD2511F53u * site;
  const uint64_t q1 = (uint64_t)0xCD9E8D57u * ((uint32_t)(q0 >> 32) ^ sh.thi[i]);
  const uint4 u = sh.u[i * 16 + (int)m];
  uint32_t c0 = (uint32_t)(q1 >> 32) ^ u.x, c1 = (uint32_t)q1, c2 = u.y ^ (uint32_t)q0, c3 = u.z;
  uint32_t k0 = sh.klo[i] + 2u * 0x9E3779B9u, k1 = sh.khi[i] + 2u * 0xBB67AE85u;
#pragma unroll
  for (int r = 2; r < 10; ++r) {
    const uint64_t p0 = (uint64_t)0xD2511F53u * c0;
    const uint64_t p1 = (uint64_t)0xCD9E8D57u * c2;
    const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ k0;
    const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ k1;
    c1 = (uint32_t)p1;
    c3 = (uint32_t)p0;
    c0 = n0;
    c2 = n2;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return make_uint4(c0, c1, c2, c3);
}

template <int D, bool P2, int T>
__global__ void __launch_bounds__(kFusedBlock) k_sweep_fused(const FusedParams fp) {
  __shared__ FusedShared sh;
  const BitsParams& p = fp.b;
  const int g = blockIdx.y;
  if (fp.early) stage_fused(sh, fp, g);
  dependent_launch_entry();
  if (!fp.early) stage_fused(sh, fp, g);
  const uint64_t live = sh.live, inv = sh.inv;
  const int nsg = sh.n;
  if (live == 0ull) return;
  const Geom geom = p.geom;
  const uint32_t N = geom.N;
  const uint64_t* Jg = p.J + (size_t)g * D * N;
  uint64_t* sp = p.spins + (size_t)g * N;  // one slot per group
  const uint32_t w_begin = blockIdx.x * p.words_per_block;
  const uint32_t w_end = min(w_begin + p.words_per_block, geom.half);
  const uint32_t sub = threadIdx.x % T, first = threadIdx.x & 31u & ~(uint32_t)(T - 1);
  for (uint32_t base = w_begin; base < w_end; base += kFusedBlock / T) {  // uniform across the block
    const uint32_t w = base + threadIdx.x / T;
    const bool valid = w < w_end;
    const Nbr n = split_neighbours_t<P2>(geom, p.colour, valid ? w : w_begin);
    const uint64_t b = sp[n.self];
    uint64_t e[2 * D];
    e[0] = b ^ sp[n.xp] ^ __ldg(Jg + n.self);
    e[1] = b ^ sp[n.xm] ^ __ldg(Jg + n.xm);
    e[2] = b ^ sp[n.yp] ^ __ldg(Jg + N + n.self);
    e[3] = b ^ sp[n.ym] ^ __ldg(Jg + N + n.ym);
    if (D == 3) {
      e[4] = b ^ sp[n.zp] ^ __ldg(Jg + 2u * N + n.self);
      e[5] = b ^ sp[n.zm] ^ __ldg(Jg + 2u * N + n.zm);
    }
    uint64_t u0, u1, u2;
    count_unsat<D>(e, u0, u1, u2);
    // a segment's lanes may hold either algorithm's planes: select over all classes
    const uint64_t always = class_select<D, 1>(sh.tpa + 32 * kMaxClasses, u0, u1, u2);
    uint64_t lt = always;
    uint64_t und = valid ? ~always & live : 0ull;
#pragma unroll 1
    for (uint32_t m0 = 0; m0 < 16u && __any_sync(0xffffffffu, und != 0ull); m0 += T) {
      uint64_t r0 = 0, r1 = 0;
#pragma unroll 1
      for (int j = 0; j < nsg; ++j) {
        const uint64_t mk = sh.mask[j];
        if (!(und & mk)) continue;
        const uint4 x = fused_block(sh, j, m0 + sub, n.site);
        const uint32_t s = sh.lane0[j];
        r0 |= (((uint64_t)x.x | ((uint64_t)x.y << 32)) << s) & mk;
        r1 |= (((uint64_t)x.z | ((uint64_t)x.w << 32)) << s) & mk;
      }
#pragma unroll
      for (int q = 0; q < 2 * T; ++q) {
        uint64_t r = (q & 1) ? r1 : r0;
        if (T > 1) r = __shfl_sync(0xffffffffu, (unsigned long long)r, (int)first + (q >> 1));
        const uint64_t tb = class_select<D, 1>(sh.tpa + (2u * m0 + (uint32_t)q) * kMaxClasses, u0, u1, u2);
        lt |= und & ~r & tb;
        und &= ~(r ^ tb);
      }
    }
    const uint64_t flip = (lt ^ inv) & live;
    if (valid && sub == 0u && flip) sp[n.self] = b ^ flip;
  }
}

// A job's couplings and initial spins, as samples 64 jgroup + b of its own
// lattice (group jgroup, slot 0 of the J and INIT streams under the job's
// key), written into lanes lane0 + b of group g.
__global__ void k_load_segment(uint64_t* spins, uint64_t* J, Geom geom, int g, uint32_t lane0, uint64_t mask,
                               uint32_t jgroup, PhiloxKeys keys) {
  const uint32_t L = (uint32_t)geom.L;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < geom.N; i += gridDim.x * blockDim.x) {
    const int x = (int)(i % L), y = (int)((i / L) % L), z = geom.D == 3 ? (int)(i / (L * L)) : 0;
    const uint32_t j = split_index(geom, x, y, z);
    for (int d = 0; d < geom.D; ++d) {
      const uint4 r = philox10(i, (uint32_t)d, (TAG_J << 28) | jgroup, 0u, keys);
      uint64_t* wp = J + ((size_t)g * geom.D + d) * geom.N + j;
      *wp = (*wp & ~mask) | ((((uint64_t)r.x | ((uint64_t)r.y << 32)) << lane0) & mask);
    }
    const uint4 r = philox10(i, 0u, (TAG_INIT << 28) | jgroup, 0u, keys);
    uint64_t* wp = spins + (size_t)g * geom.N + j;
    *wp = (*wp & ~mask) | ((((uint64_t)r.x | ((uint64_t)r.y << 32)) << lane0) & mask);
  }
}

__global__ void k_advance_segments(Segment* segs, const uint32_t* nseg, int G, uint32_t by) {
  const int total = G * kMaxSegs;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
    const int g = idx / kMaxSegs, j = idx - g * kMaxSegs;
    if ((uint32_t)j >= nseg[g]) continue;
    Segment& sg = segs[idx];
    if (sg.mask != 0ull && sg.t < sg.t_end) sg.t = min(sg.t_end, sg.t + by);
  }
}

// ---- initialisation: one Philox block gives the word of 64 samples ----

__global__ void k_init_bits(uint64_t* spins, uint64_t* J, Geom geom, int G, int slots, int jmode,
                            PhiloxKeys keys) {
  const uint64_t total = (uint64_t)G * geom.N;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t g = (uint32_t)(idx / geom.N), i = (uint32_t)(idx - (uint64_t)g * geom.N);
    const uint32_t L = (uint32_t)geom.L;
    const int x = (int)(i % L), y = (int)((i / L) % L), z = geom.D == 3 ? (int)(i / (L * L)) : 0;
    const uint32_t j = split_index(geom, x, y, z);
    for (int d = 0; d < geom.D; ++d) {
      const uint4 r = philox10(i, (uint32_t)d, (TAG_J << 28) | g, 0u, keys);
      J[((size_t)g * geom.D + d) * geom.N + j] =
          jmode == 1 ? 0ull : (jmode == 2 ? ~0ull : ((uint64_t)r.x | ((uint64_t)r.y << 32)));
    }
    for (int sg = 0; sg < slots; ++sg) {
      const uint4 r = philox10(i, 0u, (TAG_INIT << 28) | ((uint32_t)sg << 12) | g, 0u, keys);
      spins[((size_t)g * slots + sg) * geom.N + j] = (uint64_t)r.x | ((uint64_t)r.y << 32);
    }
  }
}

// ---- threshold planes: TP[g][sigma][p][u], bit l = bit (31-p) of T of the
// temperature sample 64g+l holds in slot sigma; plane 32 = (T == 2^32). ----

// Threshold planes of one 64-lane word, one warp each: thread t holds the
// thresholds of lanes t and 32 + t, and plane q is the ballot of bit 31 - q
// (plane 32: threshold 2^32, "always").  Thread q < 32 keeps plane q, and
// thread 0 also the always plane; the caller stores them.
__device__ __forceinline__ void warp_planes(uint64_t T_lo, uint64_t T_hi, uint64_t& mine, uint64_t& always) {
  const uint32_t lane = threadIdx.x & 31u;
  always = (uint64_t)__ballot_sync(0xffffffffu, T_lo >= kTwo32) |
           ((uint64_t)__ballot_sync(0xffffffffu, T_hi >= kTwo32) << 32);
  mine = 0;
#pragma unroll 4
  for (uint32_t q = 0; q < 32u; ++q) {
    const uint32_t lo = __ballot_sync(0xffffffffu, T_lo < kTwo32 && ((T_lo >> (31u - q)) & 1ull));
    const uint32_t hi = __ballot_sync(0xffffffffu, T_hi < kTwo32 && ((T_hi >> (31u - q)) & 1ull));
    if (lane == q) mine = (uint64_t)lo | ((uint64_t)hi << 32);
  }
}

// TP[g][sigma][p][u] from the per-temperature thresholds thr[k][u] of each
// lane's temperature, one warp per (group, slot, class).
__global__ void k_build_planes(uint64_t* tp, const uint64_t* thr, const int32_t* temp_of, int G, int S, int R,
                               int K, int slots) {
  const int total = G * slots * kMaxClasses;
  const uint32_t lane = threadIdx.x & 31u;
  for (int idx = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); idx < total;
       idx += (int)((gridDim.x * blockDim.x) >> 5)) {  // uniform across the warp
    const int u = idx % kMaxClasses, rest = idx / kMaxClasses;
    const int sigma = rest % slots, g = rest / slots;
    const int tslot = sigma / R, a = sigma - tslot * R;
    uint64_t T[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int s = 64 * g + 32 * h + (int)lane;
      const int k = s < S ? temp_of[((size_t)s * R + a) * K + tslot] : tslot;
      T[h] = thr[(size_t)k * kMaxClasses + u];
    }
    uint64_t mine, always;
    warp_planes(T[0], T[1], mine, always);
    uint64_t* out = tp + ((size_t)g * slots + sigma) * kPlanes * kMaxClasses + u;
    out[(size_t)lane * kMaxClasses] = mine;
    if (lane == 0) out[(size_t)32 * kMaxClasses] = always;
  }
}

// Field planes: FTP[g][sigma][p][8 f + u] from the per-temperature field
// thresholds fthr[k][(v + 2D) * 2 + f], v = 2D - 2u; classes u > 2D stay 0.
// With dilution (NF = kDiluteClasses) the class is 16 f + t, field class
// t * 2 + f; classes t > 4D stay 0.  One warp per (group, slot, class).
__global__ void k_build_field_planes(uint64_t* ftp, const uint64_t* fthr, const int32_t* temp_of, int D, int G,
                                     int S, int R, int K, int slots, int NF) {
  const int total = G * slots * NF;
  const uint32_t lane = threadIdx.x & 31u;
  for (int idx = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); idx < total;
       idx += (int)((gridDim.x * blockDim.x) >> 5)) {  // uniform across the warp
    const int c = idx % NF, rest = idx / NF;
    const int sigma = rest % slots, g = rest / slots;
    const int tslot = sigma / R, a = sigma - tslot * R;
    const bool dil = NF == kDiluteClasses;
    const int u = dil ? (c & 15) : (c & 7), f = dil ? (c >> 4) : (c >> 3);
    const bool live = dil ? u <= 4 * D : u <= 2 * D;
    const int cls = (dil ? u : 4 * D - 2 * u) * 2 + f;
    uint64_t T[2] = {0, 0};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int s = 64 * g + 32 * h + (int)lane;
      const int k = s < S ? temp_of[((size_t)s * R + a) * K + tslot] : tslot;
      if (live) T[h] = fthr[(size_t)k * kFieldClasses + cls];
    }
    uint64_t mine, always;
    warp_planes(T[0], T[1], mine, always);
    uint64_t* out = ftp + ((size_t)g * slots + sigma) * kPlanes * NF + c;
    out[(size_t)lane * NF] = mine;
    if (lane == 0) out[(size_t)32 * NF] = always;
  }
}

// ---- measurements: per-lane counts in vertical counters ----
//
// Each thread adds the 64-bit words of its sites (bits of the unsatisfied
// forward bonds as a 2-bit number, the spin-down bits, the disagreement bits
// of two replicas) into per-lane counters held as bit-planes (LaneCounter):
// four words at a time through carry-save adders, so that only one carry of
// four ripples through the upper planes, and kMeasChunk words at most before
// a flush.  A flush adds the counters of the warp's threads as bit-sliced
// numbers, a butterfly of five steps (the first splits the 64 lanes between
// the half-warps), and reads each lane's total off the planes.  At the end the
// block sums its warps in shared memory and adds one value per lane and
// quantity to the accumulators.  Per site and configuration this gives U
// (E = 2U - D N), B (M = N - 2B) and X (Q = N - 2X).
//
// Bound: load latency (64 to 128 registers for the planes and four sites in
// flight, 8 to 16 warps an SM) and integer issue.  One launch, state in L2:
// random fields L=64, 256 samples 34 -> 13.5 us; L=32, 32 temperatures x 64 x
// 2 25 -> 17.5 us; L=64, 256 x 2 22.3 -> 20 us; L=128, 256 x 2 (from memory)
// 112 us.  Two words at a time in 80 registers was slower (27 us at L=64).

constexpr int kMeasWarps = kBlock / 32;
constexpr int kMeasMaxQ = 5;     // quantities per block: U and B of two replicas and X; 2 U - O, X, F
constexpr int kMeasBatch = 4;    // words a thread adds together
constexpr int kMeasChunk = 20;   // words a thread adds between flushes: up to 3 each (a site's forward
                                 // bonds) fit 6 planes, up to 1 each fit 5
constexpr int kPlanesBond = 6, kPlanesBit = 5;

__device__ __forceinline__ uint64_t maj3(uint64_t a, uint64_t b, uint64_t c) { return (a & b) | (c & (a ^ b)); }

// c = sum bit, returns the carry of c + x + y.
__device__ __forceinline__ uint64_t csa(uint64_t& c, uint64_t x, uint64_t y) {
  const uint64_t k = maj3(x, y, c);
  c ^= x ^ y;
  return k;
}

template <int K>
struct LaneCounter {
  uint64_t c[K];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int b = 0; b < K; ++b) c[b] = 0;
  }
  // x of weight 2^B into plane B and up.
  template <int B>
  __device__ __forceinline__ void ripple(uint64_t x) {
#pragma unroll
    for (int b = B; b < K; ++b) {
      const uint64_t t = c[b] & x;
      c[b] ^= x;
      x = t;
    }
  }
  // four words of 0/1 per lane
  __device__ __forceinline__ void add1(const uint64_t (&x)[kMeasBatch]) {
    const uint64_t t0 = csa(c[0], x[0], x[1]), t1 = csa(c[0], x[2], x[3]);
    ripple<2>(csa(c[1], t0, t1));
  }
  // four 2-bit numbers s + 2 k per lane
  __device__ __forceinline__ void add2(const uint64_t (&s)[kMeasBatch], const uint64_t (&k)[kMeasBatch]) {
    const uint64_t t0 = csa(c[0], s[0], s[1]), t1 = csa(c[0], s[2], s[3]);
    const uint64_t u0 = csa(c[1], k[0], k[1]), u1 = csa(c[1], k[2], k[3]), u2 = csa(c[1], t0, t1);
    const uint64_t v0 = csa(c[2], u0, u1), v1 = c[2] & u2;
    c[2] ^= u2;
    ripple<4>(csa(c[3], v0, v1));
  }
  // Adds 2^shift sign times the warp's totals of lanes meas_lane(), + 1 to lo, hi and clears.
  __device__ __forceinline__ void flush(int shift, long long sign, long long& lo, long long& hi) {
    const uint32_t t = threadIdx.x & 31u;
    uint32_t p[K + 5], carry = 0;
#pragma unroll
    for (int b = 0; b < K; ++b) {
      const uint32_t l = (uint32_t)c[b], h = (uint32_t)(c[b] >> 32);
      const uint32_t x = (t & 16u) ? h : l, y = __shfl_xor_sync(0xffffffffu, (t & 16u) ? l : h, 16);
      p[b] = x ^ y ^ carry;
      carry = (x & y) | (carry & (x ^ y));
      c[b] = 0;
    }
    p[K] = carry;
#pragma unroll
    for (int st = 0; st < 4; ++st) {
      carry = 0;
#pragma unroll
      for (int b = 0; b < K + 1 + st; ++b) {
        const uint32_t y = __shfl_xor_sync(0xffffffffu, p[b], 8 >> st), x = p[b];
        p[b] = x ^ y ^ carry;
        carry = (x & y) | (carry & (x ^ y));
      }
      p[K + 1 + st] = carry;
    }
    const uint32_t at = 2u * (t & 15u);
    uint32_t n0 = 0, n1 = 0;
#pragma unroll
    for (int b = 0; b < K + 5; ++b) {
      n0 |= ((p[b] >> at) & 1u) << b;
      n1 |= ((p[b] >> (at + 1u)) & 1u) << b;
    }
    lo += sign * ((long long)n0 << shift);
    hi += sign * ((long long)n1 << shift);
  }
};

// First of the two sample lanes whose totals this thread holds after a flush.
__device__ __forceinline__ uint32_t meas_lane() {
  const uint32_t t = threadIdx.x & 31u;
  return 32u * (t >> 4) + 2u * (t & 15u);
}

struct MeasGeom {
  FastDiv h, L;
  uint32_t N;
};

// Split index j -> split indices of the forward neighbours x+1, y+1, z+1.
struct Fwd {
  uint32_t x, y, z;
};

template <int D>
__device__ __forceinline__ Fwd split_forward(const MeasGeom& g, uint32_t j) {
  const uint32_t h = g.h.d, L = g.L.d;
  const uint32_t rc = div_by(j, g.h), k = j - rc * h, row = rc >> 1, c = rc & 1u;
  const uint32_t z = D == 3 ? div_by(row, g.L) : 0u, y = row - z * L;
  const uint32_t xpar = (c ^ y ^ z) & 1u;
  const uint32_t o = j + (c ? 0u - h : h);  // the other colour's word of the same row and k
  Fwd f;
  f.x = o + (xpar ? (k + 1u == h ? 0u - k : 1u) : 0u);
  f.y = o + (y + 1u == L ? 0u - 2u * h * (L - 1u) : 2u * h);
  f.z = D == 3 ? o + (z + 1u == L ? 0u - 2u * h * L * (L - 1u) : 2u * h * L) : 0u;
  return f;
}

// Unsatisfied forward bonds of a site as a 2-bit number (sum, carry).
template <int D>
__device__ __forceinline__ void bond_count(uint64_t b, uint64_t nx, uint64_t ny, uint64_t nz, uint64_t Jx,
                                           uint64_t Jy, uint64_t Jz, uint64_t& s1, uint64_t& c1) {
  const uint64_t ex = b ^ nx ^ Jx, ey = b ^ ny ^ Jy;
  if (D == 3) {
    const uint64_t ez = b ^ nz ^ Jz;
    s1 = ex ^ ey ^ ez;
    c1 = maj3(ex, ey, ez);
  } else {
    s1 = ex ^ ey;
    c1 = ex & ey;
  }
}

// Block reduction of the per-thread lane totals tot[q][2] and one atomic add
// per (lane, quantity) into acc[sample][row_of(q)][field_of(q)].
__device__ __forceinline__ void block_flush(long long (*red)[64], const long long (*tot)[2], int nq, int g, int S,
                                            int64_t* acc, const int* row_off, const int* field, int row_stride) {
  const int warp = threadIdx.x >> 5;
  const uint32_t l0 = meas_lane();
  for (int q = 0; q < nq; ++q) {
    red[warp * kMeasMaxQ + q][l0] = tot[q][0];
    red[warp * kMeasMaxQ + q][l0 + 1u] = tot[q][1];
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < nq * 64; idx += kBlock) {
    const int q = idx >> 6, l = idx & 63;
    long long v = 0;
    for (int w = 0; w < kMeasWarps; ++w) v += red[w * kMeasMaxQ + q][l];
    const int s = 64 * g + l;
    if (s < S && v != 0)
      atomicAdd((unsigned long long*)&acc[((size_t)s * row_stride + row_off[q]) * kAccStride + field[q]],
                (unsigned long long)v);
  }
}

// One temperature (slot = replica): U and B of every replica and, with two
// replicas, X, in one pass.  Grid (chunks, groups), from group y0.
template <int D, int R>
__global__ void __launch_bounds__(kBlock, 2) k_measure_bits_k1(const uint64_t* __restrict__ spins,
                                                               const uint64_t* __restrict__ J, int64_t* acc,
                                                               MeasGeom geom, int S, int y0) {
  __shared__ long long red[kMeasWarps * kMeasMaxQ][64];
  const int g = y0 + blockIdx.y;
  const uint32_t N = geom.N;
  const uint64_t* Jg = J + (size_t)g * D * N;
  const uint64_t* sg = spins + (size_t)g * R * N;
  constexpr int NQ = 2 * R + (R == 2 ? 1 : 0);
  long long tot[NQ][2];
#pragma unroll
  for (int q = 0; q < NQ; ++q) tot[q][0] = tot[q][1] = 0;
  LaneCounter<kPlanesBond> cu[R];
  LaneCounter<kPlanesBit> cb[R], cx;
#pragma unroll
  for (int a = 0; a < R; ++a) {
    cu[a].zero();
    cb[a].zero();
  }
  cx.zero();
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t stride = gridDim.x * kBlock;
  uint64_t base = blockIdx.x * kBlock + (threadIdx.x & ~31u);  // uniform across the warp
  while (base < N) {
    for (int n = 0; n < kMeasChunk / kMeasBatch && base < N; ++n, base += (uint64_t)kMeasBatch * stride) {
      uint64_t s1[R][kMeasBatch], c1[R][kMeasBatch], bw[R][kMeasBatch];
#pragma unroll
      for (int q = 0; q < kMeasBatch; ++q) {
        const uint64_t jj = base + (uint64_t)q * stride + lane;
        const bool in = jj < N;
        const uint32_t j = in ? (uint32_t)jj : 0u;
        const Fwd f = split_forward<D>(geom, j);
        const uint64_t Jx = Jg[j], Jy = Jg[N + j], Jz = D == 3 ? Jg[2u * N + j] : 0ull;
#pragma unroll
        for (int a = 0; a < R; ++a) {
          const uint64_t* sp = sg + (size_t)a * N;
          bw[a][q] = sp[j];
          bond_count<D>(bw[a][q], sp[f.x], sp[f.y], D == 3 ? sp[f.z] : 0ull, Jx, Jy, Jz, s1[a][q], c1[a][q]);
          if (!in) bw[a][q] = s1[a][q] = c1[a][q] = 0;
        }
      }
#pragma unroll
      for (int a = 0; a < R; ++a) {
        cu[a].add2(s1[a], c1[a]);
        cb[a].add1(bw[a]);
      }
      if (R == 2) {
        uint64_t x[kMeasBatch];
#pragma unroll
        for (int q = 0; q < kMeasBatch; ++q) x[q] = bw[0][q] ^ bw[R - 1][q];
        cx.add1(x);
      }
    }
#pragma unroll
    for (int a = 0; a < R; ++a) {
      cu[a].flush(0, 1, tot[2 * a][0], tot[2 * a][1]);
      cb[a].flush(0, 1, tot[2 * a + 1][0], tot[2 * a + 1][1]);
    }
    if (R == 2) cx.flush(0, 1, tot[NQ - 1][0], tot[NQ - 1][1]);
  }
  int row_off[NQ], field[NQ];
#pragma unroll
  for (int a = 0; a < R; ++a) {
    row_off[2 * a] = row_off[2 * a + 1] = a;
    field[2 * a] = 0;
    field[2 * a + 1] = 1;
  }
  if (R == 2) {
    row_off[NQ - 1] = 0;
    field[NQ - 1] = 6;
  }
  block_flush(red, tot, NQ, g, S, acc, row_off, field, R);
}

// Any number of temperatures: U and B of one slot.  Grid (chunks, groups x
// slots), from row y0.
template <int D, bool EONLY = false>
__global__ void __launch_bounds__(kBlock) k_measure_bits(const uint64_t* __restrict__ spins,
                                                         const uint64_t* __restrict__ J, int64_t* acc, MeasGeom geom,
                                                         int S, int slots, int y0) {
  __shared__ long long red[kMeasWarps * kMeasMaxQ][64];
  const int gt = y0 + blockIdx.y;  // g * slots + sigma
  const int g = gt / slots, sigma = gt - g * slots;
  const uint32_t N = geom.N;
  const uint64_t* Jg = J + (size_t)g * D * N;
  const uint64_t* sp = spins + ((size_t)g * slots + sigma) * N;
  long long tot[2][2] = {{0, 0}, {0, 0}};
  LaneCounter<kPlanesBond> cu;
  LaneCounter<kPlanesBit> cb;
  cu.zero();
  cb.zero();
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t stride = gridDim.x * kBlock;
  uint64_t base = blockIdx.x * kBlock + (threadIdx.x & ~31u);  // uniform across the warp
  while (base < N) {
    for (int n = 0; n < kMeasChunk / kMeasBatch && base < N; ++n, base += (uint64_t)kMeasBatch * stride) {
      uint64_t s1[kMeasBatch], c1[kMeasBatch], bw[kMeasBatch];
#pragma unroll
      for (int q = 0; q < kMeasBatch; ++q) {
        const uint64_t jj = base + (uint64_t)q * stride + lane;
        const bool in = jj < N;
        const uint32_t j = in ? (uint32_t)jj : 0u;
        const Fwd f = split_forward<D>(geom, j);
        bw[q] = sp[j];
        bond_count<D>(bw[q], sp[f.x], sp[f.y], D == 3 ? sp[f.z] : 0ull, Jg[j], Jg[N + j],
                      D == 3 ? Jg[2u * N + j] : 0ull, s1[q], c1[q]);
        if (!in) bw[q] = s1[q] = c1[q] = 0;
      }
      cu.add2(s1, c1);
      if (!EONLY) cb.add1(bw);
    }
    cu.flush(0, 1, tot[0][0], tot[0][1]);
    if (!EONLY) cb.flush(0, 1, tot[1][0], tot[1][1]);
  }
  const int row_off[2] = {sigma, sigma}, field[2] = {0, 1};
  block_flush(red, tot, EONLY ? 1 : 2, g, S, acc, row_off, field, slots);
}

// Field models (RFIM, DAFF) of one slot, values rather than counts:
// E_J = sum over forward bonds with both ends occupied of (2 e - 1), as
// 2 U - O with U, O the per-site counts of occupied unsatisfied and occupied
// bonds (each a 2-bit sum); M = sum x s = X - 2 sum x b and F = sum sign(h)
// x s = X - 2 sum x (b ^ hb), X = sum x.  acc[0..2] = E_J, M, F.  Without
// dilution (DIL false) O = D N and X = N need no counting.
template <int D, bool DIL>
__global__ void __launch_bounds__(kBlock, 2) k_measure_field_bits(const uint64_t* __restrict__ spins,
                                                                  const uint64_t* __restrict__ J,
                                                                  const uint64_t* __restrict__ hbits,
                                                                  const uint64_t* __restrict__ xbits, int64_t* acc,
                                                                  MeasGeom geom, int S, int slots, int y0) {
  __shared__ long long red[kMeasWarps * kMeasMaxQ][64];
  const int gt = y0 + blockIdx.y;  // g * slots + sigma
  const int g = gt / slots, sigma = gt - g * slots;
  const uint32_t N = geom.N;
  const uint64_t* Jg = J + (size_t)g * D * N;
  const uint64_t* sp = spins + ((size_t)g * slots + sigma) * N;
  const uint64_t* Hg = hbits + (size_t)g * N;
  const uint64_t* Xg = xbits + (size_t)g * N;
  long long tot[3][2] = {{0, 0}, {0, 0}, {0, 0}};
  // U: occupied unsatisfied forward bonds, O: occupied forward bonds,
  // X: occupied sites, XB: occupied down spins, XF: occupied against the field
  LaneCounter<kPlanesBond> cuu, coo;
  LaneCounter<kPlanesBit> cxs, cxb, cxf;
  cuu.zero();
  coo.zero();
  cxs.zero();
  cxb.zero();
  cxf.zero();
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t stride = gridDim.x * kBlock;
  uint64_t base = blockIdx.x * kBlock + (threadIdx.x & ~31u);  // uniform across the warp
  while (base < N) {
    for (int n = 0; n < kMeasChunk / kMeasBatch && base < N; ++n, base += (uint64_t)kMeasBatch * stride) {
      uint64_t us[kMeasBatch], uc[kMeasBatch], os[kMeasBatch], oc[kMeasBatch];
      uint64_t xw[kMeasBatch], xb[kMeasBatch], xf[kMeasBatch];
#pragma unroll
      for (int q = 0; q < kMeasBatch; ++q) {
        const uint64_t jj = base + (uint64_t)q * stride + lane;
        const bool in = jj < N;
        const uint32_t j = in ? (uint32_t)jj : 0u;
        const Fwd f = split_forward<D>(geom, j);
        const uint64_t b = sp[j];
        uint64_t ux = b ^ sp[f.x] ^ Jg[j], uy = b ^ sp[f.y] ^ Jg[N + j];
        uint64_t uz = D == 3 ? b ^ sp[f.z] ^ Jg[2u * N + j] : 0ull;
        if (DIL) {
          const uint64_t xs = Xg[j];
          const uint64_t ox = xs & Xg[f.x], oy = xs & Xg[f.y], oz = D == 3 ? xs & Xg[f.z] : 0ull;
          ux &= ox;
          uy &= oy;
          uz &= oz;
          os[q] = in ? ox ^ oy ^ oz : 0ull;
          oc[q] = in ? maj3(ox, oy, oz) : 0ull;
          xw[q] = in ? xs : 0ull;
        } else {
          xw[q] = in ? ~0ull : 0ull;
        }
        us[q] = in ? ux ^ uy ^ uz : 0ull;
        uc[q] = in ? maj3(ux, uy, uz) : 0ull;
        xb[q] = xw[q] & b;
        xf[q] = xw[q] & (b ^ Hg[j]);
      }
      cuu.add2(us, uc);
      cxb.add1(xb);
      cxf.add1(xf);
      if (DIL) {
        coo.add2(os, oc);
        cxs.add1(xw);
      }
    }
    // E_J = 2U - O, M = X - 2 XB, F = X - 2 XF
    cuu.flush(1, 1, tot[0][0], tot[0][1]);
    cxb.flush(1, -1, tot[1][0], tot[1][1]);
    cxf.flush(1, -1, tot[2][0], tot[2][1]);
    if (DIL) {
      coo.flush(0, -1, tot[0][0], tot[0][1]);
      long long xl = 0, xh = 0;
      cxs.flush(0, 1, xl, xh);
      tot[1][0] += xl;
      tot[1][1] += xh;
      tot[2][0] += xl;
      tot[2][1] += xh;
    }
  }
  if (!DIL && blockIdx.x == 0 && threadIdx.x < 32u) {  // O = D N and X = N, once per lane
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      tot[0][l] -= (long long)D * N;
      tot[1][l] += N;
      tot[2][l] += N;
    }
  }
  const int row_off[3] = {sigma, sigma, sigma}, field[3] = {0, 1, 2};
  block_flush(red, tot, 3, g, S, acc, row_off, field, slots);
}

// Overlap at temperature k between replicas 0 and 1 (Sec. 4.1).  After
// parallel-tempering swaps the configuration holding temperature k differs
// per sample: lane l of temperature k compares slot slot_at[l][0][k] of
// replica 0 with slot_at[l][1][k] of replica 1.  X = disagreements per lane,
// Q = N - 2X, stored in acc[s][k*R][6]; with occupations (field models) the
// value Q = sum x (1 - 2 (w0 ^ w1)) instead of the count.
//
// Up to kOverlapTemps temperatures: a block takes 32 sites at a time.  Each
// slot's 32 words are transposed across a warp into one 32-site word per
// lane, in shared memory [slot][lane]; a thread then looks up the two slots of
// its (temperature, lane) pairs and counts the differing bits.  Every spin
// word is read once, where a pass per temperature reads them K times: K = 32,
// L = 32, 64 x 2: 58 -> 26.6 us.  Grid (chunks, groups).
constexpr int kOverlapTemps = 64;

// 32x32 bit transpose across the warp: afterwards thread j holds, in bit t,
// bit j of the word thread t passed in (five butterfly exchanges).
__device__ __forceinline__ uint32_t warp_transpose32(uint32_t x) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t M[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const uint32_t sft = 16u >> i;
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, sft);
    x = (lane & sft) ? ((x & ~M[i]) | ((y >> sft) & M[i])) : ((x & M[i]) | ((y << sft) & ~M[i]));
  }
  return x;
}

template <int PAIRS>
__global__ void __launch_bounds__(kBlock, PAIRS <= 8 ? 4 : 2) k_overlap_bits_tile(const uint64_t* __restrict__ spins,
                                                              const int32_t* __restrict__ slot_at,
                                                              const uint64_t* __restrict__ xbits, int64_t* acc,
                                                              uint32_t N, int S, int R, int K, int slots) {
  extern __shared__ uint32_t rows[];  // [2 K (+ 1 with occupations)][64]: slot t of replica a in row a K + t
  const int g = blockIdx.y;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint64_t* sg = spins + (size_t)g * slots * N;
  // this thread's pairs: p = threadIdx + 256 i, lane p mod 64 of temperature p / 64
  uint32_t at0[PAIRS], at1[PAIRS];
  int n[PAIRS];
#pragma unroll
  for (int i = 0; i < PAIRS; ++i) {
    const int p = (int)threadIdx.x + kBlock * i, k = p >> 6, l = p & 63, s = 64 * g + l;
    const bool in = k < K && s < S;
    at0[i] = 64u * (uint32_t)(in ? slot_at[((size_t)s * R + 0) * K + k] : 0) + (uint32_t)l;
    at1[i] = 64u * (uint32_t)(K + (in ? slot_at[((size_t)s * R + 1) * K + k] : 0)) + (uint32_t)l;
    n[i] = 0;
  }
  const int nrows = 2 * K + (xbits ? 1 : 0);
  for (uint32_t j0 = blockIdx.x * 32u; j0 < N; j0 += gridDim.x * 32u) {
    const uint32_t j = j0 + lane;
    for (int r0 = (int)warp; r0 < nrows; r0 += 4 * kMeasWarps) {  // four rows' loads in flight
      uint64_t w[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = r0 + q * kMeasWarps;
        w[q] = 0;
        if (j < N && r < 2 * K) {
          const int a = r >= K ? 1 : 0, t = r - a * K;
          w[q] = sg[((size_t)t * R + a) * N + j];
        } else if (j < N && r < nrows) {
          w[q] = xbits[(size_t)g * N + j];
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = r0 + q * kMeasWarps;
        if (r >= nrows) break;  // uniform across the warp
        rows[64 * r + (int)lane] = warp_transpose32((uint32_t)w[q]);
        rows[64 * r + 32 + (int)lane] = warp_transpose32((uint32_t)(w[q] >> 32));
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < PAIRS; ++i) {
      const int p = (int)threadIdx.x + kBlock * i;
      if ((p >> 6) >= K) continue;
      const uint32_t d = rows[at0[i]] ^ rows[at1[i]];
      if (xbits) {
        const uint32_t x = rows[64 * 2 * K + (p & 63)];
        n[i] += __popc(x) - 2 * __popc(x & d);
      } else {
        n[i] += __popc(d);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < PAIRS; ++i) {
    const int p = (int)threadIdx.x + kBlock * i, k = p >> 6, s = 64 * g + (p & 63);
    if (k < K && s < S && n[i] != 0)
      atomicAdd((unsigned long long*)&acc[((size_t)s * slots + (size_t)k * R) * kAccStride + 6],
                (unsigned long long)(long long)n[i]);
  }
}

// More temperatures: the word of replica a at temperature k assembled lane by
// lane, W_a = OR_t (sel[a][t] & spins[t*R + a]), sel[a][t] = lanes whose
// temperature k sits in slot t.  Grid (chunks, groups x temperatures).
__global__ void __launch_bounds__(kBlock) k_overlap_bits(const uint64_t* __restrict__ spins,
                                                         const int32_t* __restrict__ slot_at,
                                                         const uint64_t* __restrict__ xbits, int64_t* acc,
                                                         uint32_t N, int S, int R, int K, int slots) {
  extern __shared__ uint64_t sel[];  // [2][K]
  __shared__ long long red[kMeasWarps * kMeasMaxQ][64];
  const int gk = blockIdx.y;
  const int g = gk / K, k = gk - g * K;
  for (int t = threadIdx.x; t < 2 * K; t += kBlock) {
    const int a = t / K, ts = t - a * K;
    uint64_t m = 0;
    for (int l = 0; l < 64; ++l) {
      const int s = 64 * g + l;
      const int at = s < S ? slot_at[((size_t)s * R + a) * K + k] : k;
      if (at == ts) m |= 1ull << l;
    }
    sel[t] = m;
  }
  __syncthreads();
  const uint64_t* sg = spins + (size_t)g * slots * N;
  long long tot[1][2] = {{0, 0}};
  LaneCounter<kPlanesBit> cd, cw;  // disagreements (occupied), occupied sites
  cd.zero();
  cw.zero();
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t stride = gridDim.x * kBlock;
  uint64_t base = blockIdx.x * kBlock + (threadIdx.x & ~31u);  // uniform across the warp
  while (base < N) {
    for (int n = 0; n < kMeasChunk / kMeasBatch && base < N; ++n, base += (uint64_t)kMeasBatch * stride) {
      uint64_t d[kMeasBatch], x[kMeasBatch];
#pragma unroll
      for (int q = 0; q < kMeasBatch; ++q) {
        const uint64_t jj = base + (uint64_t)q * stride + lane;
        const bool in = jj < N;
        const uint32_t j = in ? (uint32_t)jj : 0u;
        uint64_t w0 = 0, w1 = 0;
        for (int t = 0; t < K; ++t) {
          const uint64_t m0 = sel[t], m1 = sel[K + t];
          if (m0) w0 |= m0 & sg[((size_t)t * R + 0) * N + j];
          if (m1) w1 |= m1 & sg[((size_t)t * R + 1) * N + j];
        }
        x[q] = !in ? 0ull : xbits ? xbits[(size_t)g * N + j] : ~0ull;
        d[q] = x[q] & (w0 ^ w1);
      }
      cd.add1(d);
      if (xbits) cw.add1(x);
    }
    if (xbits) {  // Q = sum x (1 - 2 (w0 ^ w1))
      cw.flush(0, 1, tot[0][0], tot[0][1]);
      cd.flush(1, -1, tot[0][0], tot[0][1]);
    } else {
      cd.flush(0, 1, tot[0][0], tot[0][1]);
    }
  }
  const int row_off[1] = {k * R}, field[1] = {6};
  block_flush(red, tot, 1, g, S, acc, row_off, field, slots);
}

// ---- layout conversions (natural int8 <-> bit-sliced split words) ----

__global__ void k_get_spins_bits(const uint64_t* spins, int8_t* out, Geom geom, int S, int slots) {
  const uint64_t total = (uint64_t)S * slots * geom.N;
  const uint32_t L = (uint32_t)geom.L;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t i = (uint32_t)(idx % geom.N);
    const uint64_t rest = idx / geom.N;
    const int sg = (int)(rest % slots), s = (int)(rest / slots);
    const int x = (int)(i % L), y = (int)((i / L) % L), z = geom.D == 3 ? (int)(i / (L * L)) : 0;
    const uint64_t w = spins[((size_t)(s >> 6) * slots + sg) * geom.N + split_index(geom, x, y, z)];
    out[idx] = ((w >> (s & 63)) & 1ull) ? -1 : 1;
  }
}

__global__ void k_set_spins_bits(uint64_t* spins, const int8_t* in, Geom geom, int S, int G, int slots) {
  const uint64_t total = (uint64_t)G * slots * geom.N;
  const uint32_t L = (uint32_t)geom.L;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t i = (uint32_t)(idx % geom.N);
    const uint64_t rest = idx / geom.N;
    const int sg = (int)(rest % slots), g = (int)(rest / slots);
    const int x = (int)(i % L), y = (int)((i / L) % L), z = geom.D == 3 ? (int)(i / (L * L)) : 0;
    uint64_t* wp = &spins[((size_t)g * slots + sg) * geom.N + split_index(geom, x, y, z)];
    uint64_t w = *wp;
    for (int l = 0; l < 64; ++l) {
      const int s = 64 * g + l;
      if (s >= S) break;
      const uint64_t bit = in[((size_t)s * slots + sg) * geom.N + i] < 0 ? 1ull : 0ull;
      w = (w & ~(1ull << l)) | (bit << l);
    }
    *wp = w;
  }
}

__global__ void k_get_couplings_bits(const uint64_t* J, int8_t* out, Geom geom, int S) {
  const uint64_t total = (uint64_t)S * geom.D * geom.N;
  const uint32_t L = (uint32_t)geom.L;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t i = (uint32_t)(idx % geom.N);
    const uint64_t rest = idx / geom.N;
    const int d = (int)(rest % geom.D), s = (int)(rest / geom.D);
    const int x = (int)(i % L), y = (int)((i / L) % L), z = geom.D == 3 ? (int)(i / (L * L)) : 0;
    const uint64_t w = J[((size_t)(s >> 6) * geom.D + d) * geom.N + split_index(geom, x, y, z)];
    out[idx] = ((w >> (s & 63)) & 1ull) ? -1 : 1;
  }
}

__global__ void k_set_couplings_bits(uint64_t* J, const int8_t* in, Geom geom, int S, int G) {
  const uint64_t total = (uint64_t)G * geom.D * geom.N;
  const uint32_t L = (uint32_t)geom.L;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t i = (uint32_t)(idx % geom.N);
    const uint64_t rest = idx / geom.N;
    const int d = (int)(rest % geom.D), g = (int)(rest / geom.D);
    const int x = (int)(i % L), y = (int)((i / L) % L), z = geom.D == 3 ? (int)(i / (L * L)) : 0;
    uint64_t* wp = &J[((size_t)g * geom.D + d) * geom.N + split_index(geom, x, y, z)];
    uint64_t w = *wp;
    for (int l = 0; l < 64; ++l) {
      const int s = 64 * g + l;
      if (s >= S) break;
      const uint64_t bit = in[((size_t)s * geom.D + d) * geom.N + i] < 0 ? 1ull : 0ull;
      w = (w & ~(1ull << l)) | (bit << l);
    }
    *wp = w;
  }
}

inline unsigned grid_for(uint64_t total, unsigned block = 256, unsigned cap = 152u * 16u) {
  uint64_t g = (total + block - 1) / block;
  if (g > cap) g = cap;
  if (g == 0) g = 1;
  return (unsigned)g;
}

template <int D, int ALGO, int RT, bool P2, bool Q>
cudaError_t sweep_launch(Lattice& lat, const BitsParams& p, dim3 grid) {
  const size_t smem = bits_sweep_smem(lat.R, Q);
  if (smem > 48 * 1024) {  // many replicas: opt in to more than 48 KiB of planes and queues
    // the most that any lattice needs: other threads may be launching theirs
    cudaError_t e = cudaFuncSetAttribute(k_sweep_bits<D, ALGO, RT, P2, Q>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return e;
  }
  k_sweep_bits<D, ALGO, RT, P2, Q><<<grid, kBlock, smem, lat.stream>>>(p);
  return cudaGetLastError();
}

template <int D, int ALGO, bool P2>
cudaError_t sweep_dispatch(Lattice& lat, const BitsParams& p, dim3 grid, size_t) {
  if (lat.R == 1) return sweep_launch<D, ALGO, 1, P2, ALGO == 1>(lat, p, grid);
  if (lat.R == 2) return sweep_launch<D, ALGO, 2, P2, ALGO == 1>(lat, p, grid);
  // the heat bath's queues when they fit beside the planes (up to 97 replicas)
  if (ALGO == 1 && bits_sweep_smem(lat.R, true) <= 227u * 1024u)
    return sweep_launch<D, ALGO, 0, P2, true>(lat, p, grid);
  return sweep_launch<D, ALGO, 0, P2, false>(lat, p, grid);
}

template <int D, int ALGO>
cudaError_t sweep_dispatch2(Lattice& lat, const BitsParams& p, dim3 grid, size_t smem) {
  return lat.geom.lL > 0 ? sweep_dispatch<D, ALGO, true>(lat, p, grid, smem)
                         : sweep_dispatch<D, ALGO, false>(lat, p, grid, smem);
}

template <int D, int ALGO, bool P2>
cudaError_t field_launch(Lattice& lat, const BitsParams& p, dim3 grid, size_t smem) {
  if (lat.dilute) {
    auto kern = k_sweep_bits_dilute<D, ALGO, P2>;
    if (smem > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    kern<<<grid, kBlock, smem, lat.stream>>>(p, lat.hbits, lat.xbits);
    return cudaGetLastError();
  }
  auto kern = k_sweep_bits_field<D, ALGO, P2>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  kern<<<grid, kBlock, smem, lat.stream>>>(p, lat.hbits);
  return cudaGetLastError();
}

cudaError_t field_dispatch(Lattice& lat, const BitsParams& p, dim3 grid, size_t smem, int algo) {
  const bool p2 = lat.geom.lL > 0;
  if (lat.D == 3) {
    if (algo) return p2 ? field_launch<3, 1, true>(lat, p, grid, smem) : field_launch<3, 1, false>(lat, p, grid, smem);
    return p2 ? field_launch<3, 0, true>(lat, p, grid, smem) : field_launch<3, 0, false>(lat, p, grid, smem);
  }
  if (algo) return p2 ? field_launch<2, 1, true>(lat, p, grid, smem) : field_launch<2, 1, false>(lat, p, grid, smem);
  return p2 ? field_launch<2, 0, true>(lat, p, grid, smem) : field_launch<2, 0, false>(lat, p, grid, smem);
}

// Shapes of the run-time specialised sweep (variants 2..): lockstep plane
// loop or per-warp queues entered after phase_a pairs; registers capped so
// that min_blocks blocks of 256 threads fit on an SM.
struct JitShape {
  int mode, phase_a, min_blocks, group, jreload, ufirst, block;
};
constexpr JitShape kJitShapes[] = {
    {0, 8, 3, 1, 0, 0, 256}, {0, 8, 4, 1, 0, 0, 256}, {1, 4, 3, 1, 0, 0, 256}, {1, 4, 4, 1, 0, 0, 256},
    {1, 3, 3, 1, 0, 0, 256}, {1, 5, 3, 1, 0, 0, 256}, {2, 8, 2, 1, 0, 0, 256}, {2, 8, 3, 1, 0, 0, 256},
    {0, 8, 3, 2, 0, 0, 256}, {1, 4, 3, 2, 0, 0, 256}, {1, 6, 3, 2, 0, 0, 256}, {1, 4, 4, 2, 1, 0, 256},
    {0, 8, 4, 2, 1, 0, 256}, {0, 8, 4, 1, 1, 0, 256}, {1, 4, 4, 1, 1, 0, 256}, {1, 4, 3, 2, 0, 1, 256},
    {0, 8, 4, 2, 0, 1, 256}, {0, 8, 3, 2, 0, 1, 256}, {1, 4, 7, 2, 0, 1, 128}, {1, 4, 6, 2, 0, 1, 128},
    // mode 3: the lane-queue kernel (jit_sweep_lt.cuh), blocks/SM and block size
    {3, 4, 8, 1, 0, 0, 128}, {3, 4, 6, 1, 0, 0, 128}, {3, 4, 4, 1, 0, 0, 256},
    // mode 4: its persistent form; phase_a = least colour words per block / 128
    {4, 4, 8, 1, 0, 0, 128}, {4, 1, 8, 1, 0, 0, 128}, {4, 4, 4, 1, 0, 0, 256}};
constexpr int kNumJitShapes = sizeof(kJitShapes) / sizeof(kJitShapes[0]);
static_assert(kNumJitShapes + 1 == kMaxVariant, "variants 2..kMaxVariant are the shapes");
constexpr int kAutoJitVariant = 24;  // the lane-queue kernel, 4 blocks of 256 per SM
constexpr int kLtBlock = 256, kLtBlocks = 4;  // the same shape for fields and per-lane planes

// Blocks per SM of the lane-queue field sweep: a pair of replicas with field
// words (and u3 with dilution) needs more than 64 registers.
int field_blocks(const Lattice& lat) { return lat.R == 2 ? 3 : kLtBlocks; }

// The automatic and the lane-queue variants sweep fields and per-lane planes
// with that kernel; variants 2..21 with the earlier one-word-per-thread shapes.
bool lane_queue(const Lattice& lat) { return lat.variant == 0 || lat.variant >= 22; }

// Replicas a thread of the per-lane-plane sweep does together.
int lanes_replicas(const Lattice& lat) { return lat.R % 2 == 0 ? 2 : 1; }

// Launches a colour pass of a lane-queue kernel (jit_sweep_lt.cuh): ys block
// rows, about min_blocks blocks per SM in all (one wave), whole warps of words.
// Blocks that stage threshold rows (rows: per-lane planes) have at least a block
// of words where they would have less than half of one: L=20, 100 samples x 4
// replicas, blocks of 32 words 5.7 us a pass, of 128 or 256 3.8; L=14, 64
// samples x 4 x 10 temperatures 6.2 (64 words) / 4.9 (128) / 4.3 (256); but L=20,
// 64 x 2 x 20 temperatures 6.3 (192) / 6.8 (256).
cudaError_t launch_lt(const Lattice& lat, cudaKernel_t k, BitsParams& p, uint32_t ys, int min_blocks, int block,
                      bool rows = false) {
  uint32_t w;
  if (lat.block_words) {
    w = (lat.block_words + 31u) / 32u * 32u;
  } else {
    const uint32_t per_row = std::max<uint32_t>(1u, 152u * (uint32_t)min_blocks / ys);
    w = (lat.geom.half + per_row - 1u) / per_row;
    w = std::max<uint32_t>(32u, (w + 31u) / 32u * 32u);
    if (rows && w <= (uint32_t)block / 2u) w = (uint32_t)block;
  }
  p.words_per_block = w;
  // the rows of this chain (all of them but inside a graph of several)
  const uint32_t n = lat.chains > 1 ? (uint32_t)lat.chains : 1u;
  p.y0 = ys * (uint32_t)lat.chain / n;
  const uint32_t y1 = ys * ((uint32_t)lat.chain + 1u) / n;
  void* args[] = {(void*)&p};
  return launch_dependent((const void*)k, dim3((lat.geom.half + w - 1u) / w, y1 - p.y0), dim3((unsigned)block), args,
                          0, lat.stream);
}

// The specialised kernel shape (>= 2) that variant `variant` selects on this
// lattice with lane-uniform tables (ulut_ok), or 1 for the per-lane kernel.
int jit_variant_of(const Lattice& lat, int variant, bool ulut_ok) {
  int v = variant == 0 ? kAutoJitVariant : variant;
  bool ok = lat.K == 1 && ulut_ok && v >= 2 && v < 2 + kNumJitShapes && (lat.R == 1 || lat.R == 2);
  if (ok && kJitShapes[v - 2].mode == 2 && lat.R != 2) v = 2;  // the interleaved shape needs two replicas
  return ok ? v : 1;
}

// The specialised kernel shape the next sweep uses (>= 2), or 1 for the
// precompiled per-lane kernel.
int jit_variant_for(const Lattice& lat) { return jit_variant_of(lat, lat.variant, lat.ulut_ok); }

}  // namespace

int specialised_variant(const Lattice& lat, int variant) { return jit_variant_of(lat, variant, true); }

bool persistent_variant(const Lattice& lat) {
  const int v = jit_variant_for(lat);
  return v >= 2 && kJitShapes[v - 2].mode == 4 && !lat.field && lat.flags;
}

cudaError_t launch_sweep_persistent(Lattice& lat, int inv, uint64_t t0, uint32_t nsweeps, bool* ran) {
  *ran = false;
  const int v = jit_variant_for(lat);
  if (v < 2 || kJitShapes[v - 2].mode != 4 || nsweeps == 0) return cudaSuccess;
  const JitShape& js = kJitShapes[v - 2];
  prepare_sweep_bits(lat, inv);
  if (!lat.jit) return cudaSuccess;
  int dev = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void*)lat.jit, js.block, 0) != cudaSuccess) {
    cudaGetLastError();
    return cudaSuccess;
  }
  // blocks per group: as many as are resident at once, each with at least
  // phase_a * 128 colour words and at least one row
  const uint32_t Rg = lat.N / (uint32_t)lat.L, h = (uint32_t)lat.L / 2u;
  const uint32_t resident = (uint32_t)sms * (uint32_t)per_sm;
  uint32_t cpg = resident / (uint32_t)lat.G;
  const uint32_t min_words = 128u * (uint32_t)js.phase_a;
  cpg = std::min(cpg, std::max<uint32_t>(1u, Rg * h / min_words));
  cpg = std::min(cpg, Rg);
  const uint64_t blocks = (uint64_t)cpg * (uint64_t)lat.G;
  if (cpg == 0 || blocks > (uint64_t)resident || blocks > (uint64_t)kMaxPersistBlocks) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(lat.flags, 0, (size_t)blocks * 4, lat.stream);
  if (e != cudaSuccess) return e;
  BitsParams p;
  p.spins = (uint64_t*)lat.spins;
  p.J = (const uint64_t*)lat.J;
  p.tp = lat.tp;
  p.geom = lat.geom;
  p.G = lat.G;
  p.R = lat.R;
  p.K = lat.K;
  p.slots = lat.slots;
  p.colour = 0;
  p.t_lo = (uint32_t)t0;
  p.t_hi = (uint32_t)(t0 >> 32);
  p.words_per_block = 0;
  p.keys = lat.keys;
  p.t_dev = nullptr;
  PersistParams pp;
  pp.flags = lat.flags;
  pp.err = lat.err;
  pp.npass = 2u * nsweeps;
  pp.cpg = cpg;
  pp.t0_lo = (uint32_t)t0;
  pp.t0_hi = (uint32_t)(t0 >> 32);
  pp.timeout_ns = lat.persist_timeout_ns;
  pp.skip_block = lat.persist_absent;
  void* args[] = {(void*)&p, (void*)&pp};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3((unsigned)js.block);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = lat.stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelExC(&cfg, (const void*)lat.jit, args);
  if (e == cudaErrorCooperativeLaunchTooLarge) {  // not resident at once here: per-pass kernels instead
    cudaGetLastError();
    return cudaSuccess;
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return e;
  }
  *ran = true;
  return cudaSuccess;
}

cudaKernel_t specialised_sweep_kernel(const Lattice& lat, const UniformLut& u, int algo, int v) {
  if (v < 2 || v >= 2 + kNumJitShapes) return nullptr;
  const JitShape& js = kJitShapes[v - 2];
  if (js.mode >= 3) return jit_lt_kernel(lat, u, algo, js.min_blocks, js.block, js.mode == 4);
  return jit_kernel(lat, u, algo, js.mode, js.phase_a, js.min_blocks, js.group, js.jreload, js.ufirst, js.block);
}

// Whether random fields are swept by the kernel specialised at run time:
// variants 0 (large lattices) and 2..; else by the precompiled ones.
bool field_specialised(const Lattice& lat) {
  return lat.flut_ok && lat.variant != 1 &&
         (lat.variant != 0 || (uint64_t)lat.G * lat.slots * lat.N >= (1ull << 20));
}

void prepare_sweep_bits(Lattice& lat, int inv) {
  const int algo = inv ? 1 : 0;
  if (lat.field) {
    const bool lq = lane_queue(lat);
    if (field_specialised(lat) && (lat.jitf_algo != algo || lat.jitf_lq != lq)) {
      lat.jitf = lq ? jit_lt_field_kernel(lat, algo, field_blocks(lat), kLtBlock)
                    : jit_field_kernel(lat, algo, lat.dilute && lat.R == 2 ? 2 : 3);
      lat.jitf_algo = algo;
      lat.jitf_lq = lq;
    }
    return;
  }
  const int v = jit_variant_for(lat);
  if (v >= 2 && (lat.jit_algo != algo || lat.jit_variant != v)) {
    lat.jit = specialised_sweep_kernel(lat, lat.ulut, algo, v);
    lat.jit_algo = algo;
    lat.jit_variant = v;
  }
  // the per-lane planes (also the fallback of a failed specialisation),
  // compiled for the geometry unless variant 1 asks for the precompiled kernel
  const int lq = lane_queue(lat) ? 1 : 0;
  if ((v < 2 || !lat.jit) && lat.variant != 1 && !lat.jitp_tried[algo][lq]) {
    const int rt = lat.R == 1 || lat.R == 2 ? lat.R : 0;
    const bool q = algo == 1 && bits_sweep_smem(lat.R, true) <= 227u * 1024u;
    lat.jitp[algo][lq] = lq ? jit_lt_lanes_kernel(lat, algo, lanes_replicas(lat), kLtBlocks, kLtBlock)
                            : jit_planes_kernel(lat, algo, rt, q, q ? 3 : 4, (size_t)bits_sweep_smem(lat.R, q));
    lat.jitp_tried[algo][lq] = true;
  }
}

int sweep_chains_bits(const Lattice& lat, int inv) {
  if (!lane_queue(lat)) return 1;
  uint64_t rows;
  if (lat.field) {
    if (!field_specialised(lat) || !lat.jitf) return 1;
    rows = (uint64_t)lat.G;
  } else {
    const int v = jit_variant_for(lat);
    if (v >= 2 && lat.jit && kJitShapes[v - 2].mode == 3)
      rows = (uint64_t)lat.G;
    else if (v < 2 && lat.jitp[inv ? 1 : 0][1])
      rows = (uint64_t)lat.G * lat.K * (lat.R / lanes_replicas(lat));
    else
      return 1;
  }
  if (rows < 2 || rows > 65535 || rows * lat.geom.half < kChainSites) return 1;
  return rows >= 4 ? 4 : 2;
}

cudaError_t launch_init_bits(Lattice& lat, int jmode) {
  k_init_bits<<<grid_for((uint64_t)lat.G * lat.N), 256, 0, lat.stream>>>((uint64_t*)lat.spins, (uint64_t*)lat.J,
                                                                          lat.geom, lat.G, lat.slots, jmode, lat.keys);
  return cudaGetLastError();
}

cudaError_t launch_init_sites_bits(Lattice& lat, double occupation) {
  const uint64_t T_occ = (uint64_t)std::floor(std::ldexp(occupation, 32));
  k_init_sites_bits<<<grid_for((uint64_t)lat.G * lat.N), 256, 0, lat.stream>>>(
      lat.hbits, lat.xbits, lat.geom, lat.G, lat.disorder == IANUS_DISORDER_RFIM, lat.disorder == IANUS_DISORDER_DAFF,
      T_occ, lat.keys);
  return cudaGetLastError();
}

cudaError_t launch_get_sites_bits(Lattice& lat, int8_t* dev_hs, int8_t* dev_occ) {
  k_get_sites_bits<<<grid_for((uint64_t)lat.S * lat.N), 256, 0, lat.stream>>>(lat.hbits, lat.xbits, dev_hs, dev_occ,
                                                                             lat.geom, lat.S);
  return cudaGetLastError();
}

cudaError_t launch_set_sites_bits(Lattice& lat, const int8_t* dev_hs, const int8_t* dev_occ) {
  k_set_sites_bits<<<grid_for((uint64_t)lat.G * lat.N), 256, 0, lat.stream>>>(lat.hbits, lat.xbits, dev_hs, dev_occ,
                                                                               lat.geom, lat.S, lat.G);
  return cudaGetLastError();
}

cudaError_t launch_load_segment(Lattice& lat, int group, uint32_t lane0, uint32_t n, uint32_t jgroup,
                                PhiloxKeys job_keys) {
  const uint64_t mask = (n >= 64u ? ~0ull : ((1ull << n) - 1ull)) << lane0;
  k_load_segment<<<grid_for(lat.N), 256, 0, lat.stream>>>((uint64_t*)lat.spins, (uint64_t*)lat.J, lat.geom, group,
                                                          lane0, mask, jgroup, job_keys);
  return cudaGetLastError();
}

cudaError_t launch_advance_segments(Lattice& lat, uint32_t by) {
  k_advance_segments<<<grid_for((uint64_t)lat.G * kMaxSegs, 128), 128, 0, lat.stream>>>(lat.segs, lat.nseg, lat.G, by);
  return cudaGetLastError();
}

cudaError_t launch_sweep_fused(Lattice& lat, int colour, uint32_t off, bool early) {
  FusedParams fp{};
  BitsParams& p = fp.b;
  p.spins = (uint64_t*)lat.spins;
  p.J = (const uint64_t*)lat.J;
  p.tp = lat.tp;
  p.geom = lat.geom;
  p.G = lat.G;
  p.R = 1;
  p.K = 1;
  p.slots = 1;
  p.colour = colour;
  p.t_lo = off;
  p.keys = lat.keys;
  fp.segs = lat.segs;
  fp.nseg = lat.nseg;
  fp.early = early ? 1 : 0;
  // threads a word, by 50 sweeps of 9 to 16 jobs: 8192 words (3D L=16, 4 groups)
  // 393 us with four threads, 444 with two, 496 with one; 32768 (2D L=128) 635,
  // 503, 656; 65536 (3D L=32) 926, 927, 682
  const uint32_t half = lat.geom.half;
  const uint64_t words = (uint64_t)half * (uint64_t)lat.G;
  const uint32_t T = words <= 152u * 96u ? 4u : words <= 152u * 300u ? 2u : 1u;
  const uint32_t unit = kFusedBlock / T;  // words a block takes at a time
  const uint32_t target_blocks = (152u * 12u + (uint32_t)lat.G - 1) / (uint32_t)lat.G;
  uint32_t wpb = (half + target_blocks - 1) / target_blocks;
  p.words_per_block = wpb = std::max(unit, (wpb + unit - 1) / unit * unit);
  const dim3 grid((half + wpb - 1) / wpb, (unsigned)lat.G);
  const bool p2 = lat.geom.lL > 0;
  const void* k[2][2][3] = {
      {{(const void*)k_sweep_fused<2, false, 1>, (const void*)k_sweep_fused<2, false, 2>, (const void*)k_sweep_fused<2, false, 4>},
       {(const void*)k_sweep_fused<2, true, 1>, (const void*)k_sweep_fused<2, true, 2>, (const void*)k_sweep_fused<2, true, 4>}},
      {{(const void*)k_sweep_fused<3, false, 1>, (const void*)k_sweep_fused<3, false, 2>, (const void*)k_sweep_fused<3, false, 4>},
       {(const void*)k_sweep_fused<3, true, 1>, (const void*)k_sweep_fused<3, true, 2>, (const void*)k_sweep_fused<3, true, 4>}}};
  void* args[] = {(void*)&fp};
  return launch_dependent(k[lat.D - 2][p2 ? 1 : 0][T >> 1], grid, dim3(kFusedBlock), args, 0, lat.stream);
}

cudaError_t launch_build_field_planes(Lattice& lat) {
  k_build_field_planes<<<grid_for((uint64_t)lat.G * lat.slots * lat.fpc * 32, 256), 256, 0, lat.stream>>>(
      lat.ftp, lat.fthr, lat.temp_of, lat.D, lat.G, lat.S, lat.R, lat.K, lat.slots, lat.fpc);
  return cudaGetLastError();
}

cudaError_t launch_build_planes(Lattice& lat) {
  k_build_planes<<<grid_for((uint64_t)lat.G * lat.slots * kMaxClasses * 32, 256), 256, 0, lat.stream>>>(
      lat.tp, lat.thr, lat.temp_of, lat.G, lat.S, lat.R, lat.K, lat.slots);
  return cudaGetLastError();
}

size_t sweep_bits_smem(int R) { return bits_sweep_smem(R, false); }

// Launches a sweep kernel with programmatic stream serialisation: its blocks
// may become resident while the previous kernel on the stream drains, and its
// entry (dependent_launch_entry) holds them until that kernel has completed.
// Inside a stream capture this becomes a programmatic edge of the graph.  A
// refused launch returns its error and leaves no pending error behind.
cudaError_t launch_dependent(const void* k, dim3 grid, dim3 block, void** args, size_t smem, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelExC(&cfg, k, args);
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

cudaError_t launch_sweep_bits(Lattice& lat, int colour, uint64_t t, int inv) {
  BitsParams p;
  p.spins = (uint64_t*)lat.spins;
  p.J = (const uint64_t*)lat.J;
  p.tp = lat.tp;
  p.geom = lat.geom;
  p.G = lat.G;
  p.R = lat.R;
  p.K = lat.K;
  p.slots = lat.slots;
  p.colour = colour;
  p.t_lo = (uint32_t)(t & 0xffffffffu);
  p.t_hi = (uint32_t)(t >> 32);
  p.keys = lat.keys;
  p.t_dev = lat.capturing ? lat.t_dev : nullptr;
  p.hbits = lat.hbits;
  p.xbits = lat.xbits;
  // blocks per (group, temperature slot): enough to fill the GPU ~4 deep
  const uint32_t half = lat.geom.half;
  const uint32_t gts = (uint32_t)(lat.G * lat.K);
  uint32_t target_blocks = (152u * 8u + gts - 1) / gts;
  uint32_t wpb;
  if (lat.block_words) {  // explicit shape: whole warps
    wpb = (lat.block_words + 31u) / 32u * 32u;
  } else {
    wpb = (half + target_blocks - 1) / target_blocks;
    wpb = ((wpb + kBlock - 1) / kBlock) * kBlock;
    if (wpb < (uint32_t)kBlock) wpb = kBlock;
  }
  p.words_per_block = wpb;
  dim3 grid((half + wpb - 1) / wpb, gts);
  const size_t smem = (size_t)lat.R * kPlanes * kMaxClasses * sizeof(uint64_t);
  const int algo = inv ? 1 : 0;
  if (lat.field) {
    // one temperature: the field kernel specialised at run time for the
    // lattice's tables; else per-lane planes
    if (field_specialised(lat)) {
      prepare_sweep_bits(lat, inv);
      if (lat.jitf && lane_queue(lat)) return launch_lt(lat, lat.jitf, p, (uint32_t)lat.G, field_blocks(lat), kLtBlock);
      if (lat.jitf) {
        const uint8_t* lut = (const uint8_t*)(lat.fthr + (size_t)lat.K * kFieldClasses);
        void* args[] = {(void*)&p, (void*)&p.hbits, (void*)&p.xbits, (void*)&lut};
        return launch_dependent((const void*)lat.jitf, grid, dim3(kBlock), args, 0, lat.stream);
      }
    }
    p.tp = lat.ftp;
    const size_t fsmem = (size_t)lat.R * kPlanes * lat.fpc * sizeof(uint64_t);
    return field_dispatch(lat, p, grid, fsmem, algo);
  }
  // Lane-uniform thresholds (one temperature): the kernel specialised for
  // them at run time.  Variants (ianus_set_variant): 0 = automatic (the
  // lane-queue shape with one temperature and one or two replicas, else the
  // per-lane planes; small lattices take the resident sweep before they get
  // here), 1 = per-lane planes, 2.. = a specialised kernel shape from
  // kJitShapes.  A compile costs a fraction of a second and is cached.
  const int v = jit_variant_for(lat);
  if (v >= 2) {
    const JitShape& js = kJitShapes[v - 2];
    prepare_sweep_bits(lat, inv);
    // mode 4 (persistent) passes that run one at a time use its per-pass form
    const cudaKernel_t k3 = js.mode == 4 ? jit_lt_kernel(lat, lat.ulut, algo, js.min_blocks, js.block) : lat.jit;
    if (k3 && js.mode >= 3) return launch_lt(lat, k3, p, (uint32_t)lat.G, js.min_blocks, js.block);
    if (lat.jit) {
      const uint8_t* lut_t = (const uint8_t*)(lat.thr + (size_t)lat.K * kMaxClasses);
      void* args[] = {(void*)&p, (void*)&lut_t};
      return launch_dependent((const void*)lat.jit, grid, dim3(js.block), args,
                              js.mode == 1 ? kJitSmemBytes / 256 * js.block : 0, lat.stream);
    }
  }
  // Per-lane planes: the kernel compiled for the lattice's geometry, else
  // (variant 1, or no run-time compiler) the precompiled one.
  if (lat.variant != 1) {
    prepare_sweep_bits(lat, inv);
    const cudaKernel_t k = lat.jitp[algo][lane_queue(lat) ? 1 : 0];
    if (k && lane_queue(lat)) {
      const uint64_t ys = (uint64_t)gts * (uint64_t)(lat.R / lanes_replicas(lat));
      if (ys <= 65535u) return launch_lt(lat, k, p, (uint32_t)ys, kLtBlocks, kLtBlock, true);
    } else if (k) {
      const bool q = algo == 1 && bits_sweep_smem(lat.R, true) <= 227u * 1024u;
      void* args[] = {(void*)&p};
      return launch_dependent((const void*)k, grid, dim3(kBlock), args, (size_t)bits_sweep_smem(lat.R, q), lat.stream);
    }
  }
  if (lat.D == 3)
    return algo ? sweep_dispatch2<3, 1>(lat, p, grid, smem) : sweep_dispatch2<3, 0>(lat, p, grid, smem);
  return algo ? sweep_dispatch2<2, 1>(lat, p, grid, smem) : sweep_dispatch2<2, 0>(lat, p, grid, smem);
}

// Blocks along the lattice for a measurement kernel with `ys` blocks across:
// about two blocks per SM in all, each warp taking 32 words at a time, and
// enough that a thread adds at most kMeasChunk words (one counter flush).
inline unsigned meas_blocks(uint32_t N, unsigned ys) {
  unsigned want = (152u * 2u + ys - 1u) / ys;
  const unsigned one_flush = (N + kBlock * kMeasChunk - 1) / (kBlock * kMeasChunk);
  if (want < one_flush) want = one_flush;
  const unsigned most = (N + kBlock - 1) / kBlock;
  return want < 1u ? 1u : (want > most ? most : want);
}

template <int PAIRS>
cudaError_t overlap_tile(Lattice& lat, const uint64_t* xbits) {
  const size_t smem = (size_t)(2 * lat.K + (xbits ? 1 : 0)) * 64 * sizeof(uint32_t);
  // about four blocks per SM, each tile of 32 sites once
  const unsigned tiles = (lat.N + 31u) / 32u, want = (152u * 4u + (unsigned)lat.G - 1u) / (unsigned)lat.G;
  k_overlap_bits_tile<PAIRS><<<dim3(std::min(tiles, want), (unsigned)lat.G), kBlock, smem, lat.stream>>>(
      (const uint64_t*)lat.spins, lat.slot_at, xbits, lat.acc, lat.N, lat.S, lat.R, lat.K, lat.slots);
  return cudaGetLastError();
}

template <int D>
cudaError_t counts_dispatch(Lattice& lat, bool energy_only) {
  const uint64_t* sp = (const uint64_t*)lat.spins;
  const uint64_t* J = (const uint64_t*)lat.J;
  const MeasGeom geom{fast_div((uint32_t)lat.geom.h), fast_div((uint32_t)lat.geom.L), lat.N};
  const bool one = lat.K == 1 && (lat.R == 1 || lat.R == 2) && !lat.field;  // one pass for E, M and (R == 2) Q
  const uint32_t rows = (uint32_t)(one ? lat.G : lat.G * lat.slots);
  // the rows of this chain: a multiple of its sweep's block rows (launch_lt)
  uint32_t y0 = 0, y1 = rows;
  if (lat.chains > 1) {
    const uint32_t sweep_rows = one || lat.field ? (uint32_t)lat.G : rows / (uint32_t)lanes_replicas(lat);
    const uint32_t per = rows / sweep_rows, n = (uint32_t)lat.chains;
    y0 = per * (sweep_rows * (uint32_t)lat.chain / n);
    y1 = per * (sweep_rows * ((uint32_t)lat.chain + 1u) / n);
  }
  const dim3 grid(meas_blocks(lat.N, rows), y1 - y0);
  const int y = (int)y0;
  if (one && lat.R == 2)
    k_measure_bits_k1<D, 2><<<grid, kBlock, 0, lat.stream>>>(sp, J, lat.acc, geom, lat.S, y);
  else if (one)
    k_measure_bits_k1<D, 1><<<grid, kBlock, 0, lat.stream>>>(sp, J, lat.acc, geom, lat.S, y);
  else if (lat.field && lat.dilute)
    k_measure_field_bits<D, true><<<grid, kBlock, 0, lat.stream>>>(sp, J, lat.hbits, lat.xbits, lat.acc, geom, lat.S,
                                                                   lat.slots, y);
  else if (lat.field)
    k_measure_field_bits<D, false><<<grid, kBlock, 0, lat.stream>>>(sp, J, lat.hbits, lat.xbits, lat.acc, geom, lat.S,
                                                                    lat.slots, y);
  else if (energy_only)  // U of every configuration, for the PT swap
    k_measure_bits<D, true><<<grid, kBlock, 0, lat.stream>>>(sp, J, lat.acc, geom, lat.S, lat.slots, y);
  else
    k_measure_bits<D><<<grid, kBlock, 0, lat.stream>>>(sp, J, lat.acc, geom, lat.S, lat.slots, y);
  return cudaGetLastError();
}

cudaError_t launch_measure_bits_counts(Lattice& lat, bool energy_only) {
  return lat.D == 3 ? counts_dispatch<3>(lat, energy_only) : counts_dispatch<2>(lat, energy_only);
}

bool overlap_apart(const Lattice& lat, int want_q) {
  return want_q && lat.R >= 2 && !(lat.K == 1 && lat.R == 2 && !lat.field);
}

cudaError_t launch_overlap_bits(Lattice& lat) {
  const uint64_t* xb = lat.field ? lat.xbits : nullptr;
  if (lat.K <= 16) return overlap_tile<4>(lat, xb);
  if (lat.K <= 32) return overlap_tile<8>(lat, xb);
  if (lat.K <= kOverlapTemps) return overlap_tile<kOverlapTemps / 4>(lat, xb);
  dim3 gq(meas_blocks(lat.N, (unsigned)(lat.G * lat.K)), (unsigned)(lat.G * lat.K));
  k_overlap_bits<<<gq, kBlock, 2 * lat.K * sizeof(uint64_t), lat.stream>>>(
      (const uint64_t*)lat.spins, lat.slot_at, xb, lat.acc, lat.N, lat.S, lat.R, lat.K, lat.slots);
  return cudaGetLastError();
}

cudaError_t launch_measure_bits(Lattice& lat, int want_q, bool energy_only) {
  cudaError_t e = cudaMemsetAsync(lat.acc, 0, (size_t)lat.S * lat.slots * kAccStride * sizeof(int64_t), lat.stream);
  if (e == cudaSuccess) e = launch_measure_bits_counts(lat, energy_only);
  if (e == cudaSuccess && !energy_only && overlap_apart(lat, want_q)) e = launch_overlap_bits(lat);
  return e;
}

cudaError_t launch_get_spins_bits(Lattice& lat, int8_t* dev_out) {
  k_get_spins_bits<<<grid_for((uint64_t)lat.S * lat.slots * lat.N), 256, 0, lat.stream>>>(
      (const uint64_t*)lat.spins, dev_out, lat.geom, lat.S, lat.slots);
  return cudaGetLastError();
}

cudaError_t launch_set_spins_bits(Lattice& lat, const int8_t* dev_in) {
  k_set_spins_bits<<<grid_for((uint64_t)lat.G * lat.slots * lat.N), 256, 0, lat.stream>>>(
      (uint64_t*)lat.spins, dev_in, lat.geom, lat.S, lat.G, lat.slots);
  return cudaGetLastError();
}

cudaError_t launch_get_couplings_bits(Lattice& lat, int8_t* dev_out) {
  k_get_couplings_bits<<<grid_for((uint64_t)lat.S * lat.D * lat.N), 256, 0, lat.stream>>>(
      (const uint64_t*)lat.J, dev_out, lat.geom, lat.S);
  return cudaGetLastError();
}

cudaError_t launch_set_couplings_bits(Lattice& lat, const int8_t* dev_in) {
  k_set_couplings_bits<<<grid_for((uint64_t)lat.G * lat.D * lat.N), 256, 0, lat.stream>>>(
      (uint64_t*)lat.J, dev_in, lat.geom, lat.S, lat.G);
  return cudaGetLastError();
}

}  // namespace ianus
