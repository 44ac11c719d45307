// k_words.cu -- plain (IANUS_LAYOUT_I8) lattices of many samples swept in
// bit-sliced words.
//
// A plain sweep moves and counts one byte a spin; the bit-sliced one updates 64
// samples with each instruction, from the same random numbers.  A run of sweeps
// of a plain lattice therefore packs the spins and the couplings into words,
// sweeps those (api.cu, sweep_words) and unpacks the spins: three passes over
// bytes for the run instead of several for every sweep.  Nothing is kept from
// one run to the next, since a program may write either in the lattice's buffer.
//
// The sweep is the precompiled per-lane-plane kernel, so that a plain lattice never
// waits for the run-time compiler (1.2 s for a geometry).  The lane-queue kernel
// against per-lane planes (jit_sweep_lt.cuh) would also serve every temperature
// once compiled, at 22 us for as many updates as the 38 us pass below (L=32, 64
// samples x 2 x 32 temperatures, Metropolis).  us per colour pass, 3D, heat bath (plain /
// words): L=64, 256 samples x 2 149 / 38; L=40, 100 x 2 33 / 8.7; L=100, 64 x 2
// 288 / 39; L=16, 256 x 2 10.2 / 6.1; L=24, 20 samples 8.2 / 4.5.
//
// Bound: HBM, a byte and an eighth a spin or coupling.  L=64, 256 x 2: packing 134 M
// spins and 201 M couplings 75 us in one launch of 4 bytes a thread and sample,
// sixteen loads under way (5 TB/s; 46 + 66 us in two launches of 2 bytes),
// unpacking the spins 44 us.
#include <algorithm>

#include "lattice.h"

namespace ianus {

namespace {

// Bytes and words of the spins or the couplings.
struct WordsPart {
  int8_t* bytes;    // sample s, unit u: s sample_stride + u unit_stride + site
  uint64_t* words;  // [G][units][N], split layout
  uint64_t sample_stride, unit_stride;
  uint32_t units;   // slots or dimensions
};

struct WordsParams {
  WordsPart part[2];  // spins, couplings: blockIdx.y counts the units of both
  Geom geom;
  int S;
};

// The two words of the sites 2q and 2q + 1 (natural order): even x first.
__device__ __forceinline__ void pair_words(const Geom& g, uint32_t q, uint32_t& even, uint32_t& odd) {
  const uint32_t h = (uint32_t)g.h, L = (uint32_t)g.L, row = q / h, k = q - row * h;
  const uint32_t c = g.D == 3 ? (row % L + row / L) & 1u : row & 1u;  // colour of even x
  even = (2u * row + c) * h + k;
  odd = (2u * row + 1u - c) * h + k;
}

// Thread: four neighbouring sites of a group's 64 samples, 4 bytes a sample (N
// is a multiple of 4), so that a warp's access to a sample is 128 contiguous bytes.
__global__ void __launch_bounds__(256) k_bytes_to_words(const WordsParams p) {
  const uint32_t q = blockIdx.x * blockDim.x + threadIdx.x, g = blockIdx.z;
  if (q >= p.geom.N / 4u) return;
  const bool couplings = blockIdx.y >= p.part[0].units;
  const WordsPart t = couplings ? p.part[1] : p.part[0];
  const uint32_t u = couplings ? blockIdx.y - p.part[0].units : blockIdx.y;
  const int8_t* in = t.bytes + (uint64_t)g * 64u * t.sample_stride + u * t.unit_stride + 4u * q;
  const int n = min(64, p.S - 64 * (int)g);
  uint32_t w[2][4] = {};  // half, site
#pragma unroll
  for (int hf = 0; hf < 2; ++hf)
#pragma unroll 1
    for (int l0 = 0; l0 < 32; l0 += 16) {
      uint32_t v[16];  // 16 loads under way
#pragma unroll
      for (int l = 0; l < 16; ++l) {
        const int s = 32 * hf + l0 + l;
        v[l] = s < n ? *(const uint32_t*)(in + (uint64_t)s * t.sample_stride) : 0u;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        uint32_t b = 0;
#pragma unroll
        for (int l = 0; l < 16; ++l) b |= (v[l] >> (8 * i + 7) & 1u) << l;
        w[hf][i] |= b << l0;
      }
    }
  uint64_t* out = t.words + ((uint64_t)g * t.units + u) * p.geom.N;
#pragma unroll
  for (int i = 0; i < 4; i += 2) {
    uint32_t ie, io;
    pair_words(p.geom, 2u * q + (uint32_t)i / 2u, ie, io);
    out[ie] = (uint64_t)w[0][i] | (uint64_t)w[1][i] << 32;
    out[io] = (uint64_t)w[0][i + 1] | (uint64_t)w[1][i + 1] << 32;
  }
}

__global__ void __launch_bounds__(256) k_words_to_bytes(const WordsParams p) {
  const uint32_t q = blockIdx.x * blockDim.x + threadIdx.x, u = blockIdx.y, g = blockIdx.z;
  if (q >= p.geom.half) return;
  const WordsPart& t = p.part[0];
  uint32_t ie, io;
  pair_words(p.geom, q, ie, io);
  const uint64_t* in = t.words + ((uint64_t)g * t.units + u) * p.geom.N;
  const uint64_t we = in[ie], wo = in[io];
  int8_t* out = t.bytes + (uint64_t)g * 64u * t.sample_stride + u * t.unit_stride + 2u * q;
  const int n = min(64, p.S - 64 * (int)g);
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const uint32_t e = (uint32_t)(we >> (32 * w)), o = (uint32_t)(wo >> (32 * w));
#pragma unroll 16
    for (int l = 0; l < 32; ++l) {
      if (32 * w + l >= n) continue;
      // 1 or -1: 1 - 2 b in each byte
      const uint32_t v = (e >> l & 1u ? 0xFFu : 1u) | (o >> l & 1u ? 0xFF00u : 0x100u);
      *(uint16_t*)(out + (uint64_t)(32 * w + l) * t.sample_stride) = (uint16_t)v;
    }
  }
}

WordsParams params(const Lattice& lat) {
  WordsParams p{};
  p.geom = lat.geom;
  p.S = lat.S;
  const uint64_t N = lat.N, S = (uint64_t)lat.S, D = (uint64_t)lat.D;
  p.part[0] = WordsPart{(int8_t*)lat.spins, (uint64_t*)lat.words->spins, N, S * N, (uint32_t)lat.slots};
  p.part[1] = WordsPart{(int8_t*)lat.J, (uint64_t*)lat.words->J, D * N, N, (uint32_t)lat.D};
  return p;
}

}  // namespace

cudaError_t launch_pack_words(Lattice& lat) {
  const WordsParams p = params(lat);
  const dim3 grid((lat.N / 4u + 255u) / 256u, p.part[0].units + p.part[1].units, (unsigned)(lat.S + 63) / 64u);
  k_bytes_to_words<<<grid, 256, 0, lat.stream>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_unpack_spins(Lattice& lat) {
  const WordsParams p = params(lat);
  const dim3 grid((lat.geom.half + 255u) / 256u, p.part[0].units, (unsigned)(lat.S + 63) / 64u);
  k_words_to_bytes<<<grid, 256, 0, lat.stream>>>(p);
  return cudaGetLastError();
}

// Estimated us of a run of n sweeps in words: 5 us a pass and 34 ns a thousand
// words, the conversions (the couplings', too) at 3 bytes/ns and their launches;
// against the plain sweeps' (plain_us), with a fifth in hand.
bool words_pay(const Lattice& lat, uint64_t n) {
  if (!lat.words || n < 2) return false;
  const double spins = (double)lat.S * lat.slots * lat.N, words = (double)lat.words->G * lat.slots * lat.geom.half;
  const double pass = 5.0 + 0.034e-3 * words;
  const double convert = 20.0 + (2.25 * spins + 1.125 * lat.S * lat.D * (double)lat.N) / 3e6;
  return 1.2 * (2.0 * pass * n + convert) < plain_us(lat) * n;
}

}  // namespace ianus
