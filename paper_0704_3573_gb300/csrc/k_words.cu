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
// The sweep is the precompiled per-lane-plane kernel, which needs no run-time
// compiler for a new temperature.  us per colour pass, 3D, heat bath (plain /
// words): L=64, 256 samples x 2 149 / 38; L=40, 100 x 2 33 / 8.7; L=100, 64 x 2
// 288 / 39; L=16, 256 x 2 10.2 / 6.1; L=24, 20 samples 8.2 / 4.5.
//
// Bound: HBM, a byte and an eighth a spin: 134 M spins 46 us with sixteen loads
// under way a thread (121 one by one).
#include <algorithm>

#include "lattice.h"

namespace ianus {

namespace {

struct WordsParams {
  int8_t* bytes;    // sample s, unit u: s sample_stride + u unit_stride + site
  uint64_t* words;  // [G][units][N], split layout
  uint64_t sample_stride, unit_stride;
  Geom geom;
  uint32_t units;   // slots or dimensions
  int S;
};

// The two words of the sites 2q and 2q + 1 (natural order): even x first.
__device__ __forceinline__ void pair_words(const Geom& g, uint32_t q, uint32_t& even, uint32_t& odd) {
  const uint32_t h = (uint32_t)g.h, L = (uint32_t)g.L, row = q / h, k = q - row * h;
  const uint32_t c = g.D == 3 ? (row % L + row / L) & 1u : row & 1u;  // colour of even x
  even = (2u * row + c) * h + k;
  odd = (2u * row + 1u - c) * h + k;
}

// Thread: two neighbouring sites of a group's 64 samples, 2 bytes a sample, so
// that a warp's access to a sample is 64 contiguous bytes.
__global__ void __launch_bounds__(256) k_bytes_to_words(const WordsParams p) {
  const uint32_t q = blockIdx.x * blockDim.x + threadIdx.x, u = blockIdx.y, g = blockIdx.z;
  if (q >= p.geom.half) return;
  const int8_t* in = p.bytes + (uint64_t)g * 64u * p.sample_stride + u * p.unit_stride + 2u * q;
  const int n = min(64, p.S - 64 * (int)g);
  uint32_t e[2] = {0u, 0u}, o[2] = {0u, 0u};
#pragma unroll
  for (int w = 0; w < 2; ++w)
#pragma unroll 1
    for (int l0 = 0; l0 < 32; l0 += 16) {
      uint32_t v[16];  // 16 loads under way
#pragma unroll
      for (int l = 0; l < 16; ++l) {
        const int s = 32 * w + l0 + l;
        v[l] = s < n ? *(const uint16_t*)(in + (uint64_t)s * p.sample_stride) : 0u;
      }
      uint32_t be = 0, bo = 0;
#pragma unroll
      for (int l = 0; l < 16; ++l) {
        be |= (v[l] >> 7 & 1u) << l;
        bo |= (v[l] >> 15) << l;
      }
      e[w] |= be << l0;
      o[w] |= bo << l0;
    }
  uint32_t ie, io;
  pair_words(p.geom, q, ie, io);
  uint64_t* out = p.words + ((uint64_t)g * p.units + u) * p.geom.N;
  out[ie] = (uint64_t)e[0] | (uint64_t)e[1] << 32;
  out[io] = (uint64_t)o[0] | (uint64_t)o[1] << 32;
}

__global__ void __launch_bounds__(256) k_words_to_bytes(const WordsParams p) {
  const uint32_t q = blockIdx.x * blockDim.x + threadIdx.x, u = blockIdx.y, g = blockIdx.z;
  if (q >= p.geom.half) return;
  uint32_t ie, io;
  pair_words(p.geom, q, ie, io);
  const uint64_t* in = p.words + ((uint64_t)g * p.units + u) * p.geom.N;
  const uint64_t we = in[ie], wo = in[io];
  int8_t* out = p.bytes + (uint64_t)g * 64u * p.sample_stride + u * p.unit_stride + 2u * q;
  const int n = min(64, p.S - 64 * (int)g);
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const uint32_t e = (uint32_t)(we >> (32 * w)), o = (uint32_t)(wo >> (32 * w));
#pragma unroll 16
    for (int l = 0; l < 32; ++l) {
      if (32 * w + l >= n) continue;
      // 1 or -1: 1 - 2 b in each byte
      const uint32_t v = (e >> l & 1u ? 0xFFu : 1u) | (o >> l & 1u ? 0xFF00u : 0x100u);
      *(uint16_t*)(out + (uint64_t)(32 * w + l) * p.sample_stride) = (uint16_t)v;
    }
  }
}

WordsParams params(const Lattice& lat, bool couplings) {
  WordsParams p{};
  p.geom = lat.geom;
  p.S = lat.S;
  if (couplings) {
    p.bytes = (int8_t*)lat.J;
    p.words = (uint64_t*)lat.words->J;
    p.units = (uint32_t)lat.D;
    p.sample_stride = (uint64_t)lat.D * lat.N;
    p.unit_stride = lat.N;
  } else {
    p.bytes = (int8_t*)lat.spins;
    p.words = (uint64_t*)lat.words->spins;
    p.units = (uint32_t)lat.slots;
    p.sample_stride = lat.N;
    p.unit_stride = (uint64_t)lat.S * lat.N;
  }
  return p;
}

dim3 grid_of(const Lattice& lat, uint32_t units) {
  return dim3((lat.geom.half + 255u) / 256u, units, (unsigned)(lat.S + 63) / 64u);
}

}  // namespace

cudaError_t launch_pack_spins(Lattice& lat) {
  const WordsParams p = params(lat, false);
  k_bytes_to_words<<<grid_of(lat, p.units), 256, 0, lat.stream>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_pack_couplings(Lattice& lat) {
  const WordsParams p = params(lat, true);
  k_bytes_to_words<<<grid_of(lat, p.units), 256, 0, lat.stream>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_unpack_spins(Lattice& lat) {
  const WordsParams p = params(lat, false);
  k_words_to_bytes<<<grid_of(lat, p.units), 256, 0, lat.stream>>>(p);
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
