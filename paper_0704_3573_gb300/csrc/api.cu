// api.cu -- the extern "C" entry points of libianus.so (declared and
// documented in include/ianus.h): lattice set-up, the sweep loop
// (Sec. 2.2 sweeps of the two-colour update of Sec. 3.1), acceptance-table
// uploads (Sec. 3.2), measurements (Sec. 4.1), parallel tempering,
// checkpoints and error reporting.  Host logic only; all per-site work runs
// in the kernels of k_plain.cu, k_msc.cu, k_potts.cu and k_pt.cu.
#include <atomic>
#include <cmath>
#include <functional>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "lattice.h"

using namespace ianus;

namespace {

constexpr uint32_t kDefaultSeries = 1024;
constexpr uint32_t kPtCapMax = 4096;
constexpr uint64_t kStateMagic = 0x31534e4149ull;  // "IANS1"

struct Sizes {
  int model, D, L, S, R, K, slots, layout, G, Q4, mq;
  uint32_t N, cap, pt_cap;
  bool field;
  int fpc;
  uint32_t rows;
  size_t off_wheels, wheel_bytes;
  bool poolable;
  size_t off_segs, off_nseg;
  size_t off_spins, off_J, off_thr, off_tp, off_fthr, off_ftp, off_sites, off_ptab, off_pttab, off_ptsign, off_slot,
      off_temp, off_acc_pt, off_acc, off_oE, off_oM, off_oQ, off_sw, off_sE, off_sM, off_sQ, off_err, off_tdev, off_flags, least, total;
  size_t off_masks, mask_bytes, off_wspins, off_wJ, off_wtp;
  bool words;  // room for the lattice in words
  size_t spins_bytes, J_bytes, sites_bytes;
};

constexpr size_t kMaxSmemPerBlock = 227 * 1024;

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Validates cfg and lays out the device buffer.  Returns IANUS_OK or an error.
int plan(const ianus_config* c, Sizes& z) {
  if (!c) return IANUS_EINVAL;
  if (c->abi_version != IANUS_ABI_VERSION) return IANUS_EINVAL;
  if (c->model != IANUS_EA_PM_J && c->model != IANUS_POTTS4_J && c->model != IANUS_POTTS4_PERM) return IANUS_EINVAL;
  if (c->dim != 2 && c->dim != 3 && !(c->dim == 4 && c->model == IANUS_POTTS4_PERM)) return IANUS_EINVAL;
  if (c->L < 2 || (c->L & 1) || c->L > 4096) return IANUS_EINVAL;
  if (c->n_samples < 1 || c->n_samples >= (1 << 18)) return IANUS_EINVAL;
  if (c->n_replicas < 1 || c->n_temps < 1) return IANUS_EINVAL;
  if ((long long)c->n_replicas * c->n_temps >= 4096) return IANUS_EINVAL;
  if (c->disorder < IANUS_DISORDER_PM_J || c->disorder > IANUS_DISORDER_DAFF) return IANUS_EINVAL;
  const bool field = c->disorder == IANUS_DISORDER_RFIM || c->disorder == IANUS_DISORDER_DAFF;
  if (!std::isfinite(c->field) || c->field < 0.0) return IANUS_EINVAL;
  if (!field && c->field != 0.0) return IANUS_EINVAL;
  if (c->disorder == IANUS_DISORDER_DAFF && !(c->occupation >= 0.0 && c->occupation <= 1.0)) return IANUS_EINVAL;
  if (field && c->model != IANUS_EA_PM_J) return IANUS_EINVAL;
  if (c->rng != IANUS_RNG_PHILOX && c->rng != IANUS_RNG_WHEEL) return IANUS_EINVAL;
  uint64_t N = 1;
  for (int d = 0; d < c->dim; ++d) N *= (uint64_t)c->L;
  if (N >= (1ull << 31)) return IANUS_EINVAL;
  int layout = c->layout;
  const bool potts = c->model != IANUS_EA_PM_J;
  if (layout == IANUS_LAYOUT_AUTO)
    layout = potts ? IANUS_LAYOUT_U8X4
             : c->rng == IANUS_RNG_WHEEL ? IANUS_LAYOUT_I8
                                         : IANUS_LAYOUT_BITS64;
  if (layout < IANUS_LAYOUT_I8 || layout > IANUS_LAYOUT_U8X4) return IANUS_EINVAL;
  if (!potts && layout == IANUS_LAYOUT_U8X4) return IANUS_EUNSUPPORTED;
  if (potts && layout != IANUS_LAYOUT_U8X4) return IANUS_EUNSUPPORTED;
  if (c->rng == IANUS_RNG_WHEEL && (potts || layout != IANUS_LAYOUT_I8)) return IANUS_EUNSUPPORTED;
  if (layout == IANUS_LAYOUT_BITS64 &&  // the sweep stages one block's threshold planes in shared memory
      (!field ? sweep_bits_smem(c->n_replicas)
              : (size_t)c->n_replicas * kPlanes *
                    (c->disorder == IANUS_DISORDER_DAFF ? kDiluteClasses : kFieldPlaneClasses) * 8) > kMaxSmemPerBlock)
    return IANUS_EUNSUPPORTED;
  z.model = c->model;
  z.D = c->dim;
  z.L = c->L;
  z.S = c->n_samples;
  z.R = c->n_replicas;
  z.K = c->n_temps;
  z.slots = z.R * z.K;
  z.layout = layout;
  z.N = (uint32_t)N;
  z.G = (z.S + 63) / 64;
  z.Q4 = (z.S + 3) / 4;
  z.field = field;
  z.mq = potts ? 4 : (field ? 2 : 1);
  z.cap = c->series_capacity ? c->series_capacity : kDefaultSeries;
  z.pt_cap = z.K > 1 ? (uint32_t)std::min<uint64_t>((uint64_t)z.D * N / 2 + 1, kPtCapMax) : 0;
  if (layout == IANUS_LAYOUT_I8) {
    z.spins_bytes = (size_t)z.slots * z.S * N;
    z.J_bytes = (size_t)z.S * z.D * N;
  } else if (layout == IANUS_LAYOUT_BITS64) {
    z.spins_bytes = (size_t)z.G * z.slots * N * 8;
    z.J_bytes = (size_t)z.G * z.D * N * 8;
  } else {
    z.spins_bytes = (size_t)z.slots * z.Q4 * N * 4;
    z.J_bytes = (size_t)z.Q4 * z.D * N * 4;
  }
  // I8: hs, occ int8 [S][N]; BITS64: hbits, xbits u64 [G][N]
  z.sites_bytes = !field ? 0 : layout == IANUS_LAYOUT_I8 ? (size_t)2 * z.S * N : (size_t)2 * z.G * N * 8;
  z.fpc = c->disorder == IANUS_DISORDER_DAFF ? kDiluteClasses : kFieldPlaneClasses;
  z.rows = (uint32_t)(N / (uint64_t)c->L);
  z.wheel_bytes = c->rng == IANUS_RNG_WHEEL ? (size_t)z.slots * z.S * 2 * 64 * z.rows * 4 : 0;
  const size_t SKR = (size_t)z.S * z.K * z.R;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    size_t at = o;
    o += align256(bytes);
    return at;
  };
  z.off_spins = take(z.spins_bytes);
  z.off_J = take(z.J_bytes);
  z.off_thr = take((size_t)z.K * kMaxClasses * 8 + sizeof(UniformLut));  // class thresholds, then the uniform tables
  z.off_tp = take(layout == IANUS_LAYOUT_BITS64 && !field ? (size_t)z.G * z.slots * kPlanes * kMaxClasses * 8 : 0);
  z.off_fthr = take(field ? (size_t)z.K * kFieldClasses * 8 + sizeof(FieldLut) : 0);  // then the uniform tables
  z.off_ftp = take(field && layout == IANUS_LAYOUT_BITS64 ? (size_t)z.G * z.slots * kPlanes * z.fpc * 8 : 0);
  z.off_sites = take(z.sites_bytes);
  z.off_wheels = take(z.wheel_bytes);
  // segment tables for fused serving: bit-sliced EA lattices with one replica
  // and one temperature
  z.poolable = !potts && !field && layout == IANUS_LAYOUT_BITS64 && z.R == 1 && z.K == 1;
  z.off_segs = take(z.poolable ? (size_t)z.G * kMaxSegs * sizeof(Segment) : 0);
  z.off_nseg = take(z.poolable ? (size_t)z.G * 4 : 0);
  z.off_ptab = take(layout != IANUS_LAYOUT_U8X4 ? 0
                    : c->model == IANUS_POTTS4_PERM ? (size_t)z.K * perm_table_entries(z.D) * 16
                                                    : (size_t)z.K * kPottsRows * 16);
  z.off_pttab = take((size_t)std::max(z.K - 1, 0) * z.pt_cap * 8);
  z.off_ptsign = take((size_t)std::max(z.K - 1, 1));
  z.off_slot = take((size_t)z.S * z.R * z.K * 4 * 2);  // slot_at then temp_of
  z.off_temp = z.off_slot + (size_t)z.S * z.R * z.K * 4;
  z.off_acc_pt = take((size_t)z.S * z.R * std::max(z.K - 1, 1) * 8);
  z.off_acc = take((size_t)z.S * z.slots * kAccStride * 8);
  z.off_oE = take(SKR * 8);
  z.off_oM = take(SKR * z.mq * 8);
  z.off_oQ = take((size_t)z.S * z.K * 8);
  z.off_sw = take((size_t)z.cap * 8);
  z.off_sE = take((size_t)z.cap * SKR * 8);
  z.off_sM = take((size_t)z.cap * SKR * z.mq * 8);
  z.off_sQ = take((size_t)z.cap * z.S * z.K * 8);
  z.off_err = take(8);
  z.off_tdev = take(24);
  // progress flags of the persistent one-temperature bit-sliced sweep
  z.off_flags = take(layout == IANUS_LAYOUT_BITS64 && !field && z.K == 1 ? (size_t)kMaxPersistBlocks * 4 : 0);
  z.least = o;  // the rest only makes sweeps faster
  z.mask_bytes = layout == IANUS_LAYOUT_I8 && !field && c->rng == IANUS_RNG_PHILOX && z.K == 1
                     ? packed_mask_bytes(z.N, (uint64_t)z.S * z.R)
                     : 0;
  z.off_masks = take(z.mask_bytes);
  // the same lattice in words: from 8 samples on, at most 2 GiB, replicas whose
  // threshold planes fit one block of the word sweep (up to 110), and no more
  // (group, replica) rows than a launch of the measurement takes
  const size_t wspins = (size_t)z.G * z.slots * z.N * 8, wJ = (size_t)z.G * z.D * z.N * 8;
  const size_t wtp = (size_t)z.G * z.slots * kPlanes * kMaxClasses * 8;
  z.words = layout == IANUS_LAYOUT_I8 && !field && c->rng == IANUS_RNG_PHILOX && z.K == 1 && z.S >= 8 &&
            sweep_bits_smem(z.R) <= kMaxSmemPerBlock && (z.R <= 2 || (size_t)z.G * z.slots <= 65535) && wspins + wJ + wtp <= (size_t)2 << 30;
  z.off_wspins = take(z.words ? wspins : 0);
  z.off_wJ = take(z.words ? wJ : 0);
  z.off_wtp = take(z.words ? wtp : 0);
  z.total = o;
  return IANUS_OK;
}

// A failure code usable as the return value of both the int helpers and the
// ianus_status entry points.
struct Fail {
  int v;
  operator int() const { return v; }
  operator ianus_status() const { return (ianus_status)v; }
};

Fail fail(Lattice* lat, int st) {
  if (lat && st == IANUS_ECUDA) lat->sticky = IANUS_ESTATE;
  return Fail{st};
}

#define CK(expr)                                     \
  do {                                               \
    cudaError_t e_ = (expr);                         \
    if (e_ != cudaSuccess) return fail(lat, IANUS_ECUDA); \
  } while (0)

void drop_graphs(Lattice* lat);

}  // namespace

// Bit c of t[q] is bit 31 - q of class c's threshold; `always` marks the
// classes that flip whatever the random number (threshold 2^32), `need` the
// classes whose comparison decides the flip.
UniformLut ianus::uniform_lut(int dim, int algo, const uint64_t* thr) {
  UniformLut u{};
  uint32_t always = 0, cmp = 0;
  for (int c = 0; c <= 2 * dim; ++c) {
    const uint64_t T = thr[c];
    if (T >= kTwo32) always |= 1u << c;
    else if (algo == IANUS_HEATBATH || c < dim) cmp |= 1u << c;
    for (int q = 0; q < 32; ++q)
      if (T < kTwo32 && ((T >> (31 - q)) & 1ull)) u.t[q] |= (uint8_t)(1u << c);
  }
  u.always = (uint8_t)always;
  u.need = (uint8_t)cmp;
  return u;
}

namespace {

bool beta_ok(const double* beta, int K) {
  for (int k = 0; k < K; ++k)
    if (!std::isfinite(beta[k]) || beta[k] < 0.0) return false;
  return true;
}

// Table row of one tuple of Potts counts: the thresholds, 2^32 - 1 standing
// for 2^32, and a flag for each of those.
uint4 potts_table_row(double beta, const int* n) {
  uint64_t T[3];
  potts_thresholds(beta, n, T);
  auto word = [](uint64_t t) { return t >= kTwo32 ? 0xffffffffu : (uint32_t)t; };
  return make_uint4(word(T[0]), word(T[1]), word(T[2]),
                    (T[0] >= kTwo32 ? 1u : 0u) | (T[1] >= kTwo32 ? 2u : 0u) | (T[2] >= kTwo32 ? 4u : 0u));
}

// Rebuild and upload the acceptance tables for (algo, beta).
int upload_tables(Lattice* lat, int algo, const double* beta) {
  const int K = lat->K;
  if (lat->field) {
    std::vector<uint64_t> fthr((size_t)K * kFieldClasses);
    for (int k = 0; k < K; ++k) field_thresholds(lat->D, algo, beta[k], lat->hmag, &fthr[(size_t)k * kFieldClasses]);
    CK(cudaMemcpyAsync(lat->fthr, fthr.data(), fthr.size() * 8, cudaMemcpyHostToDevice, lat->stream));
    if (lat->layout == IANUS_LAYOUT_BITS64) CK(launch_build_field_planes(*lat));
    lat->ulut_ok = false;
    lat->jit = nullptr;
    lat->jit_algo = -1;
    lat->flut_ok = false;
    lat->jitf = nullptr;
    lat->jitf_algo = -1;
    if (K == 1 && lat->layout == IANUS_LAYOUT_BITS64) {
      // one temperature: the truth tables of the specialised field kernel.
      // Without dilution the class is (u, f), field class (v + 2D) * 2 + f
      // with v = 2D - 2u, tables [f][0] bit u.  With dilution it is (t, f),
      // t = v + 2D = 8 t3 + k, tables [f][t3] bit k.
      FieldLut fl{};
      for (int f = 0; f < 2; ++f)
        for (int cls = 0; cls <= (lat->dilute ? 4 * lat->D : 2 * lat->D); ++cls) {
          const int t = lat->dilute ? cls : 4 * lat->D - 2 * cls;
          const int hi = lat->dilute ? (cls >> 3) : 0, bit = lat->dilute ? (cls & 7) : cls;
          const uint64_t T = fthr[(size_t)t * 2 + f];
          if (T >= kTwo32) {
            fl.always[f][hi] |= (uint8_t)(1u << bit);
          } else {
            fl.need[f][hi] |= (uint8_t)(1u << bit);
            for (int q = 0; q < 32; ++q)
              if ((T >> (31 - q)) & 1ull) fl.t[f][hi][q] |= (uint8_t)(1u << bit);
          }
        }
      lat->flut = fl;
      CK(cudaMemcpyAsync(lat->fthr + (size_t)K * kFieldClasses, &lat->flut, sizeof(FieldLut), cudaMemcpyHostToDevice,
                         lat->stream));
      lat->flut_ok = true;
    }
  } else if (lat->model == IANUS_EA_PM_J) {
    std::vector<uint64_t> thr((size_t)K * kMaxClasses);
    for (int k = 0; k < K; ++k) class_thresholds(lat->D, algo, beta[k], &thr[(size_t)k * kMaxClasses]);
    CK(cudaMemcpyAsync(lat->thr, thr.data(), thr.size() * 8, cudaMemcpyHostToDevice, lat->stream));
    if (lat->layout == IANUS_LAYOUT_BITS64) CK(launch_build_planes(*lat));
    lat->ulut_ok = false;
    if (K == 1) {
      lat->ulut = uniform_lut(lat->D, algo, thr.data());
      CK(cudaMemcpyAsync(lat->thr + (size_t)K * kMaxClasses, &lat->ulut, sizeof(UniformLut), cudaMemcpyHostToDevice,
                         lat->stream));
      lat->ulut_ok = true;
    }
    lat->jit = nullptr;  // specialised lazily by the first launch that wants it
    lat->jit_algo = -1;
  } else if (lat->model == IANUS_POTTS4_PERM) {
    // counts n_k in 0..2D with n0 + n1 + n2 + n3 = 2D
    const int D = lat->D;
    for (int k = 0; k < K; ++k)
      if (2.0 * D * beta[k] > 700.0) return IANUS_EINVAL;  // exp(2D beta) must stay finite
    const uint32_t NT = perm_table_entries(D);
    std::vector<uint4> tab((size_t)K * NT);
    std::memset(tab.data(), 0, tab.size() * sizeof(uint4));
    for (int k = 0; k < K; ++k)
      for (int n0 = 0; n0 <= 2 * D; ++n0)
        for (int n1 = 0; n0 + n1 <= 2 * D; ++n1)
          for (int n2 = 0; n0 + n1 + n2 <= 2 * D; ++n2) {
            const int n[4] = {n0, n1, n2, 2 * D - n0 - n1 - n2};
            tab[(size_t)k * NT + perm_row(D, n0, n1, n2)] = potts_table_row(beta[k], n);
          }
    CK(cudaMemcpyAsync(lat->ptab, tab.data(), tab.size() * sizeof(uint4), cudaMemcpyHostToDevice, lat->stream));
  } else {
    for (int k = 0; k < K; ++k)
      if (beta[k] > 100.0) return IANUS_EINVAL;  // exp(6 beta) must stay finite
    // counts with sum |n_k| <= 2D and even, as the 2D bonds of weight +-1 give
    const int m = 2 * lat->D;
    std::vector<uint4> tab((size_t)K * kPottsRows);
    std::memset(tab.data(), 0, tab.size() * sizeof(uint4));
    for (int k = 0; k < K; ++k) {
      int n[4];
      for (n[0] = -m; n[0] <= m; ++n[0])
        for (n[1] = -m; n[1] <= m; ++n[1])
          for (n[2] = -m; n[2] <= m; ++n[2])
            for (n[3] = -m; n[3] <= m; ++n[3]) {
              const int sum = std::abs(n[0]) + std::abs(n[1]) + std::abs(n[2]) + std::abs(n[3]);
              if (sum > m || (sum & 1)) continue;
              tab[(size_t)k * kPottsRows + potts_row(n[0], n[1], n[2], n[3])] = potts_table_row(beta[k], n);
            }
    }
    CK(cudaMemcpyAsync(lat->ptab, tab.data(), tab.size() * sizeof(uint4), cudaMemcpyHostToDevice, lat->stream));
  }
  if (K > 1 && lat->model == IANUS_EA_PM_J && !lat->field) {
    // PT tables: T(m) for |d| = 4m until the first zero (or the largest
    // possible |d|/4 = D N / 2).
    std::vector<uint64_t> pt((size_t)(K - 1) * lat->pt_cap, 0);
    std::vector<int8_t> sign((size_t)K - 1);
    uint32_t len = 1;
    const uint64_t mmax = (uint64_t)lat->D * lat->N / 2;
    for (int k = 0; k + 1 < K; ++k) {
      const double db = beta[k] - beta[k + 1];
      sign[k] = db > 0 ? 1 : (db < 0 ? -1 : 0);
      if (sign[k] == 0) continue;
      std::vector<uint64_t> col(lat->pt_cap);
      table_pt(beta[k], beta[k + 1], col.data(), col.size());
      uint32_t m = 0;
      while (m < lat->pt_cap && m < mmax && col[m] != 0) ++m;
      if (m == lat->pt_cap && m < mmax) return IANUS_EUNSUPPORTED;  // temperatures too close for the table
      for (uint32_t q = 0; q < m; ++q) pt[(size_t)k * lat->pt_cap + q] = col[q];
      len = std::max(len, m);
    }
    lat->pt_falls = true;
    for (int k = 0; k + 1 < K && lat->pt_falls; ++k)
      lat->pt_falls = std::is_sorted(pt.begin() + (size_t)k * lat->pt_cap, pt.begin() + (size_t)(k + 1) * lat->pt_cap,
                                     std::greater<uint64_t>());
    lat->pt_len = lat->pt_cap;  // rows are stored with stride pt_cap; zeros end each row
    (void)len;
    CK(cudaMemcpyAsync(lat->pttab, pt.data(), pt.size() * 8, cudaMemcpyHostToDevice, lat->stream));
    CK(cudaMemcpyAsync(lat->pt_sign, sign.data(), sign.size(), cudaMemcpyHostToDevice, lat->stream));
  }
  lat->beta.assign(beta, beta + K);
  lat->algo = algo;
  lat->tables_ok = true;
  drop_graphs(lat);  // captured kernels depend on the tables and the algorithm
  return IANUS_OK;
}

void acc_fresh(Lattice* lat) {
  lat->acc_ok = true;
  lat->acc_sweeps = lat->sweeps;
  lat->acc_mut = lat->mut;
}

int measure_into(Lattice* lat, int64_t* E, int64_t* M, int64_t* Q, uint64_t* sweep_out, int want_q) {
  want_q = want_q && lat->R >= 2;
  if (lat->layout == IANUS_LAYOUT_I8)
    CK(launch_measure_i8(*lat, want_q));
  else if (lat->layout == IANUS_LAYOUT_BITS64)
    CK(launch_measure_bits(*lat, want_q));
  else
    CK(launch_measure_potts(*lat, want_q));
  acc_fresh(lat);
  CK(launch_finalize(*lat, E, M, Q, sweep_out, want_q));
  return IANUS_OK;
}

int record_row(Lattice* lat) {
  const size_t SKR = (size_t)lat->S * lat->K * lat->R;
  const size_t row = (size_t)(lat->ser_count % lat->cap);
  int st = measure_into(lat, lat->ser_E + row * SKR, lat->ser_M + row * SKR * lat->mq,
                        lat->ser_Q + row * (size_t)lat->S * lat->K, lat->ser_sweep + row, 1);
  if (st) return st;
  lat->ser_count += 1;
  lat->t_dev_valid = false;
  return IANUS_OK;
}

int one_sweep(Lattice* lat, int inv) {
  const uint64_t t = lat->sweeps;
  for (int c = 0; c < 2; ++c) {
    if (lat->layout == IANUS_LAYOUT_I8)
      CK(launch_sweep_i8(*lat, c, t, inv));
    else if (lat->layout == IANUS_LAYOUT_BITS64)
      CK(launch_sweep_bits(*lat, c, t, inv));
    else
      CK(launch_sweep_potts(*lat, c, t));
  }
  lat->sweeps += 1;
  return IANUS_OK;
}

bool same_beta(const Lattice* lat, const double* beta) {
  if ((int)lat->beta.size() != lat->K) return false;
  for (int k = 0; k < lat->K; ++k)
    if (std::memcmp(&lat->beta[k], &beta[k], sizeof(double)) != 0) return false;
  return true;
}

int do_pt_swap(Lattice* lat) {
  // energies of every configuration: those of the last measurement when no
  // sweep or other change came after it, else measured (U only when
  // bit-sliced)
  if (!(lat->acc_ok && lat->acc_sweeps == lat->sweeps && lat->acc_mut == lat->mut)) {
    if (lat->layout == IANUS_LAYOUT_BITS64)
      CK(launch_measure_bits(*lat, 0, true));
    else
      CK(launch_measure_i8(*lat, 0));
    acc_fresh(lat);
  }
  CK(launch_pt_swap(*lat));
  lat->steps += 1;
  lat->t_dev_valid = false;
  if (lat->layout == IANUS_LAYOUT_BITS64) CK(launch_build_planes(*lat));
  return IANUS_OK;
}

// ---- CUDA graphs of sweep blocks ----

void drop_graphs(Lattice* lat) {
  if (!lat->graphs) return;
  for (auto& kv : *lat->graphs)
    if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
  lat->graphs->clear();
}

// Resident sweep of a bit-sliced lattice for a run of n sweeps.
enum class Resident { kNone, kBlock, kCluster };

Resident resident_kind(Lattice* lat, uint64_t n) {
  if (lat->layout != IANUS_LAYOUT_BITS64 || n < 2 || !lat->use_resident || lat->variant != 0) return Resident::kNone;
  if (resident_cluster_bits(*lat)) return Resident::kCluster;
  return resident_bits_fits(*lat) ? Resident::kBlock : Resident::kNone;
}

cudaError_t launch_resident(Lattice* lat, Resident kind, int inv, uint64_t t0, uint32_t n) {
  return kind == Resident::kCluster ? launch_resident_cluster_bits(*lat, inv, t0, n)
                                    : launch_resident_bits(*lat, inv, t0, n);
}

// What ends a captured cycle: a series row, a series row and a swap step, or a
// swap step on energies measured for it alone.
enum class Swap : uint32_t { kNone = 0, kMeasured = 1, kOnly = 2 };

// One colour pass of the chain being captured.
cudaError_t launch_pass(Lattice* lat, int colour, uint64_t t, int inv) {
  if (lat->layout == IANUS_LAYOUT_I8) return launch_sweep_i8(*lat, colour, t, inv);
  if (lat->layout == IANUS_LAYOUT_BITS64) return launch_sweep_bits(*lat, colour, t, inv);
  return launch_sweep_potts(*lat, colour, t);
}

// Captures B sweeps (2B colour kernels reading the device sweep counter at
// offsets 0..B-1), or with cycles > 0 that many times B sweeps and a
// measurement into the next series row, and the counters' advance on private
// streams.  A large lattice is captured as up to four chains, each a part of
// its configurations on a stream of its own: while one chain's pass drains and
// its next one starts, the others' blocks keep the SMs busy (L=64, 256 x 2,
// heat bath: 20.0 -> 18.2 us per colour pass; random fields L=64, 256: 14.2 ->
// 12.3).  A bit-sliced chain's counts follow its sweeps without waiting for
// the other chains (but for the overlap, which reads them all), and the
// accumulators are cleared and turned into the series row on another stream
// beside the next sweeps (L=20, 100 x 4 replicas, 100 sweeps with 10
// measurements: 1344 -> 1204 us).  With a swap each cycle ends in a
// parallel-tempering step, which needs every energy; its cycles follow one
// another.
int build_graph(Lattice* lat, int inv, uint32_t B, uint32_t cycles, Swap swap, cudaGraphExec_t* out) {
  const bool bits = lat->layout == IANUS_LAYOUT_BITS64;
  const Resident kind = cycles > 0 ? resident_kind(lat, B) : Resident::kNone;
  int chains = 1;
  if (kind != Resident::kNone) {
    chains = 1;
  } else if (bits) {
    prepare_sweep_bits(*lat, inv);  // compile before capturing
    chains = sweep_chains_bits(*lat, inv);
  } else if (lat->layout == IANUS_LAYOUT_U8X4) {
    chains = sweep_chains_potts(*lat);
  } else {
    chains = sweep_chains_i8(*lat);
  }
  const int side = cycles > 0 && bits ? kMaxChains : chains - 1;  // side streams in use
  if (!lat->cap_stream) CK(cudaStreamCreateWithFlags(&lat->cap_stream, cudaStreamNonBlocking));
  for (int k = 0; k < side; ++k)
    if ((k + 1 < chains || k + 1 == kMaxChains) && !lat->side_streams[k])
      CK(cudaStreamCreateWithFlags(&lat->side_streams[k], cudaStreamNonBlocking));
  cudaEvent_t ev = nullptr;
  CK(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
  const cudaStream_t user = lat->stream, main = lat->cap_stream, aux = lat->side_streams[kMaxChains - 1];
  const int want_q = lat->R >= 2;
  lat->capturing = true;
  lat->chains = chains;
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaStreamBeginCapture(main, cudaStreamCaptureModeThreadLocal);
  auto stream_of = [&](int k) { return k == 0 ? main : lat->side_streams[k - 1]; };
  // `to` continues after what `from` holds now
  auto after = [&](cudaStream_t to, cudaStream_t from) {
    if (e == cudaSuccess) e = cudaEventRecord(ev, from);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(to, ev, 0);
  };
  auto sweeps = [&](int k, uint32_t s0) {
    lat->chain = k;
    lat->stream = stream_of(k);
    if (kind != Resident::kNone && e == cudaSuccess) {
      e = launch_resident(lat, kind, inv, s0, B);
      return;
    }
    for (uint32_t s = s0; e == cudaSuccess && s < s0 + B; ++s)
      for (int c = 0; e == cudaSuccess && c < 2; ++c) e = launch_pass(lat, c, s, inv);
  };
  auto clear = [&]() {
    if (e == cudaSuccess)
      e = cudaMemsetAsync(lat->acc, 0, (size_t)lat->S * lat->slots * kAccStride * sizeof(int64_t), aux);
  };
  for (int k = 1; k < chains; ++k) after(stream_of(k), main);
  if (cycles == 0) {
    for (int k = 0; k < chains; ++k) sweeps(k, 0);
    for (int k = 1; k < chains; ++k) after(main, stream_of(k));
  } else if (bits) {
    after(aux, main);
    clear();
    for (uint32_t n = 0; n < cycles; ++n) {
      for (int k = 0; k < chains; ++k) {
        sweeps(k, n * B);
        after(stream_of(k), aux);  // cleared accumulators
        if (e == cudaSuccess) e = launch_measure_bits_counts(*lat, swap == Swap::kOnly);
      }
      if (swap != Swap::kNone) {
        for (int k = 1; k < chains; ++k) after(main, stream_of(k));
        lat->stream = main;
        if (swap == Swap::kMeasured) {
          if (e == cudaSuccess && overlap_apart(*lat, want_q)) e = launch_overlap_bits(*lat);
          if (e == cudaSuccess) e = launch_finalize_row(*lat, n, (uint64_t)(n + 1) * B, want_q);
        }
        if (e == cudaSuccess) e = launch_pt_swap(*lat, n);
        if (e == cudaSuccess) e = launch_build_planes(*lat);
        after(aux, main);
        if (n + 1 < cycles) clear();
        for (int k = 1; k < chains; ++k) after(stream_of(k), main);
        continue;
      }
      if (overlap_apart(*lat, want_q)) {
        for (int k = 1; k < chains; ++k) after(main, stream_of(k));
        lat->stream = main;
        if (e == cudaSuccess) e = launch_overlap_bits(*lat);
        for (int k = 1; k < chains; ++k) after(stream_of(k), main);
      }
      for (int k = 0; k < chains; ++k) after(aux, stream_of(k));
      lat->stream = aux;
      if (e == cudaSuccess) e = launch_finalize_row(*lat, n, (uint64_t)(n + 1) * B, want_q);
      if (n + 1 < cycles) clear();
    }
    for (int k = 1; k < chains; ++k) after(main, stream_of(k));
    after(main, aux);
  } else {
    for (uint32_t n = 0; n < cycles; ++n) {
      for (int k = 0; k < chains; ++k) sweeps(k, n * B);
      for (int k = 1; k < chains; ++k) after(main, stream_of(k));
      lat->stream = main;
      lat->chain = lat->chains = 0;
      const int q = swap == Swap::kOnly ? 0 : want_q;
      if (e == cudaSuccess)
        e = lat->layout == IANUS_LAYOUT_I8 ? launch_measure_i8(*lat, q) : launch_measure_potts(*lat, q);
      lat->chains = chains;
      // the next cycle's sweeps read the spins only after the measurement has,
      // and the temperatures only after the swap step has written them
      auto go_on = [&]() {
        if (n + 1 < cycles)
          for (int k = 1; k < chains; ++k) after(stream_of(k), main);
      };
      if (swap == Swap::kNone) go_on();
      if (e == cudaSuccess && swap != Swap::kOnly)
        e = launch_finalize_row(*lat, n, (uint64_t)(n + 1) * B, want_q);
      if (swap != Swap::kNone) {
        if (e == cudaSuccess) e = launch_pt_swap(*lat, n);
        go_on();
      }
    }
  }
  lat->stream = main;
  lat->chain = lat->chains = 0;
  if (e == cudaSuccess)
    e = launch_advance_tick(*lat, (uint64_t)B * std::max(cycles, 1u), swap == Swap::kOnly ? 0u : cycles,
                            swap == Swap::kNone ? 0u : cycles);
  cudaError_t e2 = cudaStreamEndCapture(main, &g);
  cudaEventDestroy(ev);
  lat->stream = user;
  lat->capturing = false;
  if (e != cudaSuccess || e2 != cudaSuccess || !g) {
    if (g) cudaGraphDestroy(g);
    cudaGetLastError();
    return IANUS_ECUDA;
  }
  e = cudaGraphInstantiate(out, g, 0);
  cudaGraphDestroy(g);
  return e == cudaSuccess ? IANUS_OK : fail(lat, IANUS_ECUDA);
}

// Lattices whose passes take longer than their launches.
bool large_lattice(const Lattice& lat) { return (uint64_t)lat.S * lat.slots * lat.N >= (1u << 22); }

// The slot of `key` when its graph exists or should be captured now, null when
// the caller should launch its kernels one by one; `uses`: times that the rest
// of this call would replay it.  Capturing costs about 3 us a node, as much as
// the launches, so a call launches what it asks for first, and a graph is
// captured when an earlier call asked for it or this one still replays it three
// times; two times where the first block of a large lattice keeps the GPU busy
// meanwhile.  First calls on a new state, against capturing at once: 154 x 154,
// 253 samples x 2, 99 sweeps 2226 -> 1148 us; L=20, 73 samples, 53 sweeps with
// 26 measurements 927 -> 646; three-dimensional Potts L=78 1508 -> 472.
GraphSlot* graph_slot(Lattice* lat, uint32_t key, uint64_t uses) {
  GraphSlot& s = (*lat->graphs)[key];  // {null, 0} when new
  if (s.exec) return &s;
  const bool large = large_lattice(*lat);
  if (s.asked == lat->calls) return uses >= (large ? 2u : 3u) ? &s : nullptr;
  if (s.asked != 0 && (!large || uses < 3)) return &s;
  s.asked = lat->calls;
  return nullptr;
}

// Sweeps per launch of the resident bit-sliced sweep: long enough that the
// launch costs nothing, short enough that no launch runs for long.
constexpr uint32_t kResidentBlock = 4096;

// Runs n sweeps (no measurement inside) through cached graphs of blocks of up
// to 64 sweeps, 16 of a large lattice (whose chains have as many nodes and whose
// graph starts are hidden); runs of less than 4 launch by launch.  The call has
// `reps` such runs left.
int sweeps_graphed(Lattice* lat, int inv, uint64_t n, uint64_t reps) {
  // small bit-sliced lattices under the automatic variant: resident sweeps,
  // many per launch, the lattice in shared memory
  if (const Resident kind = resident_kind(lat, n); kind != Resident::kNone) {
    while (n > 0) {
      const uint32_t B = (uint32_t)std::min<uint64_t>(n, kResidentBlock);
      CK(launch_resident(lat, kind, inv, lat->sweeps, B));
      lat->sweeps += B;
      lat->t_dev_valid = false;
      n -= B;
    }
    return IANUS_OK;
  }
  // the persistent one-temperature sweep: all n sweeps in launches of up to
  // 2^20 sweeps, no graphs needed (falls through when it cannot run)
  if (lat->layout == IANUS_LAYOUT_BITS64 && persistent_variant(*lat)) {
    bool ran = true;
    while (n > 0 && ran) {
      const uint32_t B = (uint32_t)std::min<uint64_t>(n, 1u << 20);
      cudaError_t e = launch_sweep_persistent(*lat, inv, lat->sweeps, B, &ran);
      if (e != cudaSuccess) return fail(lat, IANUS_ECUDA);
      if (!ran) break;
      lat->sweeps += B;
      lat->t_dev_valid = false;
      n -= B;
    }
    if (n == 0) return IANUS_OK;
  }
  const uint32_t most = large_lattice(*lat) ? 16u : 64u;
  while (n > 0) {
    const uint32_t B = (uint32_t)std::min<uint64_t>(n, most);
    GraphSlot* slot = nullptr;
    if (B >= 4 && lat->use_graphs && lat->graphs) slot = graph_slot(lat, B, n / B * reps);
    if (!slot) {
      for (uint32_t s = 0; s < B; ++s) {
        int st = one_sweep(lat, inv);
        if (st) return st;
      }
      lat->t_dev_valid = false;
      n -= B;
      continue;
    }
    if (!slot->exec) {
      const int st = build_graph(lat, inv, B, 0, Swap::kNone, &slot->exec);
      if (st) return st;
    }
    if (!lat->t_dev_valid) CK(launch_set_tick(*lat, lat->sweeps, lat->ser_count, lat->steps));
    CK(cudaGraphLaunch(slot->exec, lat->stream));
    lat->sweeps += B;
    lat->t_dev_valid = true;  // the graph advanced the counter by B
    n -= B;
  }
  return IANUS_OK;
}

// Runs up to `left` cycles of B sweeps through a captured graph and returns how
// many it ran (0: the caller goes on launch by launch).  Small lattices take
// several cycles a graph.
constexpr uint32_t kCycleKey = 1u << 30, kCycleSweeps = 64, kCycleMost = 16;

int cycles_graphed(Lattice* lat, int inv, uint32_t B, uint64_t left, Swap swap, uint32_t* ran) {
  *ran = 0;
  if (!lat->use_graphs || !lat->graphs || B > kCycleSweeps) return IANUS_OK;
  if (lat->layout == IANUS_LAYOUT_BITS64 && persistent_variant(*lat)) return IANUS_OK;
  // a graph's start costs about 6 us: hidden by 16 sweeps of a large lattice,
  // by 64 of a small one (one measured sweep a graph: L=64, 58 samples 1.4 ms
  // for 44 against 1.2 ms launched one by one)
  const uint32_t most = std::min(kCycleMost, std::max(1u, (large_lattice(*lat) ? 16u : kCycleSweeps) / B));
  uint32_t n = 1;
  while (2u * n <= most && 2u * n <= left) n *= 2u;
  for (; n > 0 && n * B >= 4u; n /= 2u) {  // shorter ones: launch by launch
    const uint32_t key = kCycleKey | (uint32_t)swap << 16 | B << 8 | n;
    GraphSlot* slot = graph_slot(lat, key, left / n);
    if (!slot) continue;
    if (!slot->exec) {
      const int st = build_graph(lat, inv, B, n, swap, &slot->exec);
      if (st) return st;
    }
    if (!lat->t_dev_valid) CK(launch_set_tick(*lat, lat->sweeps, lat->ser_count, lat->steps));
    CK(cudaGraphLaunch(slot->exec, lat->stream));
    lat->sweeps += (uint64_t)B * n;
    if (swap != Swap::kOnly) lat->ser_count += n;
    if (swap != Swap::kNone) lat->steps += n;
    lat->t_dev_valid = true;  // the graph advanced the counters
    acc_fresh(lat);
    *ran = n;
    return IANUS_OK;
  }
  return IANUS_OK;
}

struct StateHeader {
  uint64_t magic;
  uint32_t version, model, dim, L, S, R, K, layout, disorder, pad;
  uint64_t seed, sweeps, steps, spins_bytes, J_bytes, sites_bytes, wheel_bytes;
  double field, occupation;
};

}  // namespace

// ---- reads of results ----

namespace {

// Page-locked memory that small results pass through on their way to the
// caller's arrays: a copy straight into pageable memory waits for the stream and
// for the driver's own staging each time, about 8 us an array, one into
// page-locked memory is queued with the others (measure() of L=8, 64 samples x
// 2: 55 -> 38 us).  Blocks belong to one call at a time; the process keeps up to
// kPinnedMost of them, and a call that finds none copies directly.  Large arrays
// are copied directly (3.5 MB: 160 us less than staged) once their pages exist:
// the copy engine spends some 500 us on each MB of new ones, so the host touches
// them first, while the GPU is still at work (11 MB of series into new arrays,
// with the 48 swap steps that filled it: 8.7 -> 2.4 ms).
constexpr size_t kPinnedBytes = 1u << 20;
constexpr int kPinnedMost = 4;
constexpr size_t kStagedMost = 512u << 10;  // bytes of an array that is staged
constexpr size_t kPage = 4096;

class PinnedBlock {
 public:
  PinnedBlock() {
    std::lock_guard<std::mutex> lock(mutex());
    if (!idle().empty()) {
      p_ = idle().back();
      idle().pop_back();
    } else if (count() < kPinnedMost) {
      if (cudaHostAlloc(&p_, kPinnedBytes, cudaHostAllocPortable) == cudaSuccess) {
        ++count();
      } else {
        cudaGetLastError();
        p_ = nullptr;
      }
    }
  }
  ~PinnedBlock() {
    if (!p_) return;
    std::lock_guard<std::mutex> lock(mutex());
    idle().push_back(p_);  // its room was reserved below
  }
  PinnedBlock(const PinnedBlock&) = delete;
  PinnedBlock& operator=(const PinnedBlock&) = delete;
  uint8_t* data() const { return (uint8_t*)p_; }

 private:
  static std::mutex& mutex() {
    static std::mutex m;
    return m;
  }
  static int& count() {
    static int n = 0;
    return n;
  }
  static std::vector<void*>& idle() {  // never destroyed: the driver may go first
    static std::vector<void*>* v = [] {
      auto* w = new std::vector<void*>();
      w->reserve(kPinnedMost);
      return w;
    }();
    return *v;
  }
  void* p_ = nullptr;
};

struct Read {
  void* dst;  // host; null: skipped
  const void* src;
  size_t bytes;
};

// Whether a host array is pageable (others are copied to directly).
bool pageable(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeUnregistered;
}

// Copies device ranges to the host and waits for them.
int read_back(Lattice* lat, const Read* reads, int n) {
  const PinnedBlock block;
  uint8_t* const pin = block.data();
  struct Part {
    void* dst;
    size_t at, bytes;
  };
  Part parts[8];
  int np = 0;
  size_t used = 0;
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < n && e == cudaSuccess; ++i) {
    const Read& r = reads[i];
    if (!r.dst || !r.bytes) continue;
    const bool paged = pageable(r.dst);
    if (pin && paged && r.bytes <= kStagedMost && used + r.bytes <= kPinnedBytes && np < 8) {
      e = cudaMemcpyAsync(pin + used, r.src, r.bytes, cudaMemcpyDeviceToHost, lat->stream);
      parts[np++] = Part{r.dst, used, r.bytes};
      used += (r.bytes + 63) & ~(size_t)63;
      continue;
    }
    if (paged && r.bytes > kStagedMost)
      for (size_t o = 0; o < r.bytes; o += kPage) ((volatile uint8_t*)r.dst)[o] = 0;
    e = cudaMemcpyAsync(r.dst, r.src, r.bytes, cudaMemcpyDeviceToHost, lat->stream);
  }
  // also after a refused copy: the ones before it write the block until they are done
  const cudaError_t waited = cudaStreamSynchronize(lat->stream);
  CK(e);
  CK(waited);
  for (int k = 0; k < np; ++k) std::memcpy(parts[k].dst, pin + parts[k].at, parts[k].bytes);
  return IANUS_OK;
}

// What a lattice's buffer holds beyond its least only makes sweeps faster, and it
// can double a plain lattice of few samples.  The lattices of a process take up
// to kRoomMost of it, 3 % of the memory, so that a program whose lattices fill
// the GPU fits as it did without; the ones made after that do without.
constexpr size_t kRoomMost = (size_t)8 << 30;
std::atomic<size_t> room_held{0};

size_t wanted_bytes(const Sizes& z) { return z.total - z.least + room_held <= kRoomMost ? z.total : z.least; }

}  // namespace

extern "C" {

size_t ianus_required_bytes(const ianus_config* cfg) {
  Sizes z;
  if (plan(cfg, z) != IANUS_OK) return 0;
  return z.least;
}

size_t ianus_preferred_bytes(const ianus_config* cfg) {
  Sizes z;
  if (plan(cfg, z) != IANUS_OK) return 0;
  return wanted_bytes(z);
}

ianus_status ianus_lattice_create(const ianus_config* cfg, ianus_lattice** out) {
  if (!out) return IANUS_EINVAL;
  *out = nullptr;
  Sizes z;
  int st = plan(cfg, z);
  if (st) return (ianus_status)st;
  Lattice* lat = new (std::nothrow) Lattice();
  if (!lat) return IANUS_ENOMEM;
  lat->cfg = *cfg;
  lat->model = z.model;
  lat->D = z.D;
  lat->L = z.L;
  lat->S = z.S;
  lat->R = z.R;
  lat->K = z.K;
  lat->slots = z.slots;
  lat->layout = z.layout;
  lat->G = z.G;
  lat->Q4 = z.Q4;
  lat->N = z.N;
  lat->mq = z.mq;
  lat->disorder = cfg->disorder;
  lat->field = z.field;
  lat->hmag = cfg->field;
  lat->rng = cfg->rng;
  lat->rows = z.rows;
  lat->cap = z.cap;
  lat->pt_cap = z.pt_cap;
  lat->pt_len = z.pt_cap;
  lat->geom.D = z.D;
  lat->geom.L = z.L;
  lat->geom.h = z.L / 2;
  lat->geom.lh = lat->geom.lL = 0;
  if ((z.L & (z.L - 1)) == 0) {  // power of two: shift-based index arithmetic
    while ((1 << lat->geom.lL) < z.L) ++lat->geom.lL;
    lat->geom.lh = lat->geom.lL - 1;
  }
  lat->geom.N = z.N;
  lat->geom.half = z.N / 2;
  lat->stream = (cudaStream_t)cfg->cuda_stream;
  lat->keys = make_keys(cfg->seed);
  if (cudaGetDevice(&lat->dev) != cudaSuccess) {
    cudaGetLastError();
    lat->dev = 0;
  }
  lat->algo = -1;
  lat->jit_algo = -1;
  lat->jit_variant = -1;
  lat->persist_timeout_ns = 2000000000ull;  // 2 s
  lat->persist_absent = -1;
  lat->jitf_algo = -1;
  lat->mut = 0;
  lat->acc_ok = false;
  lat->bytes = !cfg->device_buffer ? wanted_bytes(z) : cfg->device_buffer_bytes < z.total ? z.least : z.total;
  if (cfg->device_buffer) {
    if (cfg->device_buffer_bytes < z.least || ((uintptr_t)cfg->device_buffer & 255u)) {
      delete lat;
      return IANUS_EINVAL;
    }
    lat->base = (uint8_t*)cfg->device_buffer;
    lat->owns_buffer = false;
  } else {
    void* p = nullptr;
    cudaError_t e = cudaMalloc(&p, lat->bytes);
    if (e == cudaErrorMemoryAllocation && z.least < lat->bytes) {
      cudaGetLastError();
      lat->bytes = z.least;
      e = cudaMalloc(&p, z.least);
    }
    if (e != cudaSuccess) {
      cudaGetLastError();
      delete lat;
      return e == cudaErrorMemoryAllocation ? IANUS_ENOMEM : IANUS_ECUDA;
    }
    lat->base = (uint8_t*)p;
    lat->owns_buffer = true;
  }
  uint8_t* b = lat->base;
  lat->spins = b + z.off_spins;
  lat->J = b + z.off_J;
  lat->thr = (uint64_t*)(b + z.off_thr);
  lat->tp = (uint64_t*)(b + z.off_tp);
  lat->fthr = (uint64_t*)(b + z.off_fthr);
  lat->ftp = (uint64_t*)(b + z.off_ftp);
  lat->hs = z.field && z.layout == IANUS_LAYOUT_I8 ? (int8_t*)(b + z.off_sites) : nullptr;
  lat->occ = z.field && z.layout == IANUS_LAYOUT_I8 ? (int8_t*)(b + z.off_sites) + (size_t)z.S * z.N : nullptr;
  lat->hbits = z.field && z.layout == IANUS_LAYOUT_BITS64 ? (uint64_t*)(b + z.off_sites) : nullptr;
  lat->xbits = lat->hbits ? lat->hbits + (size_t)z.G * z.N : nullptr;
  lat->dilute = z.field && z.layout == IANUS_LAYOUT_BITS64 && cfg->disorder == IANUS_DISORDER_DAFF;
  lat->fpc = z.fpc;
  lat->wheels = z.wheel_bytes ? (uint32_t*)(b + z.off_wheels) : nullptr;
  lat->segs = z.poolable ? (Segment*)(b + z.off_segs) : nullptr;
  lat->nseg = z.poolable ? (uint32_t*)(b + z.off_nseg) : nullptr;
  lat->ptab = (uint4*)(b + z.off_ptab);
  lat->pttab = (uint64_t*)(b + z.off_pttab);
  lat->pt_sign = (int8_t*)(b + z.off_ptsign);
  lat->slot_at = (int32_t*)(b + z.off_slot);
  lat->temp_of = (int32_t*)(b + z.off_temp);
  lat->accepted = (uint64_t*)(b + z.off_acc_pt);
  lat->acc = (int64_t*)(b + z.off_acc);
  lat->out_E = (int64_t*)(b + z.off_oE);
  lat->out_M = (int64_t*)(b + z.off_oM);
  lat->out_Q = (int64_t*)(b + z.off_oQ);
  lat->ser_sweep = (uint64_t*)(b + z.off_sw);
  lat->ser_E = (int64_t*)(b + z.off_sE);
  lat->ser_M = (int64_t*)(b + z.off_sM);
  lat->ser_Q = (int64_t*)(b + z.off_sQ);
  lat->err = (uint32_t*)(b + z.off_err);
  lat->flags = (z.layout == IANUS_LAYOUT_BITS64 && !z.field && z.K == 1) ? (uint32_t*)(b + z.off_flags) : nullptr;
  lat->t_dev = (uint64_t*)(b + z.off_tdev);
  lat->mask_bytes = lat->bytes == z.total ? z.mask_bytes : 0;
  lat->masks = lat->mask_bytes ? (uint4*)(b + z.off_masks) : nullptr;
  lat->use_graphs = true;
  lat->use_resident = true;
  lat->resident_mode = 1;
  lat->graphs = new (std::nothrow) std::map<uint32_t, GraphSlot>();

  auto bail = [&](int code) {
    if (lat->owns_buffer) cudaFree(lat->base);
    if (lat->words) delete lat->words->graphs;
    delete lat->words;
    delete lat->graphs;
    delete lat;
    return (ianus_status)code;
  };
  if (z.poolable) {
    lat->segs_host = new (std::nothrow) std::vector<Segment>((size_t)z.G * kMaxSegs);
    lat->nseg_host = new (std::nothrow) std::vector<uint32_t>((size_t)z.G, 0u);
    lat->tp_host = new (std::nothrow) std::vector<uint64_t>((size_t)z.G * kPlanes * kMaxClasses, 0ull);
    if (!lat->segs_host || !lat->nseg_host || !lat->tp_host) {
      delete lat->segs_host;
      delete lat->nseg_host;
      delete lat->tp_host;
      return bail(IANUS_ENOMEM);
    }
  }
  if (cudaMemsetAsync(lat->base, 0, z.least, lat->stream) != cudaSuccess) return bail(IANUS_ECUDA);
  {
    std::vector<int32_t> perm((size_t)z.S * z.R * z.K);
    for (size_t c = 0; c < perm.size(); ++c) perm[c] = (int32_t)(c % z.K);
    if (cudaMemcpyAsync(lat->slot_at, perm.data(), perm.size() * 4, cudaMemcpyHostToDevice, lat->stream) !=
            cudaSuccess ||
        cudaMemcpyAsync(lat->temp_of, perm.data(), perm.size() * 4, cudaMemcpyHostToDevice, lat->stream) !=
            cudaSuccess)
      return bail(IANUS_ECUDA);
  }
  // couplings: the J stream (EA), +1 (ferromagnet, RFIM) or -1 (DAFF)
  const int jmode = cfg->disorder == IANUS_DISORDER_PM_J ? 0 : (cfg->disorder == IANUS_DISORDER_DAFF ? 2 : 1);
  cudaError_t e;
  if (lat->layout == IANUS_LAYOUT_I8)
    e = launch_init_i8(*lat, jmode);
  else if (lat->layout == IANUS_LAYOUT_BITS64)
    e = launch_init_bits(*lat, jmode);
  else
    e = launch_init_potts(*lat, jmode);
  if (e == cudaSuccess && lat->field)
    e = lat->layout == IANUS_LAYOUT_I8 ? launch_init_sites_i8(*lat, cfg->occupation)
                                       : launch_init_sites_bits(*lat, cfg->occupation);
  if (e == cudaSuccess && lat->wheels) e = launch_init_wheels(*lat);
  if (e != cudaSuccess || cudaStreamSynchronize(lat->stream) != cudaSuccess) return bail(IANUS_ECUDA);
  if (z.words && lat->bytes == z.total) {
    // everything but the spins, the couplings and the planes is shared
    lat->words = new (std::nothrow) Lattice(*lat);
    if (lat->words) {
      Lattice* w = lat->words;
      w->layout = IANUS_LAYOUT_BITS64;
      w->spins = b + z.off_wspins;
      w->J = b + z.off_wJ;
      w->tp = (uint64_t*)(b + z.off_wtp);
      w->masks = nullptr;
      w->mask_bytes = 0;
      w->owns_buffer = false;
      w->variant = 1;  // no run-time compiler: plain sweeps take new temperatures as they come
      w->graphs = new (std::nothrow) std::map<uint32_t, GraphSlot>();
    }
  }
  lat->room = lat->bytes - z.least;
  room_held += lat->room;
  *out = reinterpret_cast<ianus_lattice*>(lat);
  return IANUS_OK;
}

#define GET_LAT(h)                                          \
  Lattice* lat = reinterpret_cast<Lattice*>(h);             \
  if (!lat) return IANUS_EINVAL;                            \
  if (lat->sticky) return (ianus_status)lat->sticky;

// Whether a run of n sweeps of a small plain lattice is resident.
static bool resident_i8_run(Lattice& lat, uint64_t n, uint32_t measure_every) {
  return lat.use_resident && resident_i8_fits(lat) && (lat.R == 1 || measure_every == 0) && n >= 2 &&
         (lat.resident_mode != 1 || packed_i8_pays(lat, n) || resident_i8_pays(lat, measure_every));
}

static ianus_status sweep_words(Lattice* lat, int32_t algo, const double* beta, uint64_t nsweeps,
                                uint32_t measure_every);

// ianus_sweep within a call that makes `reps` more of the same.
static ianus_status sweep_run(Lattice* lat, int32_t algo, const double* beta, uint64_t nsweeps,
                              uint32_t measure_every, uint64_t reps) {
  if (lat->pool) return IANUS_EINVAL;  // a pool is driven by ianus_sweep_segments
  if (!beta || (algo != IANUS_METROPOLIS && algo != IANUS_HEATBATH)) return IANUS_EINVAL;
  if (!beta_ok(beta, lat->K)) return IANUS_EINVAL;
  if (lat->model != IANUS_EA_PM_J && algo == IANUS_METROPOLIS) return IANUS_EUNSUPPORTED;
  if (!lat->tables_ok || lat->algo != algo || !same_beta(lat, beta)) {
    int st = upload_tables(lat, algo, beta);
    if (st) return (ianus_status)st;
  }
  const int inv = algo == IANUS_HEATBATH;
  if (resident_i8_run(*lat, nsweeps, measure_every)) {
    // small plain lattice: whole configurations in shared memory, many sweeps per launch
    uint64_t left = nsweeps;
    while (left > 0) {
      const uint32_t n = (uint32_t)std::min<uint64_t>(left, 65536);
      if (lat->resident_mode == 1 && packed_i8_pays(*lat, n))
        CK(launch_packed_i8(*lat, inv, n, measure_every));
      else
        CK(launch_resident_i8(*lat, inv, n, measure_every));
      if (measure_every)  // measured sweeps t+1 in (sweeps, sweeps + n] with (t+1) % every == 0
        lat->ser_count += (lat->sweeps + n) / measure_every - lat->sweeps / measure_every;
      lat->sweeps += n;
      lat->t_dev_valid = false;
      left -= n;
    }
    return IANUS_OK;
  }
  if (lat->words && lat->use_resident && lat->resident_mode == 1 && lat->variant == 0 && words_pay(*lat, nsweeps))
    return sweep_words(lat, algo, beta, nsweeps, measure_every);
  uint64_t left = nsweeps;
  while (left > 0) {
    if (measure_every && lat->sweeps % measure_every == 0 && left >= measure_every) {
      uint32_t ran = 0;
      int st = cycles_graphed(lat, inv, measure_every, left / measure_every, Swap::kNone, &ran);
      if (st) return (ianus_status)st;
      left -= (uint64_t)ran * measure_every;
      if (ran) continue;
    }
    uint64_t chunk = left;  // sweeps up to the next measurement point
    if (measure_every) chunk = std::min<uint64_t>(chunk, measure_every - lat->sweeps % measure_every);
    int st = sweeps_graphed(lat, inv, chunk, measure_every ? reps * std::max<uint64_t>(1, left / measure_every) : reps);
    if (st) return (ianus_status)st;
    left -= chunk;
    if (measure_every && lat->sweeps % measure_every == 0) {
      st = record_row(lat);
      if (st) return (ianus_status)st;
    }
  }
  return IANUS_OK;
}

// A plain lattice's sweeps in words: the counters and the series are the
// lattice's own.
static ianus_status sweep_words(Lattice* lat, int32_t algo, const double* beta, uint64_t nsweeps,
                                uint32_t measure_every) {
  Lattice* w = lat->words;
  CK(launch_pack_words(*lat));
  w->use_graphs = lat->use_graphs;
  w->sweeps = lat->sweeps;
  w->ser_count = lat->ser_count;
  w->steps = lat->steps;
  w->t_dev_valid = false;
  w->acc_ok = false;
  w->calls += 1;
  w->sticky = 0;
  const ianus_status st = sweep_run(w, algo, beta, nsweeps, measure_every, 1);
  lat->t_dev_valid = false;
  lat->acc_ok = false;
  if (w->sticky) {  // a refused launch inside a sweep: the state is lost
    lat->sticky = w->sticky;
    return st;
  }
  // also after a capture that failed: the words hold the sweeps counted so far
  CK(launch_unpack_spins(*lat));
  lat->sweeps = w->sweeps;
  lat->ser_count = w->ser_count;
  return st;
}

ianus_status ianus_sweep(ianus_lattice* h, int32_t algo, const double* beta, uint64_t nsweeps,
                         uint32_t measure_every) {
  GET_LAT(h);
  lat->calls += 1;
  return sweep_run(lat, algo, beta, nsweeps, measure_every, 1);
}

ianus_status ianus_pt_swap(ianus_lattice* h) {
  GET_LAT(h);
  if (lat->pool) return IANUS_EINVAL;
  if (lat->K < 2 || !lat->tables_ok) return IANUS_EINVAL;
  if (lat->model != IANUS_EA_PM_J || lat->field) return IANUS_EUNSUPPORTED;
  return (ianus_status)do_pt_swap(lat);
}

ianus_status ianus_sweep_pt(ianus_lattice* h, int32_t algo, const double* beta, uint64_t nsweeps,
                            uint32_t swap_every, uint32_t measure_every) {
  GET_LAT(h);
  if (swap_every == 0 || nsweeps % swap_every != 0) return IANUS_EINVAL;
  if (lat->K < 2) return IANUS_EINVAL;
  if (lat->model != IANUS_EA_PM_J || lat->field) return IANUS_EUNSUPPORTED;
  lat->calls += 1;
  for (uint64_t n = 0; n < nsweeps; n += swap_every) {
    // cycles that end in a measurement (or none) and a swap, once the first
    // has checked the arguments and brought the tables up to date
    if (n > 0 && swap_every <= kCycleSweeps && !resident_i8_run(*lat, swap_every, measure_every) &&
        (measure_every == 0 || (measure_every == swap_every && lat->sweeps % swap_every == 0))) {
      uint32_t ran = 0;
      const int st = cycles_graphed(lat, algo == IANUS_HEATBATH, swap_every, (nsweeps - n) / swap_every,
                                    measure_every ? Swap::kMeasured : Swap::kOnly, &ran);
      if (st) return (ianus_status)st;
      if (ran) {
        n += (uint64_t)(ran - 1u) * swap_every;
        continue;
      }
    }
    ianus_status st = sweep_run(lat, algo, beta, swap_every, measure_every, (nsweeps - n) / swap_every);
    if (st) return st;
    st = ianus_pt_swap(h);
    if (st) return st;
  }
  return IANUS_OK;
}

ianus_status ianus_measure(ianus_lattice* h, int64_t* energy, int64_t* magnetisation, int64_t* overlap) {
  GET_LAT(h);
  if (overlap && lat->R < 2) return IANUS_EINVAL;
  int st = measure_into(lat, lat->out_E, lat->out_M, lat->out_Q, nullptr, overlap != nullptr);
  if (st) return (ianus_status)st;
  const size_t SKR = (size_t)lat->S * lat->K * lat->R;
  const Read reads[] = {{energy, lat->out_E, SKR * 8},
                        {magnetisation, lat->out_M, SKR * lat->mq * 8},
                        {overlap, lat->out_Q, (size_t)lat->S * lat->K * 8}};
  return (ianus_status)read_back(lat, reads, 3);
}

ianus_status ianus_read_series(ianus_lattice* h, uint64_t* sweep, int64_t* energy, int64_t* magnetisation,
                               int64_t* overlap, size_t cap_rows, size_t* n_rows, int32_t clear) {
  GET_LAT(h);
  const uint64_t first = std::max<uint64_t>(lat->ser_first, lat->ser_count > lat->cap ? lat->ser_count - lat->cap : 0);
  uint64_t n = lat->ser_count - first;
  if (n > cap_rows) n = cap_rows;
  const size_t SKR = (size_t)lat->S * lat->K * lat->R, SK = (size_t)lat->S * lat->K;
  // the rows are contiguous in the ring except where it wraps: at most two
  // copies per array
  Read reads[8];
  int nr = 0;
  for (uint64_t r = 0; r < n;) {
    const size_t pos = (size_t)((first + r) % lat->cap);
    const size_t m = (size_t)std::min<uint64_t>(n - r, lat->cap - pos);
    if (sweep) reads[nr++] = {sweep + r, lat->ser_sweep + pos, m * 8};
    if (energy) reads[nr++] = {energy + r * SKR, lat->ser_E + pos * SKR, m * SKR * 8};
    if (magnetisation)
      reads[nr++] = {magnetisation + r * SKR * lat->mq, lat->ser_M + pos * SKR * lat->mq, m * SKR * lat->mq * 8};
    if (overlap && lat->R >= 2) reads[nr++] = {overlap + r * SK, lat->ser_Q + pos * SK, m * SK * 8};
    r += m;
  }
  const int st = read_back(lat, reads, nr);
  if (st) return (ianus_status)st;
  if (n_rows) *n_rows = (size_t)n;
  if (clear) lat->ser_first = lat->ser_count;
  return IANUS_OK;
}

static ianus_status staged_get(Lattice* lat, int8_t* host, size_t bytes,
                               cudaError_t (*fn)(Lattice&, int8_t*)) {
  int8_t* d = nullptr;
  if (cudaMalloc(&d, bytes) != cudaSuccess) {
    cudaGetLastError();
    return IANUS_ENOMEM;
  }
  cudaError_t e = fn(*lat, d);
  if (e == cudaSuccess) e = cudaMemcpyAsync(host, d, bytes, cudaMemcpyDeviceToHost, lat->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(lat->stream);
  cudaFree(d);
  return e == cudaSuccess ? IANUS_OK : (ianus_status)fail(lat, IANUS_ECUDA);
}

static ianus_status staged_set(Lattice* lat, const int8_t* host, size_t bytes,
                               cudaError_t (*fn)(Lattice&, const int8_t*)) {
  int8_t* d = nullptr;
  if (cudaMalloc(&d, bytes) != cudaSuccess) {
    cudaGetLastError();
    return IANUS_ENOMEM;
  }
  cudaError_t e = cudaMemcpyAsync(d, host, bytes, cudaMemcpyHostToDevice, lat->stream);
  if (e == cudaSuccess) e = fn(*lat, d);
  if (e == cudaSuccess) e = cudaStreamSynchronize(lat->stream);
  cudaFree(d);
  return e == cudaSuccess ? IANUS_OK : (ianus_status)fail(lat, IANUS_ECUDA);
}

ianus_status ianus_get_spins_i8(ianus_lattice* h, int8_t* host) {
  GET_LAT(h);
  if (!host) return IANUS_EINVAL;
  const size_t bytes = (size_t)lat->S * lat->slots * lat->N;
  auto fn = lat->layout == IANUS_LAYOUT_I8 ? launch_get_spins_i8
            : lat->layout == IANUS_LAYOUT_BITS64 ? launch_get_spins_bits : launch_get_spins_potts;
  return staged_get(lat, host, bytes, fn);
}

ianus_status ianus_set_spins_i8(ianus_lattice* h, const int8_t* host) {
  GET_LAT(h);
  lat->mut += 1;  // the state changes other than by sweeps
  if (!host) return IANUS_EINVAL;
  const size_t bytes = (size_t)lat->S * lat->slots * lat->N;
  for (size_t i = 0; i < bytes; ++i) {
    const int v = host[i];
    if (lat->model == IANUS_EA_PM_J ? (v != 1 && v != -1) : (v < 0 || v > 3)) return IANUS_EINVAL;
  }
  auto fn = lat->layout == IANUS_LAYOUT_I8 ? launch_set_spins_i8
            : lat->layout == IANUS_LAYOUT_BITS64 ? launch_set_spins_bits : launch_set_spins_potts;
  return staged_set(lat, host, bytes, fn);
}

ianus_status ianus_get_couplings_i8(ianus_lattice* h, int8_t* host) {
  GET_LAT(h);
  if (!host) return IANUS_EINVAL;
  const size_t bytes = (size_t)lat->S * lat->D * lat->N;
  auto fn = lat->layout == IANUS_LAYOUT_I8 ? launch_get_couplings_i8
            : lat->layout == IANUS_LAYOUT_BITS64 ? launch_get_couplings_bits : launch_get_couplings_potts;
  return staged_get(lat, host, bytes, fn);
}

ianus_status ianus_set_couplings_i8(ianus_lattice* h, const int8_t* host) {
  GET_LAT(h);
  lat->mut += 1;  // the state changes other than by sweeps
  if (!host) return IANUS_EINVAL;
  const size_t bytes = (size_t)lat->S * lat->D * lat->N;
  for (size_t i = 0; i < bytes; ++i) {
    if (lat->model == IANUS_POTTS4_PERM) {  // the four 2-bit fields must be 0, 1, 2, 3 in some order
      const uint32_t c = (uint8_t)host[i];
      const uint32_t seen = (1u << (c & 3u)) | (1u << ((c >> 2) & 3u)) | (1u << ((c >> 4) & 3u)) | (1u << (c >> 6));
      if (seen != 0xFu) return IANUS_EINVAL;
    } else if (host[i] != 1 && host[i] != -1) {
      return IANUS_EINVAL;
    }
  }
  auto fn = lat->layout == IANUS_LAYOUT_I8 ? launch_set_couplings_i8
            : lat->layout == IANUS_LAYOUT_BITS64 ? launch_set_couplings_bits : launch_set_couplings_potts;
  return staged_set(lat, host, bytes, fn);
}

ianus_status ianus_get_sites_i8(ianus_lattice* h, int8_t* hsign, int8_t* occupied) {
  GET_LAT(h);
  if (lat->model != IANUS_EA_PM_J) return IANUS_EUNSUPPORTED;
  const size_t n = (size_t)lat->S * lat->N;
  if (!lat->field) {
    if (hsign) std::memset(hsign, 1, n);
    if (occupied) std::memset(occupied, 1, n);
    return IANUS_OK;
  }
  std::vector<int8_t> hs(n), occ(n, 1);
  ianus_status st;
  if (lat->layout == IANUS_LAYOUT_I8) {
    int8_t* d = nullptr;
    if (cudaMalloc(&d, 2 * n) != cudaSuccess) {
      cudaGetLastError();
      return IANUS_ENOMEM;
    }
    cudaError_t e = launch_get_sites_i8(*lat, d, d + n);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hs.data(), d, n, cudaMemcpyDeviceToHost, lat->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(occ.data(), d + n, n, cudaMemcpyDeviceToHost, lat->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(lat->stream);
    cudaFree(d);
    st = e == cudaSuccess ? IANUS_OK : (ianus_status)fail(lat, IANUS_ECUDA);
  } else {
    int8_t* d = nullptr;
    if (cudaMalloc(&d, 2 * n) != cudaSuccess) {
      cudaGetLastError();
      return IANUS_ENOMEM;
    }
    cudaError_t e = launch_get_sites_bits(*lat, d, d + n);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hs.data(), d, n, cudaMemcpyDeviceToHost, lat->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(occ.data(), d + n, n, cudaMemcpyDeviceToHost, lat->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(lat->stream);
    cudaFree(d);
    st = e == cudaSuccess ? IANUS_OK : (ianus_status)fail(lat, IANUS_ECUDA);
  }
  if (st) return st;
  if (hsign) std::memcpy(hsign, hs.data(), n);
  if (occupied) std::memcpy(occupied, occ.data(), n);
  return IANUS_OK;
}

ianus_status ianus_set_sites_i8(ianus_lattice* h, const int8_t* hsign, const int8_t* occupied) {
  GET_LAT(h);
  lat->mut += 1;  // the state changes other than by sweeps
  if (!lat->field) return IANUS_EUNSUPPORTED;
  const size_t n = (size_t)lat->S * lat->N;
  for (size_t i = 0; hsign && i < n; ++i)
    if (hsign[i] != 1 && hsign[i] != -1) return IANUS_EINVAL;
  for (size_t i = 0; occupied && i < n; ++i)
    if (occupied[i] != 0 && occupied[i] != 1) return IANUS_EINVAL;
  if (lat->layout == IANUS_LAYOUT_BITS64 && !lat->dilute) {  // the random-field model has no empty sites
    for (size_t i = 0; occupied && i < n; ++i)
      if (occupied[i] != 1) return IANUS_EUNSUPPORTED;
  }
  const bool bits = lat->layout == IANUS_LAYOUT_BITS64;
  int8_t* d = nullptr;
  if (cudaMalloc(&d, 2 * n) != cudaSuccess) {
    cudaGetLastError();
    return IANUS_ENOMEM;
  }
  cudaError_t e = bits ? launch_get_sites_bits(*lat, d, d + n) : launch_get_sites_i8(*lat, d, d + n);  // keep the rest
  if (e == cudaSuccess && hsign) e = cudaMemcpyAsync(d, hsign, n, cudaMemcpyHostToDevice, lat->stream);
  if (e == cudaSuccess && occupied) e = cudaMemcpyAsync(d + n, occupied, n, cudaMemcpyHostToDevice, lat->stream);
  if (e == cudaSuccess) e = bits ? launch_set_sites_bits(*lat, d, d + n) : launch_set_sites_i8(*lat, d, d + n);
  if (e == cudaSuccess) e = cudaStreamSynchronize(lat->stream);
  cudaFree(d);
  return e == cudaSuccess ? IANUS_OK : (ianus_status)fail(lat, IANUS_ECUDA);
}

// ---- fused serving: jobs in lanes of a pool lattice ----

static int segment_find(const Lattice* lat, int group, int lane0) {
  const uint32_t ns = (*lat->nseg_host)[group];
  for (uint32_t j = 0; j < ns; ++j)
    if ((int)(*lat->segs_host)[(size_t)group * kMaxSegs + j].lane0 == lane0) return (int)j;
  return -1;
}

static ianus_status upload_group(Lattice* lat, int group) {
  CK(cudaMemcpyAsync(lat->segs + (size_t)group * kMaxSegs, lat->segs_host->data() + (size_t)group * kMaxSegs,
                     kMaxSegs * sizeof(Segment), cudaMemcpyHostToDevice, lat->stream));
  CK(cudaMemcpyAsync(lat->nseg + group, lat->nseg_host->data() + group, 4, cudaMemcpyHostToDevice, lat->stream));
  CK(cudaMemcpyAsync(lat->tp + (size_t)group * kPlanes * kMaxClasses,
                     lat->tp_host->data() + (size_t)group * kPlanes * kMaxClasses,
                     kPlanes * kMaxClasses * sizeof(uint64_t), cudaMemcpyHostToDevice, lat->stream));
  // the host copies may change again before the copy runs: wait for it
  CK(cudaStreamSynchronize(lat->stream));
  return IANUS_OK;
}

ianus_status ianus_segment_load(ianus_lattice* h, int32_t group, int32_t lane0, int32_t n, uint64_t seed,
                                int32_t job_group, int32_t algo, double beta, uint64_t nsweeps) {
  GET_LAT(h);
  lat->mut += 1;  // the state changes other than by sweeps
  if (!lat->segs) return IANUS_EUNSUPPORTED;
  if (group < 0 || group >= lat->G || lane0 < 0 || n < 1 || lane0 + n > 64) return IANUS_EINVAL;
  if (job_group < 0 || job_group >= 4096) return IANUS_EINVAL;
  if ((algo != IANUS_METROPOLIS && algo != IANUS_HEATBATH) || !std::isfinite(beta) || beta < 0.0) return IANUS_EINVAL;
  const uint64_t mask = (n >= 64 ? ~0ull : ((1ull << n) - 1ull)) << lane0;
  uint32_t& ns = (*lat->nseg_host)[group];
  for (uint32_t j = 0; j < ns; ++j)
    if ((*lat->segs_host)[(size_t)group * kMaxSegs + j].mask & mask) return IANUS_EINVAL;  // lanes taken
  if (ns >= (uint32_t)kMaxSegs) return IANUS_EINVAL;
  if (!lat->pool) {
    lat->pool = true;
    drop_graphs(lat);
  }
  const PhiloxKeys keys = make_keys(seed);
  CK(launch_load_segment(*lat, group, (uint32_t)lane0, (uint32_t)n, (uint32_t)job_group, keys));
  // per-lane thresholds of the job's (algo, beta), as its own lattice would use
  uint64_t thr[kMaxClasses];
  class_thresholds(lat->D, algo, beta, thr);
  uint64_t* tp = lat->tp_host->data() + (size_t)group * kPlanes * kMaxClasses;
  for (int u = 0; u < kMaxClasses; ++u) {
    for (int q = 0; q < kPlanes; ++q) tp[q * kMaxClasses + u] &= ~mask;
    if (u > 2 * lat->D) continue;
    if (thr[u] >= kTwo32) {
      tp[32 * kMaxClasses + u] |= mask;
    } else {
      for (int q = 0; q < 32; ++q)
        if ((thr[u] >> (31 - q)) & 1ull) tp[q * kMaxClasses + u] |= mask;
    }
  }
  Segment sg{};
  sg.mask = mask;
  sg.t = 0;
  sg.t_end = nsweeps;
  sg.key_lo = (uint32_t)(seed & 0xffffffffu);
  sg.key_hi = (uint32_t)(seed >> 32);
  sg.lane0 = (uint32_t)lane0;
  sg.inv = algo == IANUS_HEATBATH ? 1u : 0u;
  sg.jgroup = (uint32_t)job_group;
  (*lat->segs_host)[(size_t)group * kMaxSegs + ns] = sg;
  ns += 1;
  return upload_group(lat, group);
}

ianus_status ianus_segment_release(ianus_lattice* h, int32_t group, int32_t lane0) {
  GET_LAT(h);
  lat->mut += 1;  // the state changes other than by sweeps
  if (!lat->segs || group < 0 || group >= lat->G) return IANUS_EINVAL;
  const int j = segment_find(lat, group, lane0);
  if (j < 0) return IANUS_EINVAL;
  uint32_t& ns = (*lat->nseg_host)[group];
  Segment* base = lat->segs_host->data() + (size_t)group * kMaxSegs;
  base[j] = base[ns - 1];  // keep the table compact; order is immaterial
  base[ns - 1] = Segment{};
  ns -= 1;
  return upload_group(lat, group);
}

ianus_status ianus_segment_state(ianus_lattice* h, int32_t group, int32_t lane0, uint64_t* sweeps_done,
                                 uint64_t* sweeps_requested) {
  GET_LAT(h);
  if (!lat->segs || group < 0 || group >= lat->G) return IANUS_EINVAL;
  const int j = segment_find(lat, group, lane0);
  if (j < 0) return IANUS_EINVAL;
  const Segment& sg = (*lat->segs_host)[(size_t)group * kMaxSegs + j];
  if (sweeps_done) *sweeps_done = sg.t;
  if (sweeps_requested) *sweeps_requested = sg.t_end;
  return IANUS_OK;
}

// n sweeps of a pool's segments, whose counters advance at the end.  Inside a
// capture nothing but the sweeps runs between them, so all but the first pass
// stage their tables early.
static int fused_sweeps(Lattice* lat, uint32_t n, bool captured) {
  for (uint32_t k = 0; k < n; ++k) {
    CK(launch_sweep_fused(*lat, 0, k, captured && k > 0));
    CK(launch_sweep_fused(*lat, 1, k, captured));
  }
  CK(launch_advance_segments(*lat, n));
  return IANUS_OK;
}

ianus_status ianus_sweep_segments(ianus_lattice* h, uint64_t nsweeps) {
  GET_LAT(h);
  lat->mut += 1;  // the state changes other than by sweeps
  if (!lat->segs) return IANUS_EUNSUPPORTED;
  lat->calls += 1;
  uint64_t left = nsweeps;
  const bool resident = nsweeps >= 2 && lat->use_resident && resident_fused_fits(*lat);
  while (left > 0) {
    const uint32_t B = (uint32_t)std::min<uint64_t>(left, resident ? kResidentBlock : 64);
    GraphSlot* slot = nullptr;
    if (!resident && B >= 4 && lat->use_graphs && lat->graphs) slot = graph_slot(lat, (1u << 31) | B, left / B);
    if (resident) {
      CK(launch_resident_fused(*lat, B));
    } else if (!slot) {
      const int st = fused_sweeps(lat, B, false);
      if (st) return (ianus_status)st;
    } else {
      if (!slot->exec) {
        if (!lat->cap_stream) CK(cudaStreamCreateWithFlags(&lat->cap_stream, cudaStreamNonBlocking));
        cudaStream_t user = lat->stream;
        lat->stream = lat->cap_stream;
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamBeginCapture(lat->cap_stream, cudaStreamCaptureModeThreadLocal);
        int st = IANUS_OK;
        if (e == cudaSuccess) st = fused_sweeps(lat, B, true);
        cudaError_t e2 = cudaStreamEndCapture(lat->cap_stream, &g);
        lat->stream = user;
        if (e != cudaSuccess || e2 != cudaSuccess || st != IANUS_OK || !g ||
            cudaGraphInstantiate(&slot->exec, g, 0) != cudaSuccess) {
          if (g) cudaGraphDestroy(g);
          cudaGetLastError();
          return IANUS_ECUDA;
        }
        cudaGraphDestroy(g);
      }
      CK(cudaGraphLaunch(slot->exec, lat->stream));
    }
    // the host copy follows the device counters: every live segment advances
    for (int g = 0; g < lat->G; ++g)
      for (uint32_t j = 0; j < (*lat->nseg_host)[g]; ++j) {
        Segment& sg = (*lat->segs_host)[(size_t)g * kMaxSegs + j];
        sg.t = std::min<uint64_t>(sg.t_end, sg.t + B);
      }
    left -= B;
  }
  return IANUS_OK;
}

ianus_status ianus_get_pt_state(ianus_lattice* h, int32_t* slot_at, uint64_t* accepted, uint64_t* swap_steps) {
  GET_LAT(h);
  const size_t n = (size_t)lat->S * lat->R * lat->K;
  const Read reads[] = {{slot_at, lat->slot_at, n * 4},
                        {lat->K > 1 ? accepted : nullptr, lat->accepted, (size_t)lat->S * lat->R * (lat->K - 1) * 8}};
  const int st = read_back(lat, reads, 2);
  if (st) return (ianus_status)st;
  if (swap_steps) *swap_steps = lat->steps;
  return IANUS_OK;
}

ianus_status ianus_get_sweeps(ianus_lattice* h, uint64_t* sweeps) {
  GET_LAT(h);
  if (!sweeps) return IANUS_EINVAL;
  *sweeps = lat->sweeps;
  return IANUS_OK;
}

ianus_status ianus_get_state(ianus_lattice* h, void* host_buf, size_t cap, size_t* n) {
  GET_LAT(h);
  if (lat->pool) return IANUS_EUNSUPPORTED;  // segment tables are not part of the blob
  Sizes z;
  plan(&lat->cfg, z);
  const size_t perm = (size_t)lat->S * lat->R * lat->K * 4;
  const size_t accb = (size_t)lat->S * lat->R * std::max(lat->K - 1, 1) * 8;
  const size_t need =
      sizeof(StateHeader) + 2 * perm + accb + z.J_bytes + z.spins_bytes + z.sites_bytes + z.wheel_bytes;
  if (n) *n = need;
  if (!host_buf) return IANUS_OK;
  if (cap < need) return IANUS_EINVAL;
  StateHeader hd{};
  hd.magic = kStateMagic;
  hd.version = IANUS_ABI_VERSION;
  hd.model = (uint32_t)lat->model;
  hd.dim = (uint32_t)lat->D;
  hd.L = (uint32_t)lat->L;
  hd.S = (uint32_t)lat->S;
  hd.R = (uint32_t)lat->R;
  hd.K = (uint32_t)lat->K;
  hd.layout = (uint32_t)lat->layout;
  hd.disorder = (uint32_t)lat->cfg.disorder;
  hd.seed = lat->cfg.seed;
  hd.sweeps = lat->sweeps;
  hd.steps = lat->steps;
  hd.spins_bytes = z.spins_bytes;
  hd.J_bytes = z.J_bytes;
  hd.sites_bytes = z.sites_bytes;
  hd.wheel_bytes = z.wheel_bytes;
  hd.field = lat->cfg.field;
  hd.occupation = lat->cfg.occupation;
  uint8_t* o = (uint8_t*)host_buf;
  std::memcpy(o, &hd, sizeof hd);
  o += sizeof hd;
  CK(cudaMemcpyAsync(o, lat->slot_at, perm, cudaMemcpyDeviceToHost, lat->stream));
  o += perm;
  CK(cudaMemcpyAsync(o, lat->temp_of, perm, cudaMemcpyDeviceToHost, lat->stream));
  o += perm;
  CK(cudaMemcpyAsync(o, lat->accepted, accb, cudaMemcpyDeviceToHost, lat->stream));
  o += accb;
  CK(cudaMemcpyAsync(o, lat->J, z.J_bytes, cudaMemcpyDeviceToHost, lat->stream));
  o += z.J_bytes;
  CK(cudaMemcpyAsync(o, lat->spins, z.spins_bytes, cudaMemcpyDeviceToHost, lat->stream));
  o += z.spins_bytes;
  if (z.sites_bytes) CK(cudaMemcpyAsync(o, lat->base + z.off_sites, z.sites_bytes, cudaMemcpyDeviceToHost, lat->stream));
  o += z.sites_bytes;
  if (z.wheel_bytes)
    CK(cudaMemcpyAsync(o, lat->base + z.off_wheels, z.wheel_bytes, cudaMemcpyDeviceToHost, lat->stream));
  CK(cudaStreamSynchronize(lat->stream));
  return IANUS_OK;
}

ianus_status ianus_set_state(ianus_lattice* h, const void* host_buf, size_t n) {
  Lattice* lat = reinterpret_cast<Lattice*>(h);
  if (!lat || !host_buf) return IANUS_EINVAL;
  Sizes z;
  plan(&lat->cfg, z);
  const size_t perm = (size_t)lat->S * lat->R * lat->K * 4;
  const size_t accb = (size_t)lat->S * lat->R * std::max(lat->K - 1, 1) * 8;
  const size_t need =
      sizeof(StateHeader) + 2 * perm + accb + z.J_bytes + z.spins_bytes + z.sites_bytes + z.wheel_bytes;
  if (n < need) return IANUS_ESTATE;
  StateHeader hd;
  std::memcpy(&hd, host_buf, sizeof hd);
  if (hd.magic != kStateMagic || hd.version != IANUS_ABI_VERSION || hd.model != (uint32_t)lat->model ||
      hd.dim != (uint32_t)lat->D || hd.L != (uint32_t)lat->L || hd.S != (uint32_t)lat->S ||
      hd.R != (uint32_t)lat->R || hd.K != (uint32_t)lat->K || hd.layout != (uint32_t)lat->layout ||
      hd.seed != lat->cfg.seed || hd.spins_bytes != z.spins_bytes || hd.J_bytes != z.J_bytes ||
      hd.disorder != (uint32_t)lat->cfg.disorder || hd.sites_bytes != z.sites_bytes ||
      hd.wheel_bytes != z.wheel_bytes ||
      std::memcmp(&hd.field, &lat->cfg.field, sizeof(double)) != 0)
    return IANUS_ESTATE;
  const uint8_t* in = (const uint8_t*)host_buf + sizeof hd;
  lat->sticky = 0;
  lat->mut += 1;  // the state changes other than by sweeps
  CK(cudaMemcpyAsync(lat->slot_at, in, perm, cudaMemcpyHostToDevice, lat->stream));
  in += perm;
  CK(cudaMemcpyAsync(lat->temp_of, in, perm, cudaMemcpyHostToDevice, lat->stream));
  in += perm;
  CK(cudaMemcpyAsync(lat->accepted, in, accb, cudaMemcpyHostToDevice, lat->stream));
  in += accb;
  CK(cudaMemcpyAsync(lat->J, in, z.J_bytes, cudaMemcpyHostToDevice, lat->stream));
  in += z.J_bytes;
  CK(cudaMemcpyAsync(lat->spins, in, z.spins_bytes, cudaMemcpyHostToDevice, lat->stream));
  in += z.spins_bytes;
  if (z.sites_bytes) CK(cudaMemcpyAsync(lat->base + z.off_sites, in, z.sites_bytes, cudaMemcpyHostToDevice, lat->stream));
  in += z.sites_bytes;
  if (z.wheel_bytes)
    CK(cudaMemcpyAsync(lat->base + z.off_wheels, in, z.wheel_bytes, cudaMemcpyHostToDevice, lat->stream));
  CK(cudaMemsetAsync(lat->err, 0, 4, lat->stream));
  // The tables depend on beta and the algorithm only, the per-lane planes
  // also on the restored temperature permutation: those are rebuilt in
  // place, so that the tables, the specialised kernels and the captured
  // sweep graphs stay valid.
  if (lat->tables_ok && lat->layout == IANUS_LAYOUT_BITS64)
    CK(lat->field ? launch_build_field_planes(*lat) : launch_build_planes(*lat));
  CK(cudaStreamSynchronize(lat->stream));
  lat->sweeps = hd.sweeps;
  lat->steps = hd.steps;
  lat->t_dev_valid = false;
  return IANUS_OK;
}

ianus_status ianus_synchronize(ianus_lattice* h) {
  GET_LAT(h);
  CK(cudaStreamSynchronize(lat->stream));
  uint32_t err = 0;
  CK(cudaMemcpy(&err, lat->err, 4, cudaMemcpyDeviceToHost));
  if (err & ERR_TIMEOUT) {
    lat->sticky = IANUS_ESTATE;
    return IANUS_ETIMEOUT;
  }
  if (err) {
    lat->sticky = IANUS_ESTATE;
    return IANUS_ESTATE;
  }
  return IANUS_OK;
}

ianus_status ianus_set_variant(ianus_lattice* h, int32_t variant) {
  GET_LAT(h);
  if (variant < 0 || variant > kMaxVariant) return IANUS_EINVAL;
  if (lat->variant != variant) drop_graphs(lat);
  lat->variant = variant;
  return IANUS_OK;
}

ianus_status ianus_prepare_sweep(ianus_lattice* h, int32_t algo, const double* beta, int32_t variant,
                                 int32_t* ready) {
  Lattice* lat = reinterpret_cast<Lattice*>(h);
  if (!lat || !beta || !ready) return IANUS_EINVAL;
  *ready = 0;
  if ((algo != IANUS_METROPOLIS && algo != IANUS_HEATBATH) || variant < 0 || variant > kMaxVariant) return IANUS_EINVAL;
  if (!beta_ok(beta, lat->K)) return IANUS_EINVAL;
  // only the bit-sliced +-J sweep at one temperature has specialised kernels
  if (lat->model != IANUS_EA_PM_J || lat->layout != IANUS_LAYOUT_BITS64 || lat->field || lat->pool || lat->K != 1)
    return IANUS_OK;
  const int v = specialised_variant(*lat, variant);
  if (v < 2) return IANUS_OK;
  uint64_t thr[kMaxClasses];
  class_thresholds(lat->D, algo, beta[0], thr);
  const UniformLut u = uniform_lut(lat->D, algo, thr);
  int prev = -1;
  if (cudaGetDevice(&prev) != cudaSuccess) {
    cudaGetLastError();
    prev = -1;
  }
  if (prev != lat->dev && cudaSetDevice(lat->dev) != cudaSuccess) {
    cudaGetLastError();
    return IANUS_ECUDA;
  }
  *ready = specialised_sweep_kernel(*lat, u, algo, v) ? 1 : 0;
  if (prev >= 0 && prev != lat->dev) cudaSetDevice(prev);
  cudaGetLastError();
  return IANUS_OK;
}

ianus_status ianus_set_persistent_wait(ianus_lattice* h, uint64_t timeout_ns, int32_t absent_block) {
  GET_LAT(h);
  if (timeout_ns == 0 || absent_block < -1) return IANUS_EINVAL;
  lat->persist_timeout_ns = timeout_ns;
  lat->persist_absent = absent_block;
  return IANUS_OK;
}

ianus_status ianus_set_block_words(ianus_lattice* h, uint32_t words_per_block) {
  GET_LAT(h);
  if (words_per_block > (1u << 24)) return IANUS_EINVAL;
  if (lat->block_words != words_per_block) drop_graphs(lat);
  lat->block_words = words_per_block;
  return IANUS_OK;
}

ianus_status ianus_set_graphs(ianus_lattice* h, int32_t enable) {
  GET_LAT(h);
  lat->use_graphs = enable != 0;
  return IANUS_OK;
}

ianus_status ianus_set_resident(ianus_lattice* h, int32_t enable) {
  GET_LAT(h);
  if (enable < 0 || enable > 3) return IANUS_EINVAL;
  // captured cycles hold the resident sweep that was chosen for them
  if (lat->use_resident != (enable != 0) || (enable && lat->resident_mode != enable)) drop_graphs(lat);
  lat->use_resident = enable != 0;
  if (enable) lat->resident_mode = enable;
  return IANUS_OK;
}

ianus_status ianus_destroy(ianus_lattice* h) {
  Lattice* lat = reinterpret_cast<Lattice*>(h);
  if (!lat) return IANUS_OK;
  cudaStreamSynchronize(lat->stream);
  drop_graphs(lat);
  delete lat->graphs;
  if (Lattice* w = lat->words) {
    drop_graphs(w);
    delete w->graphs;
    if (w->cap_stream) cudaStreamDestroy(w->cap_stream);
    for (cudaStream_t s : w->side_streams)
      if (s) cudaStreamDestroy(s);
    delete w;
  }
  delete lat->segs_host;
  delete lat->nseg_host;
  delete lat->tp_host;
  if (lat->cap_stream) cudaStreamDestroy(lat->cap_stream);
  for (cudaStream_t s : lat->side_streams)
    if (s) cudaStreamDestroy(s);
  room_held -= lat->room;
  if (lat->owns_buffer) cudaFree(lat->base);
  delete lat;
  return IANUS_OK;
}

const char* ianus_status_string(int32_t status) {
  switch (status) {
    case IANUS_OK: return "ok";
    case IANUS_EINVAL: return "invalid argument";
    case IANUS_ENOMEM: return "out of memory";
    case IANUS_ECUDA: return "CUDA runtime error";
    case IANUS_ETIMEOUT: return "bounded device wait expired";
    case IANUS_EUNSUPPORTED: return "unsupported configuration";
    case IANUS_ESTATE: return "lattice in error state or bad state blob";
    default: return "unknown status";
  }
}

}  // extern "C"
