// jit.cu -- run-time specialisation of the bit-sliced sweep for one set of
// lane-uniform thresholds (see jit_sweep.cuh).  NVRTC (loaded with dlopen,
// so the library also loads where it is absent) compiles the kernel for
// sm_103a with the lattice's truth tables as immediates; the cubin is loaded
// with cudaLibraryLoadData and launched with programmatic stream
// serialisation (launch_dependent in k_msc.cu).  Kernels are
// cached per (device, dimension, algorithm, replicas, power-of-two side,
// tables).  When NVRTC is unavailable or compilation fails, jit_kernel()
// returns null and the caller keeps the precompiled per-lane-plane kernel.
// Compilation runs outside the cache's lock, so several threads may compile
// different kernels at once (ianus_prepare_sweep on worker threads); a thread
// that asks for a kernel another thread is compiling waits for that result.
#include <dlfcn.h>

#include <condition_variable>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "jit_sources.h"  // generated by build.py: kJitCommonSrc, kJitSweepSrc, kJitFieldSrc, kJitPlanesSrc,
                          // kJitSweepLtSrc
#include "lattice.h"

namespace ianus {
namespace {

typedef struct _nvrtcProgram* NvProg;
struct Nvrtc {
  int (*create)(NvProg*, const char*, const char*, int, const char* const*, const char* const*) = nullptr;
  int (*compile)(NvProg, int, const char* const*) = nullptr;
  int (*cubin_size)(NvProg, size_t*) = nullptr;
  int (*cubin)(NvProg, char*) = nullptr;
  int (*destroy)(NvProg*) = nullptr;
  bool ok = false;
};

Nvrtc load_nvrtc() {
  Nvrtc n;
  const char* names[] = {"libnvrtc.so.13", "libnvrtc.so", "/usr/local/cuda/lib64/libnvrtc.so.13"};
  void* h = nullptr;
  for (const char* nm : names)
    if ((h = dlopen(nm, RTLD_NOW | RTLD_LOCAL)) != nullptr) break;
  if (!h) return n;
  n.create = (decltype(n.create))dlsym(h, "nvrtcCreateProgram");
  n.compile = (decltype(n.compile))dlsym(h, "nvrtcCompileProgram");
  n.cubin_size = (decltype(n.cubin_size))dlsym(h, "nvrtcGetCUBINSize");
  n.cubin = (decltype(n.cubin))dlsym(h, "nvrtcGetCUBIN");
  n.destroy = (decltype(n.destroy))dlsym(h, "nvrtcDestroyProgram");
  n.ok = n.create && n.compile && n.cubin_size && n.cubin && n.destroy;
  return n;
}

Nvrtc& nvrtc() {
  static Nvrtc n = load_nvrtc();
  return n;
}

struct JitEntry {
  bool done = false;
  cudaKernel_t kern = nullptr;
};
std::mutex g_jit_mu;
std::condition_variable g_jit_cv;
std::map<std::string, JitEntry> g_jit_cache;  // entries are never erased: references stay valid

// NVRTC compile of preamble + src (which includes common.cuh) for sm_103a,
// cubin load and kernel lookup; null on any failure (no sticky error left).
cudaKernel_t compile_load(int dev, const std::string& pre, const char* src, const char* src_name, const char* name,
                          int max_dyn_smem) {
  cudaKernel_t kern = nullptr;
  Nvrtc& nv = nvrtc();
  if (nv.ok) {
    const char* hdr_src[] = {kJitCommonSrc, src};
    const char* hdr_name[] = {"common.cuh", src_name};
    NvProg prog = nullptr;
    if (nv.create(&prog, pre.c_str(), "ianus_jit.cu", 2, hdr_src, hdr_name) == 0) {
      const char* opts[] = {"--gpu-architecture=sm_103a", "-std=c++17"};
      size_t n = 0;
      if (nv.compile(prog, 2, opts) == 0 && nv.cubin_size(prog, &n) == 0 && n > 0) {
        std::vector<char> bin(n);
        cudaLibrary_t libh = nullptr;
        if (nv.cubin(prog, bin.data()) == 0 &&
            cudaLibraryLoadData(&libh, bin.data(), nullptr, nullptr, 0, nullptr, nullptr, 0) == cudaSuccess) {
          if (cudaLibraryGetKernel(&kern, libh, name) != cudaSuccess ||
              (max_dyn_smem > 0 && cudaKernelSetAttributeForDevice(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                                   max_dyn_smem, dev) != cudaSuccess))
            kern = nullptr;
        }
      }
      nv.destroy(&prog);
    }
  }
  cudaGetLastError();  // a failed compile/load leaves no sticky error; the caller falls back
  return kern;
}

// The kernel for (device, preamble): from the cache, or compiled by this
// thread (outside the lock), or awaited from the thread compiling it.
cudaKernel_t compile_cached(int dev, const std::string& pre, const char* src, const char* src_name, const char* name,
                            int max_dyn_smem) {
  const std::string key = std::to_string(dev) + "\n" + pre;
  {
    std::unique_lock<std::mutex> lock(g_jit_mu);
    auto it = g_jit_cache.find(key);
    if (it != g_jit_cache.end()) {
      JitEntry& e = it->second;
      g_jit_cv.wait(lock, [&e] { return e.done; });
      return e.kern;
    }
    g_jit_cache.emplace(key, JitEntry{});
  }
  const cudaKernel_t kern = compile_load(dev, pre, src, src_name, name, max_dyn_smem);
  {
    std::lock_guard<std::mutex> lock(g_jit_mu);
    JitEntry& e = g_jit_cache[key];
    e.kern = kern;
    e.done = true;
  }
  g_jit_cv.notify_all();
  return kern;
}

}  // namespace

cudaKernel_t jit_kernel(const Lattice& lat, const UniformLut& u, int algo, int mode, int phase_a, int min_blocks,
                        int group, int jreload, int ufirst, int block) {
  if (lat.K != 1 || (lat.R != 1 && lat.R != 2)) return nullptr;  // one temperature
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
  std::string pre;
  pre += "#define IANUS_JIT_D " + std::to_string(lat.D) + "\n";
  pre += "#define IANUS_JIT_ALGO " + std::to_string(algo) + "\n";
  pre += "#define IANUS_JIT_R " + std::to_string(lat.R) + "\n";
  pre += "#define IANUS_JIT_P2 " + std::to_string(lat.geom.lL > 0 ? 1 : 0) + "\n";
  pre += "#define IANUS_JIT_LUTS ";
  for (int q = 0; q < 32; ++q) pre += std::to_string((unsigned)u.t[q]) + (q < 31 ? "," : "\n");
  pre += "#define IANUS_JIT_ALWAYS " + std::to_string((unsigned)u.always) + "\n";
  pre += "#define IANUS_JIT_NEED " + std::to_string((unsigned)u.need) + "\n";
  pre += "#define IANUS_JIT_MODE " + std::to_string(mode) + "\n";
  pre += "#define IANUS_JIT_PHASEA " + std::to_string(phase_a) + "\n";
  pre += "#define IANUS_JIT_MINB " + std::to_string(min_blocks) + "\n";
  pre += "#define IANUS_JIT_GROUP " + std::to_string(group) + "\n";
  pre += "#define IANUS_JIT_JRELOAD " + std::to_string(jreload) + "\n";
  pre += "#define IANUS_JIT_UFIRST " + std::to_string(ufirst) + "\n";
  pre += "#define IANUS_JIT_BLOCK " + std::to_string(block) + "\n";
  pre += "#define IANUS_JIT_L " + std::to_string(lat.L) + "\n";
  pre += "#define IANUS_JIT_LH " + std::to_string(lat.geom.lh) + "\n";
  pre += "#define IANUS_JIT_LL " + std::to_string(lat.geom.lL) + "\n";
  pre += "#include \"jit_sweep.cuh\"\n";
  return compile_cached(dev, pre, kJitSweepSrc, "jit_sweep.cuh", "ianus_jit_sweep", (int)kJitSmemBytes);
}

cudaKernel_t jit_field_kernel(const Lattice& lat, int algo, int min_blocks) {
  if (!lat.flut_ok || lat.K != 1 || (lat.R != 1 && lat.R != 2)) return nullptr;  // one temperature
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
  std::string pre;
  pre += "#define IANUS_JIT_D " + std::to_string(lat.D) + "\n";
  pre += "#define IANUS_JIT_ALGO " + std::to_string(algo) + "\n";
  pre += "#define IANUS_JIT_R " + std::to_string(lat.R) + "\n";
  pre += "#define IANUS_JIT_P2 " + std::to_string(lat.geom.lL > 0 ? 1 : 0) + "\n";
  pre += "#define IANUS_JIT_MINB " + std::to_string(min_blocks) + "\n";
  pre += "#define IANUS_JIT_DILUTE " + std::to_string(lat.dilute ? 1 : 0) + "\n";
  pre += "#define IANUS_JIT_L " + std::to_string(lat.L) + "\n";
  pre += "#define IANUS_JIT_LH " + std::to_string(lat.geom.lh) + "\n";
  pre += "#define IANUS_JIT_LL " + std::to_string(lat.geom.lL) + "\n";
  for (int f = 0; f < 2; ++f)
    for (int h = 0; h < 2; ++h) {
      const std::string fh = std::to_string(f) + std::to_string(h);
      pre += "#define IANUS_JIT_LUT" + fh + " ";
      for (int q = 0; q < 32; ++q) pre += std::to_string((unsigned)lat.flut.t[f][h][q]) + (q < 31 ? "," : "\n");
      pre += "#define IANUS_JIT_ALWAYS" + fh + " " + std::to_string((unsigned)lat.flut.always[f][h]) + "\n";
      pre += "#define IANUS_JIT_NEED" + fh + " " + std::to_string((unsigned)lat.flut.need[f][h]) + "\n";
    }
  pre += "#include \"jit_field.cuh\"\n";
  return compile_cached(dev, pre, kJitFieldSrc, "jit_field.cuh", "ianus_jit_field_sweep", 0);
}

cudaKernel_t jit_planes_kernel(const Lattice& lat, int algo, int rt, bool queue, int min_blocks, size_t smem) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
  std::string pre;
  pre += "#define IANUS_JIT_PLANES 1\n";
  pre += "#define IANUS_JIT_D " + std::to_string(lat.D) + "\n";
  pre += "#define IANUS_JIT_ALGO " + std::to_string(algo) + "\n";
  pre += "#define IANUS_JIT_RT " + std::to_string(rt) + "\n";
  pre += "#define IANUS_JIT_P2 " + std::to_string(lat.geom.lL > 0 ? 1 : 0) + "\n";
  pre += "#define IANUS_JIT_Q " + std::to_string(queue ? 1 : 0) + "\n";
  pre += "#define IANUS_JIT_MINB " + std::to_string(min_blocks) + "\n";
  pre += "#define IANUS_JIT_L " + std::to_string(lat.L) + "\n";
  pre += "#define IANUS_JIT_LH " + std::to_string(lat.geom.lh) + "\n";
  pre += "#define IANUS_JIT_LL " + std::to_string(lat.geom.lL) + "\n";
  pre += "#include \"sweep_planes.cuh\"\n";
  // R is a launch parameter when rt = 0, so one compiled kernel serves every
  // replica count: allow it all the shared memory a block may have
  (void)smem;
  return compile_cached(dev, pre, kJitPlanesSrc, "sweep_planes.cuh", "ianus_jit_planes_sweep", 227 * 1024);
}

// Preamble of jit_sweep_lt.cuh but for its thresholds, RT replicas a thread.
static std::string lt_preamble(const Lattice& lat, int algo, int rt, int min_blocks, int block) {
  std::string pre;
  pre += "#define IANUS_JIT_D " + std::to_string(lat.D) + "\n";
  pre += "#define IANUS_JIT_ALGO " + std::to_string(algo) + "\n";
  pre += "#define IANUS_JIT_R " + std::to_string(rt) + "\n";
  pre += "#define IANUS_JIT_P2 " + std::to_string(lat.geom.lL > 0 ? 1 : 0) + "\n";
  pre += "#define IANUS_JIT_MINB " + std::to_string(min_blocks) + "\n";
  pre += "#define IANUS_JIT_BLOCK " + std::to_string(block) + "\n";
  pre += "#define IANUS_JIT_L " + std::to_string(lat.L) + "\n";
  pre += "#define IANUS_JIT_LH " + std::to_string(lat.geom.lh) + "\n";
  pre += "#define IANUS_JIT_LL " + std::to_string(lat.geom.lL) + "\n";
  return pre;
}

static std::string bytes_list(const uint8_t* t) {
  std::string s;
  for (int q = 0; q < 32; ++q) s += std::to_string((unsigned)t[q]) + (q < 31 ? "," : "\n");
  return s;
}

static cudaKernel_t lt_compile(const std::string& pre, bool persist) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
  const std::string all = pre + "#define IANUS_JIT_PERSIST " + (persist ? "1" : "0") + "\n" +
                          "#include \"jit_sweep_lt.cuh\"\n";
  return compile_cached(dev, all, kJitSweepLtSrc, "jit_sweep_lt.cuh",
                        persist ? "ianus_jit_sweep_ltp" : "ianus_jit_sweep_lt", 0);
}

cudaKernel_t jit_lt_kernel(const Lattice& lat, const UniformLut& u, int algo, int min_blocks, int block,
                           bool persist) {
  if (lat.K != 1 || (lat.R != 1 && lat.R != 2)) return nullptr;  // one temperature
  std::string pre = lt_preamble(lat, algo, lat.R, min_blocks, block);
  pre += "#define IANUS_JIT_LUTS " + bytes_list(u.t);
  pre += "#define IANUS_JIT_ALWAYS " + std::to_string((unsigned)u.always) + "\n";
  pre += "#define IANUS_JIT_NEED " + std::to_string((unsigned)u.need) + "\n";
  return lt_compile(pre, persist);
}

cudaKernel_t jit_lt_field_kernel(const Lattice& lat, int algo, int min_blocks, int block) {
  if (!lat.flut_ok || lat.K != 1 || (lat.R != 1 && lat.R != 2)) return nullptr;  // one temperature
  std::string pre = lt_preamble(lat, algo, lat.R, min_blocks, block);
  pre += "#define IANUS_JIT_FIELD " + std::to_string(lat.dilute ? 2 : 1) + "\n";
  for (int f = 0; f < 2; ++f)
    for (int h = 0; h < 2; ++h) {
      const std::string fh = std::to_string(f) + std::to_string(h);
      pre += "#define IANUS_JIT_LUT" + fh + " " + bytes_list(lat.flut.t[f][h]);
      pre += "#define IANUS_JIT_ALWAYS" + fh + " " + std::to_string((unsigned)lat.flut.always[f][h]) + "\n";
      pre += "#define IANUS_JIT_NEED" + fh + " " + std::to_string((unsigned)lat.flut.need[f][h]) + "\n";
    }
  return lt_compile(pre, false);
}

cudaKernel_t jit_lt_lanes_kernel(const Lattice& lat, int algo, int rt, int min_blocks, int block) {
  return lt_compile(lt_preamble(lat, algo, rt, min_blocks, block) + "#define IANUS_JIT_LANES 1\n", false);
}

}  // namespace ianus
