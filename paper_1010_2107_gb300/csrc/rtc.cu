// rtc.cu -- user integrands compiled at run time.
//
// Step 3 of Sec. 2.1 evaluates the user's integrand inside the sampling
// kernel; the paper's users write it as device code and rebuild.  Here the
// integrand is CUDA C++ source handed to vegas_create_user: NVRTC compiles it
// together with this library's own kernel templates (k_sample, k_dump,
// k_spring with the exact dimension compiled in) to an sm_103a cubin, which
// is loaded as a CUDA library; the kernel handles then take the place of the
// built-in registry entries, so every other step (reduction, refinement,
// graphs, SPRING) is unchanged.  libnvrtc is opened on first use, so the
// library itself does not depend on it.
#include <dlfcn.h>
#include <nvrtc.h>

#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <system_error>
#include <thread>
#include <vector>

#include "kernels.h"
#include "sample_kernel.cuh"
#include "rtc_sources.inc"  // generated by the build: kRtcHeaders[] = {include name, text}

namespace gv {
namespace {

// The entry points of libnvrtc this file calls.
struct Nvrtc {
  decltype(&nvrtcCreateProgram) create = nullptr;
  decltype(&nvrtcDestroyProgram) destroy = nullptr;
  decltype(&nvrtcCompileProgram) compile = nullptr;
  decltype(&nvrtcGetProgramLogSize) log_size = nullptr;
  decltype(&nvrtcGetProgramLog) log = nullptr;
  decltype(&nvrtcGetCUBINSize) cubin_size = nullptr;
  decltype(&nvrtcGetCUBIN) cubin = nullptr;
  decltype(&nvrtcAddNameExpression) add_name = nullptr;
  decltype(&nvrtcGetLoweredName) lowered = nullptr;
  decltype(&nvrtcGetErrorString) err = nullptr;
};

// Opens libnvrtc once per process (the CUDA 13 soname first).
const Nvrtc* nvrtc(std::string* why) {
  static std::once_flag once;
  static Nvrtc api;
  static bool ok = false;
  static std::string fail;
  std::call_once(once, [] {
    std::vector<std::string> names = {"libnvrtc.so.13", "libnvrtc.so"};
    for (const char* env : {"CUDA_HOME", "CUDA_PATH"})
      if (const char* root = getenv(env)) names.push_back(std::string(root) + "/lib64/libnvrtc.so.13");
    names.push_back("/usr/local/cuda/lib64/libnvrtc.so.13");
    void* h = nullptr;
    for (const std::string& n : names)
      if ((h = dlopen(n.c_str(), RTLD_NOW | RTLD_LOCAL))) break;
    if (!h) {
      fail = "cannot load the run-time compiler libnvrtc (CUDA 13)";
      return;
    }
    bool all = true;
    auto sym = [&](auto& fp, const char* name) {
      fp = reinterpret_cast<std::remove_reference_t<decltype(fp)>>(dlsym(h, name));
      all = all && fp != nullptr;
    };
    sym(api.create, "nvrtcCreateProgram");
    sym(api.destroy, "nvrtcDestroyProgram");
    sym(api.compile, "nvrtcCompileProgram");
    sym(api.log_size, "nvrtcGetProgramLogSize");
    sym(api.log, "nvrtcGetProgramLog");
    sym(api.cubin_size, "nvrtcGetCUBINSize");
    sym(api.cubin, "nvrtcGetCUBIN");
    sym(api.add_name, "nvrtcAddNameExpression");
    sym(api.lowered, "nvrtcGetLoweredName");
    sym(api.err, "nvrtcGetErrorString");
    if (!all) {
      fail = "libnvrtc lacks an entry point this library needs";
      return;
    }
    ok = true;
  });
  if (!ok && why) *why = fail;
  return ok ? &api : nullptr;
}

// Kernels of one program: which are built and their names.
enum { K_SAMPLE = 0, K_FROZEN = 1, K_SPRING = 2, K_DUMP = 3, K_COL = 4, K_COUNT = 5 };

struct Shape {
  int prec, ybits, d;
  bool spec;
};

// The sampling kernel evaluates two points at a time per thread when it is
// the specialised FP32 kernel with d <= 8 (kPairPoints): its tiles are then
// multiples of two points.
static_assert(kPairPoints<float, 8, true> && !kPairPoints<float, 9, true> && !kPairPoints<double, 4, true> &&
                  !kPairPoints<float, 4, false>,
              "pair rule of the specialised sampling kernel");
int spec_ppt_min(const Shape& s) { return s.spec && s.prec != VG_FP64 && s.d <= 8 ? 2 : 1; }

// Kernels of a shape's program: the column-histogram kernel exists for the
// specialised FP32 form with compensated sums.
int kernel_count(const Shape& s) { return s.spec && s.prec == VG_FP32_ACCCOMP ? K_COUNT : K_COL; }

// The kernels are compiled as two or three programs at the same time, which is
// what a first use of a source waits for (two-peak Gaussian, d = 8, on 16 Arm
// cores: FP32 form 700 ms against 1410 as one program, FP64 950 against 1900).
constexpr int kPrograms = 3;
int program_of(int k) { return k == K_COL ? 2 : (k == K_FROZEN || k == K_SPRING ? 1 : 0); }
int program_count(const Shape& s) { return program_of(kernel_count(s) - 1) == 2 ? 3 : 2; }

// Template arguments (T, ACC) of the precision.
const char* type_of(int prec) { return prec == VG_FP64 ? "double" : "float"; }
int acc_of(int prec) { return prec == VG_FP64 ? 0 : (prec == VG_FP32_ACC64 ? 1 : 2); }

std::string name_expr(int k, const Shape& s) {
  const std::string T = type_of(s.prec), D = std::to_string(s.d), Y = std::to_string(s.ybits);
  const std::string sp = s.spec ? "true" : "false";
  switch (k) {
    case K_SAMPLE:
    case K_FROZEN:
      return "&gv::k_sample<" + T + ", " + D + ", gv::UserIntegrand, " + std::to_string(acc_of(s.prec)) + ", " + Y +
             ", " + sp + (k == K_SAMPLE ? ", true>" : ", false>");
    case K_COL:
      return "&gv::k_sample_col<" + D + ", gv::UserIntegrand, true>";
    case K_SPRING:
      return "&gv::k_spring<" + T + ", " + D + ", gv::UserIntegrand, " + Y + ", " + sp + ">";
    default:
      return "&gv::k_dump<" + T + ", " + D + ", gv::UserIntegrand, " + Y + ">";
  }
}

// The program: the kernel templates, the layout checks of the argument
// blocks against this side's, the user's source (its own line numbers in
// the log), and the functor that adapts vegas_user_f to the integrand
// interface (x in registers, constants in shared memory).
std::string program_text(const char* source) {
  std::string p = "#include \"sample_kernel.cuh\"\n";
  p += "static_assert(sizeof(gv::SampleArgs) == " + std::to_string(sizeof(SampleArgs)) +
       " && sizeof(gv::SpringArgs) == " + std::to_string(sizeof(SpringArgs)) +
       " && sizeof(gv::DumpArgs) == " + std::to_string(sizeof(DumpArgs)) +
       ", \"kernel argument layout differs from the host's\");\n";
  p += "#line 1 \"vegas_user_f\"\n";
  p += source;
  p += "\n#line 1 \"vegas_user_glue\"\n"
       "namespace gv {\n"
       "template <typename T, int DM> struct UserIntegrand {\n"
       "  static __device__ __forceinline__ T eval(const T (&x)[DM], int d, const T* P) {\n"
       "    return ::vegas_user_f<T>(&x[0], d, P);\n"
       "  }\n"
       "};\n"
       "}  // namespace gv\n";
  return p;
}

struct Compiled {
  std::vector<char> cubin[kPrograms];
  std::string lowered[K_COUNT];
};

// NVRTC compile of program `part` of one shape (its own entries of *out);
// VEGAS_EINVAL with the log for a source error.
int compile_part(const char* source, const Shape& s, int part, Compiled* out, std::string* why) {
  const Nvrtc* api = nvrtc(why);
  if (!api) return VEGAS_ECUDA;
  const int nh = (int)(sizeof kRtcHeaders / sizeof kRtcHeaders[0]);
  std::vector<const char*> names(nh), texts(nh);
  for (int i = 0; i < nh; ++i) {
    names[i] = kRtcHeaders[i][0];
    texts[i] = kRtcHeaders[i][1];
  }
  const std::string text = program_text(source);
  nvrtcProgram prog = nullptr;
  nvrtcResult r = api->create(&prog, text.c_str(), "vegas_user.cu", nh, texts.data(), names.data());
  if (r != NVRTC_SUCCESS) {
    *why = std::string("nvrtcCreateProgram: ") + api->err(r);
    return VEGAS_ECUDA;
  }
  std::unique_ptr<nvrtcProgram, void (*)(nvrtcProgram*)> guard(&prog, [](nvrtcProgram* p) {
    if (*p) nvrtc(nullptr)->destroy(p);
  });
  std::string exprs[K_COUNT];
  for (int k = 0; k < kernel_count(s); ++k) {
    if (program_of(k) != part) continue;
    exprs[k] = name_expr(k, s);
    if ((r = api->add_name(prog, exprs[k].c_str())) != NVRTC_SUCCESS) {
      *why = std::string("nvrtcAddNameExpression: ") + api->err(r);
      return VEGAS_ECUDA;
    }
  }
  // -default-device: the generic lambdas inside the kernels are device code
  const char* opts[] = {"-arch=sm_103a", "-std=c++17", "-lineinfo", "-default-device"};
  r = api->compile(prog, (int)(sizeof opts / sizeof opts[0]), opts);
  if (r != NVRTC_SUCCESS) {
    size_t n = 0;
    std::string log;
    if (api->log_size(prog, &n) == NVRTC_SUCCESS && n > 1) {
      log.resize(n);
      api->log(prog, &log[0]);
      log.resize(n - 1);
    }
    *why = "user integrand does not compile (" + std::string(api->err(r)) + "):\n" + log;
    return r == NVRTC_ERROR_COMPILATION ? VEGAS_EINVAL : VEGAS_ECUDA;
  }
  size_t n = 0;
  if ((r = api->cubin_size(prog, &n)) != NVRTC_SUCCESS || n == 0) {
    *why = "nvrtcGetCUBINSize failed";
    return VEGAS_ECUDA;
  }
  out->cubin[part].resize(n);
  if ((r = api->cubin(prog, out->cubin[part].data())) != NVRTC_SUCCESS) {
    *why = std::string("nvrtcGetCUBIN: ") + api->err(r);
    return VEGAS_ECUDA;
  }
  for (int k = 0; k < kernel_count(s); ++k) {
    if (program_of(k) != part) continue;
    const char* low = nullptr;
    if ((r = api->lowered(prog, exprs[k].c_str(), &low)) != NVRTC_SUCCESS || !low) {
      *why = "nvrtcGetLoweredName failed for " + exprs[k];
      return VEGAS_ECUDA;
    }
    out->lowered[k] = low;
  }
  return VEGAS_OK;
}

// All programs of one shape; the first part that fails gives status and reason.
int compile(const char* source, const Shape& s, Compiled* out, std::string* why) {
  int st[kPrograms] = {VEGAS_OK, VEGAS_OK, VEGAS_OK};
  std::string reason[kPrograms];
  auto part = [&](int i) {
    try {
      st[i] = compile_part(source, s, i, out, &reason[i]);
    } catch (...) {  // (out of memory: nothing may leave a thread, or this library)
      st[i] = VEGAS_ENOMEM;
    }
  };
  std::thread others[kPrograms - 1];
  const int n = program_count(s);
  for (int i = 1; i < n; ++i) {
    try {
      others[i - 1] = std::thread(part, i);
    } catch (const std::system_error&) {  // no thread to be had: one after another
      part(i);
    }
  }
  part(0);
  for (std::thread& t : others)
    if (t.joinable()) t.join();
  for (int i = 0; i < n; ++i)
    if (st[i] != VEGAS_OK) {
      *why = reason[i];
      return st[i];
    }
  return VEGAS_OK;
}

// Shared memory of the column-histogram kernel: its layout depends on the
// compile-time bound, here the dimension itself.
template <int D>
size_t col_smem_upto(int d, int N, int nwarps) {
  if constexpr (D > kMaxDim) {
    return 0;
  } else {
    return d == D ? ColSmem<D, true>::total(d, N, nwarps) : col_smem_upto<D + 1>(d, N, nwarps);
  }
}
size_t col_smem_user(int d, int N, int nwarps) { return col_smem_upto<1>(d, N, nwarps); }

std::string cache_key(const char* source, const Shape& s) {
  return std::to_string(s.prec) + "," + std::to_string(s.ybits) + "," + std::to_string(s.d) + "," +
         (s.spec ? "1" : "0") + "\n" + source;
}

// Compiled programs and loaded modules, for the life of the process (a
// module's kernels may sit in captured graphs of any live context).
std::mutex g_mu;
std::map<std::string, std::shared_ptr<Compiled>> g_compiled;
std::map<std::string, KernelEntry> g_loaded;

int compiled_for(const char* source, const Shape& s, std::shared_ptr<Compiled>* out, std::string* why) {
  const std::string key = cache_key(source, s);
  {
    std::lock_guard<std::mutex> lk(g_mu);
    auto it = g_compiled.find(key);
    if (it != g_compiled.end()) {
      *out = it->second;
      return VEGAS_OK;
    }
  }
  auto c = std::make_shared<Compiled>();
  const int st = compile(source, s, c.get(), why);  // outside the lock: seconds
  if (st != VEGAS_OK) return st;
  std::lock_guard<std::mutex> lk(g_mu);
  *out = g_compiled.emplace(key, c).first->second;
  return VEGAS_OK;
}

int check_shape(int prec, int ybits, int d, std::string* why) {
  if (prec < VG_FP64 || prec > VG_FP32_ACCCOMP) {
    *why = "unknown precision " + std::to_string(prec);
    return VEGAS_EINVAL;
  }
  if (ybits != 24 && ybits != 53) {
    *why = "ybits must be 24 or 53";
    return VEGAS_EINVAL;
  }
  if (d < 1 || d > kMaxDim) {
    *why = "ndim " + std::to_string(d) + " outside 1.." + std::to_string(kMaxDim);
    return VEGAS_EINVAL;
  }
  return VEGAS_OK;
}

}  // namespace

int rtc_user_entry(const char* source, int prec, int ybits, int d, bool spec, KernelEntry* out, std::string* why) {
  int st = check_shape(prec, ybits, d, why);
  if (st != VEGAS_OK) return st;
  // the specialised kernels exist for 24-bit words and the FP64 or
  // compensated FP32 sums (as for the built-in integrands)
  const Shape s{prec, ybits, d, spec && ybits == 24 && acc_of(prec) != 1};
  const std::string key = cache_key(source, s);
  {
    std::lock_guard<std::mutex> lk(g_mu);
    auto it = g_loaded.find(key);
    if (it != g_loaded.end()) {
      *out = it->second;
      return VEGAS_OK;
    }
  }
  std::shared_ptr<Compiled> c;
  if ((st = compiled_for(source, s, &c, why)) != VEGAS_OK) return st;
  cudaLibrary_t lib[kPrograms] = {};
  auto unload = [&]() {
    for (cudaLibrary_t l : lib)
      if (l) cudaLibraryUnload(l);
  };
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < program_count(s) && e == cudaSuccess; ++i)
    e = cudaLibraryLoadData(&lib[i], c->cubin[i].data(), nullptr, nullptr, 0, nullptr, nullptr, 0);
  if (e != cudaSuccess) {
    unload();
    *why = std::string("cudaLibraryLoadData: ") + cudaGetErrorString(e);
    return VEGAS_ECUDA;
  }
  cudaKernel_t k[K_COUNT] = {};
  for (int i = 0; i < kernel_count(s) && e == cudaSuccess; ++i)
    e = cudaLibraryGetKernel(&k[i], lib[program_of(i)], c->lowered[i].c_str());
  if (e != cudaSuccess) {
    unload();
    *why = std::string("cudaLibraryGetKernel: ") + cudaGetErrorString(e);
    return VEGAS_ECUDA;
  }
  KernelEntry ke{};
  ke.sample = (const void*)k[K_SAMPLE];
  ke.frozen = (const void*)k[K_FROZEN];
  ke.sample_spec = s.spec ? ke.sample : nullptr;
  ke.frozen_spec = s.spec ? ke.frozen : nullptr;
  ke.spring = (const void*)k[K_SPRING];
  ke.spring_spec = s.spec ? ke.spring : nullptr;
  ke.dump = (const void*)k[K_DUMP];
  ke.sample_col_exact = (const void*)k[K_COL];
  ke.smem_col = &col_smem_user;
  ke.smem = prec == VG_FP64 ? &sample_smem_bytes<double, 0>
                            : (prec == VG_FP32_ACC64 ? &sample_smem_bytes<float, 1> : &sample_smem_bytes<float, 2>);
  ke.smem_nobins = prec == VG_FP64 ? &sample_smem_nobins<double, 0>
                                   : (prec == VG_FP32_ACC64 ? &sample_smem_nobins<float, 1>
                                                            : &sample_smem_nobins<float, 2>);
  ke.dm = d;
  ke.max_threads = s.spec ? kSampleMaxThreads<true> : kSampleMaxThreads<false>;
  ke.spec_ppt_min = spec_ppt_min(s);
  ke.grad = ke.grad_spec = nullptr;
  ke.grad_nt = 0;
  ke.grad_smem = nullptr;
  std::lock_guard<std::mutex> lk(g_mu);
  auto ins = g_loaded.emplace(key, ke);
  if (!ins.second) unload();  // another thread loaded it first
  *out = ins.first->second;
  return VEGAS_OK;
}

int rtc_user_compile(const char* source, int prec, int ybits, int d, bool spec, std::string* why) {
  int st = check_shape(prec, ybits, d, why);
  if (st != VEGAS_OK) return st;
  const Shape s{prec, ybits, d, spec && ybits == 24 && acc_of(prec) != 1};
  std::shared_ptr<Compiled> c;
  return compiled_for(source, s, &c, why);
}

}  // namespace gv
