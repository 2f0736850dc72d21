// Host stand-ins for the device side of csrc/api.cu.  Memory is real (but untouched) address space; a kernel launch only
// checks which bytes it would read and write: every access lies in one allocation, what is read is what the right launch
// before left there, and a host buffer that a copy may still be reading is neither freed nor written.
// Sizes that depend on the kernels (groups, CTAs) are asked of the real library.
#include <dlfcn.h>
#include <sys/mman.h>

#include <atomic>
#include <chrono>
#include <functional>
#include <map>
#include <mutex>
#include <set>
#include <string>
#include <thread>
#include <vector>

#include "cuda_runtime.h"
#include "ops.h"

struct SimStream { int unused; };
struct SimEvent { long at; };
struct SimGraph { std::vector<std::function<void()>> ops; };

namespace {

typedef uintptr_t U;
struct State {
  std::map<U, size_t> dev, pinned;
  std::map<U, std::pair<U, std::string>> tag;  // [first, (end, last writer)
  struct Copy { U lo, hi; std::vector<unsigned char> at_call; };
  std::vector<Copy> pending;  // host sources of queued copies
  std::vector<std::string> bad;
  long launches = 0;
  bool values = true;  // whether what a launch reads is checked, not only where
  void* real = nullptr;
};
State* S = new State();
std::atomic<int> hold_N{0};  // the synthesis of this lattice waits
thread_local SimGraph* capture = nullptr;  // capture mode is thread-local
std::recursive_mutex mu;
#define LOCK std::lock_guard<std::recursive_mutex> lock(mu)

void fault(const std::string& m) {
  if (S->bad.size() < 20) S->bad.push_back(m);
}
bool inside(const std::map<U, size_t>& a, U p, size_t n) {
  auto it = a.upper_bound(p);
  if (it == a.begin()) return false;
  --it;
  return p + n <= it->first + it->second;
}
void check(const char* who, const void* p, size_t n) {
  if (!inside(S->dev, (U)p, n)) fault(std::string(who) + ": outside of its allocation");
}
void cut(U p) {  // no interval spans p
  auto it = S->tag.upper_bound(p);
  if (it == S->tag.begin()) return;
  --it;
  if (it->first < p && it->second.first > p) {
    S->tag[p] = it->second;
    it->second.first = p;
  }
}
void wr(const char* who, const void* p, size_t n, const std::string& t) {
  check(who, p, n);
  cut((U)p);
  cut((U)p + n);
  S->tag.erase(S->tag.lower_bound((U)p), S->tag.lower_bound((U)p + n));
  S->tag[(U)p] = {(U)p + n, t};
}
std::string rd(const char* who, const void* p, size_t n) {  // the one writer of [p, p + n)
  check(who, p, n);
  U at = (U)p;
  std::string t;
  auto it = S->tag.upper_bound(at);
  if (it != S->tag.begin()) --it;
  for (; it != S->tag.end() && at < (U)p + n; ++it) {
    if (it->second.first <= at) continue;
    if (it->first > at || (!t.empty() && t != it->second.second)) break;
    t = it->second.second;
    at = it->second.first;
  }
  if (at < (U)p + n && S->values) fault(std::string(who) + ": reads what '" + t + "' did not write all of");
  return t;
}
void want(const char* who, const std::string& got, const std::string& start) {
  if (S->values && got.compare(0, start.size(), start)) fault(std::string(who) + ": reads '" + got + "', not '" + start + "'");
}
cudaError_t launch(std::function<void()> f) {
  LOCK;
  if (capture) capture->ops.push_back(f);
  else {
    S->launches++;
    f();
  }
  return cudaSuccess;
}
std::string num(const void* p) { return std::to_string((unsigned long long)p); }
const char* c(const void* p) { return (const char*)p; }
void on_free(void* p) {
  LOCK;
  for (auto& q : S->pending)
    if (p && q.lo == (U)p) fault("a buffer is freed while a queued copy may still read it");
}

}  // namespace

// Host buffers of the library (bound inside this shared object).
void operator delete(void* p) noexcept {
  if (S) on_free(p);
  free(p);
}
void operator delete(void* p, size_t) noexcept { operator delete(p); }

const char* cudaGetErrorString(cudaError_t) { return "simulated"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
  LOCK;
  *p = mmap(nullptr, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (*p == MAP_FAILED) return cudaErrorMemoryAllocation;
  S->dev[(U)*p] = n;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  LOCK;
  auto it = S->dev.find((U)p);
  if (it == S->dev.end()) return cudaSuccess;
  wr("free", p, it->second, "");
  S->tag.erase((U)p);
  munmap(p, it->second);
  S->dev.erase(it);
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) {
  LOCK;
  *p = calloc(1, n);
  S->pinned[(U)*p] = n;
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  LOCK;
  on_free(p);
  S->pinned.erase((U)p);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) { return check("memset", p, n), memset(p, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int, size_t n, cudaStream_t) {
  return launch([=] { wr("memset", p, n, "zero"); });
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) {
  LOCK;
  cudaStreamSynchronize(nullptr);
  check("copy", k == cudaMemcpyHostToDevice ? d : s, n);
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  LOCK;
  check("copy", k == cudaMemcpyHostToDevice ? d : s, n);
  if (k == cudaMemcpyHostToDevice) {
    for (auto& q : S->pending)
      if ((U)s < q.hi && (U)s + n > q.lo) fault("a buffer is used again while a queued copy may still read it");
    S->pending.push_back({(U)s, (U)s + n, std::vector<unsigned char>((const unsigned char*)s, (const unsigned char*)s + n)});
  }
  if (n <= (1 << 20)) memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = new SimStream(), cudaSuccess; }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) { return *s = new SimStream(), cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int* least, int* greatest) { return *least = 0, *greatest = -5, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return delete s, cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) {
  LOCK;
  std::vector<State::Copy> p;
  p.swap(S->pending);
  for (auto& q : p)
    if (memcmp((const void*)q.lo, q.at_call.data(), q.hi - q.lo)) fault("a buffer changed before its copy was over");
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, int) { return capture = new SimGraph(), cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return *g = capture, capture = nullptr, cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
  return *e = new SimGraph(*g), cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
  for (auto& f : e->ops) launch(f);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return delete g, cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t g) { return delete g, cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = new SimEvent(), cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return delete e, cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { return e->at = S->launches, cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {  // a launch takes a millisecond
  return *ms = (float)(b->at - a->at), cudaSuccess;
}

namespace sigw {

template <typename R, typename... A>
static R ask(const char* name32, const char* name64, bool f64, A... a) {
  typedef R (*Fn)(A...);
  return ((Fn)dlsym(S->real, f64 ? name64 : name32))(a...);
}
#define ASK(R, fn, args, ...) \
  ask<R>("_ZN4sigw5OpsRTIfE" fn "E" args, "_ZN4sigw5OpsRTIdE" fn "E" args, sizeof(T) == 8, __VA_ARGS__)

template <typename T> LaunchShape OpsRT<T>::shape(int N) { return ASK(LaunchShape, "5shape", "i", N); }
template <typename T> int OpsRT<T>::rows_blocks(int N) { return ASK(int, "11rows_blocks", "i", N); }
template <typename T> int OpsRT<T>::variants(int N) { return ASK(int, "8variants", "i", N); }
template <typename T> int OpsRT<T>::p3_variants(int N) { return ASK(int, "11p3_variants", "i", N); }
template <typename T> bool OpsRT<T>::fused(int N, int v) { return ASK(bool, "5fused", "ii", N, v); }
template <typename T> int OpsRT<T>::last_groups(int N, int v, int n) { return ASK(int, "11last_groups", "iii", N, v, n); }

template <typename T> struct Size {
  size_t cel = 2 * sizeof(T), f, h, r;  // a packed and a standard half spectrum, a real field (one realisation)
  explicit Size(size_t N) : f(N * N * (N / 2) * cel), h(N * N * (N / 2 + 1) * cel), r(N * N * N * sizeof(T)) {}
};

// ---- synthesis and utility passes
template <typename T>
cudaError_t OpsRT<T>::rows_r2c_noise(int N, void* Y, const uint64_t* seeds, int b, const void*, cudaStream_t) {
  while (hold_N == N) std::this_thread::sleep_for(std::chrono::milliseconds(1));
  return launch([=] { check("noise", seeds, 8 * b); wr("noise", Y, b * Size<T>(N).f, "Y"); });
}
template <typename T>
cudaError_t OpsRT<T>::rows_r2c_real(int N, const void*, void* Y, int b, const void*, cudaStream_t) {
  return launch([=] { wr("rows", Y, b * Size<T>(N).f, "Y"); });
}
template <typename T>
cudaError_t OpsRT<T>::rows_r2c_map(int N, const void* R, void* Y, int b, const MapArgs* m, const double*,
                                   unsigned long long*, const void*, cudaStream_t, const void* R2, const void* R3) {
  return launch([=] {
    check("map", m, sizeof(MapArgs) * b);
    for (const void* x : {R, R2, R3})
      if (x) want("map", rd("map", x, b * Size<T>(N).r), "R");
    wr("map", Y, b * Size<T>(N).f, "Y");
  });
}
template <typename T>
cudaError_t OpsRT<T>::rows_r2c_square(int N, const void* R, void* Y, int b, const void*, cudaStream_t) {
  return launch([=] { want("square", rd("square", R, b * Size<T>(N).r), "R"); wr("square", Y, b * Size<T>(N).f, "Y"); });
}
template <typename T>
cudaError_t OpsRT<T>::rows_c2r(int N, const void* Y, void* R, int b, double, double*, const void*, cudaStream_t) {
  return launch([=] {
    std::string t = rd("c2r", Y, b * Size<T>(N).f);
    want("c2r", t, "Y");
    wr("c2r", R, b * Size<T>(N).r, "R" + t.substr(1));
  });
}
template <typename T>
cudaError_t OpsRT<T>::pass(int N, void* Y, int, int, int b, const void*, cudaStream_t) {
  return launch([=] { want("pass", rd("pass", Y, b * Size<T>(N).f), "Y"); });
}
template <typename T>
cudaError_t OpsRT<T>::unpack(int N, const void* Y, void* X, int b, const void*, long, double, int, cudaStream_t) {
  return launch([=] { want("unpack", rd("unpack", Y, b * Size<T>(N).f), "Y"); wr("unpack", X, b * Size<T>(N).h, "X"); });
}
template <typename T>
cudaError_t OpsRT<T>::pass_pack(int N, const void* X, void* Y, int b, const void*, cudaStream_t, double) {
  return launch([=] {
    std::string t;
    for (int i = 0; i < b; ++i) t = rd("pack", c(X) + i * Size<T>(N).h, Size<T>(N).h);
    want("pack", t, "X");
    wr("pack", Y, b * Size<T>(N).f, "Y" + t.substr(1));
    want("pack", rd("pack", X, Size<T>(N).h), "X");  // not written over
  });
}

// ---- hot path: T and W carry their kernel (its tables) and shell (its cell table) from pass to pass
template <typename T>
cudaError_t OpsRT<T>::p1(int N, const void* phi, void* Ta, void* Tb, const int16_t* lut, const void* tab, int nm1, int a0,
                         int nb, int batch, const void*, int variant, cudaStream_t) {
  return launch([=] {
    const Size<T> z(N);
    want("P1", rd("P1", phi, batch * z.h), "X");
    check("P1 tables", tab, (size_t)(a0 + nb) * nm1 * sizeof(T));
    const std::string id = " " + num(tab) + " " + num(lut) + " terms " + std::to_string(a0) + "+" + std::to_string(nb) +
                           (fused(N, variant) ? " fused" : "");
    wr("P1", Ta, batch * nb * z.f, "Ta" + id);
    wr("P1", Tb, batch * nb * z.f, "Tb" + id);
    want("P1", rd("P1", phi, batch * z.h), "X");
    want("P1", rd("P1", Ta, batch * nb * z.f), "Ta");
  });
}
static std::string owner(const std::string& t) {  // kernel and shell
  const size_t a = t.find(' '), b = t.find(' ', a + 1), e = t.find(' ', b + 1);
  return t.substr(a, e == std::string::npos ? e : e - a);
}
template <typename T>
cudaError_t OpsRT<T>::p2(int N, const void* Ta, const void* Tb, void* W, int n_alpha, int a0, int nb, int batch,
                         const void*, int*, long long, cudaStream_t) {
  return launch([=] {
    const Size<T> z(N);
    const std::string t = rd("P2", Ta, batch * nb * z.f), id = owner(t);
    const std::string terms = " terms " + std::to_string(a0) + "+" + std::to_string(nb);
    if (S->values && t != "Ta" + id + terms) fault("P2 reads '" + t + "' for" + terms);
    const std::string u = rd("P2", Tb, batch * nb * z.f);
    if (S->values && u != "Tb" + id + terms) fault("P2: Tb is not Ta's");
    if (a0 % 2 || (nb % 2 && a0 + nb < n_alpha)) fault("P2: a pair is split");
    const size_t np = (n_alpha + 1) / 2, row = 2 * z.f;
    for (int b = 0; b < batch; ++b)
      for (int a = a0; a < a0 + nb; a += 2)
        for (int f = 0; f < 3; ++f)
          if (f != 1 || a + 1 < n_alpha) wr("P2", c(W) + (((size_t)b * np + a / 2) * 3 + f) * row, row, "W" + id);
    rd("P2", Ta, batch * nb * z.f);  // not written over
    if (rd("P2", Tb, batch * nb * z.f) != u) fault("P2 writes over its input");
  });
}
template <typename T>
cudaError_t OpsRT<T>::p3(int N, const void* W, const void* sigma, int n_alpha, void* F, int groups, long fgs, int n_c,
                         int batch, const void*, int*, long long, int, cudaStream_t) {
  return launch([=] {
    const Size<T> z(N);
    check("P3 sigma", sigma, n_alpha * sizeof(T));
    const size_t np = (n_alpha + 1) / 2, row = 2 * z.f;
    std::string id;
    auto input = [&] {
      for (int b = 0; b < batch; ++b)
        for (int a = 0; a < n_alpha; a += 2)
          for (int f = 0; f < 3; ++f)
            if (f != 1 || a + 1 < n_alpha) {
              const std::string t = rd("P3", c(W) + (((size_t)b * np + a / 2) * 3 + f) * row, row);
              want("P3", t, "W");
              if (id.empty()) id = owner(t);
              if (owner(t) != id) fault("P3: rows of another kernel or shell");
            }
    };
    input();
    const size_t n = (size_t)6 * batch * N * N * (n_c + 1) * z.cel;
    if (groups < 1 || groups > (int)np) fault("P3: groups");
    for (int g = 0; g < groups; ++g) wr("P3", c(F) + g * fgs * z.cel, n, "F" + id);
    input();
  });
}
template <typename T>
cudaError_t OpsRT<T>::p23(int N, const void* Ta, const void* Tb, const void* sigma, int n_alpha, void* F, int groups,
                          long fgs, int n_c, int batch, const void*, int*, long long, cudaStream_t) {
  return launch([=] {
    const Size<T> z(N);
    const size_t n = (size_t)6 * batch * N * N * (n_c + 1) * z.cel;
    check("P23 sigma", sigma, n_alpha * sizeof(T));
    const std::string t = rd("P23", Ta, batch * n_alpha * z.f), id = owner(t);
    const std::string all = id + " terms 0+" + std::to_string(n_alpha) + " fused";
    if (t != "Ta" + all || rd("P23", Tb, batch * n_alpha * z.f) != "Tb" + all) fault("P23 reads '" + t + "'");
    for (int g = 0; g < groups; ++g) wr("P23", c(F) + g * fgs * z.cel, n, "F" + id);
    rd("P23", Ta, batch * n_alpha * z.f);  // not written over
    rd("P23", Tb, batch * n_alpha * z.f);
  });
}
static void n1_range(int N, int n_c, int* nk1) { *nk1 = (n_c < N / 2 ? n_c : N / 2) - (n_c < N / 2 ? -n_c : 1 - N / 2) + 1; }
template <typename T>
cudaError_t OpsRT<T>::f2(int N, const void* F, int groups, long fgs, void* F2, int n_c, int nf, const void*, cudaStream_t) {
  return launch([=] {
    const Size<T> z(N);
    int nk1;
    n1_range(N, n_c, &nk1);
    const size_t in = (size_t)6 * N * N * (n_c + 1) * z.cel, out = (size_t)6 * N * nk1 * (n_c + 1) * z.cel;
    std::vector<std::string> ids;
    for (int b = 0; b < nf; ++b)
      for (int g = 0; g < groups; ++g) {
        const std::string t = rd("F2", c(F) + g * fgs * z.cel + b * in, in);
        want("F2", t, "F ");
        if (g == 0) ids.push_back(owner(t));
        if (owner(t) != ids[b]) fault("F2: parts of different fields");
      }
    for (int b = 0; b < nf; ++b) wr("F2", c(F2) + b * out, out, "F2" + ids[b]);
    for (int b = 0; b < nf; ++b)
      for (int g = 0; g < groups; ++g) want("F2", rd("F2", c(F) + g * fgs * z.cel + b * in, in), "F ");
  });
}
template <typename T>
cudaError_t OpsRT<T>::f3(int N, const void* F2, int n_c, double* part, long pbs, long ms, int nm, int batch, const void*,
                         cudaStream_t, void* Xj) {
  const LaunchShape sh = shape(N);
  return launch([=] {
    const Size<T> z(N);
    int nk1;
    n1_range(N, n_c, &nk1);
    const size_t in = (size_t)6 * N * nk1 * (n_c + 1) * z.cel;
    const size_t blk = (size_t)((n_c + sh.tc_f3) / sh.tc_f3) * nk1;
    for (int b = 0; b < nm * batch; ++b) {
      const std::string t = rd("F3", c(F2) + b * in, in);
      want("F3", t, "F2");
      wr("F3", part + (b % batch) * pbs + (b / batch) * ms, blk * 8, "part" + owner(t));
      if (Xj) {
        want("F3 amplitudes", rd("F3", c(Xj) + 2 * b * z.h, 2 * z.h), "zero");
        wr("F3", c(Xj) + 2 * b * z.h, 2 * z.h, "X" + owner(t));
      }
    }
    for (int b = 0; b < nm * batch; ++b) want("F3", rd("F3", c(F2) + b * in, in), "F2");
  });
}
template <typename T>
cudaError_t OpsRT<T>::subvol(int N, int M, const void* R, int nf, double* out, cudaStream_t) {
  return launch([=] {
    const size_t per = (size_t)M * M * M * (N / M);
    for (int i = 0; i < nf; ++i) {
      want("subvol", rd("subvol", c(R) + i * Size<T>(N).r, Size<T>(N).r), "R ");
      wr("subvol", out + i * per, per * 8, "energies");
    }
  });
}
template struct OpsRT<float>;
template struct OpsRT<double>;

cudaError_t launch_reduce_mean(const double*, int, double*, int, double, cudaStream_t) { return launch([] {}); }
cudaError_t launch_amp(const PzArgs* pz, void* amp, long n, double, int, int prec, int b, cudaStream_t) {
  return launch([=] { check("amp", pz, sizeof(PzArgs) * b); wr("amp", amp, b * n * prec / 8, "amp"); });
}

}  // namespace sigw

// The shells' partial sums: both kernels of the shell, from the tables of its n_c.
static void fin(const double* part, long pbs, int maxblk, const std::vector<int>& shells, int N, int tc3, int batch,
                const void* out) {
  for (int b = 0; b < batch; ++b)
    for (size_t s = 0; s < shells.size(); ++s) {
      int nk1;
      sigw::n1_range(N, shells[s], &nk1);
      const size_t blk = (size_t)((shells[s] + tc3) / tc3) * nk1;
      const std::string a = rd("fin", part + b * pbs + (2 * s) * maxblk, blk * 8);
      const std::string d = rd("fin", part + b * pbs + (2 * s + 1) * maxblk, blk * 8);
      want("fin", a, "part ");
      want("fin", d, "part ");
      if (a.substr(a.rfind(' ')) != d.substr(d.rfind(' ')) || a == d) fault("fin: '" + a + "' beside '" + d + "'");
      if (strtoull(a.c_str() + 5, nullptr, 10) > strtoull(d.c_str() + 5, nullptr, 10)) fault("fin: kernels exchanged");
    }
  wr("fin", out, (size_t)batch * shells.size() * 32, "results");
}
namespace sigw {
cudaError_t launch_fin(const double* part, long pbs, int maxblk, int ns, const ShellList& l, const double*, int N, double,
                       int tc3, double* out, int batch, cudaStream_t) {
  return launch([=] { fin(part, pbs, maxblk, std::vector<int>(l.n_c, l.n_c + ns), N, tc3, batch, out); });
}
}  // namespace sigw

extern "C" {
int sigw_fft3d_noalloc() { return 3; }  // the plan-free transform is not simulated
void sim_init(const char* real) { S->real = dlopen(real, RTLD_NOW | RTLD_LOCAL); }
void sim_hold(int N) { hold_N = N; }
void sim_check_values(int on) { S->values = on; }  // off: the autotuner times launches on what is there
long sim_launches() { return S->launches; }
size_t sim_device_bytes() {
  size_t n = 0;
  for (auto& a : S->dev) n += a.second;
  return n;
}
// The faults since the last call, one a line.
const char* sim_faults() {
  static std::string all;
  all.clear();
  for (auto& m : S->bad) all += m + "\n";
  S->bad.clear();
  return all.c_str();
}
}
