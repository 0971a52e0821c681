// Test helper (host code only): the runtime of qfs_api.cu over a fake device.  The CUDA calls it makes are replaced by
// counting stand-ins, the kernel launchers by recorders, so that tests/test_host_runtime.py can check on the CPU what a
// call allocates and launches, at memory limits too.
//
//   host_runtime SCENARIO...   a scenario is "key=value,..."; prints one JSON line for each
#include <cuda_runtime.h>

#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <string>
#include <vector>

namespace fake {
constexpr int kSms = 152;
size_t limit = ~size_t(0), live = 0, peak = 0;
std::map<uintptr_t, size_t> blocks;
uintptr_t next = 1 << 20;
std::vector<std::string> launches;
int crews[4], rounds;   // of the last fused launch

cudaError_t alloc(void **p, size_t n) {
  if (live + n > limit) return cudaErrorMemoryAllocation;
  *p = reinterpret_cast<void *>(next);
  blocks[next] = n;
  next += (n + 511) & ~size_t(255);
  live += n;
  peak = live > peak ? live : peak;
  return cudaSuccess;
}
cudaError_t release(void *p) {
  auto it = blocks.find(reinterpret_cast<uintptr_t>(p));
  if (it == blocks.end()) return cudaErrorInvalidValue;
  live -= it->second;
  blocks.erase(it);
  return cudaSuccess;
}
cudaError_t properties(cudaDeviceProp *d, int) {
  *d = cudaDeviceProp{};
  d->multiProcessorCount = kSms;
  d->totalGlobalMem = size_t(284208) << 20;
  d->major = 10;
  d->minor = 3;
  return cudaSuccess;
}
// CTAs per SM: 228 KB of shared memory, 1 KB of it per CTA for the system, at most `by_registers`
int per_sm(size_t smem, int by_registers) {
  const int fit = (int)((228 << 10) / (smem + 1024));
  return fit < by_registers ? fit : by_registers;
}
void record(const char *format, ...) {
  char line[200];
  va_list a;
  va_start(a, format);
  std::vsnprintf(line, sizeof(line), format, a);
  va_end(a);
  launches.push_back(line);
}
}  // namespace fake

#include "qfs_kernels.cuh"
#include "qfs_matmul.cuh"
#include "qfs_polypow.cuh"
#include "qfs_reduced.cuh"
#include "qfs_screen.cuh"
#include "qfs_staged.cuh"
#include "qfs_theta_matrix.cuh"

namespace qfs {
#define FAKE_FORM(F)                                                                                                   \
  template <>                                                                                                          \
  cudaError_t FormLauncher<F>::fused(const FusedParams &prm, int grid, size_t smem, cudaStream_t, bool) {              \
    fake::record("fused form=%d grid=%d crew=%d smem=%zu classes=%d", F, grid, prm.crew, smem, prm.classes != nullptr); \
    for (int i = 0; i < 4; ++i) fake::crews[i] = prm.crews[i];                                                         \
    fake::rounds = prm.crew_rounds;                                                                                    \
    return cudaSuccess;                                                                                                \
  }                                                                                                                    \
  template <>                                                                                                          \
  cudaError_t FormLauncher<F>::occupancy(int *n, size_t smem, bool) {                                                  \
    *n = fake::per_sm(smem, F == 2 ? 3 : 2);                                                                           \
    return cudaSuccess;                                                                                                \
  }                                                                                                                    \
  template <>                                                                                                          \
  cudaError_t FormLauncher<F>::crews(int *n, int crew, size_t smem) {                                                  \
    *n = fake::kSms * fake::per_sm(smem, 2) / crew;                                                                    \
    return cudaSuccess;                                                                                                \
  }                                                                                                                    \
  template <>                                                                                                          \
  cudaError_t FormLauncher<F>::debug(int, const uint8_t *, int, int8_t *, uint32_t *, uint32_t *, uint32_t *,          \
                                     DebugPtrs, cudaStream_t, int) {                                                   \
    return cudaSuccess;                                                                                                \
  }
FAKE_FORM(0)
FAKE_FORM(1)
FAKE_FORM(2)

cudaError_t screen_launch(const FusedParams &, int, int64_t *, unsigned long long *, int, cudaStream_t) {
  fake::record("screen");
  return cudaSuccess;
}
cudaError_t reduced_launch(int, const FusedParams &, int, cudaStream_t) {
  fake::record("reduced");
  return cudaSuccess;
}
cudaError_t staged_occupancy(int, int *n) {
  *n = 2;
  return cudaSuccess;
}
size_t staged_survivor_bytes(int) { return 1 << 20; }
cudaError_t staged_run(const StagedPlan &, int, const uint8_t *, int8_t *, int64_t, int, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t theta_matrix_launch(int, const uint8_t *, int n, int crew, uint8_t *, uint32_t *, size_t, int *, uint32_t *,
                                cudaStream_t) {
  fake::record("theta_matrix n=%d crew=%d", n, crew);
  return cudaSuccess;
}
size_t matmul_scratch_bytes(int, int n, int m, int k) { return (size_t)(n + m) * k; }
cudaError_t matmul_mod_launch(int, int n, int m, int k, const uint8_t *A, const uint8_t *, uint8_t *C, uint8_t *, int,
                              uint32_t *, cudaStream_t) {
  fake::record("matmul n=%d m=%d k=%d a=%zu c=%zu", n, m, k, (size_t)(uintptr_t)A, (size_t)(uintptr_t)C);
  return cudaSuccess;
}
int polypow_primes(uint64_t, int) { return 5; }
int polypow_primes_at_once(int, int, int nprimes) { return nprimes; }
size_t polypow_scratch_words(int, int, int, int at_once) { return size_t(at_once) << 20; }
void polypow_plan(int, int, int, uint64_t *, uint64_t *) {}
cudaError_t polypow_launch(int, int, int, int at_once, const uint32_t *, uint32_t *, uint32_t *, cudaStream_t) {
  fake::record("poly_power at_once=%d", at_once);
  return cudaSuccess;
}
int noalloc_take_counters(uint32_t *, unsigned long long *) { return 0; }
}  // namespace qfs

#undef cudaGetDeviceProperties
#define cudaGetDeviceProperties(p, d) fake::properties(p, d)
#define cudaGetDevice(p) (*(p) = 0, cudaSuccess)
#define cudaSetDevice(d) ((void)(d), cudaSuccess)
#define cudaGetLastError() cudaSuccess
#define cudaDeviceSynchronize() cudaSuccess
#define cudaThreadExchangeStreamCaptureMode(m) ((void)(m), cudaSuccess)
#define cudaMalloc(p, n) fake::alloc(reinterpret_cast<void **>(p), n)
#define cudaFree(p) fake::release(p)
#define cudaMemset(p, v, n) ((void)(p), cudaSuccess)
#define cudaMemsetAsync(p, v, n, s) ((void)(p), cudaSuccess)
#define cudaEventCreate(e) ((void)(e), cudaSuccess)
#define cudaEventDestroy(e) ((void)(e), cudaSuccess)
#define cudaEventRecord(e, s) ((void)(e), cudaSuccess)
#define cudaEventSynchronize(e) ((void)(e), cudaSuccess)
#define cudaEventElapsedTime(ms, a, b) (*(ms) = 1.f, cudaSuccess)
#include "qfs_api.cu"

namespace {
std::map<std::string, std::string> parse(const char *s) {
  std::map<std::string, std::string> m;
  std::string t = s, k, v;
  for (size_t i = 0; i <= t.size();) {
    size_t e = t.find(',', i);
    if (e == std::string::npos) e = t.size();
    const std::string kv = t.substr(i, e - i);
    const size_t q = kv.find('=');
    m[kv.substr(0, q)] = kv.substr(q + 1);
    i = e + 1;
  }
  return m;
}
}  // namespace

int main(int argc, char **argv) {
  static uint8_t rows[35];
  static int8_t out[1];
  for (int a = 1; a < argc; ++a) {
    auto m = parse(argv[a]);
    auto num = [&](const char *k, long long d) { return m.count(k) ? std::atoll(m[k].c_str()) : d; };
    qfs_shutdown();
    fake::launches.clear();
    fake::limit = m.count("limit") ? (size_t)num("limit", 0) : ~size_t(0);
    fake::live = fake::peak = 0;
    int rc = -1;
    const std::string op = m["op"];
    if (m.count("after")) qfs_plan_prepare((int)num("after", 7), 1);   // an earlier call's workspace
    if (op == "heights") {   // groups p1, n1, p2, n2, ...
      qfs_group_t g[QFS_MAX_GROUPS];
      int n = 0;
      for (; n < QFS_MAX_GROUPS; ++n) {
        const std::string i = std::to_string(n + 1);
        if (!m.count("p" + i)) break;
        g[n] = qfs_group_t{(int)num(("p" + i).c_str(), 0), num(("n" + i).c_str(), 1), rows, out};
      }
      qfs_options_t o{};
      o.form = (int)num("form", QFS_FORM_DP4A);
      o.power = (int)num("power", QFS_POWER_CHAIN);
      o.workspace_budget = (size_t)num("budget", 0);
      o.max_ctas = (int)num("max_ctas", 0);
      rc = qfs_heights_multi_ex(n, g, 10, &o, nullptr);
    } else if (op == "joint") {   // crews of a launch over several primes: survivors n1, n2, ... of groups p1 > p2 > ...
      FusedGroup g[kMaxGroups] = {};
      unsigned long long n_list[kMaxGroups] = {};
      int n = 0;
      for (; m.count("p" + std::to_string(n + 1)); ++n) {
        g[n].p = (int)num(("p" + std::to_string(n + 1)).c_str(), 0);
        n_list[n] = (unsigned long long)num(("n" + std::to_string(n + 1)).c_str(), 0);
      }
      rc = (int)joint_items(n, g, n_list, (int)num("crew", 8), num("ctas", 304), 3);
    } else if (op == "sweep_autotune") {
      int dense = -1, ctas = -1;
      float ms = 0;
      rc = qfs_sweep_autotune((int)num("form", QFS_FORM_DP4A), (int)num("p", 7), num("n", 1), rows, &dense, &ctas, &ms);
      fake::record("best dense_min=%d ctas=%d", dense, ctas);
      qfs_sweep_tune_set((int)num("form", QFS_FORM_DP4A), (int)num("p", 7), 0, 0);
    } else if (op == "prepare") {
      rc = qfs_plan_prepare((int)num("p", 7), num("n", 0));
    } else if (op == "theta_matrix") {
      rc = qfs_theta_matrix((int)num("p", 7), num("n", 1), rows, rows, nullptr);
    } else if (op == "matmul") {   // operands at made-up addresses, which nothing reads
      rc = qfs_matmul_mod(11, (int)num("n", 1), (int)num("m", 1), (int)num("k", 1), reinterpret_cast<uint8_t *>(1 << 20),
                          rows, reinterpret_cast<uint8_t *>(1 << 20), nullptr);
    } else if (op == "poly_power") {
      static uint32_t c[4], limbs[1];
      rc = qfs_poly_power(1, c, 2, limbs, nullptr);
    }
    std::printf("{\"crews\": [%d, %d, %d, %d], \"crew_for\": [", fake::crews[0], fake::crews[1], fake::crews[2],
                fake::crews[3]);
    for (int n = 0; n <= 700; ++n) std::printf("%s%d", n ? ", " : "", crew_for(n, fake::crews, fake::rounds));
    std::printf("], \"rc\": %d, \"live\": %zu, \"peak\": %zu, \"launches\": [", rc, fake::live, fake::peak);
    for (size_t i = 0; i < fake::launches.size(); ++i) std::printf("%s\"%s\"", i ? ", " : "", fake::launches[i].c_str());
    std::printf("]}\n");
  }
  return 0;
}
