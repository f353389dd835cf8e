// Host-only run of the lockstep engine with a fake CUDA runtime: device memory is
// host memory and launches are only counted. Compiled and read by
// tests/test_growth_cpu.py.
//   growth   the k-th allocation after the server's creation fails; one line per k:
//            what the failed step left behind and how the retry ended
//   count    the launches that ascg_server_info reports, and those made, for a server
//            with one system of each size
//   memory   the most device bytes held while systems run, beside what they need
//   tune     the exponent passes and tensor-core Grams that the autotuner makes, by rows
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <iterator>
#include <map>
#include <string>
#include <vector>

namespace fake {
int count = 0, fail_at = -1;
std::map<void*, size_t> live;
size_t held = 0, peak = 0;
cudaError_t alloc(void** p, size_t n) {
  if (++count == fail_at) {
    *p = nullptr;
    return cudaErrorMemoryAllocation;
  }
  *p = std::calloc(1, n ? n : 1);
  live[*p] = n;
  held += n;
  peak = held > peak ? held : peak;
  return cudaSuccess;
}
cudaError_t release(void* p) {
  if (p) held -= live[p];
  live.erase(p);
  std::free(p);
  return cudaSuccess;
}
cudaError_t host(void** p, size_t n) {
  *p = std::calloc(1, n ? n : 1);
  return cudaSuccess;
}
cudaError_t ok() { return cudaSuccess; }
cudaError_t copy(void* d, const void* s, size_t n) {
  if (!d || !s) return cudaErrorInvalidValue;
  std::memcpy(d, s, n);
  return cudaSuccess;
}
}  // namespace fake

#define cudaMalloc(p, n) fake::alloc((void**)(p), n)
#define cudaFree(p) fake::release((void*)(p))
#define cudaMallocHost(p, n) fake::host((void**)(p), n)
#define cudaFreeHost(p) (std::free((void*)(p)), cudaSuccess)
#define cudaMemcpyAsync(d, s, n, k, st) fake::copy(d, s, n)
#define cudaMemsetAsync(p, v, n, st) (std::memset(p, v, n), cudaSuccess)
#define cudaMemset2DAsync(...) fake::ok()
#define cudaStreamSynchronize(s) fake::ok()
#define cudaStreamCreateWithPriority(p, f, q) (*(p) = nullptr, cudaSuccess)
#define cudaStreamDestroy(s) fake::ok()
#define cudaStreamWaitEvent(...) fake::ok()
#define cudaStreamBeginCapture(s, m) cudaErrorNotSupported
#define cudaEventCreateWithFlags(p, f) (*(p) = nullptr, cudaSuccess)
#define cudaEventCreate(p) (*(p) = nullptr, fake::ok())
#define cudaEventElapsedTime(p, a, b) (*(p) = 1.0f, fake::ok())
#define cudaEventRecord(...) fake::ok()
#define cudaEventQuery(e) fake::ok()
#define cudaEventSynchronize(e) fake::ok()
#define cudaEventDestroy(e) fake::ok()
#define cudaGetDevice(p) (*(p) = 0, cudaSuccess)
#define cudaGetLastError() fake::ok()
#define cudaDeviceGetStreamPriorityRange(a, b) (*(a) = *(b) = 0, cudaSuccess)
#define cudaGraphExecDestroy(g) fake::ok()

#define private public
#include "lockstep.cu"
#undef private

namespace ascg {
std::string last;
void set_last_error(const std::string& m) { last = m; }
ascg_status check_options(const ascg_options&) { return ASCG_OK; }
ascg_status op_split_desc(ascg_op op, SysDesc* d, int* device, double* row_len) {
  std::memset(d, 0, sizeof(*d));
  d->n = (int64_t)(uintptr_t)op;  // the handle is the row count
  *device = 0;
  *row_len = 4.0;
  return ASCG_OK;
}
int gram_grid() { return 152; }
bool gram_tc_applies(int w) { return w >= kGramTcMinW && w <= kMaxW; }
bool gram_tc_aligned(const double*, int64_t) { return true; }
// every table a launch is given has to be there
int missing = 0;
int64_t calls = 0, exponents = 0, grams = 0;
void want(const void* p) { missing += p == nullptr; }
cudaError_t launch_mpk_items(const SysDesc* a, const RowItem* b, int, const int* c, int, bool, int*, cudaStream_t) {
  ++calls;
  want(a), want(b), want(c);
  return cudaSuccess;
}
cudaError_t launch_mpk_items_both(const SysDesc* a, const RowItem* b, int, const int* c, int, cudaStream_t) {
  ++calls;
  want(a), want(b), want(c);
  return cudaSuccess;
}
cudaError_t launch_tc_items_exponents(int, const double*, int64_t, const GramPiece* a, int n, const int*, int*,
                                      cudaStream_t) {
  exponents += n > 0;
  calls += n > 0;
  want(a);
  return cudaSuccess;
}
cudaError_t launch_gram_items(int, const SysDesc*, const GramItem* a, int, const int*, double* b, int, bool,
                              cudaStream_t) {
  ++calls;
  want(a), want(b);
  return cudaSuccess;
}
cudaError_t launch_gram_items_finalize(int, const double* a, const int*, const int*, const int*, int, double*, int64_t,
                                       bool, cudaStream_t) {
  ++calls;
  want(a);
  return cudaSuccess;
}
cudaError_t launch_gram_tc_items(int, const double*, int64_t, int64_t, const GramPiece* a, int, const int*, const int*,
                                 double* b, unsigned long long* c, unsigned* d, cudaStream_t) {
  ++grams;
  ++calls;
  want(a), want(b), want(c), want(d);
  return cudaSuccess;
}
// a block takes one step; a system converges at its sixth
cudaError_t launch_block_ctrl_batch(const double*, int64_t, const double*, const double*, const double*, BlockState* st,
                                    int count, int, int, double*, int64_t, double*, int, double*, int, double*,
                                    unsigned*, cudaStream_t) {
  ++calls;
  for (int q = 0; q < count; ++q) {
    st[q].s_k = st[q].active ? 1 : 0;
    st[q].converged = st[q].m + 1 >= 6;
  }
  return cudaSuccess;
}
cudaError_t launch_recover_items(int, const SysDesc*, const RowItem* a, int, const int*, const double*, int64_t,
                                 cudaStream_t) {
  ++calls;
  want(a);
  return cudaSuccess;
}
cudaError_t launch_residual_items(const SysDesc*, const RowItem* a, int, const int*, int, cudaStream_t) {
  ++calls;
  want(a);
  return cudaSuccess;
}
// ||b||^2 = ||r||^2 = 1: every system needs blocks
cudaError_t launch_seg_sumsq(const SysDesc*, const int* list, int n, int, double* out, cudaStream_t) {
  ++calls;
  for (int i = 0; i < n; ++i) out[list[i]] = 1.0;
  return cudaSuccess;
}
cudaError_t launch_fill_uniform(double*, int64_t, uint64_t, cudaStream_t) { return cudaSuccess; }
}  // namespace ascg

int count_launches() {
  for (int64_t n : {700, 3000, 250000, 1100000}) {
    ascg_options o{};
    o.method = ASCG_ADAPTIVE;
    o.s_max = o.s0 = o.f = 8;
    o.max_iters = 100;
    ascg_server srv = nullptr;
    if (ascg_server_create(&o, (int64_t)1 << 30, 4, nullptr, &srv) != ASCG_OK) return 2;
    ascg::calls = 0;
    ascg_completion c[8];
    int nd = 0, na = 1, np = 0;
    double b = 0, x = 0;
    if (ascg_server_submit(srv, (ascg_op)(uintptr_t)n, &b, &x, 1e-8, 1) != ASCG_OK) return 3;
    while (na + np > 0)
      if (ascg_server_step(srv, c, 8, &nd, &na, &np) != ASCG_OK) return 4;
    ascg_server_stats st;
    ascg_server_info(srv, &st);
    std::printf("n %lld reported %lld made %lld\n", (long long)n, (long long)st.launches, (long long)ascg::calls);
    ascg_server_destroy(srv);
  }
  return 0;
}

// Rounds of requests on one server, each drained before the next comes.
int memory() {
  const std::vector<std::vector<int64_t>> rounds = {
      std::vector<int64_t>(16, 1000), {64000, 65000, 30000}, {200000, 120000}, {600000}, std::vector<int64_t>(16, 5000)};
  for (int s : {2, 8, 16}) {
    ascg_options o{};
    o.method = ASCG_ADAPTIVE;
    o.s_max = o.s0 = o.f = s;
    o.max_iters = 100;
    ascg_server srv = nullptr;
    fake::peak = fake::held;
    const size_t before = fake::held;
    if (ascg_server_create(&o, (int64_t)1 << 30, 16, nullptr, &srv) != ASCG_OK) return 2;
    int64_t git[3] = {0, 0, 0}, tit[3] = {0, 0, 0}, units[3] = {0, 0, 0};
    double b = 0, x = 0;
    for (const auto& r : rounds) {
      for (int64_t n : r)
        if (ascg_server_submit(srv, (ascg_op)(uintptr_t)n, &b, &x, 1e-8, 1) != ASCG_OK) return 3;
      ascg_completion c[32];
      int nd = 0, na = 1, np = 0;
      while (na + np > 0) {
        if (ascg_server_step(srv, c, 32, &nd, &na, &np) != ASCG_OK) return 4;
        for (int g = 0; g < 3; ++g) {
          const ascg::Lockstep& e = srv->group[g].eng;
          git[g] = std::max(git[g], (int64_t)e.gitems_.size());
          tit[g] = std::max(tit[g], (int64_t)e.titems_.size());
          units[g] = std::max(units[g], (int64_t)e.ritems_.size());
        }
      }
    }
    std::printf("s %d arena %zu peak %zu gitems %lld titems %lld units %lld split %lld\n", s, srv->arena.bytes_total(),
                fake::peak - before, (long long)(git[0] + git[1] + git[2]), (long long)(tit[0] + tit[1] + tit[2]),
                (long long)(units[0] + units[1] + units[2]),
                (long long)(std::min<int64_t>(tit[0], 256) + std::min<int64_t>(tit[1], 256) + std::min<int64_t>(tit[2], 256)));
    ascg_server_destroy(srv);
  }
  return 0;
}

int tune() {
  int64_t rows = 0;
  double table[3 * 16];
  int nrow = 0;
  if (ascg_tune_gram_schedule(4, &rows, table, 16, &nrow, nullptr) != ASCG_OK) return 2;
  std::printf("sizes %d grams %lld exponents %lld\n", nrow, (long long)ascg::grams, (long long)ascg::exponents);
  return 0;
}

int growth() {
  for (int k = 1; k < 40; ++k) {
    ascg_options o{};
    o.method = ASCG_ADAPTIVE;
    o.s_max = o.s0 = o.f = 8;
    o.max_iters = 100;
    ascg_server srv = nullptr;
    fake::fail_at = -1;
    if (ascg_server_create(&o, 64 << 20, 16, nullptr, &srv) != ASCG_OK) return 2;
    ascg::missing = 0;
    ascg_completion c[8];
    int nd = 0, na = 0, np = 0, status = 0, done = 0, after = 0, pend = 0;
    double b = 0, x = 0;
    // a small system first, still running when the larger ones come
    ascg_server_submit(srv, (ascg_op)(uintptr_t)3000, &b, &x, 1e-8, 0);
    ascg_server_step(srv, c, 8, &nd, &na, &np);
    done += nd;
    ascg_server_submit(srv, (ascg_op)(uintptr_t)30000, &b, &x, 1e-8, 1);
    ascg_server_submit(srv, (ascg_op)(uintptr_t)100000, &b, &x, 1e-8, 2);
    ascg_server_submit(srv, (ascg_op)(uintptr_t)40000, &b, &x, 1e-8, 3);
    fake::fail_at = fake::count + k;
    bool hit = false;
    for (int step = 0; step < 50; ++step) {
      const ascg_status st = ascg_server_step(srv, c, 8, &nd, &na, &np);
      if (st != ASCG_OK) {
        hit = true;
        status = st;
        after = srv->running;
        pend = (int)srv->queue.size();
        continue;
      }
      done += nd;
      if (na == 0 && np == 0) break;
    }
    std::printf("k %d hit %d status %d running %d queued %d done %d missing %d used %zu\n", k, hit, status, after, pend,
                done, ascg::missing, srv->arena.bytes_used());
    ascg_server_destroy(srv);
    if (!hit) break;
  }
  std::printf("leaked %zu\n", fake::live.size());
  return 0;
}

int main(int argc, char** argv) {
  const std::string what = argc > 1 ? argv[1] : "";
  return what == "growth" ? growth() : what == "count" ? count_launches() : what == "memory" ? memory() : what == "tune" ? tune() : 1;
}
