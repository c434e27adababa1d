// Test helper (built by tests/test_host_on_fake_cuda.py): the library's host
// code (host.cpp, server.cpp, encoder.cpp) over a CUDA runtime and kernel
// launchers that run on the CPU. Device memory is heap memory filled with
// 0xAB, which nothing may take for initialised; every runtime call and every
// launch can be made to fail; every launch checks that the memory it is given
// is allocated, large enough and in the state that the kernels rely on.
//
// usage: host_on_fake_cuda calls <FASTQ file>   each entry point, with each of
//          its runtime calls failing in turn, and then called again
//        host_on_fake_cuda server <FASTQ file>  requests go on while the serving
//          engine reads a batch's error word back, and a handle's launch
//          configuration may change while it is served; batches whose end
//          cannot be read end with an error
//        host_on_fake_cuda depth <file>  prints the depth class of its
//          whole-file decode (team_depth)
//        host_on_fake_cuda blocks <file>  the blocks of a line (line_block),
//          for short lines and for lines of almost 4 GiB
// prints "ok" lines and exits 1 at the first violation.
#include <cuda_runtime.h>

#include <atomic>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <fstream>
#include <functional>
#include <future>
#include <iterator>
#include <map>
#include <mutex>
#include <string>

#include "archive.h"

namespace {

#define REQUIRE(c)                                                    \
  do {                                                                \
    if (!(c)) {                                                       \
      std::printf("violated at line %d: %s\n", __LINE__, #c);         \
      std::fflush(stdout);                                            \
      std::_Exit(1);                                                  \
    }                                                                 \
  } while (0)

std::mutex g_mu;
std::map<const uint8_t *, size_t> g_mem;  // allocations of device memory
std::atomic<int> g_fail_at{-1}, g_calls{0};

// the next runtime call: fails when it is the one that the test chose
cudaError_t call() { return g_calls++ == g_fail_at ? cudaErrorUnknown : cudaSuccess; }

bool live(const void *p, size_t bytes) {
  if (!bytes) return true;
  const uint8_t *b = static_cast<const uint8_t *>(p);
  std::lock_guard<std::mutex> lk(g_mu);
  auto it = g_mem.upper_bound(b);
  if (!b || it == g_mem.begin()) return false;
  --it;
  return b + bytes <= it->first + it->second;
}

cudaError_t give(void **p, size_t n) {
  if (cudaError_t e = call()) return e;
  uint8_t *b = static_cast<uint8_t *>(std::malloc(n));
  std::memset(b, 0xAB, n);
  std::lock_guard<std::mutex> lk(g_mu);
  g_mem[b] = n;
  *p = b;
  return cudaSuccess;
}

cudaError_t take(void *p) {
  std::lock_guard<std::mutex> lk(g_mu);
  if (p) REQUIRE(g_mem.erase(static_cast<uint8_t *>(p)) == 1);
  std::free(p);
  return cudaSuccess;
}

std::atomic<bool> g_lost{false}, g_unreadable{false};  // every event's, every copy to the host's error
std::function<void()> g_on_read_back;  // called inside every copy to the host

}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 0, cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { return give(p, n); }
cudaError_t cudaFree(void *p) { return take(p); }
cudaError_t cudaMallocHost(void **p, size_t n) {
  if (cudaError_t e = call()) return e;
  return *p = std::malloc(n), cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind k) {
  if (cudaError_t e = call()) return e;
  if (k != cudaMemcpyDeviceToHost) REQUIRE(live(d, n));
  if (k != cudaMemcpyHostToDevice) REQUIRE(live(s, n));
  if (k == cudaMemcpyDeviceToHost && g_on_read_back) g_on_read_back();
  if (k == cudaMemcpyDeviceToHost && g_unreadable) return cudaErrorUnknown;
  return std::memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemset(void *d, int v, size_t n) {
  if (cudaError_t e = call()) return e;
  REQUIRE(live(d, n));
  return std::memset(d, v, n), cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  if (cudaError_t e = call()) return e;
  return *s = reinterpret_cast<cudaStream_t>(std::malloc(1)), cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { return std::free(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t e, unsigned) { return e ? call() : cudaErrorInvalidValue; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *ev, unsigned) {
  if (cudaError_t e = call()) return e;
  return *ev = reinterpret_cast<cudaEvent_t>(std::malloc(1)), cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) { return std::free(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { return e ? call() : cudaErrorInvalidValue; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { return e ? cudaSuccess : cudaErrorInvalidValue; }
cudaError_t cudaEventQuery(cudaEvent_t e) {
  return !e ? cudaErrorInvalidValue : g_lost ? cudaErrorLaunchFailure : cudaSuccess;
}
// (memory pools: not offered, so that buffers come from cudaMalloc)
cudaError_t cudaMallocFromPoolAsync(void **, size_t, cudaMemPool_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaFreeAsync(void *, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *, const cudaMemPoolProps *) { return cudaErrorNotSupported; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaErrorNotSupported; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaErrorNotSupported; }
}

namespace aceapex {

int decode_grid(int, int) { return 152; }
static uint32_t g_depth;

static bool archive_ok(const DevArchive &A) {
  return live(A.dir, 24 * (size_t)A.n_seg) && live(A.lut, kLutBytes) && live(A.flags, 8 * (size_t)A.n_seg) &&
         (!A.n_seg || live(A.payload, 1));
}

cudaError_t launch_begin(uint32_t *g, uint32_t *e, uint32_t *c, cudaStream_t) {
  if (cudaError_t r = call()) return r;
  REQUIRE(live(g, 4) && live(e, 4) && live(c, 4));
  *e = ++*g;
  *c = 0;
  return cudaSuccess;
}
cudaError_t launch_set_pages(uint32_t *page, const WorkItem *work, uint32_t n, cudaStream_t) {
  if (cudaError_t r = call()) return r;
  REQUIRE(live(work, 8 * (size_t)n));
  for (uint32_t i = 0; i < n; ++i) {
    REQUIRE(live(page + work[i].seg, 4));
    page[work[i].seg] = i;
  }
  return cudaSuccess;
}
cudaError_t launch_begin_list(const WorkList &list, WorkItem *work, uint32_t *page, uint32_t *g, uint32_t *e,
                              uint32_t *c, cudaStream_t st) {
  REQUIRE(live(work, 8 * (size_t)list.n));
  for (uint32_t i = 0; i < list.n; ++i) work[i] = WorkItem{0, list.seg[i]};
  if (cudaError_t r = launch_set_pages(page, work, list.n, st)) return r;
  return launch_begin(g, e, c, st);
}
cudaError_t launch_clear_pages(uint32_t *page, const WorkItem *work, uint32_t n, cudaStream_t) {
  if (cudaError_t r = call()) return r;
  REQUIRE(live(work, 8 * (size_t)n));
  for (uint32_t i = 0; i < n; ++i) {
    REQUIRE(live(page + work[i].seg, 4));
    page[work[i].seg] = 0xFFFFFFFFu;
  }
  return cudaSuccess;
}
cudaError_t launch_init_flags(uint64_t *flags, const SegRec *dir, uint64_t n, cudaStream_t) {
  if (cudaError_t r = call()) return r;
  REQUIRE(live(flags, 8 * n) && live(dir, 24 * n));
  for (uint64_t s = 0; s < n; ++s) flags[s] = (uint64_t)dir[s].level << 32;
  return cudaSuccess;
}
cudaError_t launch_window_order(const SegRec *dir, uint64_t n, uint64_t per, uint32_t, WorkItem *out, cudaStream_t) {
  if (cudaError_t r = call()) return r;
  REQUIRE(per && live(dir, 24 * n) && live(out, 8 * n));
  for (uint64_t s = 0; s < n; ++s) out[s] = WorkItem{0, (uint32_t)s};
  return cudaSuccess;
}
cudaError_t launch_decode(const DecodeLaunch &L, int grid, int, cudaStream_t) {
  if (cudaError_t r = call()) return r;
  REQUIRE(grid > 0 && archive_ok(L.arc0) && live(L.work, 8 * (size_t)L.n_work));
  REQUIRE(live(L.err, 4) && live(L.epoch, 4) && live(L.counter, 4));
  g_depth = L.team_depth;
  REQUIRE(L.max_stage <= L.stage_cap || live(L.scratch, (size_t)L.scratch_warps * kStageBytes));
  for (uint32_t i = 0; i < L.n_work; ++i) {
    REQUIRE(L.work[i].seg < L.arc0.n_seg);
    if (L.view0.page) REQUIRE(live(L.view0.page + L.work[i].seg, 4) && L.view0.page[L.work[i].seg] < L.n_work);
  }
  if (L.view0.page)
    for (uint32_t s = 0; s < L.arc0.n_seg; ++s) REQUIRE(L.view0.page[s] == 0xFFFFFFFFu || L.view0.page[s] < L.arc0.n_seg);
  if (L.view0.page) REQUIRE(live(L.view0.slot_base, (size_t)L.n_work << L.arc0.log2_S));
  else if (L.view0.mask != ~uint64_t(0)) REQUIRE(live(L.view0.base, L.view0.mask + 1));
  else REQUIRE(live(L.view0.base, 1));
  return cudaSuccess;
}
cudaError_t launch_batch(const DecodeLaunch &L, uint32_t n, uint32_t, int, cudaStream_t) {
  if (cudaError_t r = call()) return r;
  REQUIRE(live(L.arcs, n * sizeof(DevArchive)) && live(L.views, n * sizeof(OutView)));
  for (uint32_t i = 0; i < n; ++i)
    REQUIRE(archive_ok(L.arcs[i]) && live(L.arcs[i].order, 8 * (size_t)L.arcs[i].n_seg) &&
            live(L.views[i].base, L.arcs[i].n));
  return cudaSuccess;
}
cudaError_t launch_gather(OutView v, uint32_t, uint64_t lo, uint64_t hi, uint8_t *dst, uint32_t *page,
                          const WorkItem *work, uint32_t n, cudaStream_t st) {
  REQUIRE(v.page == page && live(dst, hi - lo));
  return launch_clear_pages(page, work, n, st);
}
cudaError_t launch_gather_bases(OutView, uint32_t, uint64_t, uint32_t, uint32_t, uint64_t n, uint8_t *dst,
                                uint32_t *page, const WorkItem *work, uint32_t n_work, cudaStream_t st) {
  REQUIRE(live(dst, n));
  return launch_clear_pages(page, work, n_work, st);
}
cudaError_t launch_copy_view(OutView a, OutView b, uint32_t, uint64_t, uint64_t, cudaStream_t) {
  REQUIRE(live(a.slot_base, 1) && live(b.base, b.mask + 1));
  return call();
}
cudaError_t launch_multi_gather(const GatherJob *jobs, uint32_t n, uint64_t, cudaStream_t) {
  if (cudaError_t r = call()) return r;
  REQUIRE(live(jobs, n * sizeof(GatherJob)));
  for (uint32_t i = 0; i < n; ++i) REQUIRE(live(jobs[i].dst, jobs[i].n));
  return cudaSuccess;
}
cudaError_t launch_fastq_interleave(const uint8_t *const base[4], const uint64_t len[4], uint32_t *counts,
                                    uint64_t *offs, uint32_t *const nl[4], const uint64_t cap[4], uint32_t *err,
                                    uint8_t *out, cudaStream_t) {
  uint64_t chunks = 0, n = 0;
  for (int k = 0; k < 4; ++k) {
    REQUIRE(live(base[k], (len[k] + 15) & ~uint64_t(15)) && live(nl[k], 4 * cap[k]));
    chunks += (len[k] + 65535) / 65536;
    n += len[k];
  }
  REQUIRE(live(counts, 4 * chunks) && live(offs, 8 * (chunks + 4)) && live(err, 4) && live(out, n));
  return call();
}
static void closure_ok(const ClosureDev &C, uint32_t gen) {
  REQUIRE(live(C.dep_ptr, 8 * ((size_t)C.n_seg + 1)) && live(C.dir, 24 * (size_t)C.n_seg) && live(C.err, 4));
  REQUIRE(C.dep_ptr[0] == 0 && live(C.deps, 4 * C.dep_ptr[C.n_seg]) && live(C.found, 4 * kClosureFound));
  REQUIRE(live(C.mark, 4 * (size_t)C.n_seg) && live(C.list, 4 * (size_t)C.n_seg));
  for (uint32_t s = 0; s < C.n_seg; ++s) REQUIRE(C.mark[s] <= gen);
}
cudaError_t launch_closure_seed(ClosureDev C, uint32_t s_lo, uint32_t n, uint32_t top, uint32_t gen, cudaStream_t) {
  if (cudaError_t r = call()) return r;
  closure_ok(C, gen);
  for (uint32_t l = 0; l <= top; ++l) C.found[l] = 0;
  C.found[top + 1] = n;
  for (uint32_t i = 0; i < n; ++i) C.mark[C.list[i] = s_lo + i] = gen;
  return cudaSuccess;
}
cudaError_t launch_closure_expand(ClosureDev C, uint32_t level, uint32_t top, uint32_t gen, cudaStream_t) {
  if (cudaError_t r = call()) return r;
  closure_ok(C, gen);
  uint32_t n = 0;
  for (uint32_t l = level + 1; l <= top + 1; ++l) n += C.found[l];
  for (uint32_t i = 0; i < n; ++i) {
    const uint32_t s = C.list[i];
    REQUIRE(s < C.n_seg);
    if (C.dir[s].level != level) continue;
    for (uint64_t k = C.dep_ptr[s]; k < C.dep_ptr[s + 1]; ++k)
      if (C.mark[C.deps[k]] != gen) {
        C.mark[C.deps[k]] = gen;
        C.list[n + C.found[level]++] = C.deps[k];
      }
  }
  return cudaSuccess;
}
cudaError_t launch_closure_order(ClosureDev C, uint32_t top, WorkItem *work, uint32_t *page, uint32_t *n_out,
                                 cudaStream_t) {
  if (cudaError_t r = call()) return r;
  uint32_t n = 0;
  for (uint32_t l = 1; l <= top + 1; ++l) n += C.found[l];
  REQUIRE(live(work, 8 * (size_t)n) && live(n_out, 4));
  for (uint32_t i = 0; i < n; ++i) {
    work[i] = WorkItem{0, C.list[i]};
    page[C.list[i]] = i;
  }
  *n_out = n;
  return cudaSuccess;
}
cudaError_t launch_window_crc(OutView v, uint64_t, uint64_t, uint32_t *crc, uint32_t *sums, uint32_t, cudaStream_t) {
  REQUIRE(live(v.base, v.mask + 1) && live(crc, 4) && live(sums, 8) && sums[0] == 0 && sums[1] == 0);
  return call();
}

}  // namespace aceapex

namespace {

std::vector<uint8_t> encoded(const uint8_t *d, uint64_t n, uint32_t log2_B, uint64_t D = 0) {
  void *o = nullptr;
  uint64_t len = 0;
  REQUIRE(aceapex_encode(d, n, log2_B, 16, 8, D, nullptr, 0, 0, &o, &len) == ACEAPEX_OK);
  std::vector<uint8_t> a(static_cast<uint8_t *>(o), static_cast<uint8_t *>(o) + len);
  aceapex_free(o);
  return a;
}

struct Opened {
  std::vector<aceapex_archive *> as;
  explicit Opened(const std::vector<const std::vector<uint8_t> *> &v) {
    for (const auto *a : v) {
      as.push_back(nullptr);
      REQUIRE(aceapex_open(a->data(), a->size(), 0, &as.back()) == ACEAPEX_OK);
    }
  }
  ~Opened() {
    for (aceapex_archive *a : as) aceapex_close(a);
  }
};

// f on new handles, with its k-th runtime call failing, for every k; then
// twice more without a failure, which has to work
void each_failure(const char *name, const std::vector<const std::vector<uint8_t> *> &v,
                  const std::function<int(std::vector<aceapex_archive *> &)> &f) {
  int k = 0;
  for (bool more = true; more; ++k) {
    Opened o(v);
    g_calls = 0;
    g_fail_at = k;
    f(o.as);  // (some failures have no consequence: a status is not asked for)
    more = g_calls > k;
    g_fail_at = -1;
    for (int again = 0; again < 2; ++again)
      if (f(o.as) != ACEAPEX_OK) {
        std::printf("%s: a call after a failure of runtime call %d fails\n", name, k);
        std::exit(1);
      }
  }
  std::printf("ok %s (%d calls)\n", name, k - 1);
}

void calls(const std::vector<uint8_t> &in) {
  const uint64_t n = in.size();
  const auto wide = encoded(in.data(), n, 12), small = encoded(in.data(), 300'000, 14);
  const auto bounded = encoded(in.data(), 1'000'000, 14, 1 << 16);
  std::vector<uint8_t> lines(n);
  uint64_t len[4], at = 0;
  aceapex_fastq_split(in.data(), 300'000, lines.data(), len);
  std::vector<std::vector<uint8_t>> parts;
  for (int k = 0; k < 4; ++k) {
    parts.push_back(encoded(lines.data() + at, len[k], 14));
    at += len[k];
  }
  void *out = nullptr;
  REQUIRE(cudaMalloc(&out, n) == cudaSuccess);
  std::vector<uint8_t> host(n);
  const auto range = [&](uint64_t lo, uint64_t hi) {
    return [=](std::vector<aceapex_archive *> &a) { return aceapex_decode_range(a[0], lo, hi, out, n, nullptr); };
  };
  each_failure("open and close", {}, [&](auto &) {
    aceapex_archive *a = nullptr;
    const int rc = aceapex_open(bounded.data(), bounded.size(), 0, &a);
    aceapex_close(a);
    return rc;
  });
  each_failure("host to host", {}, [&](auto &) {
    return aceapex_decode_host(bounded.data(), bounded.size(), 0, host.data(), n, 1 << 17);
  });
  each_failure("range, closure walked on the host", {&small}, range(100'000, 100'400));
  each_failure("range, closure found on the device", {&wide}, range(n - 1'200'000, n));
  each_failure("whole file", {&small}, [&](auto &a) { return aceapex_decode_all(a[0], out, n, nullptr, nullptr); });
  each_failure("ring", {&bounded}, [&](auto &a) {
    return aceapex_stream_range(a[0], 1 << 17, 1'000'000, 1 << 19, 1 << 17, static_cast<uint32_t *>(out), nullptr);
  });
  each_failure("batch", {&small, &bounded}, [&](auto &a) {
    void *outs[2] = {out, static_cast<uint8_t *>(out) + 300'000};
    return aceapex_decode_batch(a.data(), 2, outs, nullptr);
  });
  each_failure("line streams", {&parts[0], &parts[1], &parts[2], &parts[3]},
               [&](auto &a) { return aceapex_decode_fastq_streams(a.data(), out, n, nullptr); });
  each_failure("to host, two window sizes", {&bounded}, [&](auto &a) {
    int rc = aceapex_decode_all_to_host(a[0], host.data(), n, 1 << 17, nullptr);
    const int rc2 = aceapex_decode_all_to_host(a[0], host.data(), n, 1 << 18, nullptr);
    const int rc3 = aceapex_decode_all_to_host(a[0], host.data(), n, 1 << 17, nullptr);
    return rc ? rc : rc2 ? rc2 : rc3;
  });
  take(out);
  REQUIRE(g_mem.size() <= 1);  // (the device's epoch word stays)
}

// Submits `n` ranges of the archive to a server and waits for them; returns
// how many ended with a status other than OK.
int serve(aceapex_server *S, int n, void *out) {
  std::vector<uint64_t> tickets(n);
  int bad = 0;
  for (int i = 0; i < n; ++i)
    REQUIRE(aceapex_server_submit(S, 0, 100 * i, 100 * i + 1000, out, 1000, &tickets[i]) == ACEAPEX_OK);
  for (uint64_t t : tickets) {
    int done = 0;
    bad += aceapex_server_poll(S, t, 1, &done, nullptr) != ACEAPEX_OK;
    REQUIRE(done);
  }
  return bad;
}

void server(const std::vector<uint8_t> &in) {
  const auto arc = encoded(in.data(), 300'000, 14);
  Opened o({&arc});
  void *out = nullptr;
  REQUIRE(cudaMalloc(&out, 1000) == cudaSuccess);
  aceapex_server *S = nullptr;
  REQUIRE(aceapex_server_create(o.as.data(), 1, 64 << 20, 4, &S) == ACEAPEX_OK);
  g_on_read_back = [&] {
    aceapex_server_stats st;
    auto other = std::async(std::launch::async, [&] { return aceapex_server_get_stats(S, &st); });
    REQUIRE(other.wait_for(std::chrono::seconds(10)) == std::future_status::ready);
  };
  REQUIRE(serve(S, 50, out) == 0);
  aceapex_server_destroy(S);
  g_on_read_back = nullptr;
  // a handle whose stage is made smaller while it is served
  REQUIRE(aceapex_set_launch(o.as[0], 0, 0, 0) == ACEAPEX_OK);
  REQUIRE(aceapex_server_create(o.as.data(), 1, 64 << 20, 4, &S) == ACEAPEX_OK);
  REQUIRE(aceapex_set_launch(o.as[0], 0, 0, 16) == ACEAPEX_OK);
  REQUIRE(serve(S, 50, out) == 0);
  // batches whose end or whose error word cannot be read end with an error
  for (std::atomic<bool> *f : {&g_lost, &g_unreadable}) {
    *f = true;
    REQUIRE(serve(S, 50, out) == 50);
    *f = false;
    REQUIRE(serve(S, 50, out) == 0);
  }
  aceapex_server_destroy(S);
  take(out);
  std::printf("ok requests go on while an error word is read back\n");
}

// the blocks' parts follow one another, fill their blocks and end with the line
void blocks() {
  const auto check = [](uint32_t al, uint32_t len, uint32_t b) {
    const LineBlock p = line_block(al, len, b);
    const uint64_t begin = 16 * (uint64_t)b, end = begin + 16;  // of the block, al bytes before the line's start
    const uint64_t from = std::max<uint64_t>(begin, al) - al, to = std::min<uint64_t>(end - al, len);
    REQUIRE(p.from == from && p.n == to - from && p.o == from + al - begin && p.n >= 1 && p.o + p.n <= 16);
  };
  for (uint32_t al = 0; al < 16; ++al) {
    REQUIRE(line_blocks(al, 0) == 0);
    for (uint32_t len = 1; len < 200; ++len) {
      REQUIRE(line_blocks(al, len) == (al + len + 15) / 16);
      for (uint32_t b = 0; b < line_blocks(al, len); ++b) check(al, len, b);
    }
    for (uint32_t less = 1; less < 40; ++less) {
      const uint32_t len = 0u - less;
      REQUIRE(line_blocks(al, len) == ((uint64_t)al + len + 15) / 16);
      for (uint32_t k = 0; k < 4; ++k) check(al, len, k), check(al, len, line_blocks(al, len) - 1 - k);
    }
  }
  std::printf("ok blocks\n");
}

void depth(const std::vector<uint8_t> &in) {
  const auto arc = encoded(in.data(), in.size(), 14);
  Opened o({&arc});
  void *out = nullptr;
  REQUIRE(cudaMalloc(&out, in.size()) == cudaSuccess);
  REQUIRE(aceapex_decode_all(o.as[0], out, in.size(), nullptr, nullptr) == ACEAPEX_OK);
  std::printf("depth %u\n", g_depth);
}

}  // namespace

int main(int argc, char **argv) {
  if (argc != 3) return 2;
  std::ifstream f(argv[2], std::ios::binary);
  std::vector<uint8_t> in((std::istreambuf_iterator<char>(f)), std::istreambuf_iterator<char>());
  if (std::string(argv[1]) == "calls") calls(in);
  else if (std::string(argv[1]) == "server") server(in);
  else if (std::string(argv[1]) == "blocks") blocks();
  else depth(in);
  return 0;
}
