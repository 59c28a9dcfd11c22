// Runs the blocks of a kernel launch one after the other, each thread of a
// block a fibre.  A fibre runs until it waits; the order in which the fibres
// of a block go on is shuffled (EMU_SEED), so that nothing can lean on it.
// Device allocations are filled with a pattern and end at a page that may not
// be touched.
#include "cuda_runtime.h"

#include <csetjmp>
#include <map>
#include <mutex>
#include <string>
#include <sys/mman.h>
#include <ucontext.h>

namespace emu {

int tid;
dim3 bdim, bidx, gdim;
char* dyn;
uint64_t slot[1024], block_serial, block_epoch, warp_epoch[32];

namespace {

enum Wait { kRun, kWarp, kWarpMem, kBlock, kDone };
constexpr size_t kStack = 256 << 10;
constexpr int kPattern = 0xA5;

struct Fibre {
  void* stack;
  Wait want;
  bool begun;
  jmp_buf at;
};

std::recursive_mutex mu;
std::vector<Fibre> fib;
std::function<void()>* body;
jmp_buf scheduler;
ucontext_t scheduler_ctx, first_ctx;
uint64_t rng = getenv("EMU_SEED") ? strtoull(getenv("EMU_SEED"), nullptr, 10) * 0x9E3779B97F4A7C15ull | 1 : 1;
bool capturing;
std::vector<std::function<void()>>* recorded;
std::map<void*, std::pair<void*, size_t>> mapped;
std::map<std::string, long>& reports() {
  static std::map<std::string, long> r;
  return r;
}

uint64_t random64() {
  rng ^= rng << 13;
  rng ^= rng >> 7;
  rng ^= rng << 17;
  return rng;
}

void wait(Wait w) {
  Fibre& me = fib[tid];
  me.want = w;
  if (!_setjmp(me.at)) _longjmp(scheduler, 1);
}

void entry() {
  (*body)();
  wait(kDone);
}

// Runs fibre t until it waits.  (The first time through its context, later
// by longjmp, which needs no system call.)
void resume(int t) {
  tid = t;
  Fibre& f = fib[t];
  if (_setjmp(scheduler)) return;
  if (f.begun) _longjmp(f.at, 1);
  f.begun = true;
  getcontext(&first_ctx);
  first_ctx.uc_stack.ss_sp = f.stack;
  first_ctx.uc_stack.ss_size = kStack;
  first_ctx.uc_link = &scheduler_ctx;
  makecontext(&first_ctx, entry, 0);
  setcontext(&first_ctx);
}

void run_block(int threads) {
  ++block_serial;
  ++block_epoch;
  for (auto& e : warp_epoch) ++e;
  for (int t = 0; t < threads; ++t) {
    fib[t].want = kRun;
    fib[t].begun = false;
  }
  for (;;) {
    bool progress = false;
    const uint64_t r = random64();
    for (int i = 0; i < threads; ++i) {
      const int at = (int)((i + r % threads) % threads), t = r >> 40 & 1 ? threads - 1 - at : at;
      if (fib[t].want != kRun) continue;
      progress = true;
      if (!(r >> (8 + (t >> 5)) & 1)) resume(t);  // about half of the warps go on in a sweep
    }
    bool all_block = true, all_done = true;
    for (int w = 0; w < threads; w += 32) {
      bool warp = true, live = false, mem = false;
      for (int t = w; t < min(w + 32, threads); ++t) {
        const Wait x = fib[t].want;
        all_done &= x == kDone;
        all_block &= x == kBlock || x == kDone;
        if (x == kDone) continue;
        live = true;
        warp &= x == kWarp || x == kWarpMem;
        mem |= x == kWarpMem;
      }
      if (!live || !warp) continue;
      progress = true;
      if (mem) ++warp_epoch[w >> 5];
      for (int t = w; t < min(w + 32, threads); ++t)
        if (fib[t].want != kDone) fib[t].want = kRun;
    }
    if (all_done) return;
    if (all_block) {
      progress = true;
      ++block_epoch;
      for (auto& e : warp_epoch) ++e;
      for (int t = 0; t < threads; ++t)
        if (fib[t].want != kDone) fib[t].want = kRun;
    }
    if (!progress) {
      fprintf(stderr, "emu: the threads of a block wait for each other\n");
      abort();
    }
  }
}

}  // namespace

void wait_warp(bool orders_memory) { wait(orders_memory ? kWarpMem : kWarp); }
void wait_block() { wait(kBlock); }
void nap() { wait(kRun); }
void report(const char* what) { ++reports()[what]; }

void launch(dim3 g, dim3 b, size_t smem, std::function<void()> kernel) {
  enqueue([=]() mutable {
    std::lock_guard<std::recursive_mutex> lk(mu);
    if (smem > 232448 || b.x > 1024) {
      fprintf(stderr, "emu: %zu bytes of shared memory, %u threads\n", smem, b.x);
      abort();
    }
    gdim = g;
    bdim = b;
    body = &kernel;
    while (fib.size() < b.x) {
      Fibre f{};
      f.stack = mmap(nullptr, kStack, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
      fib.push_back(f);
    }
    dyn = static_cast<char*>(device_alloc(smem));
    for (unsigned blk = 0; blk < g.x; ++blk) {
      bidx = dim3(blk);
      memset(dyn, kPattern, smem);
      run_block((int)b.x);
    }
    device_free(dyn);
  });
}

void enqueue(std::function<void()> work) {
  if (capturing)
    recorded->push_back(work);
  else
    work();
}

void* device_alloc(size_t n) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  const size_t page = 4096, bytes = (n + 15) & ~(size_t)15, total = ((bytes + page - 1) & ~(page - 1)) + 2 * page;
  char* m = static_cast<char*>(mmap(nullptr, total, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0));
  mprotect(m, page, PROT_NONE);
  mprotect(m + total - page, page, PROT_NONE);
  char* p = m + total - page - bytes;
  memset(p, kPattern, bytes);
  mapped[p] = {m, total};
  return p;
}

void device_free(void* p) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  const auto it = mapped.find(p);
  if (it == mapped.end()) return;
  munmap(it->second.first, it->second.second);
  mapped.erase(it);
}

}  // namespace emu

cudaError_t cudaStreamBeginCapture(cudaStream_t, int) {
  emu::capturing = true;
  emu::recorded = new std::vector<std::function<void()>>();
  return 0;
}

cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  emu::capturing = false;
  *g = emu::recorded;
  return 0;
}

// Accesses of watched shared memory that were reported since the last call.
extern "C" long emu_take_reports() {
  long n = 0;
  for (const auto& r : emu::reports()) {
    fprintf(stderr, "emu: %ld times a %s\n", r.second, r.first.c_str());
    n += r.second;
  }
  emu::reports().clear();
  return n;
}
