/* cudaMalloc and cudaFree of libqcd under a limit, for test_gpu_memory.py (preloaded: the library's calls come
 * here, all others pass through).  An allocation beyond the limit, or the one chosen to fail, gets
 * cudaErrorMemoryAllocation without the runtime being asked. */
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
#include <string.h>

enum { MOST = 4096, MEMORY_ALLOCATION = 2 };
static struct { void* p; size_t n; } held[MOST];
static size_t limit, live, peak;
static long count, fail_at;

static void* runtime(const char* name) {
  static void* lib;
  if (!lib) lib = dlopen("libcudart.so.13", RTLD_LAZY);
  return dlsym(lib, name);
}

static int from_library(void* caller) {
  Dl_info i;
  return dladdr(caller, &i) && i.dli_fname && strstr(i.dli_fname, "libqcd");
}

int cudaMalloc(void** p, size_t n) {
  static int (*real)(void**, size_t);
  if (!real) real = (int (*)(void**, size_t))runtime("cudaMalloc");
  if (!from_library(__builtin_return_address(0))) return real(p, n);
  count++;
  if ((limit && live + n > limit) || (fail_at && count == fail_at)) return MEMORY_ALLOCATION;
  int e = real(p, n);
  if (e) return e;
  for (int k = 0; k < MOST; k++)
    if (!held[k].p) {
      held[k].p = *p;
      held[k].n = n;
      break;
    }
  live += n;
  if (live > peak) peak = live;
  return 0;
}

int cudaFree(void* p) {
  static int (*real)(void*);
  if (!real) real = (int (*)(void*))runtime("cudaFree");
  for (int k = 0; p && k < MOST; k++)
    if (held[k].p == p) {
      live -= held[k].n;
      held[k].p = NULL;
    }
  return real(p);
}

/* a new run: at most `most` bytes held at a time (0: any number), the `which`th allocation fails (0: none) */
void alloc_limit(size_t most, long which) {
  limit = most;
  fail_at = which;
  count = 0;
  peak = live;
}
size_t alloc_peak(void) { return peak; }
long alloc_count(void) { return count; }
