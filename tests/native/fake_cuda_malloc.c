/* Test aid, preloaded into a child process: cudaMalloc refuses (with the error
 * of a full device) what is larger than a limit, and remembers the largest size
 * it was asked for.  The requests it lets through go to the CUDA runtime. */
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>

static size_t limit = 0, asked = 0;

void fake_malloc_limit(size_t bytes) { limit = bytes; }
size_t fake_malloc_asked(void) { size_t a = asked; asked = 0; return a; }

int cudaMalloc(void **p, size_t bytes) {
  static int (*real)(void **, size_t) = NULL;
  if (!real) {
    void *rt = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
    if (!rt) rt = dlopen("libcudart.so.13", RTLD_LAZY);
    if (!rt || !(real = (int (*)(void **, size_t))dlsym(rt, "cudaMalloc"))) return 2;
  }
  if (bytes > asked) asked = bytes;
  if (limit && bytes > limit) return 2; /* cudaErrorMemoryAllocation */
  return real(p, bytes);
}
