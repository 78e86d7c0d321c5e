/* Preloaded before the CUDA runtime: makes one later call of
 * cudaStreamWaitEvent or cudaEventRecord return an error without being made
 * (fail_after(which, n): the n-th one from now; 0 turns it off). */
#define _GNU_SOURCE
#include <dlfcn.h>

static int left[2];

void fail_after(int which, int n) { left[which] = n; }

static int fails(int which) { return left[which] > 0 && --left[which] == 0; }

int cudaStreamWaitEvent(void* stream, void* event, unsigned flags) {
  static int (*real)(void*, void*, unsigned);
  if (!real) real = (int (*)(void*, void*, unsigned))dlsym(RTLD_NEXT, "cudaStreamWaitEvent");
  return fails(0) ? 999 : real(stream, event, flags);
}

int cudaEventRecord(void* event, void* stream) {
  static int (*real)(void*, void*);
  if (!real) real = (int (*)(void*, void*))dlsym(RTLD_NEXT, "cudaEventRecord");
  return fails(1) ? 999 : real(event, stream);
}
