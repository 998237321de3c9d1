/* cudaMalloc and cudaFree of a library linked with --wrap: the allocation that
 * fake_arm names fails as if the device had no memory left. */
#include <stddef.h>

int __real_cudaMalloc(void **p, size_t bytes);
int __real_cudaFree(void *p);

static int count, fail_at = -1, live;

void fake_arm(int k) { count = 0; fail_at = k; }
int fake_count(void) { return count; }
int fake_live(void) { return live; }

int __wrap_cudaMalloc(void **p, size_t bytes) {
  if (count++ == fail_at) {
    *p = 0;
    return 2; /* cudaErrorMemoryAllocation */
  }
  const int e = __real_cudaMalloc(p, bytes);
  live += e == 0;
  return e;
}

int __wrap_cudaFree(void *p) {
  live -= p != 0;
  return __real_cudaFree(p);
}
