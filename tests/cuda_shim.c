/* Preloaded between libupmpm.so and the CUDA runtime by the tests that need a
 * call to be slow or to fail where on a real machine that is a matter of luck:
 *   SHIM_ATTR_SLEEP_US  microseconds that cudaFuncSetAttribute takes longer,
 *   shim_set_budget(b)  bytes that cudaMalloc may still hand out (negative: any),
 *                       which cudaMemGetInfo then calls free.
 * A refused allocation is passed on as one that no device can serve, so that the
 * runtime's own error state is the one of a real failure. */
#define _GNU_SOURCE
#include <dlfcn.h>
#include <pthread.h>
#include <stddef.h>
#include <stdlib.h>
#include <unistd.h>

#define MAXLIVE 65536
static pthread_mutex_t lock = PTHREAD_MUTEX_INITIALIZER;
static struct {
  void *p;
  size_t n;
} live[MAXLIVE];
static int nlive;
static long long budget = -1, used, refused;

static void *real(const char *name) {
  void *h = dlopen("libcudart.so.13", RTLD_LAZY);
  void *f = h ? dlsym(h, name) : NULL;
  if (!f) abort();
  return f;
}

/* bytes handed out and not yet freed; allocations refused so far */
long long shim_used(void) { return used; }
long long shim_refused(void) { return refused; }
void shim_set_budget(long long b) {
  pthread_mutex_lock(&lock);
  budget = b < 0 ? -1 : used + b;
  refused = 0;
  pthread_mutex_unlock(&lock);
}

int cudaMalloc(void **p, size_t n) {
  int (*f)(void **, size_t) = (int (*)(void **, size_t))real("cudaMalloc");
  pthread_mutex_lock(&lock);
  const int no = budget >= 0 && used + (long long)n > budget;
  if (no) ++refused;
  int rc = f(p, no ? (size_t)1 << 60 : n);
  if (!no && rc == 0) {
    if (nlive == MAXLIVE) abort();
    live[nlive].p = *p;
    live[nlive++].n = n;
    used += (long long)n;
  }
  pthread_mutex_unlock(&lock);
  return rc;
}

int cudaFree(void *p) {
  int (*f)(void *) = (int (*)(void *))real("cudaFree");
  pthread_mutex_lock(&lock);
  for (int i = 0; p && i < nlive; ++i)
    if (live[i].p == p) {
      used -= (long long)live[i].n;
      live[i] = live[--nlive];
      break;
    }
  pthread_mutex_unlock(&lock);
  return f(p);
}

int cudaMemGetInfo(size_t *avail, size_t *total) {
  int (*f)(size_t *, size_t *) = (int (*)(size_t *, size_t *))real("cudaMemGetInfo");
  const int rc = f(avail, total);
  pthread_mutex_lock(&lock);
  if (rc == 0 && budget >= 0) {
    const long long left = budget > used ? budget - used : 0;
    if ((long long)*avail > left) *avail = (size_t)left;
  }
  pthread_mutex_unlock(&lock);
  return rc;
}

int cudaFuncSetAttribute(const void *func, int attr, int value) {
  int (*f)(const void *, int, int) = (int (*)(const void *, int, int))real("cudaFuncSetAttribute");
  const int rc = f(func, attr, value);
  const char *us = getenv("SHIM_ATTR_SLEEP_US");
  if (us) usleep((useconds_t)atoi(us));
  return rc;
}
