/* A device allocator with a limit, loaded before the CUDA runtime's users so that their cudaMalloc,
 * cudaFree and cudaMemGetInfo bind here.  Calls go on to the runtime; an allocation is answered with
 * "out of memory" by the host alone where it would pass the limit, or is the one picked to fail. */
#define _GNU_SOURCE
#include <dlfcn.h>
#include <pthread.h>
#include <stddef.h>

enum { OK = 0, INVALID = 1, NO_MEMORY = 2, MAX = 1 << 16 };
static pthread_mutex_t lock = PTHREAD_MUTEX_INITIALIZER;
static void* ptr[MAX];
static size_t size[MAX];
static size_t in_use, limit = (size_t)-1;
static long countdown = -1, calls, bad_frees;

static void* real(const char* name) {
    static void* lib;
    if (!lib) lib = dlopen("libcudart.so.13", RTLD_NOW | RTLD_NOLOAD);
    if (!lib) lib = dlopen("libcudart.so.13", RTLD_NOW);
    return dlsym(lib, name);
}

int cudaMalloc(void** p, size_t n) {
    int (*f)(void**, size_t) = (int (*)(void**, size_t))real("cudaMalloc");
    pthread_mutex_lock(&lock);
    int e = NO_MEMORY;
    ++calls;
    const int pick = countdown >= 0 && countdown-- == 0;
    if (!pick && (limit == (size_t)-1 || in_use + n <= limit)) {
        e = f(p, n);
        for (int i = 0; e == OK && i < MAX; ++i)
            if (!ptr[i]) {
                ptr[i] = *p;
                size[i] = n;
                in_use += n;
                break;
            }
    }
    pthread_mutex_unlock(&lock);
    return e;
}

int cudaFree(void* p) {
    int (*f)(void*) = (int (*)(void*))real("cudaFree");
    if (!p) return f(p);
    pthread_mutex_lock(&lock);
    int e = INVALID, i = 0;
    while (i < MAX && ptr[i] != p) ++i;
    if (i < MAX) {
        e = f(p);
        in_use -= size[i];
        ptr[i] = NULL;
    } else {
        ++bad_frees;   /* not a live allocation: kept from the runtime */
    }
    pthread_mutex_unlock(&lock);
    return e;
}

int cudaMemGetInfo(size_t* free_, size_t* total) {
    int (*f)(size_t*, size_t*) = (int (*)(size_t*, size_t*))real("cudaMemGetInfo");
    const int e = f(free_, total);
    if (e == OK && limit != (size_t)-1) *free_ = limit > in_use ? limit - in_use : 0;
    return e;
}

void fake_limit(size_t bytes) { limit = bytes; }
void fake_fail(long n) { countdown = n; }         /* the n-th allocation from now fails; -1 none */
size_t fake_in_use(void) { return in_use; }
long fake_calls(void) { return calls; }
long fake_bad_frees(void) { return bad_frees; }
