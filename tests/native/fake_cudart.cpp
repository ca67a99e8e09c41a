// The CUDA runtime calls of the library's host code, without a device: memory comes from the host's heap, launches do
// nothing, the call that a test chooses returns an error, and limits on shared memory are noted beside what launches ask for.
// (No CUDA header: its inline wrappers would be defined twice.)
#include <stdio.h>
#include <stdlib.h>

#include <map>
#include <set>

std::set<void *> fake_live;
std::map<const void *, std::set<int>> fake_limits;       // dynamic shared memory allowed, of each kernel
std::map<const void *, std::set<size_t>> fake_shared;    // ... and asked for
unsigned fake_blocks;                                    // of the last launch in a row of its grid
int fake_calls = 0, fake_fail_at = 0, fake_last_error = 0;

static int step()
{
    if (++fake_calls != fake_fail_at) return 0;
    return fake_last_error = 999;                             // cudaErrorUnknown
}

extern "C" {
int cudaMalloc(void **p, size_t n)
{
    const int e = step();
    if (e == 0) fake_live.insert(*p = malloc(n));
    return e;
}
int cudaFree(void *p)
{
    if (p && !fake_live.erase(p)) {
        printf("freed, but not allocated\n");
        exit(1);
    }
    free(p);
    return 0;
}
int cudaMemGetInfo(size_t *avail, size_t *all) { *avail = *all = (size_t)1 << 30; return step(); }
int cudaStreamSynchronize(void *) { return step(); }
int cudaDeviceSynchronize(void) { return step(); }
int cudaLaunchKernel() { return step(); }                // (arguments are left where the caller put them)
struct fake_config { unsigned grid[3], block[3]; size_t shared; };
int cudaLaunchKernelExC(const fake_config *c, const void *kernel, void **)
{
    fake_shared[kernel].insert(c->shared);
    fake_blocks = c->grid[0];
    return step();
}
int cudaFuncSetAttribute(const void *kernel, int, int bytes)
{
    fake_limits[kernel].insert(bytes);
    return step();
}
int cudaMemsetAsync(void *, int, size_t, void *) { return step(); }
int cudaGetLastError(void) { const int e = fake_last_error; fake_last_error = 0; return e; }
const char *cudaGetErrorString(int) { return "injected"; }
unsigned __cudaPushCallConfiguration() { return 0; }
int __cudaPopCallConfiguration() { return 0; }
void **__cudaRegisterFatBinary(void *) { static void *handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction() {}
void __cudaRegisterVar() {}
}
