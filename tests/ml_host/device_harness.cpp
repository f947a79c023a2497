// Test harness: device_once.h against a fake of the two runtime calls it makes.  Built by the tests as a host-only
// shared library without the CUDA runtime (linked with -Bsymbolic: a runtime loaded in the process must not answer);
// the product never loads it.
#include "device_once.h"

static int g_device, g_sets, g_bytes;
static cudaError_t g_get, g_set;

extern "C" cudaError_t cudaGetDevice(int* d) {
    *d = g_device;
    return g_get;
}
extern "C" cudaError_t cudaFuncSetAttribute(const void*, enum cudaFuncAttribute, int bytes) {
    ++g_sets;
    g_bytes = bytes;
    return g_set;
}
static void kernel_a() {}
static void kernel_b() {}

extern "C" {
// asks for kernel a or b on a device; the fake calls return get and set.  Returns the status.
int device_allow(int which, int device, int bytes, int get, int set) {
    g_device = device, g_get = (cudaError_t)get, g_set = (cudaError_t)set;
    return (int)(which ? ddamg::allow_smem<kernel_b>(bytes) : ddamg::allow_smem<kernel_a>(bytes));
}
int device_sets() { return g_sets; }
int device_bytes() { return g_bytes; }
}
