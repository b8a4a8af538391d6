/* The calls of the CUDA runtime that the products' host code makes, for tests without a device.  The driver's entry point takes a while to be
 * found, and the tensor map encoder refuses threads that have not been bound to a device, as the real one does. */
#include <string.h>
#include <unistd.h>

static __thread int bound;
static int encode(void) { return bound ? 0 : 201; }   /* CUDA_ERROR_INVALID_CONTEXT */
int fake_bound(void) { return bound; }
void fake_bind(void) { bound = 1; }

int cudaGetDriverEntryPoint(const char *name, void **fn, unsigned long long flags, int *found)
{
    (void)flags;
    usleep(200000);
    *fn = strcmp(name, "cuTensorMapEncodeTiled") ? 0 : (void *)encode;
    *found = 0;
    return 0;
}
int cudaGetDriverEntryPointByVersion(const char *name, void **fn, unsigned version, unsigned long long flags, int *found)
{
    (void)version;
    return cudaGetDriverEntryPoint(name, fn, flags, found);
}
int cudaGetDevice(int *dev) { *dev = 0; return 0; }
int cudaSetDevice(int dev) { bound = 1; return dev != 0; }
int cudaDeviceGetAttribute(int *value, int attr, int dev) { (void)attr; (void)dev; *value = 148; return 0; }
int cudaFuncSetAttribute(const void *f, int attr, int value) { (void)f; (void)attr; (void)value; return 0; }
int cudaGetSymbolAddress(void **p, const void *symbol) { (void)symbol; *p = (void *)(1 << 20); return 0; }
int cudaLaunchKernelExC(const void *config, const void *f, void **args) { (void)config; (void)f; (void)args; bound = 1; return 0; }
int cudaMemcpyAsync(void) { return 0; }
int cudaMemsetAsync(void) { return 0; }
int cudaLaunchKernel(void) { return 0; }
int cudaGetLastError(void) { return 0; }
int cudaStreamIsCapturing(void *stream, int *status) { (void)stream; *status = 0; return 0; }
void **__cudaRegisterFatBinary(void *f) { static void *handle; (void)f; return &handle; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void) {}
void __cudaRegisterVar(void) {}
int __cudaPopCallConfiguration(void) { return 0; }
