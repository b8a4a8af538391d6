/* The calls of the CUDA runtime that the quantizers' host code makes, for tests without a device: launches return what a
 * test has set, and the last error is kept as the runtime keeps it. */
static int launch_result, last_error;
void fake_set(int result, int last) { launch_result = result; last_error = last; }
int fake_last_error(void) { return last_error; }

int cudaLaunchKernelExC(const void *config, const void *f, void **args)
{
    (void)config; (void)f; (void)args;
    if (launch_result) last_error = launch_result;
    return launch_result;
}
int cudaLaunchKernel(void) { return cudaLaunchKernelExC(0, 0, 0); }
int cudaGetLastError(void) { int e = last_error; last_error = 0; return e; }
int cudaStreamIsCapturing(void *stream, int *status) { (void)stream; *status = 0; return 0; }
void **__cudaRegisterFatBinary(void *f) { static void *handle; (void)f; return &handle; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void) {}
void __cudaRegisterVar(void) {}
int __cudaPopCallConfiguration(void) { return 0; }
