/* A CUDA runtime of two fake devices with different numbers of SMs, for host
 * code that is checked without a GPU: it records the kernels whose attributes
 * were set on each device and refuses (cudaErrorInvalidValue) the launch of
 * one that was not opted in on the current device. */
#include <stdlib.h>

enum { kDevices = 2, kMax = 64 };
static const int kSms[kDevices] = {152, 80};
int fake_device = 0;              /* the current device                     */
unsigned fake_grid = 0;           /* CTAs of the last launch                */
static const void* opted[kDevices][kMax];
static int n_opted[kDevices];

int cudaGetDevice(int* dev) { *dev = fake_device; return 0; }
int cudaDeviceGetAttribute(int* v, int attr, int dev) { (void)attr; *v = kSms[dev]; return 0; }
int cudaGetLastError(void) { return 0; }
int cudaFuncSetAttribute(const void* f, int attr, int v) {
  (void)attr; (void)v;
  if (n_opted[fake_device] == kMax) abort();
  opted[fake_device][n_opted[fake_device]++] = f;
  return 0;
}
/* cfg begins with the grid's three extents */
int cudaLaunchKernelExC(const void* cfg, const void* f, void** args) {
  (void)args;
  fake_grid = *(const unsigned*)cfg;
  for (int i = 0; i < n_opted[fake_device]; ++i)
    if (opted[fake_device][i] == f) return 0;
  return 1;
}

/* what the objects' start-up refers to */
int cudaOccupancyMaxActiveClusters(int* n, const void* f, const void* cfg) {
  (void)f; (void)cfg; *n = 0; return 0;
}
void** __cudaRegisterFatBinary(void* p) { static void* h; (void)p; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterFunction(void) {}
void __cudaRegisterVar(void) {}
int __cudaPushCallConfiguration(void) { return 0; }
int __cudaPopCallConfiguration(void) { return 0; }
int __cudaGetKernel(void** k, const void* f) { *k = (void*)f; return 0; }
int __cudaLaunchKernel(void) { return 0; }
char __cudaInitModule(void** h) { (void)h; return 1; }
