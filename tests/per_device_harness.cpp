// Host build of csrc/per_device.h with a fake CUDA runtime of several devices
// (test infrastructure of tests/test_per_device.py): the runtime calls below
// stand in for libcudart's and count what each device was asked.
#include "per_device.h"

static int g_device = 0, g_limit_calls[128], g_occ_calls[128], g_fail = 0;

extern "C" cudaError_t cudaGetDevice(int* d) {
  *d = g_device;
  return cudaSuccess;
}
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) {
  ++g_limit_calls[g_device];
  return g_fail ? cudaErrorInvalidValue : cudaSuccess;
}
extern "C" cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
  ++g_occ_calls[g_device];
  *n = g_device % 3;  // another answer on each device, zero among them
  return g_fail ? cudaErrorInvalidValue : cudaSuccess;
}

static PerDevice limit, blocks;
static void kernel(int) {}

extern "C" void set_device(int d) { g_device = d; }
extern "C" void set_fail(int f) { g_fail = f; }
extern "C" int ask_limit() { return hf_smem_limit(limit, &kernel, 60000); }
extern "C" int ask_blocks() { return hf_resident_blocks(blocks, &kernel, 128, 0); }
extern "C" int limit_calls(int d) { return g_limit_calls[d]; }
extern "C" int blocks_calls(int d) { return g_occ_calls[d]; }
