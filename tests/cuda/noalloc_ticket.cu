// The allocation-free residual with its arrival count in reach: a test sets
// what a call that overlapped another may have left in it.
#include "noalloc.cu"

extern "C" int noalloc_add_arrivals(int k) {
  NoAllocScratch s;
  if (cudaDeviceSynchronize() || cudaMemcpyFromSymbol(&s, g_noalloc, sizeof(s))) return 1;
  s.ticket += k;
  return cudaMemcpyToSymbol(g_noalloc, &s, sizeof(s)) != cudaSuccess;
}
