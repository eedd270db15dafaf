// One CTA that polls words whose flag nothing sets, with a small limit: the wait of
// the persistent decode step must give up, report it and make later waits return at once.
#include "persist_wait.cuh"

__global__ void poll_kernel(const uint4* words, PersistGrid* g, int* err, int* out, uint32_t limit) {
  __shared__ int abort_flag;
  volatile int* s_abort = &abort_flag;
  if (threadIdx.x == 0) *s_abort = 0;
  __syncthreads();
  uint4 w[2];
  auto src = [&](int i) { return words + 2 * threadIdx.x + i; };
  poll_vecs<2>(w, src, 0u, g, s_abort, err, limit);  // the zeroed words carry flag 0: no wait
  const int first = *s_abort;
  __syncthreads();
  poll_vecs<2>(w, src, 7u, g, s_abort, err, limit);
  __syncthreads();
  const int second = *s_abort;
  poll_vecs<2>(w, src, 7u, g, s_abort, err, 0xffffffffu);  // no limit of its own: the abort ends it
  if (threadIdx.x == 0) {
    out[0] = first;
    out[1] = second;
    out[2] = static_cast<int>(g->abort);
  }
}

// out: abort seen before and after the wait, the grid's abort word, the error word, the CUDA status.
extern "C" int run_poll(int limit, int* out) {
  const int threads = 64;
  uint4* words = nullptr;
  int* mem = nullptr;  // PersistGrid, error word, results
  cudaError_t e = cudaMalloc(&words, 2 * threads * sizeof(uint4));
  if (e == cudaSuccess) e = cudaMalloc(&mem, 64);
  if (e == cudaSuccess) e = cudaMemset(words, 0, 2 * threads * sizeof(uint4));
  if (e == cudaSuccess) e = cudaMemset(mem, 0, 64);
  if (e == cudaSuccess) {
    poll_kernel<<<1, threads>>>(words, reinterpret_cast<PersistGrid*>(mem), mem + 8, mem + 9, limit);
    e = cudaDeviceSynchronize();
  }
  if (e == cudaSuccess) e = cudaMemcpy(out, mem + 9, 12, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(out + 3, mem + 8, 4, cudaMemcpyDeviceToHost);
  cudaFree(words);
  cudaFree(mem);
  return static_cast<int>(e);
}
