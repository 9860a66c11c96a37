// ws_multi.cu -- dispatch of the persistent multi-table kernels by menu entry.
#include "ws_multi.cuh"

namespace ws {

cudaError_t launch_multi_0(int kind, const MultiGroup& g, cudaStream_t s, int num_sms);
cudaError_t launch_multi_1(int kind, const MultiGroup& g, cudaStream_t s, int num_sms);
cudaError_t launch_multi_2(int kind, const MultiGroup& g, cudaStream_t s, int num_sms);
cudaError_t launch_multi_3(int kind, const MultiGroup& g, cudaStream_t s, int num_sms);
cudaError_t launch_multi_4(int kind, const MultiGroup& g, cudaStream_t s, int num_sms);
cudaError_t launch_multi_5(int kind, const MultiGroup& g, cudaStream_t s, int num_sms);
cudaError_t launch_multi_6(int kind, const MultiGroup& g, cudaStream_t s, int num_sms);
cudaError_t launch_multi_7(int kind, const MultiGroup& g, cudaStream_t s, int num_sms);

namespace {
__global__ void count_kernel(Counters* ctr, u64* count) {
  const u64 c = ctr->count;
  ctr->live = c;  // as below
  *count = c;
}

__global__ void counts_kernel(const MultiItem* items, u32 n, u64* counts) {
  const u32 i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const u64 c = items[i].tv.ctr->count;
  items[i].tv.ctr->live = c;  // items outside the menu ran as single-table mixed kernels, which do not note it
  counts[i] = c;
}
}  // namespace

cudaError_t launch_counts(const MultiItem* items, u32 n, u64* counts, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  counts_kernel<<<(n + 127) / 128, 128, 0, s>>>(items, n, counts);
  return cudaGetLastError();
}

cudaError_t launch_count(const TableView& tv, u64* count, cudaStream_t s) {
  count_kernel<<<1, 1, 0, s>>>(tv.ctr, count);
  return cudaGetLastError();
}

cudaError_t launch_multi(int cfg, int kind, const MultiGroup& g, cudaStream_t s, int num_sms) {
  switch (cfg) {
    case 0: return launch_multi_0(kind, g, s, num_sms);
    case 1: return launch_multi_1(kind, g, s, num_sms);
    case 2: return launch_multi_2(kind, g, s, num_sms);
    case 3: return launch_multi_3(kind, g, s, num_sms);
    case 4: return launch_multi_4(kind, g, s, num_sms);
    case 5: return launch_multi_5(kind, g, s, num_sms);
    case 6: return launch_multi_6(kind, g, s, num_sms);
    case 7: return launch_multi_7(kind, g, s, num_sms);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ws
