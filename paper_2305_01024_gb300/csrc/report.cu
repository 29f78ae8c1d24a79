// report.cu -- hands the fault report over to the host (the records of
// Section 4.2.1's events and their counters).
#include "internal.cuh"

namespace ftg {

// The report's header, its first records and a flag (if given) to `out`
// (page-locked host memory), then the counters back to zero.  One small launch in place of a
// copy to pageable memory and two clears, which with the gaps between them
// took 30 us of every call that returns a report.
__global__ void __launch_bounds__(256) report_collect_kernel(DevReport* rep, const ftgemm_fault_record* __restrict__ recs,
                                                             const int* flag, HostReport* out) {
  const DevReport r = *rep;
  const int words = min(min(r.n_records, r.capacity), HostReport::kRecords) * (int)(sizeof(ftgemm_fault_record) / 16);
  const uint4* src = reinterpret_cast<const uint4*>(recs);
  uint4* dst = reinterpret_cast<uint4*>(out->recs);
  for (int i = threadIdx.x; i < words; i += blockDim.x) dst[i] = src[i];
  __syncthreads();  // every thread has read the header
  if (threadIdx.x == 0) {
    out->r = r;
    out->flag = flag ? *flag : 0;
    DevReport z{};
    z.capacity = r.capacity;
    *rep = z;
  }
}

cudaError_t launch_report_collect(DevReport* rep, const ftgemm_fault_record* recs, const int* flag, HostReport* out,
                                  cudaStream_t st) {
  report_collect_kernel<<<1, 256, 0, st>>>(rep, recs, flag, out);
  return cudaGetLastError();
}

}  // namespace ftg
