// FP32 row passes in a second CTA shape: 256 threads x 8 values per line
// instead of 128 x 16 (the same lines per CTA, so the same grids, shared
// memory and partial-sum counts), radix-8 stages instead of radix-16.  Half
// the values per thread shortens each CTA's dependent chain, which pays on
// grids of up to two CTAs per SM and costs on larger ones; rows_w8 (chain.cuh)
// holds the rule and its measurements, fl_plan_autotune may ask for this one
// throughout.  64 registers, four CTAs per SM (at two it cost twice as much on
// full grids).  Compiled apart from ops.cu so that the two build in parallel.
#include "chain.cuh"

namespace fl {

void launch_rows_fwd_w8(const RowsFwdArgs<float>& a, int grid, size_t smem, cudaStream_t s) {
  pdl_launch(k_rows_fwd<float, kRowsW8Threads, 8>, grid, kRowsW8Threads, smem, s, a);
}

void launch_rows_inv_w8(const RowsInvArgs<float>& a, int grid, size_t smem, cudaStream_t s) {
  pdl_launch(k_rows_inv<float, kRowsW8Threads, 8>, grid, kRowsW8Threads, smem, s, a);
}

void launch_dst_rows_w8(const DstRowsArgs<float>& a, int grid, size_t smem, cudaStream_t s) {
  pdl_launch(a.odd ? k_dst_rows_odd<float, kRowsW8Threads, 8>
             : a.perm ? k_dst_rows_prime<float, kRowsW8Threads, 8> : k_dst_rows<float, kRowsW8Threads, 8>,
             grid, kRowsW8Threads, smem, s, a);
}

cudaError_t configure_rows_w8() {
  cudaError_t e = cudaSuccess;
  for (const void* f : {reinterpret_cast<const void*>(&k_rows_fwd<float, kRowsW8Threads, 8>),
                        reinterpret_cast<const void*>(&k_rows_inv<float, kRowsW8Threads, 8>),
                        reinterpret_cast<const void*>(&k_dst_rows<float, kRowsW8Threads, 8>),
                        reinterpret_cast<const void*>(&k_dst_rows_odd<float, kRowsW8Threads, 8>),
                        reinterpret_cast<const void*>(&k_dst_rows_prime<float, kRowsW8Threads, 8>)}) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout,
                               cudaSharedmemCarveoutMaxShared);
  }
  return e;
}

}  // namespace fl
