// The same for the wide tensor-core pass (D <= 256, K <= 4,096).
#include "../../paper_1309_0215_gb300/csrc/k_kmeans_wide.cu"

namespace mrgb {
cudaError_t kt_begin(KTimer*, cudaStream_t) { return cudaSuccess; }
cudaError_t kt_end(KTimer*, cudaStream_t) { return cudaSuccess; }
}  // namespace mrgb

namespace {
__global__ void put_operands(const float* c, uint32_t d, uint32_t k, uint8_t* bop) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < k * d) mrgb::tc::put_operand(bop, d, i / d, i % d, c[i]);
}
}  // namespace

extern "C" uint64_t km_wide_operands(uint32_t d, uint32_t k) { return mrgb::km_wide_operand_bytes(d, k); }

// bop: km_wide_operands bytes, cleared; zeros: 4,096 of them; the rest as for km_tc_sums,
// sums: [tiles 128][chunks 256].
extern "C" int km_wide_sums(const float* x, uint32_t n, uint32_t d, const float* c, uint32_t k, const float* zeros,
                            uint8_t* bop, uint32_t* work, float* sums) {
  using namespace mrgb;
  DevInfo di;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&di.smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = allow_smem<km_wide_assign_kernel<true>>(di);
  if (e != cudaSuccess) return (int)e;
  put_operands<<<(k * d + 255) / 256, 256>>>(c, d, k, bop);
  if ((e = cudaGetLastError()) != cudaSuccess) return (int)e;
  const uint32_t tiles = (n + TM - 1) / TM;
  return (int)launch_pdl(km_wide_assign_kernel<true>, dim3(tiles < 100 ? tiles : 100), dim3(WD_THREADS), wide_smem(k),
                         (cudaStream_t) nullptr, x, n, d, k, (const uint8_t*)bop, zeros, zeros,
                         reinterpret_cast<const unsigned int*>(zeros), work + 16, (uint32_t*)nullptr, work + 16 + n,
                         work, reinterpret_cast<KmFew*>(work + 16 + 2 * n), work + 1,
                         reinterpret_cast<unsigned long long*>(work + 2), sums, pipe::SPIN_LIMIT,
                         (unsigned int*)nullptr);
}
