// The sums of the tensor-core distance pass for D <= 64, K <= 256, as the pass
// itself forms them (its kernel with SUMS on): what the error bound charges.
#include "../../paper_1309_0215_gb300/csrc/k_kmeans_tc.cu"

namespace mrgb {
cudaError_t kt_begin(KTimer*, cudaStream_t) { return cudaSuccess; }
cudaError_t kt_end(KTimer*, cudaStream_t) { return cudaSuccess; }
}  // namespace mrgb

// zeros: 1,024 of them; work: 5 n + 16 words, cleared; sums: [tiles 128][256].
// All device memory, on the legacy stream.
extern "C" int km_tc_sums(const float* x, uint32_t n, uint32_t d, const float* c, uint32_t k, const float* zeros,
                          uint32_t* work, float* sums, int terms) {
  using namespace mrgb;
  const uint32_t tiles = (n + tc::TM - 1) / tc::TM;
  auto launch = terms == 1 ? launch_km_tc_kernel<1, true> : launch_km_tc_kernel<3, true>;
  return (int)launch(x, n, d, c, k, zeros, zeros, reinterpret_cast<const unsigned int*>(zeros), work + 16, nullptr,
                     work + 16 + n, work, reinterpret_cast<KmFew*>(work + 16 + 2 * n), work + 1,
                     reinterpret_cast<unsigned long long*>(work + 2), sums, (int)(tiles < 100 ? tiles : 100), nullptr,
                     pipe::SPIN_LIMIT, 0, nullptr, nullptr, nullptr, KmBounds{});
}
