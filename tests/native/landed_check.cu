// Check of wait_landed, the wait for copies in flight at a CTA's end, on the GPU:
// with the abort flag set (where wait_phase returns at once) it waits for a bulk
// copy, whose bytes are then all there; on a barrier that nothing completes it
// gives up after its limit and records the timeout.  Prints "ok" and exits 0.
#include <cstdio>
#include <vector>

#include "tc_common.cuh"

using namespace symctr;

constexpr int kPieces = 6, kPiece = 16384, kBytes = kPieces * kPiece;

__global__ void check_kernel(const uint32_t* src, uint32_t* out, unsigned* res) {
  extern __shared__ __align__(128) uint8_t buf[];
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ Ctl ctl;
  if (threadIdx.x == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    ctl.abort = 1;
    ctl.err = res + 2;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(&bars[0], kBytes);
    for (int i = 0; i < kPieces; ++i)
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
              su32(buf + i * kPiece)),
          "l"((const uint8_t*)src + i * kPiece), "r"(kPiece), "r"(su32(&bars[0]))
          : "memory");
    res[0] = wait_landed(&bars[0], 0, &ctl) ? 1 : 0;
    if (!res[0]) wait_landed(&bars[0], 0, &ctl);
  }
  __syncthreads();
  if (mbar_test(&bars[0], 0))
    for (int i = threadIdx.x; i < kBytes / 4; i += blockDim.x) out[i] = ((const uint32_t*)buf)[i];
  if (threadIdx.x == 0) {
    res[3] = res[2];
    res[1] = wait_landed(&bars[1], 0, &ctl, 2000000) ? 1 : 0;
  }
}

int main() {
  std::vector<uint32_t> want(kBytes / 4), got(kBytes / 4);
  for (size_t i = 0; i < want.size(); ++i) want[i] = (uint32_t)(i * 2654435761u + 1);
  uint32_t *src = nullptr, *out = nullptr;
  unsigned* res = nullptr;
  unsigned r[4] = {};
  cudaError_t e = cudaMalloc(&src, kBytes);
  if (e == cudaSuccess) e = cudaMalloc(&out, kBytes);
  if (e == cudaSuccess) e = cudaMalloc(&res, sizeof(r));
  if (e == cudaSuccess) e = cudaMemset(out, 0, kBytes);
  if (e == cudaSuccess) e = cudaMemset(res, 0, sizeof(r));
  if (e == cudaSuccess) e = cudaMemcpy(src, want.data(), kBytes, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(check_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBytes);
  if (e == cudaSuccess) {
    check_kernel<<<1, 128, kBytes>>>(src, out, res);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(got.data(), out, kBytes, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(r, res, sizeof(r), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) {
    std::printf("%s\n", cudaGetErrorString(e));
    return 1;
  }
  const bool ok = r[0] == 1 && r[1] == 0 && r[2] == DEVERR_TIMEOUT && r[3] == 0 && got == want;
  std::printf(ok ? "ok\n" : "landed %u, unfinished %u, error words %u %u, data %d\n", r[0], r[1], r[2], r[3],
              (int)(got == want));
  return ok ? 0 : 1;
}
