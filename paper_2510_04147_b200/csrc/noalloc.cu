// ssd_gemm_bf16_noalloc: the skinny projection GEMM for callers that must not allocate.
//
// Some hosts of this library cannot call cudaMalloc while they run: a serving process that gave the
// whole device to its own memory arena at start-up has nothing left for the driver to hand out, and a
// latency-critical loop cannot afford a call that may block on the device or fail for lack of memory.
// For them a call is ONE kernel launch and a synchronisation: the K splits of a tile are a thread-block cluster that sums
// its parts on chip and writes the result, so there is no scratch memory to clear, share or run out of, and the error
// word is page-locked host memory that the kernel writes through.  (Before: a memset, the projection into a scratch
// array in the library image, a summing kernel and a copy of the error word - 32 us for a call of 8 x 256 x 256, 42 us
// for 77 x 4100 x 3592 in three splits.)
#include "../../include/ssd.h"
#include "error_words.h"
#include "kernels.h"

#include <atomic>
#include <mutex>

namespace {

constexpr size_t kLimitFloats = ((size_t)1 << 20) - 64;      // of split_k * rows * n: the interface's limit
constexpr int kMaxDevices = 64;

// Error words of the calls in flight, one page of this library's own memory, page-locked and mapped on first use.
constexpr int kErrWords = 1024;
alignas(4096) int g_err_words[kErrWords];
ssd::ErrorWords<kErrWords> g_err_loans;

std::mutex g_setup_mutex;
std::atomic<int*> g_err_dev[kMaxDevices] = {};               // the page's address on each device

// resolved on the first call per device
int* err_words_on_current_device() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
  if (int* p = g_err_dev[dev].load(std::memory_order_acquire)) return p;
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  if (int* p = g_err_dev[dev].load(std::memory_order_acquire)) return p;
  if (ssd::gemm_tc_init() != 0) return nullptr;
  static bool registered = false;
  if (!registered) {
    if (cudaHostRegister(g_err_words, sizeof(g_err_words), cudaHostRegisterMapped | cudaHostRegisterPortable) != cudaSuccess) return nullptr;
    registered = true;
  }
  void* p = nullptr;
  if (cudaHostGetDevicePointer(&p, g_err_words, 0) != cudaSuccess) return nullptr;
  g_err_dev[dev].store(reinterpret_cast<int*>(p), std::memory_order_release);
  return reinterpret_cast<int*>(p);
}

}  // namespace

extern "C" int ssd_gemm_bf16_noalloc(const void* x_dev, const void* w_dev, float* out_dev, int32_t rows, int32_t n,
                                     int32_t k, int32_t split_k, void* cuda_stream) {
  if (!x_dev || !w_dev || !out_dev) return SSD_ERR_INVALID_ARG;
  if (rows < 1 || n < 1 || k < 8 || (k % 8) || split_k < 1 || split_k > 8) return SSD_ERR_SHAPE;
  if ((size_t)split_k * (size_t)rows * (size_t)n > kLimitFloats) return SSD_ERR_OVERFLOW;
  int* const err_dev = err_words_on_current_device();
  if (!err_dev) return SSD_ERR_CUDA;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  struct Loan {
    const int slot = g_err_loans.borrow();
    ~Loan() { g_err_loans.give_back(slot); }
  } const loan;
  volatile int* word = g_err_words + loan.slot;
  *word = 0;
  ssd::GemmArgs g{};
  g.x = (const bf16*)x_dev; g.w = (const bf16*)w_dev; g.R = rows; g.N = n; g.K = k; g.x_pitch = k; g.w_pitch = k;
  g.splits = split_k; g.epi = split_k > 1 ? ssd::EPI_SUM : ssd::EPI_PARTIAL; g.out = out_dev; g.err_flag = err_dev + loan.slot;
  g.plain_launch = 1;
  const int rc = ssd::launch_gemm_tc(st, g);
  if (rc != 0) return rc;
  if (cudaStreamSynchronize(st) != cudaSuccess) return SSD_ERR_CUDA;
  return *word ? SSD_ERR_TIMEOUT : SSD_OK;
}
