// c2t_row_argmax_static: the arg-max pass with its scratch memory in a fixed device array of
// this library, for callers that cannot allocate device memory.  See include/c2t.h.
#include <mutex>

#include "c2t_internal.h"

namespace c2t {
namespace {

constexpr int kStaticMaxRows = C2T_STATIC_MAX_ROWS;
constexpr int kStaticMaxVocab = C2T_STATIC_MAX_VOCAB;
constexpr int kMaxDevices = 64;

// What the CTAs of a call leave for the one that finishes last.
struct StaticScratch {
  ArgmaxPieces pieces[kMaxArgmaxCtas];
  unsigned ticket;                                            // 0 between calls (and when the library is loaded)
};

// The scratch itself.  Every GPU that loads the library holds these 8 KB until the process exits.
static __device__ __align__(256) unsigned char g_static_scratch[sizeof(StaticScratch)];

// Host side: the array's name is only a handle here; the device address comes from
// cudaGetSymbolAddress, once per device, with that device current.
struct PerDevice {
  StaticScratch *scratch = nullptr;
  int grid = 0;
};
PerDevice g_dev[kMaxDevices];
std::mutex g_dev_mutex;

}  // namespace
}  // namespace c2t

using namespace c2t;

extern "C" int c2t_row_argmax_static(const void *logits_dev, int32_t rows, int32_t vocab, int32_t dtype,
                                     int64_t row_stride, int32_t *argmax_dev, void *stream) {
  if (!logits_dev || !argmax_dev || rows < 1 || vocab < 1) return C2T_EINVAL;
  if (dtype != C2T_F32 && dtype != C2T_BF16) return C2T_EINVAL;
  if (rows > kStaticMaxRows || vocab > kStaticMaxVocab) return C2T_ERANGE;   // beyond the fixed scratch
  if (row_stride < vocab) return C2T_EINVAL;
  const int eb = dtype == C2T_BF16 ? 2 : 4;
  if ((reinterpret_cast<uintptr_t>(logits_dev) & 15) || (row_stride * eb) % 16) return C2T_EALIGN;

  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { cudaGetLastError(); return C2T_ECUDA; }
  PerDevice pd;
  {
    std::lock_guard<std::mutex> lock(g_dev_mutex);
    if (!g_dev[dev].scratch) {   // first call on this device: look the array's device address up
      void *ptr = nullptr;
      int sms = 0;
      if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || !ptr ||
          cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
        cudaGetLastError();
        return C2T_ECUDA;
      }
      g_dev[dev].scratch = static_cast<StaticScratch *>(ptr);
      g_dev[dev].grid = sms * kPassCtasPerSm < kMaxArgmaxCtas ? sms * kPassCtasPerSm : kMaxArgmaxCtas;
    }
    pd = g_dev[dev];
  }

  if (launch_row_argmax(logits_dev, row_stride, rows, vocab, dtype, pd.scratch->pieces, &pd.scratch->ticket, argmax_dev,
                        pd.grid, (cudaStream_t)stream) != cudaSuccess)
    return C2T_ECUDA;                                         // (address arithmetic on device pointers, never dereferenced here)
  return C2T_OK;
}
