// Launch accounting and optional per-kernel CUDA-event timing (diagnostics; off by default).
// Launches may come from several host threads; select, reset and read may not run next to them.
#include <string.h>

#include "cvlc_common.cuh"

namespace cvlc {

namespace {
const char* const kKernelNames[kNumKernelIds] = {
    "k_zero_words", "k_client", "k_hist", "k_plan_threshold", "k_plan_fit", "k_plan_tune", "k_encode_init", "k_select", "k_select_lookback", "k_rank_split",
    "k_rank", "k_rank_rest", "k_sort", "k_pack", "k_decode_prepare", "k_fill_zero", "k_prefetch_l2", "k_decode", "k_noalloc_publish_status",
    "k_selftest", "k_hist_check", "k_apply", "k_plan_literal", "k_ec_accumulate", "k_pack_unframed", "k_decode_unframed"};

std::atomic<unsigned long long> g_launches[kNumKernelIds];
std::atomic<int> g_prof_kernel{-1};  // kernel id being timed; kNumKernelIds = every kernel; -1 = off
uint32_t g_prof_capacity = 0;
std::atomic<uint32_t> g_prof_count{0};  // pairs given out; beyond the capacity: launches that found none
cudaEvent_t* g_prof_events = nullptr;  // 2 per timed launch
int* g_prof_ids = nullptr;             // kernel id of every timed launch
}  // namespace

int launch_begin(int id, cudaStream_t st) {
  g_launches[id].fetch_add(1, std::memory_order_relaxed);
  const int timed = g_prof_kernel.load(std::memory_order_relaxed);
  if (timed != id && timed != kNumKernelIds) return -1;
  if (g_prof_count.load(std::memory_order_relaxed) >= g_prof_capacity) return -1;
  const uint32_t pair = g_prof_count.fetch_add(1, std::memory_order_relaxed);
  if (pair >= g_prof_capacity) return -1;
  cudaEventRecord(g_prof_events[2 * pair], st);
  return (int)pair;
}

void launch_end(int id, int pair, cudaStream_t st) {
  if (pair < 0) return;
  cudaEventRecord(g_prof_events[2 * pair + 1], st);
  g_prof_ids[pair] = id;
}

}  // namespace cvlc

using namespace cvlc;

static int kernel_id_of(const char* name) {
  for (int i = 0; i < kNumKernelIds; ++i)
    if (strcmp(name, kKernelNames[i]) == 0) return i;
  return -1;
}

extern "C" {

unsigned long long cvlc_launch_count(const char* kernel_name) {
  unsigned long long total = 0;
  for (int i = 0; i < kNumKernelIds; ++i)
    if (!kernel_name || !kernel_name[0] || strcmp(kernel_name, kKernelNames[i]) == 0) total += g_launches[i].load(std::memory_order_relaxed);
  return total;
}

int cvlc_profile_select(const char* kernel_name, uint32_t max_launches) {
  if (g_prof_events) {
    for (uint32_t i = 0; i < 2 * g_prof_capacity; ++i) cudaEventDestroy(g_prof_events[i]);
    delete[] g_prof_events;
    delete[] g_prof_ids;
    g_prof_events = nullptr;
    g_prof_ids = nullptr;
  }
  g_prof_kernel = -1;
  g_prof_capacity = 0;
  g_prof_count = 0;
  if (!kernel_name || !kernel_name[0] || max_launches == 0) return CVLC_OK;
  const int id = (strcmp(kernel_name, "*") == 0) ? (int)kNumKernelIds : kernel_id_of(kernel_name);
  if (id < 0) return CVLC_ERR_INVALID_ARG;
  g_prof_events = new cudaEvent_t[2 * (size_t)max_launches];
  g_prof_ids = new int[max_launches];
  for (uint32_t i = 0; i < 2 * max_launches; ++i)
    if (cudaEventCreate(&g_prof_events[i]) != cudaSuccess) return CVLC_ERR_CUDA;
  g_prof_capacity = max_launches;
  g_prof_kernel = id;
  return CVLC_OK;
}

int cvlc_profile_reset(void) {
  g_prof_count = 0;
  return CVLC_OK;
}

int cvlc_profile_read(const char* kernel_name, uint32_t* launches, double* total_ms) {
  if (!launches || !total_ms) return CVLC_ERR_INVALID_ARG;
  *launches = 0;
  *total_ms = 0.0;
  const int want = (!kernel_name || !kernel_name[0] || strcmp(kernel_name, "*") == 0) ? -1 : kernel_id_of(kernel_name);
  if (kernel_name && kernel_name[0] && strcmp(kernel_name, "*") != 0 && want < 0) return CVLC_ERR_INVALID_ARG;
  if (cudaDeviceSynchronize() != cudaSuccess) return CVLC_ERR_CUDA;
  const uint32_t taken = g_prof_count < g_prof_capacity ? (uint32_t)g_prof_count : g_prof_capacity;
  for (uint32_t i = 0; i < taken; ++i) {
    if (want >= 0 && g_prof_ids[i] != want) continue;
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, g_prof_events[2 * i], g_prof_events[2 * i + 1]) != cudaSuccess) return CVLC_ERR_CUDA;
    *total_ms += (double)ms;
    *launches += 1;
  }
  return CVLC_OK;
}

}  // extern "C"
