// corr_static.cu -- corr_xcorr_static: one block's visibilities with no
// allocation at all.
//
// Some callers of this library cannot allocate device memory: code that runs
// inside a framework which owns the whole device memory pool (an allocation
// outside that pool can exceed its budget), and code on a real-time path where
// the implicit synchronisation of cudaMalloc/cudaFree would stall work already
// queued on the device.  For them this entry point runs the X-engine kernel on
// one block with every piece of scratch memory the kernel needs (its tile
// schedule and its status word) held in a file-scope device array of fixed
// size, and writes the visibilities straight into the caller's buffer.  It
// calls no cudaMalloc, cudaFree or other allocating routine, on the device or
// on the host.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include "corr.h"
#include "xe_internal.h"
#include "xe_sched.h"

namespace {

// The scratch: [status word, padded to 256 bytes][problem descriptor,
// padded to 128 bytes][tile schedule].
static __device__ __align__(256) unsigned char g_static_scratch[CORR_STATIC_SCRATCH_BYTES];

constexpr int kStatusBytes = 256;
constexpr int kProbBytes = 128;
static_assert(sizeof(xe::XProb) <= kProbBytes, "problem descriptor slot");
constexpr int kMaxStaticUnits =
    (CORR_STATIC_SCRATCH_BYTES - kStatusBytes - kProbBytes) / (int)sizeof(xe::XUnit);
static_assert(kMaxStaticUnits >= 4, "scratch must hold the schedule of up to 256 inputs");

constexpr int kMaxDevices = 64;
std::mutex g_setup_mutex;
unsigned char *g_scratch_addr[kMaxDevices];  // device address of the array, per device
int g_smem_optin[kMaxDevices];
int g_n_sm[kMaxDevices];
unsigned long long g_timeout_ns = 2000000000ull;  // device-side wait limit (CORR_TIMEOUT_MS)

// The schedule and problem descriptor of one call, passed by value in the
// parameters of the set-up kernel below (so nothing is copied from host
// memory, which a captured copy would read again at replay).
constexpr int kMaxCallUnits = xe::kMaxWindowUnits;
struct StaticPlan {
  xe::XProb prob;
  xe::XUnit units[kMaxCallUnits];
  int n_units;
};

// Writes the call's problem descriptor and schedule into the scratch array
// and clears the status word.  One block; the X-engine launch that follows on
// the same stream reads them.
__global__ void static_setup_kernel(const __grid_constant__ StaticPlan plan, xe::XProb *d_prob,
                                    xe::XUnit *d_units, int *d_status) {
  static_assert(sizeof(xe::XUnit) % 4 == 0 && sizeof(xe::XProb) % 4 == 0, "word copies");
  const uint32_t *src = reinterpret_cast<const uint32_t *>(plan.units);
  uint32_t *dst = reinterpret_cast<uint32_t *>(d_units);
  const int n_words = plan.n_units * (int)(sizeof(xe::XUnit) / 4);
  for (int k = threadIdx.x; k < n_words; k += blockDim.x) dst[k] = src[k];
  const uint32_t *ps = reinterpret_cast<const uint32_t *>(&plan.prob);
  uint32_t *pd = reinterpret_cast<uint32_t *>(d_prob);
  for (int k = threadIdx.x; k < (int)(sizeof(xe::XProb) / 4); k += blockDim.x) pd[k] = ps[k];
  if (threadIdx.x == 0) *d_status = 0;
}

int rc_of(cudaError_t e) { return e == cudaSuccess ? CORR_OK : CORR_ECUDA; }

// Once per device, with that device current: resolve the array's device
// address (in host code the array's name is only a host-side stand-in) and
// the limits the launch needs.
int setup_device(int dev) {
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  if (g_scratch_addr[dev]) return CORR_OK;
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) return CORR_ECUDA;
  if (prop.major != 10 || prop.minor != 3) return CORR_EARCH;
  int optin = 0;
  if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return CORR_ECUDA;
  void *addr = nullptr;
  if (cudaGetSymbolAddress(&addr, g_static_scratch) != cudaSuccess || !addr) return CORR_ECUDA;
  if (const char *env = std::getenv("CORR_TIMEOUT_MS")) {
    const long long ms = std::atoll(env);
    if (ms > 0) g_timeout_ns = (unsigned long long)ms * 1000000ull;
  }
  // the kernels' shared-memory limit, which stays set (in every call, nine
  // instances took 2.9 of 14.6 us of host time)
  if (xe::cmac_set_smem(optin) != cudaSuccess) return CORR_ECUDA;
  g_smem_optin[dev] = optin;
  g_n_sm[dev] = prop.multiProcessorCount;
  g_scratch_addr[dev] = static_cast<unsigned char *>(addr);
  return CORR_OK;
}

}  // namespace

extern "C" int corr_xcorr_static(const uint8_t *d_block, int n_ant, int n_pol, int n_chan,
                                 int block_len, int64_t *d_vis, void *stream) {
  if (!d_block || !d_vis || n_ant <= 0 || n_chan <= 0 || block_len <= 0 ||
      (n_pol != 1 && n_pol != 2))
    return CORR_EINVAL;
  const long long N = (long long)n_ant * n_pol;
  if (N > CORR_STATIC_MAX_INPUTS || block_len > CORR_STATIC_MAX_BLOCK_LEN || block_len % 16 != 0)
    return CORR_EINVAL;
  if ((reinterpret_cast<uintptr_t>(d_block) & 15u) || (reinterpret_cast<uintptr_t>(d_vis) & 15u))
    return CORR_EINVAL;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return CORR_ECUDA;
  if (dev < 0 || dev >= kMaxDevices) return CORR_EINVAL;
  int rc = setup_device(dev);
  if (rc != CORR_OK) return rc;

  StaticPlan plan;
  std::memset(&plan, 0, sizeof(plan));
  xe::XUnit *units = plan.units;
  int n_tpl = xe::window_units((int)N, units);
  // Where even every stage of every unit on an SM of its own leaves more than
  // half of them idle, units of one tile: a unit's tiles are folded one after
  // the other (64 inputs, 8 channels: 64 samples 13.1 -> 10.6 us a call, 1024
  // 13.2 -> 10.6; 5 inputs, 256 channels, 16 samples 9.4 -> 8.5; the one-channel
  // A/Q units of before took 10.1, 17.3 and 8.7).
  const long long stages = (block_len + xe::kPkSamples - 1) / xe::kPkSamples;
  if (2 * stages * xe::channel_units(n_chan, units[0].n_chan) <= g_n_sm[dev])
    n_tpl = xe::window_units((int)N, units, 1);
  if (n_tpl > kMaxStaticUnits) return CORR_EINVAL;
  plan.n_units = n_tpl;
  int max_z = 0, max_pk = 0, max_sum = 0;
  for (int k = 0; k < n_tpl; ++k) {
    max_z = std::max(max_z, units[k].z_rows);
    max_pk = std::max(max_pk, units[k].pk_bytes);
    max_sum = std::max(max_sum, units[k].n_sum);
  }
  const int optin = g_smem_optin[dev];
  xe::StageLayout L;
  if (!xe::stage_layout(max_z, max_pk, max_sum, optin, xe::kMaxZStages, &L)) return CORR_EINVAL;

  cudaStream_t st = static_cast<cudaStream_t>(stream);
  unsigned char *scratch = g_scratch_addr[dev];
  int *d_status = reinterpret_cast<int *>(scratch);
  xe::XProb *d_prob = reinterpret_cast<xe::XProb *>(scratch + kStatusBytes);
  xe::XUnit *d_units = reinterpret_cast<xe::XUnit *>(scratch + kStatusBytes + kProbBytes);
  const size_t vis_bytes = (size_t)n_chan * (size_t)(N * (N + 1) / 2) * 16;
  xe::XProb &prob = plan.prob;
  prob.units = d_units;
  prob.acc = d_vis;
  prob.n_pairs = N * (N + 1) / 2;
  prob.n_in = (int)N;
  prob.n_chan = n_chan;
  prob.chunks_per_block = (block_len + xe::kChunkSamples - 1) / xe::kChunkSamples;
  prob.pk_per_block = (block_len + xe::kPkSamples - 1) / xe::kPkSamples;
  prob.map0 = 0;
  // the scratch keeps the previous call's contents: rewrite the schedule and
  // the problem and clear the status word (a set-up kernel that receives
  // them by value), and start the visibilities, which the X-engine
  // accumulates into, from zero
  static_setup_kernel<<<1, 128, 0, st>>>(plan, d_prob, d_units, d_status);
  if ((rc = rc_of(cudaGetLastError())) != CORR_OK ||
      (rc = rc_of(cudaMemsetAsync(d_vis, 0, vis_bytes, st))) != CORR_OK)
    return rc;

  xe::XMaps maps;
  std::memset(&maps, 0, sizeof(maps));
  const int ch_rows = units[0].seg[0].ch_rows ? units[0].seg[0].ch_rows : xe::kTileInputs;
  if (!xe::encode_block_map(d_block, block_len, (int)N, n_chan, block_len, maps.m[0], ch_rows))
    return CORR_ECUDA;

  xe::XParams p;
  std::memset(&p, 0, sizeof(p));
  p.probs = d_prob;
  p.items = nullptr;  // units (or their fold windows), dealt round-robin over the CTAs
  p.cta_first = nullptr;
  p.implicit_n_tpl = n_tpl;
  p.implicit_chan_step = units[0].n_chan;
  p.implicit_n_chan = xe::channel_units(n_chan, units[0].n_chan);
  p.implicit_npk = prob.pk_per_block;
  // Items per unit: as many as keep every fp32 partial exact, or more where
  // that shortens the modelled run (rounds of items over the SMs, each a piece
  // of the heaviest unit and its fold).
  const long long n_units = (long long)n_tpl * p.implicit_n_chan;
  const int min_seg = (p.implicit_npk + xe::kMaxFoldStages - 1) / xe::kMaxFoldStages;
  long long best = 0;
  for (int seg = min_seg; seg <= std::min(p.implicit_npk, 32 * min_seg); ++seg) {
    const long long rounds = (n_units * seg + g_n_sm[dev] - 1) / g_n_sm[dev];
    const long long piece = (p.implicit_npk + seg - 1) / seg;
    const long long t = rounds * (piece * xe::kChunksPerPk * xe::chunk_cost(units[0]) +
                                  xe::kFold * units[0].work);
    if (seg == min_seg || t < best) best = t, p.implicit_nseg = seg;
  }
  p.status = d_status;
  p.timeout_ns = g_timeout_ns;
  p.z_stages = L.z_stages;
  p.pk_stages = L.pk_stages;
  p.z_stage_bytes = L.z_stage_bytes;
  p.pk_stage_bytes = L.pk_stage_bytes;
  p.sum_rows = L.sum_rows;
  p.gram = units[0].gram;
  const long long n_work = n_units * p.implicit_nseg;
  const int grid = (int)std::min<long long>(n_work, g_n_sm[dev]);
  return rc_of(xe::launch_cmac(maps, p, grid, L.smem_bytes, st));
}
