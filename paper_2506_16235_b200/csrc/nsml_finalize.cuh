// What the select kernels share (nsml_list.cuh: the exact top-k of a candidate
// list; nsml_small.cuh: of a bucket in shared memory; nsml_grid.cuh: of most of a
// large bucket): their parameters, the payload header, a survivor's value on its way
// out (Alg. 2 Step 1 "quantize" for fp16), the grid barrier.
//
// The grid select is the only kernel whose blocks meet at grid barriers and have
// to be co-resident (cooperative launch).  Every barrier wait is bounded: when it
// runs out the block records NSML_ERR_TIMEOUT and leaves; the others then time out
// as well.
#pragma once

#include "nsml_codec.cuh"
#include "nsml_common.cuh"
#include "nsml_compact.cuh"
#include "nsml_select.cuh"

namespace nsml {

struct FinalizeParams {
  unsigned long long n, k;
  int bits;
  Ctl* ctl;
  unsigned int* hist;                // [4][kMaxBins]
  unsigned int tiles;
  TileList list;
  float* raw_val;
  float* residual;                   // local accumulation in one call: holds gradient + residual; what the payload carries is taken out
  unsigned char* payload;
  PayloadLayout P;
};

// All blocks arrive, then all leave.  `target` = barrier ordinal * gridDim.x.
// SH: any shared-memory struct with an int member `ok`.  max_polls: polls after which the wait gives up.
template <class SH>
__device__ __forceinline__ bool grid_barrier(Ctl* ctl, unsigned int target, SH& sh, int max_polls = kMaxPolls) {
  __syncthreads();
  if (threadIdx.x == 0) {
    // Arrive with release, wait with acquire (both at device scope): what the block wrote before the
    // __syncthreads above is visible to every block that leaves the wait, without full fences.
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(&ctl->barrier), "r"(1u) : "memory");
    int ok = 1, polls = 0;
    for (;;) {
      unsigned int seen;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&ctl->barrier) : "memory");
      if (seen >= target) break;
      if (++polls > max_polls) { ok = 0; break; }
      if (polls > 256) __nanosleep(64);
    }
    if (!ok) set_status(&ctl->status, NSML_ERR_TIMEOUT);
    sh.ok = ok;
  }
  __syncthreads();
  return sh.ok != 0;
}

// Self-test of the bounded wait: every block arrives once at a barrier whose target is one arrival more
// than the grid can deliver, so each wait runs out after max_polls polls, the status word becomes
// NSML_ERR_TIMEOUT and the kernel returns by itself.
struct BarrierProbeShared { int ok; };
static __global__ void __launch_bounds__(32) k_barrier_probe(Ctl* ctl, int max_polls) {
  __shared__ BarrierProbeShared sh;
  grid_barrier(ctl, gridDim.x + 1u, sh, max_polls);
}

// Clears the control block and the histograms of a workspace (what the sample
// kernel does on the list path) ahead of the grid select.
static __global__ void __launch_bounds__(kCta) k_clear(uint4* __restrict__ region, unsigned int count16, int keep_status) {
  pdl_wait();
  pdl_launch_dependents();
  for (unsigned int i = blockIdx.x * kCta + threadIdx.x; i < count16; i += gridDim.x * kCta)
    region[i] = make_uint4((i == 0 && keep_status) ? reinterpret_cast<const unsigned int*>(region)[0] : 0u, 0u, 0u, 0u);
}

__device__ __forceinline__ void write_header(const FinalizeParams& p) {
  nsml_payload_header h;
  h.magic = NSML_PAYLOAD_MAGIC;
  h.version = NSML_PAYLOAD_VERSION;
  h.n = p.n;
  h.k = p.k;
  h.bits = (uint32_t)p.bits;
  h.qblock = NSML_QBLOCK;
  h.nblocks = p.P.nblocks;
  h.idx_off = p.P.idx_off;
  h.val_off = p.P.val_off;
  h.scale_off = p.P.scale_off;
  *reinterpret_cast<nsml_payload_header*>(p.payload) = h;
}

// A survivor's value on its way out: float32 and fp16 values go straight to their payload position (Alg. 2
// Step 1 "quantize" for fp16); int8 values are parked in raw_val until their block of 1024 is complete.
__device__ __forceinline__ void put_value(const FinalizeParams& p, unsigned long long pos, uint32_t bits) {
  if (p.bits == NSML_BITS_FP32) reinterpret_cast<uint32_t*>(p.payload + p.P.val_off)[pos] = bits;
  else if (p.bits == NSML_BITS_FP16) reinterpret_cast<uint16_t*>(p.payload + p.P.val_off)[pos] = encode_f16(__uint_as_float(bits));
  else p.raw_val[pos] = __uint_as_float(bits);
}
// What a receiver reconstructs of a float32 or fp16 value, taken out of it (one float32 subtraction).  Callers leave
// out +0.0 only: there nothing changes, and it may stand for a pruned parameter, whose sum in the residual stays.
// -0.0 is a sum like any other and leaves -0.0 - (-0.0) = +0.0.
__device__ __forceinline__ float not_carried(const FinalizeParams& p, uint32_t bits) {
  const float v = __uint_as_float(bits);
  return __fsub_rn(v, p.bits == NSML_BITS_FP32 ? v : decode_f16(encode_f16(v)));
}

}  // namespace nsml
