// Builds the gather tables of gather.cuh on the device, one warp per 32 states.
#include "gather.cuh"

namespace hphi {

namespace {

constexpr int kGtWarps = 4;
constexpr int kGtMaxDeg = 256;

// W lanes share one pass over the banks (W entries of 128 / W bytes cover them): 32 for 4-byte
// entries, 16 for 8-byte and 8 for 16-byte ones.  nbr[q * nbr_stride + k] is term q of state k,
// target | phase << shift.  rec[(group * stride + out0 + k) * 4 + slot % 4]; hdr[(out0 + k) / 32].
template <int W>
__global__ void __launch_bounds__(kGtWarps * 32) k_gather_table(const uint32_t* __restrict__ nbr, int64_t nbr_stride,
                                                                const uint8_t* __restrict__ deg, int n, int shift,
                                                                int n_phase, uint32_t zero0, uint16_t* __restrict__ rec,
                                                                int64_t stride, int64_t out0, int max_slots,
                                                                uint4* __restrict__ hdr) {
  __shared__ int s_use[kGtWarps][32], s_load[kGtWarps][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t k0 = ((int64_t)blockIdx.x * kGtWarps + wid) * 32;
  if (k0 >= n) return;  // the whole warp
  const int64_t k = k0 + lane;
  int* use = s_use[wid] + (lane / W) * W;    // of this lane's bank pass
  int* load = s_load[wid] + (lane / W) * W;
  uint16_t list[kGtMaxDeg];
  const int d = k < n ? deg[k] : 0;
  const uint32_t mask = (1u << shift) - 1u;
  int base = 0;
  uint32_t ends[kGatherPhases];
  for (int f = 0; f < kGatherPhases; ++f) {
    if (f < n_phase) {
      int cnt = 0;
      for (int q = 0; q < d; ++q) {
        const uint32_t e = nbr[q * nbr_stride + k];
        if ((int)(e >> shift) == f) list[cnt++] = (uint16_t)(e & mask);
      }
      s_load[wid][lane] = 0;
      __syncwarp();
      for (int i = 0; i < cnt; ++i) atomicAdd(&load[list[i] % W], 1);
      const int m = __reduce_max_sync(0xffffffffu, cnt);
      for (int q = 0; q < m; ++q) {
        s_use[wid][lane] = 0;
        __syncwarp();
        const int left = m - q;
        int mine = -1;
        // lanes that have a term for every slot left choose first, one lane of a pass at a time
        for (int sweep = 0; sweep < 2; ++sweep) {
          for (int i = 0; i < W; ++i) {
            if ((lane % W) == ((i + q) % W) && mine < 0 && cnt > 0 && (sweep == 1 || cnt >= left)) {
              int best = 0, key = 1 << 30;
              for (int c = 0; c < cnt; ++c) {
                const int b = list[c] % W, kk = use[b] * 4096 - load[b];
                if (kk < key) {
                  key = kk;
                  best = c;
                }
              }
              const int b = list[best] % W;
              if (cnt >= left || use[b] == 0) {
                mine = list[best];
                list[best] = list[--cnt];
                use[b] += 1;
                load[b] -= 1;
              }
            }
            __syncwarp();
          }
        }
        if (mine < 0) {  // a zero entry in an unused bank (one exists: this lane uses none)
          int b = 0;
          while (b < W - 1 && use[b] != 0) ++b;
          mine = (int)zero0 + (int)((uint32_t)(b - (int)zero0) % W);
        }
        __syncwarp();
        const int s = base + q;
        if (s < max_slots) rec[((int64_t)(s >> 2) * stride + out0 + k) * 4 + (s & 3)] = (uint16_t)mine;
      }
      base += m;
    }
    ends[f] = (uint32_t)base;
  }
  for (int s = base; s & 3; ++s)
    if (s < max_slots) rec[((int64_t)(s >> 2) * stride + out0 + k) * 4 + (s & 3)] = (uint16_t)zero0;
  if (lane == 0)
    hdr[(out0 + k0) / 32] = make_uint4(ends[0] | (ends[1] << 16), ends[2] | (ends[3] << 16), ends[4] | (ends[5] << 16),
                                       ends[6] | (ends[7] << 16));
}

}  // namespace

Status build_gather_table(const uint32_t* nbr, int64_t nbr_stride, const uint8_t* deg, int n, int shift, int n_phase,
                          int zero0, int entry_bytes, uint2* rec, int64_t stride, int64_t out0, int max_slots,
                          uint4* hdr, cudaStream_t st) {
  if (n <= 0) return {};
  const int g = (n + 32 * kGtWarps - 1) / (32 * kGtWarps);
  uint16_t* r = reinterpret_cast<uint16_t*>(rec);
#define HPHI_GT(WW)                                                                                           \
  k_gather_table<WW><<<g, kGtWarps * 32, 0, st>>>(nbr, nbr_stride, deg, n, shift, n_phase, (uint32_t)zero0, r, \
                                                  stride, out0, max_slots, hdr)
  switch (gather_lanes(entry_bytes)) {
    case 32: HPHI_GT(32); break;
    case 16: HPHI_GT(16); break;
    default: HPHI_GT(8);
  }
#undef HPHI_GT
  HPHI_CUDA_TRY(cudaGetLastError());
  return {};
}

}  // namespace hphi
