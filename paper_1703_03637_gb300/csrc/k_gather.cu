// Builds the gather tables of gather.cuh on the device, one warp per 32 states.
#include <algorithm>

#include "gather.cuh"

namespace hphi {

namespace {

constexpr int kGtWarps = 4;

// W lanes share one pass over the banks (W entries of 128 / W bytes cover them): 32 for 4-byte
// entries, 16 for 8-byte and 8 for 16-byte ones.  nbr[q * nbr_stride + k] is term q of state k,
// target | phase << shift.  rec[(group * stride + out0 + k) * 4 + slot % 4]; hdr[(out0 + k) / 32].
//
// Lanes choose one after another, so a choice is made by the W lanes together: each weighs a share of
// the chooser's terms, and lane b of a pass keeps the state of bank b.  The lists (cap terms a lane) lie
// in shared memory, term by term across the lanes.  Bound by the latency of the choices; 12,870
// states of the 16-site Hubbard cluster: 107 us instead of 171 us with every lane searching its own list.
template <int W>
__global__ void __launch_bounds__(kGtWarps * 32) k_gather_table(const uint32_t* __restrict__ nbr, int64_t nbr_stride,
                                                                const uint8_t* __restrict__ deg, int n, int shift,
                                                                int n_phase, uint32_t zero0, uint16_t* __restrict__ rec,
                                                                int64_t stride, int64_t out0, int max_slots, int cap,
                                                                uint4* __restrict__ hdr) {
  extern __shared__ uint16_t s_list[];  // [kGtWarps][cap][32]
  __shared__ int s_load[kGtWarps][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t k0 = ((int64_t)blockIdx.x * kGtWarps + wid) * 32;
  if (k0 >= n) return;  // the whole warp
  const int64_t k = k0 + lane;
  const int g0 = (lane / W) * W, me = lane % W;  // this lane's bank pass and its place there
  constexpr unsigned kGroup = W == 32 ? 0xffffffffu : (1u << W) - 1u;
  int* load = s_load[wid] + g0;
  uint16_t* list = s_list + (size_t)wid * cap * 32;  // term c of lane l at list[c * 32 + l]
  const int d = k < n ? min((int)deg[k], cap) : 0;
  const uint32_t mask = (1u << shift) - 1u;
  int base = 0;
  uint32_t ends[kGatherPhases];
  for (int f = 0; f < kGatherPhases; ++f) {
    if (f < n_phase) {
      int cnt = 0;
      for (int q = 0; q < d; ++q) {
        const uint32_t e = nbr[q * nbr_stride + k];
        if ((int)(e >> shift) == f) list[(cnt++) * 32 + lane] = (uint16_t)(e & mask);
      }
      s_load[wid][lane] = 0;
      __syncwarp();
      for (int i = 0; i < cnt; ++i) atomicAdd(&load[list[i * 32 + lane] % W], 1);
      __syncwarp();  // all lanes' terms are counted
      const int m = __reduce_max_sync(0xffffffffu, cnt);
      int useb, loadb = s_load[wid][lane];  // bank `me` of this bank pass: uses in the slot, terms left
      for (int q = 0; q < m; ++q) {
        useb = 0;
        const int left = m - q;
        int mine = -1;
        // lanes that have a term for every slot left choose first, one lane of a pass at a time
        for (int sweep = 0; sweep < 2; ++sweep) {
          const unsigned all = __ballot_sync(0xffffffffu, mine < 0 && cnt > 0 && (sweep == 1 || cnt >= left));
          const unsigned grp = (all >> g0) & kGroup;
          const int rot = q % W;  // the order starts at a lane that moves with the slot
          unsigned todo = rot ? ((grp >> rot) | (grp << (W - rot))) & kGroup : grp;
          while (__any_sync(0xffffffffu, todo != 0u)) {
            const bool some = todo != 0u;
            const int o = some ? (__ffs(todo) - 1 + rot) % W : me;  // the chooser's place
            todo &= todo - 1u;
            int ocnt = __shfl_sync(0xffffffffu, cnt, g0 + o);
            if (!some) ocnt = 0;
            int key = 0x7fffffff, cx = 0;  // demand of the bank, then the term's place: the first best one
#pragma unroll 4
            for (int c0 = 0; c0 < left; c0 += W) {  // (no lane has more than `left` terms)
              const int c = c0 + me;
              const int x = c < ocnt ? list[c * 32 + g0 + o] : 0;
              const int v = __shfl_sync(0xffffffffu, useb * 4096 - loadb, g0 + x % W);
              const int kk = c < ocnt ? v * 256 + c : 0x7fffffff;
              if (kk < key) {
                key = kk;
                cx = x;
              }
            }
            int best = key;
            if constexpr (W == 32) {
              best = __reduce_min_sync(0xffffffffu, key);
            } else {
#pragma unroll
              for (int off = W / 2; off > 0; off >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, off));
            }
            const int x = __shfl_sync(0xffffffffu, cx, g0 + (best & (W - 1)));
            const int ub = __shfl_sync(0xffffffffu, useb, g0 + x % W);
            if (some && (ocnt >= left || ub == 0)) {
              if (me == x % W) {
                useb += 1;
                loadb -= 1;
              }
              if (me == o) {
                mine = x;
                --cnt;
                list[(best & 255) * 32 + lane] = list[cnt * 32 + lane];
              }
            }
            __syncwarp();
          }
        }
        const unsigned used = (__ballot_sync(0xffffffffu, useb != 0) >> g0) & kGroup;
        if (mine < 0) {  // a zero entry in an unused bank (one exists: this lane uses none)
          const int b = used == kGroup ? W - 1 : __ffs(~used) - 1;
          mine = (int)zero0 + (int)((uint32_t)(b - (int)zero0) % W);
        }
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

Status build_gather_table(const uint32_t* nbr, int64_t nbr_stride, const uint8_t* deg, int max_deg, int n, int shift,
                          int n_phase, int zero0, int entry_bytes, uint2* rec, int64_t stride, int64_t out0, int max_slots,
                          uint4* hdr, cudaStream_t st) {
  if (n <= 0) return {};
  max_deg = std::max(1, std::min(max_deg, 255));
  const int g = (n + 32 * kGtWarps - 1) / (32 * kGtWarps);
  uint16_t* r = reinterpret_cast<uint16_t*>(rec);
  const size_t smem = sizeof(uint16_t) * kGtWarps * 32 * (size_t)max_deg;
#define HPHI_GT(WW)                                                                                                 \
  HPHI_CUDA_TRY(cudaFuncSetAttribute(k_gather_table<WW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));  \
  k_gather_table<WW><<<g, kGtWarps * 32, smem, st>>>(nbr, nbr_stride, deg, n, shift, n_phase, (uint32_t)zero0, r,    \
                                                     stride, out0, max_slots, max_deg, hdr)
  switch (gather_lanes(entry_bytes)) {
    case 32: {
      HPHI_GT(32);
      break;
    }
    case 16: {
      HPHI_GT(16);
      break;
    }
    default: {
      HPHI_GT(8);
    }
  }
#undef HPHI_GT
  HPHI_CUDA_TRY(cudaGetLastError());
  return {};
}

}  // namespace hphi
