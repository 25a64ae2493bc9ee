// Backward kernels of libbysdf.
//
// k_backward: per-material parameter gradients.  Each record's forward pass
// is recomputed and differentiated (bysdf_grad.cuh).  KIND: the 8-column basic
// set, the 15-column extended set, or the basic set with the upstream gradient
// of an L2 loss (its value a ninth accumulated column, flushed to the
// per-material loss).
//
// k_dirgrad: the per-record vector-Jacobian products with respect to the
// record's directions; no reduction.
//
// Reduction.  A warp keeps one material's sums in registers, a partial sum
// per lane, and flushes them when the material changes: 16 columns are folded
// across the lanes with 16 shuffles (each step halves the columns a lane
// holds), then one atomic per column.  Material-sorted tiles change material
// rarely.  Records in any order are taken by material within the tile (a
// counting sort across the warp), so that a tile of 512 records of 8
// materials is flushed 8 times; per-record atomics on shared accumulators,
// whose lanes meet in a few addresses, cost more than the gradients.
#include "bysdf_launch.h"

namespace bysdf {

// Sums of each of NP (<= 16) per-lane columns over the warp; lane k returns
// column k's sum (0 for k >= NP).  Step o hands the half of the columns that
// the partner keeps to it, so the steps cost 8, 4, 2, 1 shuffles, and one more
// adds the two lanes that hold the same column.
template <int NP>
__device__ __forceinline__ float warp_columns(const float* acc, int lane) {
  float v[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = k < NP ? acc[k] : 0.f;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    const bool hi = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (k < o) {
        const float give = hi ? v[k] : v[k + o], keep = hi ? v[k + o] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
      }
    }
  }
  const float s = v[0] + __shfl_xor_sync(0xffffffffu, v[0], 16);
  return lane < 16 ? s : 0.f;
}

// Records of a tile in any material order, listed by material (`shift` drops
// low bits of the id when there are more than 32: records of one bucket then
// come in any order, which the flush allows).  Ids out of range are listed
// with material 0 (they contribute nothing).
__device__ __forceinline__ void material_order(const KArgs& a, int64_t begin, int64_t end,
                                               int lane, uint16_t* list, uint32_t* hist) {
  const int count = (int)(end - begin);
  const uint32_t lt = (1u << lane) - 1u;
  int shift = 0;
  while (((a.n_mat - 1) >> shift) >= 32) ++shift;
  auto bucket = [&](int e) {
    int mm = __ldg(a.mat_id + begin + e);
    mm = (mm >= 0 && mm < a.n_mat) ? mm : 0;
    return (uint32_t)(mm >> shift);
  };
  hist[lane] = 0u;
  __syncwarp();
#pragma unroll 1
  for (int e0 = 0; e0 < count; e0 += 32) {
    const int e = e0 + lane;
    const uint32_t b = e < count ? bucket(e) : 32u;
    const uint32_t peers = __match_any_sync(0xffffffffu, b);
    if (b < 32u && lane == __ffs(peers) - 1) hist[b] += (uint32_t)__popc(peers);
    __syncwarp();
  }
  // exclusive scan of the bucket counts (lane = bucket)
  const uint32_t h = hist[lane];
  uint32_t incl = h;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  hist[lane] = incl - h;
  __syncwarp();
#pragma unroll 1
  for (int e0 = 0; e0 < count; e0 += 32) {
    const int e = e0 + lane;
    const uint32_t b = e < count ? bucket(e) : 32u;
    const uint32_t peers = __match_any_sync(0xffffffffu, b);
    const uint32_t base = b < 32u ? hist[b] : 0u;
    __syncwarp();
    if (b < 32u) {
      list[base + (uint32_t)__popc(peers & lt)] = (uint16_t)e;
      if (lane == __ffs(peers) - 1) hist[b] = base + (uint32_t)__popc(peers);
    }
    __syncwarp();
  }
}

template <int BLOCK, int MINB, int KIND>
__global__ void __launch_bounds__(BLOCK, MINB) k_backward(const KArgs a) {
  constexpr int NP = KbCols<KIND>::acc;      // accumulated columns
  constexpr int NG = KbCols<KIND>::grad;     // gradient columns of grad_params
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ uint64_t bars[2 * (BLOCK / 32)];
  // records in any order: per-CTA accumulators behind the tables, then each
  // warp's record list and bucket counts
  float* sacc = reinterpret_cast<float*>(smem + (size_t)a.n_mat * a.sstride);
  const bool any_order = a.mode == MODE_ALL_SMEM;
  if (any_order) {
    for (int k = threadIdx.x; k < a.n_mat * NP; k += BLOCK) sacc[k] = 0.f;
  }
  uint8_t* mine = smem + a.order_off + (threadIdx.x >> 5) * kBwdOrderBytes;
  uint32_t* hist = reinterpret_cast<uint32_t*>(mine);
  uint16_t* list = reinterpret_cast<uint16_t*>(mine + 32 * sizeof(uint32_t));
  const bool listed = any_order && a.mat_id != nullptr && a.n_mat > 1;
  float acc[NP];
#pragma unroll
  for (int k = 0; k < NP; ++k) acc[k] = 0.f;
  int cur = -1;  // the material the sums belong to (-1: none yet)
  auto flush = [&](int lane) {
    if (cur < 0) return;
    const float v = warp_columns<NP>(acc, lane);
#pragma unroll
    for (int k = 0; k < NP; ++k) acc[k] = 0.f;
    if (lane >= NP || v == 0.f) return;
    if (any_order) {
      atomicAdd(&sacc[cur * NP + lane], v);
    } else if (lane < NG) {
      atomicAdd(a.grad_params + (size_t)cur * NG + lane, v);
    } else if (a.loss_mat) {
      atomicAdd(a.loss_mat + cur, v);
    }
  };
  persistent_loop<BLOCK>(a, smem, bars,
                             [&](int64_t begin, int64_t end, int mat, uint8_t* slot, int lane,
                                 int tile) {
    if (listed) material_order(a, begin, end, lane, list, hist);
    if (mat >= 0 && cur != mat) {
      if (!a.partials) flush(lane);
      cur = mat;
    }
    const int count = (int)(end - begin);
    // rolled: one copy of the (large) record body
#pragma unroll 1
    for (int e0 = 0; e0 < count; e0 += 32) {
      const int e = e0 + lane;
      bool active = e < count;
      const int64_t i = begin + (active ? (listed ? (int)list[e] : e) : 0);
      active = active && bounds_ok(i >= 0 && i < a.n);
      int mm = 0;
      float g[NP];
#pragma unroll
      for (int k = 0; k < NP; ++k) g[k] = 0.f;
      if (active) {
        Record q;
        load_record(a, i, true, false, q);
        const uint8_t* tb;
        if (mat >= 0) {
          q.mat = mm = mat;
          tb = slot;
        } else {
          q.mat = a.mat_id ? __ldcg(a.mat_id + i) : 0;
          mm = (q.mat >= 0 && q.mat < a.n_mat) ? q.mat : 0;
          tb = smem + (size_t)mm * a.sstride;
        }
        const MatDev* m = reinterpret_cast<const MatDev*>(tb);
        backward_record<KIND, NP>(a, *m, reinterpret_cast<const float2*>(m + 1), i, q, g);
      }
      if (mat >= 0) {
#pragma unroll
        for (int k = 0; k < NP; ++k) acc[k] += g[k];
        continue;
      }
      // the lanes whose record is of the current material add to its sums;
      // while others are left, the sums are flushed and the next is current
      bool left = active;
      for (;;) {
        const bool add = left && mm == cur;
#pragma unroll
        for (int k = 0; k < NP; ++k) acc[k] += add ? g[k] : 0.f;
        left = left && !add;
        const unsigned rest = __ballot_sync(0xffffffffu, left);
        if (!rest) break;
        flush(lane);
        cur = __shfl_sync(0xffffffffu, mm, __ffs(rest) - 1);
      }
    }
    if (a.partials) {
      // deterministic: this tile's sums, in a fixed order
      const float v = warp_columns<NP>(acc, lane);
      if (lane < NP) a.partials[(size_t)tile * NP + lane] = v;
#pragma unroll
      for (int k = 0; k < NP; ++k) acc[k] = 0.f;
    }
    __syncwarp();  // the list is rewritten by the next tile
  });
  if (!a.partials) flush(threadIdx.x & 31);
  if (any_order) {
    __syncthreads();
    for (int k = threadIdx.x; k < a.n_mat * NP; k += BLOCK) {
      if (sacc[k] == 0.f) continue;
      const int mm = k / NP, c = k - mm * NP;
      if (c < NG) atomicAdd(a.grad_params + (size_t)mm * NG + c, sacc[k]);
      else if (a.loss_mat) atomicAdd(a.loss_mat + mm, sacc[k]);
    }
  }
}

// Fixed-order reduction of per-tile partials: one warp per material sums its
// tiles lane-strided, then a shuffle tree (deterministic for a given launch
// shape).
__global__ void k_reduce_partials(const KArgs a) {
  const int m = blockIdx.x, lane = threadIdx.x;
  const int np = a.n_param;
  const int t0 = a.tile_start[m], t1 = a.tile_start[m + 1];
  float acc[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) acc[k] = 0.f;
  for (int t = t0 + lane; t < t1; t += 32) {
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if (k < np) acc[k] += a.partials[(size_t)t * np + k];
  }
  // gradient columns to grad_params; the L2 backward's loss column to loss_mat
  const int ng = a.target ? np - 1 : np;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    float v = acc[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0 && k < ng) a.grad_params[(size_t)m * ng + k] = v;
    if (lane == 0 && k == ng && k < np && a.loss_mat) a.loss_mat[m] = v;
  }
}

template <int BLOCK, int MINB>
__global__ void __launch_bounds__(BLOCK, MINB) k_dirgrad(const KArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ uint64_t bars[2 * (BLOCK / 32)];
  persistent_loop<BLOCK>(a, smem, bars,
                             [&](int64_t begin, int64_t end, int mat, uint8_t* slot, int lane,
                                 int) {
#pragma unroll 1
    for (int64_t i = begin + lane; i < end; i += 32) {
      if (!bounds_ok(i >= 0 && i < a.n)) continue;
      Record q;
      load_record(a, i, true, false, q);
      const uint8_t* tb;
      if (mat >= 0) {
        q.mat = mat;
        tb = slot;
      } else {
        q.mat = a.mat_id ? __ldcg(a.mat_id + i) : 0;
        const int mm = (q.mat >= 0 && q.mat < a.n_mat) ? q.mat : 0;
        tb = smem + (size_t)mm * a.sstride;
      }
      const MatDev* m = reinterpret_cast<const MatDev*>(tb);
      float g[6];
      backward_record<KB_DIRS, 6>(a, *m, reinterpret_cast<const float2*>(m + 1), i, q, g);
      const int64_t n = a.n;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (a.grad_wi) __stcs(a.grad_wi + c * n + i, g[c]);
        if (a.grad_wo) __stcs(a.grad_wo + c * n + i, g[3 + c]);
      }
    }
  });
}

// occupancy 0: registers as needed (8 warps per SM at 256 threads);
// occupancy 1: at most 128 registers (16 warps per SM; the rest spills).
template <int KIND>
static const void* bwd_fn_t(int block, int occ) {
  switch (block) {
    case 128: return occ ? (const void*)k_backward<128, 4, KIND> : (const void*)k_backward<128, 1, KIND>;
    case 256: return occ ? (const void*)k_backward<256, 2, KIND> : (const void*)k_backward<256, 1, KIND>;
    case 512: return (const void*)k_backward<512, 1, KIND>;
  }
  return nullptr;
}
static const void* bwd_fn(int block, int occ, int kind) {
  switch (kind) {
    case KB_BASIC: return bwd_fn_t<KB_BASIC>(block, occ);
    case KB_EXT: return bwd_fn_t<KB_EXT>(block, occ);
    case KB_L2: return bwd_fn_t<KB_L2>(block, occ);
  }
  return nullptr;
}
static const void* dir_fn(int block) {
  switch (block) {
    case 128: return (const void*)k_dirgrad<128, 1>;
    case 256: return (const void*)k_dirgrad<256, 1>;
    case 512: return (const void*)k_dirgrad<512, 1>;
  }
  return nullptr;
}

cudaError_t set_backward_smem_limit(int block, int occ, int kind, size_t smem, size_t optin) {
  const void* f = bwd_fn(block, occ, kind);
  return f ? raise_smem_limit(f, smem, optin) : cudaErrorInvalidValue;
}

cudaError_t backward_occupancy(int block, int occ, int kind, size_t smem, int* ctas) {
  const void* f = bwd_fn(block, occ, kind);
  if (!f) return cudaErrorInvalidValue;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, f, block, smem);
}

cudaError_t launch_backward(const KArgs& a, int block, int occ, int kind, int grid, size_t smem,
                            cudaStream_t st) {
  const void* f = bwd_fn(block, occ, kind);
  if (!f) return cudaErrorInvalidValue;
  void* args[] = {const_cast<KArgs*>(&a)};
  return cudaLaunchKernel(f, dim3(grid), dim3(block), args, smem, st);
}

cudaError_t launch_reduce_partials(const KArgs& a, cudaStream_t st) {
  k_reduce_partials<<<a.n_mat, 32, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t set_dirgrad_smem_limit(int block, size_t smem, size_t optin) {
  const void* f = dir_fn(block);
  return f ? raise_smem_limit(f, smem, optin) : cudaErrorInvalidValue;
}

cudaError_t dirgrad_occupancy(int block, size_t smem, int* ctas) {
  const void* f = dir_fn(block);
  if (!f) return cudaErrorInvalidValue;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, f, block, smem);
}

cudaError_t launch_dirgrad(const KArgs& a, int block, int grid, size_t smem, cudaStream_t st) {
  const void* f = dir_fn(block);
  if (!f) return cudaErrorInvalidValue;
  void* args[] = {const_cast<KArgs*>(&a)};
  return cudaLaunchKernel(f, dim3(grid), dim3(block), args, smem, st);
}

}  // namespace bysdf
