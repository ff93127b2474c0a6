// crmc_state.cu -- the configuration read back in particle-id order, on the
// device (sm_103a): the occupied cell slots are mapped to ids, input particles
// (ids below n_input, dense) are placed by a prefix count over the ids present,
// inserted ions (ids >= 2^32) by their rank among the ion ids (tiles of 1024
// sorted by a CTA each, then every key looked up in every tile; a device-wide
// radix sort past 16,384 ions), and every requested array is written in the
// caller's layout by many CTAs.
//
// Between two reads the id marks (present[]), the counts of their chunks and
// the ion counter are zero: the rank and ordering kernels clear what the mark
// kernel set.
//
// 13 polyelectrolyte boxes (11,000 inserted ions each) into device arrays:
// 377 us with a thread per slot (76), ranks by counting all pairs of keys (251)
// and two CTAs writing (49); now 66 us (16, 21 + 17 and 13).  A box of 87,000
// particles: the marks 38 -> 18 and the writing 202 -> 8 us.
#include <cuda_runtime.h>

#include <cub/device/device_radix_sort.cuh>

#include <algorithm>
#include <cstdint>

#include "crmc_device.cuh"
#include "crmc_kernels.h"

namespace crmc {

namespace {

constexpr int ORDER_THREADS = STATE_CHUNK;  // a thread per id of a chunk
constexpr int RANK_TILE = 1024;  // ion keys per rank-counting tile

// every particle: input ids mark their slot (slot + 1) and count in their
// chunk, inserted ions append (key, slot) to the ion list (one atomic per
// warp); the key keeps the order of the ids: (id >> 32) << lo_bits | (id &
// 0xffffffff), as the low word of an inserted id stays below 2^lo_bits.  One
// warp per 32 cells, a lane per particle.
__device__ __forceinline__ void mark_cells(const SysParams &P, const StateBufs &B, int c) {
  const int lane = threadIdx.x & 31;
  if (c - lane >= P.ncell) return;  // whole warp
  const int n = c < P.ncell ? P.cnt[c] : 0;
  int incl = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  for (int j0 = 0; j0 < total; j0 += 32) {
    const int j = j0 + lane;
    int lo = 0;  // the first of the 32 cells whose inclusive count exceeds j
#pragma unroll
    for (int st = 16; st > 0; st >>= 1) {
      const int v = __shfl_sync(0xffffffffu, incl, lo + st - 1);
      if (v <= j) lo += st;
    }
    lo = min(lo, 31);
    const int before = __shfl_sync(0xffffffffu, incl - n, lo);
    const bool have = j < total;
    const int g = (c - lane + lo) * P.cap + (j - before);
    const unsigned long long id = have ? P.pid[g] : 0ull;
    const bool ion = have && id >= (unsigned long long)B.n_input;
    if (have && !ion) {
      B.present[id] = g + 1;
      atomicAdd(&B.chunk[id / ORDER_THREADS], 1);
    }
    const unsigned m = __ballot_sync(0xffffffffu, ion);
    if (m == 0u) continue;
    const int leader = __ffs(m) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(B.n_ions, __popc(m));
    base = __shfl_sync(0xffffffffu, base, leader);
    const int o = base + __popc(m & ((1u << lane) - 1u));
    if (ion && o < B.cap) {  // (more ions than slots: the host sees the count and reports it)
      B.ion_key[o] = ((id >> 32) << B.lo_bits) | (id & 0xffffffffull);
      B.ion_val[o] = g;
    }
  }
}

__global__ void __launch_bounds__(256) k_state_mark(SysParams P, StateBufs B) {
  mark_cells(P, B, blockIdx.x * blockDim.x + threadIdx.x);
}

// Tile blockIdx.x of the n ion keys sorted in place with its slots by one CTA: a
// bitonic network over the next power of two, padded with the largest key, a
// key per thread (of its 55 steps over 1024 keys the 15 between warps go through
// shared memory, the others are shuffles).  The CTA past the last tile turns the
// chunks' counts into their exclusive prefix sums (chunk_base) and clears them.
__device__ __forceinline__ void sort_tile(const StateBufs &B, int n) {
  __shared__ unsigned long long ks[RANK_TILE];
  __shared__ int vs[RANK_TILE];
  const int t = threadIdx.x;
  if (blockIdx.x == gridDim.x - 1) {
    const int nch = (B.n_input + ORDER_THREADS - 1) / ORDER_THREADS;
    int *sum = vs;
    int carry = 0;
    for (int c0 = 0; c0 < nch; c0 += RANK_TILE) {
      const int v = c0 + t < nch ? B.chunk[c0 + t] : 0;
      sum[t] = v;
      __syncthreads();
      for (int o = 1; o < RANK_TILE; o <<= 1) {
        const int y = t >= o ? sum[t - o] : 0;
        __syncthreads();
        sum[t] += y;
        __syncthreads();
      }
      if (c0 + t < nch) {
        B.chunk_base[c0 + t] = carry + sum[t] - v;
        B.chunk[c0 + t] = 0;
      }
      carry += sum[RANK_TILE - 1];
      __syncthreads();
    }
    return;
  }
  const int i = blockIdx.x * RANK_TILE + t;
  if ((int)blockIdx.x * RANK_TILE >= n) return;  // the whole CTA
  unsigned long long k = i < n ? B.ion_key[i] : ~0ull;
  int v = i < n ? B.ion_val[i] : 0;
  const int m = min(n - (int)blockIdx.x * RANK_TILE, RANK_TILE);  // the tile's keys
  for (int size = 2; size < 2 * m; size <<= 1)
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      unsigned long long k2;
      int v2;
      if (stride >= 32) {
        __syncthreads();
        ks[t] = k;
        vs[t] = v;
        __syncthreads();
        k2 = ks[t ^ stride];
        v2 = vs[t ^ stride];
      } else {
        k2 = __shfl_xor_sync(0xffffffffu, k, stride);
        v2 = __shfl_xor_sync(0xffffffffu, v, stride);
      }
      if (((t & stride) == 0) == ((t & size) == 0) ? k2 < k : k2 > k) {
        k = k2;
        v = v2;
      }
    }
  if (i < n) {
    B.ion_key[i] = k;
    B.ion_val[i] = v;
  }
}

// the slot of each rank among the n ion keys (distinct): CTA x takes the keys
// of tile x, whose rank is the number of smaller keys in every sorted tile
__device__ __forceinline__ void rank_tile(const StateBufs &B, int n) {
  __shared__ unsigned long long ks[RANK_TILE];
  const int t = threadIdx.x, i = blockIdx.x * RANK_TILE + t;
  if ((int)blockIdx.x * RANK_TILE >= n) return;  // the whole CTA
  const unsigned long long k = i < n ? B.ion_key[i] : 0ull;
  int rank = t;  // the smaller keys of its own tile
  for (int j0 = 0; j0 < n; j0 += RANK_TILE) {
    if (j0 == (int)blockIdx.x * RANK_TILE) continue;
    __syncthreads();
    ks[t] = j0 + t < n ? B.ion_key[j0 + t] : ~0ull;
    __syncthreads();
    int lo = 0;  // keys of the tile below k
#pragma unroll
    for (int st = RANK_TILE / 2; st > 0; st >>= 1)
      if (ks[lo + st - 1] < k) lo += st;
    rank += lo + (ks[lo] < k ? 1 : 0);
  }
  if (i < n) B.ion_rank[rank] = B.ion_val[i];
}

__global__ void __launch_bounds__(RANK_TILE) k_ion_sort(StateBufs B, int n) { sort_tile(B, n); }
__global__ void __launch_bounds__(RANK_TILE) k_ion_rank(StateBufs B, int n) { rank_tile(B, n); }
// (in a batch the counter is read from the copy that the sort leaves, so that
// the ordering kernel can clear it for the next read)
__global__ void __launch_bounds__(RANK_TILE) k_ion_sort_batch(const StateBufs *__restrict__ bufs) {
  const StateBufs &B = bufs[blockIdx.y];
  const int n_ions = *B.n_ions;
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *B.n_found = n_ions;
  sort_tile(B, min(n_ions, min(B.cap, STATE_BLOCK_SORT_MAX)));
}
__global__ void __launch_bounds__(RANK_TILE) k_ion_rank_batch(const StateBufs *__restrict__ bufs) {
  const StateBufs &B = bufs[blockIdx.y];
  rank_tile(B, min(*B.n_found, min(B.cap, STATE_BLOCK_SORT_MAX)));
}

__device__ __forceinline__ void emit(const SysParams &P, const StateBufs &B, int g, int o) {
  const float4 p = P.pos[g];
  const int info = P.info[g];
  const int t = info & INFO_TYPE_MASK;
  const int ionised = (info & INFO_ION_BIT) ? 1 : 0;
  if (B.xyz) { B.xyz[3 * o] = p.x; B.xyz[3 * o + 1] = p.y; B.xyz[3 * o + 2] = p.z; }
  if (B.vel) {
    const float4 v = B.vel_src[g];
    B.vel[3 * o] = v.x; B.vel[3 * o + 1] = v.y; B.vel[3 * o + 2] = v.z;
  }
  if (B.frc) {
    const float4 f = B.frc_src ? B.frc_src[g] : make_float4(0.f, 0.f, 0.f, 0.f);
    B.frc[3 * o] = f.x; B.frc[3 * o + 1] = f.y; B.frc[3 * o + 2] = f.z;
  }
  if (B.id) B.id[o] = P.pid[g];
  if (B.type) B.type[o] = t;
  if (B.state) B.state[o] = (int8_t)ionised;
  if (B.cls) B.cls[o] = (info >> INFO_CLS_SHIFT) & 3;
  if (B.site && (t == CR_ACID || t == CR_BASE)) B.site[info >> INFO_SITE_SHIFT] = (int8_t)ionised;
}

// Chunk c of the input ids (1024 consecutive ids, one per thread), written and
// unmarked: a present id's place is the number of present ids before it --
// those of the chunks before and, by ballots and a scan of the warps' counts,
// of its own -- so that consecutive threads write consecutive entries.
// all: every input id is present, so the chunks before are full.
__device__ __forceinline__ void order_inputs(const SysParams &P, const StateBufs &B, int c, bool all) {
  __shared__ int part[ORDER_THREADS / 32];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, i = c * ORDER_THREADS + t;
  const int g = i < B.n_input ? B.present[i] - 1 : -1;
  const unsigned bal = __ballot_sync(0xffffffffu, g >= 0);
  if (lane == 0) part[w] = __popc(bal);
  __syncthreads();
  if (w == 0) {  // inclusive scan of the warps' counts
    int v = part[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += y;
    }
    part[lane] = v;
  }
  __syncthreads();
  if (g >= 0) {
    emit(P, B, g, (all ? c * ORDER_THREADS : B.chunk_base[c]) + (w > 0 ? part[w - 1] : 0) + __popc(bal & ((1u << lane) - 1u)));
    B.present[i] = 0;
  }
  if (t == 0) B.chunk[c] = 0;
}

// CTA x < input_chunks: a chunk of the input ids; the others 1024 ions each,
// after the input ids in id order (slot: the slots by rank)
__device__ __forceinline__ void order_cta(const SysParams &P, const StateBufs &B, int input_chunks, int n_present,
                                          int n_ions, const int *slot) {
  if ((int)blockIdx.x < input_chunks) {
    if ((int)blockIdx.x * ORDER_THREADS < B.n_input) order_inputs(P, B, blockIdx.x, n_present == B.n_input);
    return;
  }
  const int r = ((int)blockIdx.x - input_chunks) * ORDER_THREADS + (int)threadIdx.x;
  if (r < n_ions) emit(P, B, slot[r], n_present + r);
}

// (counts from the host, which has read the ion counter)
__global__ void __launch_bounds__(ORDER_THREADS) k_state_order(SysParams P, StateBufs B, int input_chunks,
                                                               int n_present, int n_ions, const int *slot) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *B.n_ions = 0;  // the count came to the host as n_ions
  order_cta(P, B, input_chunks, n_present, n_ions, slot);
}

// Every replica of a batch (blockIdx.y) at once, the counts read on the
// device: n from the kind counts, n_ions from the mark kernel.  A replica
// whose ions exceed the tile ranking (or whose counts are inconsistent) gets
// n_out = -1 and only its marks cleared.  n_out and err_out receive each
// replica's particle count and error word.  one_tile: no ranks were formed, and
// a replica of more ions than a tile, whose order is the ranks', is one of those.
__global__ void __launch_bounds__(256) k_state_mark_batch(const SysParams *__restrict__ reps,
                                                          const StateBufs *__restrict__ bufs) {
  mark_cells(reps[blockIdx.y], bufs[blockIdx.y], blockIdx.x * blockDim.x + threadIdx.x);
}

__global__ void __launch_bounds__(ORDER_THREADS) k_state_order_batch(const SysParams *__restrict__ reps,
                                                                     const StateBufs *__restrict__ bufs,
                                                                     int input_chunks, int one_tile,
                                                                     long long *n_out, int *err_out) {
  const int r = blockIdx.y;
  const SysParams &P = reps[r];
  const StateBufs &B = bufs[r];
  const long long *cn = B.counts;
  const long long n = cn[K_A0] + cn[K_A1] + cn[K_B0] + cn[K_B1] + cn[K_XP] + cn[K_XM] + cn[K_SP] + cn[K_SM] + B.n_other;
  const int n_ions = *B.n_found;
  const long long n_present = n - n_ions;
  const bool ok = n_ions >= 0 && n_ions <= (one_tile ? RANK_TILE : STATE_BLOCK_SORT_MAX) && n <= B.cap && n_present >= 0 &&
                  n_present <= B.n_input && *P.err == 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    n_out[r] = ok ? n : -1;
    err_out[r] = *P.err;
    *B.n_ions = 0;
  }
  if (ok) {
    order_cta(P, B, input_chunks, (int)n_present, n_ions, n_ions <= RANK_TILE ? B.ion_val : B.ion_rank);
  } else {
    const int i = blockIdx.x * ORDER_THREADS + threadIdx.x;
    if ((int)blockIdx.x < input_chunks && i < B.n_input) B.present[i] = 0;
  }
}

}  // namespace

cudaError_t launch_state_mark(const SysParams &P, const StateBufs &B, cudaStream_t s) {
  k_state_mark<<<(P.ncell + 255) / 256, 256, 0, s>>>(P, B);
  return cudaGetLastError();
}

size_t state_sort_temp_bytes(int cap) {
  if (cap <= STATE_BLOCK_SORT_MAX) return 0;
  size_t bytes = 0;
  cub::DoubleBuffer<unsigned long long> k(nullptr, nullptr);
  cub::DoubleBuffer<int> v(nullptr, nullptr);
  if (cub::DeviceRadixSort::SortPairs(nullptr, bytes, k, v, cap) != cudaSuccess) return 0;
  return bytes;
}

cudaError_t launch_state_order(const SysParams &P, const StateBufs &B, int n_present, int n_ions, int end_bit,
                               cudaStream_t s, int *launches) {
  int n_launch = 1;
  const int *slot = B.ion_rank;
  const bool wide = n_ions > STATE_BLOCK_SORT_MAX;
  // (the chunks' prefix sums come from the sort kernel's last CTA, also without
  // ions; a configuration as it was given -- no ion inserted, no id gone -- needs
  // neither, and the launch would cost a small read 5 of 70 us)
  const unsigned nt = wide ? 0u : (unsigned)((n_ions + RANK_TILE - 1) / RANK_TILE);
  if (n_ions > 0 || n_present != B.n_input) {
    k_ion_sort<<<nt + 1, RANK_TILE, 0, s>>>(B, wide ? 0 : n_ions);
    ++n_launch;
  }
  if (wide) {  // many ions: device-wide radix sort
    if (!B.sort_tmp || !B.ion_key_alt || !B.ion_val_alt) return cudaErrorInvalidValue;
    cub::DoubleBuffer<unsigned long long> k(B.ion_key, B.ion_key_alt);
    cub::DoubleBuffer<int> v(B.ion_val, B.ion_val_alt);
    size_t bytes = B.sort_tmp_bytes;
    cudaError_t e = cub::DeviceRadixSort::SortPairs(B.sort_tmp, bytes, k, v, n_ions, 0, end_bit, s);
    if (e != cudaSuccess) return e;
    slot = v.Current();
    n_launch += (end_bit + 7) / 8 + 2;  // histogram, scan and one pass per 8 bits
  } else if (nt == 1) {  // one tile: its order is the ranks'
    slot = B.ion_val;
  } else if (nt > 1) {
    k_ion_rank<<<nt, RANK_TILE, 0, s>>>(B, n_ions);
    ++n_launch;
  }
  const int ic = (B.n_input + ORDER_THREADS - 1) / ORDER_THREADS, oc = (n_ions + ORDER_THREADS - 1) / ORDER_THREADS;
  k_state_order<<<std::max(ic + oc, 1), ORDER_THREADS, 0, s>>>(P, B, ic, n_present, n_ions, slot);
  if (launches) *launches += n_launch;
  return cudaGetLastError();
}

cudaError_t launch_state_batch(const SysParams *d_reps, const StateBufs *d_bufs, int n_rep, int max_cells,
                               int max_input, int max_cap, bool one_tile, long long *d_n_out, int *d_err_out,
                               cudaStream_t s) {
  const unsigned R = (unsigned)n_rep;
  if (max_cells > 0) k_state_mark_batch<<<dim3((max_cells + 255) / 256, R), 256, 0, s>>>(d_reps, d_bufs);
  const unsigned nt = (unsigned)((std::min(max_cap, STATE_BLOCK_SORT_MAX) + RANK_TILE - 1) / RANK_TILE);
  k_ion_sort_batch<<<dim3(nt + 1, R), RANK_TILE, 0, s>>>(d_bufs);
  if (nt > 1 && !one_tile) k_ion_rank_batch<<<dim3(nt, R), RANK_TILE, 0, s>>>(d_bufs);
  const int ic = (max_input + ORDER_THREADS - 1) / ORDER_THREADS;
  const int gx = std::max(ic + (int)nt, 1);
  k_state_order_batch<<<dim3((unsigned)gx, R), ORDER_THREADS, 0, s>>>(d_reps, d_bufs, ic, one_tile ? 1 : 0, d_n_out,
                                                                              d_err_out);
  return cudaGetLastError();
}

}  // namespace crmc
