// Neighbour lists on the GPU from element connectivity: the node adjacency of a triangle or
// tetrahedral mesh (two nodes are neighbours when an element contains both), as the sorted,
// symmetric CSR rows the FTLE kernels read.  The paper computes the neighbour list on the host
// and names accelerating it as future work (Section 2.2, Conclusions); this moves that
// preparation step onto the device for meshes that arrive without adjacency.
//
// 1. every element appends its number to the bounded slot list of each of its vertices (a full list
//    sets an overflow flag, never writes past its slots; an out-of-range vertex is counted and its
//    element skipped);
// 2. each node's row is the sorted union of its elements' other vertices (more raw entries,
//    duplicates included, than the list has slots: the overflow flag), a block's rows packed into
//    one stretch and their lengths scanned within the block;
// 3. one block scans the blocks' totals; 4. each block's stretch is copied into col_idx and its row
//    offsets into row_ptr.
#include <stdint.h>
#include <string.h>

#include "capi_internal.cuh"

namespace ftle {
namespace {

struct CsrBuildFlags {
  unsigned int overflow;
  unsigned int bad_vertex;
  unsigned long long nnz;
};

// The vertices of element e (v of them; 16-byte-aligned quadruples in one load).
__device__ __forceinline__ void load_element(const int32_t* __restrict__ elems, int v, bool vec, int64_t e,
                                             int32_t* vert) {
  if (vec) {
    const int4 q = __ldg(reinterpret_cast<const int4*>(elems) + e);
    vert[0] = q.x, vert[1] = q.y, vert[2] = q.z, vert[3] = q.w;
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) vert[q] = q < v ? __ldg(elems + e * v + q) : -1;
  }
}

// One returned atomic and one store per element and vertex, the element's number; appending the other
// vertices instead (12 atomics and stores a tetrahedron, or 4 atomics and 12 stores) is bound by
// the scattered accesses: 674 and 420 us for 5.14 M tetrahedra of 96^3 nodes, 221 now (the eight scattered
// accesses of an element, a line each, take the first-level caches about 140).  One atomic for a warp's equal
// vertices (match_any) loses 10-20 % on meshes whose elements come cell by cell.  Element numbers fit
// a slot up to 2^32 elements; beyond that (WIDE) the vertices themselves are appended.
template <bool WIDE>
__global__ void __launch_bounds__(256) k_elem_pairs(int64_t n_elem, int v, const int32_t* __restrict__ elems,
                                                    int64_t n_nodes, int cap, int32_t* __restrict__ slots,
                                                    int32_t* __restrict__ raw, CsrBuildFlags* flags) {
  const bool vec = v == 4 && ((uintptr_t)elems & 15) == 0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n_elem; e += (int64_t)gridDim.x * blockDim.x) {
    int32_t vert[4];
    load_element(elems, v, vec, e, vert);
    bool ok = true;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < v && (vert[q] < 0 || vert[q] >= n_nodes)) ok = false;
    if (!ok) {
      atomicAdd(&flags->bad_vertex, 1u);
      continue;
    }
    int at[4], cnt[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {  // the element's atomics first, all in flight together
      cnt[p] = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) cnt[p] += p < v && q < v && vert[p] != vert[q];
      if (!WIDE && cnt[p]) cnt[p] = 1;
      at[p] = cnt[p] ? atomicAdd(raw + vert[p], cnt[p]) : 0;
    }
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      if (!cnt[p]) continue;
      if (at[p] > cap - cnt[p]) atomicOr(&flags->overflow, 1u);
      int32_t* row = slots + (int64_t)vert[p] * cap;
      if constexpr (WIDE) {
        int s = at[p];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q < v && vert[p] != vert[q]) {
            if ((unsigned)s < (unsigned)cap) row[s] = vert[q];
            ++s;
          }
      } else {
        if ((unsigned)at[p] < (unsigned)cap) row[at[p]] = (int32_t)(uint32_t)e;
      }
    }
  }
}

// Rows of a block of kRowBlock nodes, one per thread: the other vertices of the node's elements go
// one by one into a hash table in shared memory (kRowSlots places in buckets of two, one load a probe;
// a column per thread), the next four elements' numbers loading meanwhile.  A tetrahedral row has 72 raw
// and 14 distinct entries, so most raw ones cost one probe.  The distinct ones are sorted in registers,
// the same exchanges in every lane: by a network of 8 or 16 behind a move to the column's head when the
// longest of the warp's rows fits it, of 32 from the table as it lies otherwise.  96^3 nodes: 182 us;
// 233 with the network of 32 throughout, 391 with one place a probe and an insertion sort in the
// column (14 of 32 lanes active on average; 23 with the network of 32), 7545 with the raw entries sorted in
// global memory (72^2 / 4 moves a row).  What bounds it now is the first-level cache, where each lane's
// element is a line of its own.  The block's lists are packed in shared memory and go, in node
// order, to the start of the block's slots (their place in row_ptr is then the block's start plus an
// offset scanned here, and their copy into col_idx is one contiguous stretch).  A row with more than
// kRowList distinct entries is built where its slots lie instead, and its block's rows all stay in
// their own slots (kBlockSpread in the block's total).  The total takes the place of the block's first
// two raw counts, which this block alone reads.
constexpr int kRowBlock = 128;
constexpr int kRowSlots = 32;  // in buckets of two
constexpr int kRowList = 28;   // distinct entries the table takes
constexpr int64_t kBlockSpread = (int64_t)1 << 62;

__device__ __forceinline__ int64_t* block_total(int32_t* raw, int64_t block) {
  return reinterpret_cast<int64_t*>(raw + block * kRowBlock);
}

// Sorts N values in registers (Batcher's odd-even merge sort: 19, 63 and 191 exchanges for 8, 16 and 32,
// the same for every lane).
template <int N>
__device__ __forceinline__ void sort_net(uint32_t* r) {
#pragma unroll
  for (int p = 1; p < N; p <<= 1)
#pragma unroll
    for (int k = p; k >= 1; k >>= 1)
#pragma unroll
      for (int j = k % p; j + k < N; j += 2 * k)
#pragma unroll
        for (int i = 0; i < k; ++i)
          if (i + j + k < N && (i + j) / (2 * p) == (i + j + k) / (2 * p)) {
            const uint32_t lo = min(r[i + j], r[i + j + k]), hi = max(r[i + j], r[i + j + k]);
            r[i + j] = lo;
            r[i + j + k] = hi;
          }
}

// Inclusive scan over the warp.
__device__ __forceinline__ int64_t warp_scan(int64_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int64_t t = __shfl_up_sync(0xffffffffu, v, off);
    if (lane >= off) v += t;
  }
  return v;
}

// Inclusive scan over a block of 32 W threads (every thread calls it); total: the block's sum.
template <int W>
__device__ __forceinline__ int64_t block_scan(int64_t v, int64_t& total) {
  __shared__ int64_t s_warp[W];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t x = warp_scan(v);
  if (lane == 31) s_warp[w] = x;
  __syncthreads();
  int64_t before = 0;
  total = 0;
#pragma unroll
  for (int q = 0; q < W; ++q) {
    const int64_t t = s_warp[q];
    if (q < w) before += t;
    total += t;
  }
  __syncthreads();
  return x + before;
}

template <bool WIDE>
__global__ void __launch_bounds__(kRowBlock, 9) k_row_unique(int64_t n_nodes, int v, const int32_t* __restrict__ elems,
                                                          int cap, int32_t* __restrict__ slots,
                                                          int32_t* __restrict__ raw, int32_t* __restrict__ row_ptr,
                                                          CsrBuildFlags* flags) {
  __shared__ __align__(16) int2 s_tab[kRowSlots / 2][kRowBlock];
  const bool vec = v == 4 && ((uintptr_t)elems & 15) == 0;
  const int t = threadIdx.x;
  const int64_t first = (int64_t)blockIdx.x * kRowBlock, i = first + t;
  int32_t* row = slots + i * cap;
  const int k = i < n_nodes ? max(0, min(raw[i], cap)) : 0;
  // the raw neighbours of slot entry x: up to 3 of an element's vertices, or x itself; -1: none
  constexpr int E = WIDE ? 1 : 3;
  auto expand = [&](int32_t x, int32_t* nb) {
    if constexpr (WIDE) {
      nb[0] = x;
    } else {
      int32_t vert[4];
      load_element(elems, v, vec, (int64_t)(uint32_t)x, vert);
      int32_t last = vert[3] == (int32_t)i ? -1 : vert[3];  // takes the place of the node itself
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const bool self = vert[q] == (int32_t)i;
        nb[q] = self ? last : vert[q];
        last = self ? -1 : last;
      }
    }
  };
  int u = 0, n_raw = 0;
  bool fits = true;
  static_assert(kRowSlots == 32 && kRowList < kRowSlots, "the hash keeps four bits and never fills the table");
#pragma unroll
  for (int h = 0; h < kRowSlots / 2; ++h) s_tab[h][t] = make_int2(-1, -1);
  int32_t x[4];
  auto load4 = [&](int a0) {
    if ((cap & 3) == 0) {  // the row starts on 16 bytes: one load for four entries
      const int4 r = *reinterpret_cast<const int4*>(row + a0);
      x[0] = r.x, x[1] = r.y, x[2] = r.z, x[3] = r.w;
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) x[q] = a0 + q < k ? row[a0 + q] : 0;
    }
  };
  if (k > 0) load4(0);
  for (int a0 = 0; a0 < k && fits; a0 += 4) {
    int32_t nb[4][E];
#pragma unroll
    for (int q = 0; q < 4; ++q) {  // four elements' loads in flight
#pragma unroll
      for (int r = 0; r < E; ++r) nb[q][r] = -1;
      if (a0 + q < k) expand(x[q], nb[q]);
    }
    if (a0 + 4 < k) load4(a0 + 4);
#pragma unroll
    for (int q = 0; q < 4 * E; ++q) {
      const int32_t y = nb[q / E][q % E];
      if (y < 0 || !fits) continue;
      ++n_raw;
      int h = (int)(((uint32_t)y * 0x9E3779B1u) >> 28);  // 4 bits: kRowSlots / 2
      int2 z = s_tab[h][t];
      while (z.x != y && z.y != y && z.y >= 0) {  // kRowList < kRowSlots: an empty place is always met
        h = (h + 1) & (kRowSlots / 2 - 1);
        z = s_tab[h][t];
      }
      const bool fresh = z.x != y && z.y != y;
      fits = !fresh || u < kRowList;
      if (fresh && fits) reinterpret_cast<int32_t*>(&s_tab[h][t])[z.x < 0 ? 0 : 1] = y;
      u += fresh && fits;
    }
  }
  uint32_t list[kRowSlots];  // the distinct entries, sorted; empty places (all ones) come last
  const int u_max = __reduce_max_sync(0xffffffffu, u);  // of the warp's rows
  if (u_max <= 16) {  // the entries to the head of the column, and a smaller network
    int32_t* col = reinterpret_cast<int32_t*>(&s_tab[0][t]);
    auto place = [](int w) { return (w >> 1) * (2 * kRowBlock) + (w & 1); };
    int w = 0;
#pragma unroll
    for (int h = 0; h < kRowSlots / 2; ++h) {
      const int2 z = s_tab[h][t];
      if (z.x >= 0) col[place(w++)] = z.x;
      if (z.y >= 0) col[place(w++)] = z.y;
    }
#pragma unroll
    for (int a = 0; a < 16; ++a) list[a] = a < w ? (uint32_t)col[place(a)] : ~0u;
#pragma unroll
    for (int a = 16; a < kRowSlots; ++a) list[a] = ~0u;
    if (u_max <= 8)
      sort_net<8>(list);
    else
      sort_net<16>(list);
  } else {
#pragma unroll
    for (int h = 0; h < kRowSlots / 2; ++h) {
      const int2 z = s_tab[h][t];
      list[2 * h] = (uint32_t)z.x;
      list[2 * h + 1] = (uint32_t)z.y;
    }
    sort_net<kRowSlots>(list);
  }
  if (!fits) {
    // The row's entries move to the end of its slots and the sorted list grows from the start: it
    // never reaches the entries still to come, since each of them stands for at least one raw
    // neighbour and the raw ones fit the slots (beyond that, the overflow flag is set and the
    // list is cut).
    u = n_raw = 0;
    const int base = cap - k;
    for (int a = k - 1; a >= 0; --a) row[base + a] = row[a];
    for (int a = 0; a < k; ++a) {
      int32_t nb[E];
      const int room = base + a + 1;
      expand(row[base + a], nb);
      for (int r = 0; r < E; ++r) {
        const int32_t y = nb[r];
        if (y < 0) continue;
        ++n_raw;
        int lo = 0, hi = u;
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (row[mid] < y)
            lo = mid + 1;
          else
            hi = mid;
        }
        if ((lo < u && row[lo] == y) || u >= room) continue;
        for (int b = u; b > lo; --b) row[b] = row[b - 1];
        row[lo] = y;
        ++u;
      }
    }
  }
  if (n_raw > cap) {
    atomicOr(&flags->overflow, 1u);
    u = min(u, cap);
  }
  const bool spread = __syncthreads_or(!fits);  // every row has been read
  int64_t total;
  const int64_t off = block_scan<kRowBlock / 32>(u, total) - u;
  if (i < n_nodes) row_ptr[i] = (int32_t)off;
  if (spread) {
    if (fits) {
#pragma unroll
      for (int a = 0; a < kRowList; ++a)
        if (a < u) row[a] = (int32_t)list[a];
    }
  } else {  // packed in shared memory first (the tables have been read), then written in order
    int32_t* s_pack = reinterpret_cast<int32_t*>(s_tab);
#pragma unroll
    for (int a = 0; a < kRowList; ++a)
      if (a < u) s_pack[off + a] = (int32_t)list[a];
    __syncthreads();
    for (int a = t; a < (int)total; a += kRowBlock) slots[first * cap + a] = s_pack[a];
  }
  if (t == 0) *block_total(raw, blockIdx.x) = total | (spread ? kBlockSpread : 0);
}

// Exclusive scan of the blocks' totals in place, by one block, which replaces them by the blocks' starts:
// kSumEach totals a thread at a time, all loaded before the first is used (the chain of loads is what
// bounds this: 12 us for 6912 totals, 19 when each was read before the next).
constexpr int kSumThreads = 1024;
constexpr int kSumEach = 8;

__global__ void __launch_bounds__(kSumThreads) k_scan_sums(int64_t nb, int64_t n_nodes, int32_t* __restrict__ raw,
                                                           int32_t* __restrict__ row_ptr, CsrBuildFlags* flags) {
  int64_t before = 0;
  for (int64_t b0 = 0; b0 < nb; b0 += kSumThreads * kSumEach) {
    const int64_t lo = b0 + (int64_t)threadIdx.x * kSumEach;
    int64_t v[kSumEach], sum = 0;
#pragma unroll
    for (int q = 0; q < kSumEach; ++q) v[q] = lo + q < nb ? *block_total(raw, lo + q) : 0;
#pragma unroll
    for (int q = 0; q < kSumEach; ++q) sum += v[q] & ~kBlockSpread;
    int64_t total;
    int64_t run = before + block_scan<kSumThreads / 32>(sum, total) - sum;
#pragma unroll
    for (int q = 0; q < kSumEach; ++q) {
      if (lo + q < nb) *block_total(raw, lo + q) = run | (v[q] & kBlockSpread);
      run += v[q] & ~kBlockSpread;
    }
    before += total;
  }
  if (threadIdx.x == 0) {
    flags->nnz = (unsigned long long)before;
    row_ptr[n_nodes] = (int32_t)before;
  }
}

// Row offsets and neighbours of a block of nodes to their places.
__global__ void __launch_bounds__(kRowBlock) k_compact(int64_t n_nodes, int cap, const int32_t* __restrict__ slots,
                                                       int32_t* __restrict__ raw, int32_t* __restrict__ row_ptr,
                                                       int32_t* __restrict__ col_idx, int64_t nnz_cap,
                                                       const CsrBuildFlags* flags) {
  const int64_t nb = gridDim.x, b = blockIdx.x, first = b * kRowBlock, i = first + threadIdx.x;
  const int64_t v = *block_total(raw, b), start = v & ~kBlockSpread;
  const int64_t end = b + 1 < nb ? *block_total(raw, b + 1) & ~kBlockSpread : (int64_t)flags->nnz;
  const int64_t off = i < n_nodes ? row_ptr[i] : 0;
  if (v & kBlockSpread) {
    __shared__ int64_t s_off[kRowBlock + 1];
    s_off[threadIdx.x] = i < n_nodes ? off : end - start;
    if (threadIdx.x == 0) s_off[kRowBlock] = end - start;
    __syncthreads();
    for (int64_t a = off; i < n_nodes && a < s_off[threadIdx.x + 1]; ++a)
      if (start + a < nnz_cap) col_idx[start + a] = slots[i * cap + (a - off)];
  } else {
    for (int64_t a = threadIdx.x; a < end - start && start + a < nnz_cap; a += kRowBlock)
      col_idx[start + a] = slots[first * cap + a];
  }
  if (i < n_nodes) row_ptr[i] = (int32_t)(start + off);
}

struct CsrLayout {
  size_t flags = 0, raw = 0, slots = 0, total = 0;
};

CsrLayout csr_layout(int64_t n_nodes, int cap) {
  CsrLayout L;
  size_t off = 0;
  L.flags = off;
  off += align256(sizeof(CsrBuildFlags));
  L.raw = off;
  off += align256(sizeof(int32_t) * (size_t)(n_nodes > 0 ? n_nodes : 1));
  L.slots = off;
  off += align256(sizeof(int32_t) * (size_t)(n_nodes > 0 ? n_nodes : 1) * (size_t)cap);
  L.total = off;
  return L;
}

}  // namespace
}  // namespace ftle

using namespace ftle;

extern "C" {

size_t ftle_csr_workspace_bytes(int64_t n_nodes, int32_t max_row) {
  if (n_nodes < 0 || max_row < 1) return 0;
  return csr_layout(n_nodes, max_row).total;
}

int ftle_csr_from_elements(int64_t n_nodes, int64_t n_elem, int32_t verts_per_elem, const int32_t* elems,
                           int32_t max_row, int32_t* row_ptr, int32_t* col_idx, int64_t nnz_cap, int64_t* nnz_out,
                           void* workspace, size_t workspace_bytes, void* stream) {
  int rc;
  if (n_nodes < 0 || n_nodes >= (int64_t)INT32_MAX || n_elem < 0)
    return fail(FTLE_ERANGE, "n_nodes must be in [0, 2^31 - 1) and n_elem >= 0");
  if (verts_per_elem < 2 || verts_per_elem > 4) return fail(FTLE_EINVAL, "verts_per_elem must be 2, 3 or 4");
  if (max_row < 1 || max_row > 4096) return fail(FTLE_EINVAL, "max_row must be in [1, 4096]");
  if (!row_ptr || !nnz_out || (n_elem > 0 && !elems) || (nnz_cap > 0 && !col_idx))
    return fail(FTLE_EINVAL, "NULL pointer argument");
  const CsrLayout L = csr_layout(n_nodes, max_row);
  if ((rc = check_workspace(workspace, workspace_bytes, L.total))) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  char* w = reinterpret_cast<char*>(workspace);
  CsrBuildFlags* flags = reinterpret_cast<CsrBuildFlags*>(w + L.flags);
  int32_t* raw = reinterpret_cast<int32_t*>(w + L.raw);
  int32_t* slots = reinterpret_cast<int32_t*>(w + L.slots);
  FTLE_CUDA_CHECK(cudaMemsetAsync(flags, 0, sizeof(CsrBuildFlags), s));
  FTLE_CUDA_CHECK(cudaMemsetAsync(raw, 0, sizeof(int32_t) * (size_t)(n_nodes > 0 ? n_nodes : 1), s));
  const bool wide = n_elem > (int64_t)UINT32_MAX;
  if (n_elem > 0) {
    const int grid = grid_for(n_elem, 256, 8);
    if (wide)
      k_elem_pairs<true><<<grid, 256, 0, s>>>(n_elem, verts_per_elem, elems, n_nodes, max_row, slots, raw, flags);
    else
      k_elem_pairs<false><<<grid, 256, 0, s>>>(n_elem, verts_per_elem, elems, n_nodes, max_row, slots, raw, flags);
    FTLE_LAUNCH_CHECK("k_elem_pairs launch");
  }
  const int64_t nb = (n_nodes + kRowBlock - 1) / kRowBlock;
  if (n_nodes > 0) {
    if (wide)
      k_row_unique<true><<<(unsigned)nb, kRowBlock, 0, s>>>(n_nodes, verts_per_elem, elems, max_row, slots, raw, row_ptr,
                                                            flags);
    else
      k_row_unique<false><<<(unsigned)nb, kRowBlock, 0, s>>>(n_nodes, verts_per_elem, elems, max_row, slots, raw,
                                                             row_ptr, flags);
    FTLE_LAUNCH_CHECK("k_row_unique launch");
  }
  k_scan_sums<<<1, kSumThreads, 0, s>>>(nb, n_nodes, raw, row_ptr, flags);
  FTLE_LAUNCH_CHECK("k_scan_sums launch");
  if (n_nodes > 0) {
    k_compact<<<(unsigned)nb, kRowBlock, 0, s>>>(n_nodes, max_row, slots, raw, row_ptr, col_idx, nnz_cap, flags);
    FTLE_LAUNCH_CHECK("k_compact launch");
  }
  CsrBuildFlags h;
  FTLE_CUDA_CHECK(cudaMemcpyAsync(&h, flags, sizeof h, cudaMemcpyDeviceToHost, s));
  FTLE_CUDA_CHECK(cudaStreamSynchronize(s));
  *nnz_out = (int64_t)h.nnz;
  if (h.bad_vertex) return fail(FTLE_EINVAL, "%u elements reference a vertex outside [0, n_nodes)", h.bad_vertex);
  if (h.overflow) return fail(FTLE_ERANGE, "a node has more than max_row = %d element pair entries", max_row);
  if (h.nnz > (unsigned long long)INT32_MAX) return fail(FTLE_ERANGE, "nnz %llu beyond int32", h.nnz);
  if ((int64_t)h.nnz > nnz_cap) return fail(FTLE_ERANGE, "nnz %llu exceeds col_idx capacity %lld", h.nnz, (long long)nnz_cap);
  return FTLE_OK;
}

}  // extern "C"
