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
// the scattered accesses: 674 and 420 us for 5.14 M tetrahedra of 96^3 nodes, 223 now.  Element numbers fit
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
// one by one into a hash table of kRowSlots places in shared memory (a column per thread, so the
// lanes of a warp never share a bank); the distinct ones are then sorted in the column's head.  A
// tetrahedral row has ~72 raw and 14 distinct entries, so most raw ones cost one probe: for 96^3
// nodes 391 us, against 419 with halving into a sorted list and 7545 with the raw ones sorted in
// global memory (72^2 / 4 moves a row).  What bounds it now is instruction issue with 14 of 32
// lanes active on average (probing and sorting diverge).  The block's lists are then packed, in node order, from the start
// of the block's slots (their place in row_ptr is then the block's start plus an offset scanned
// here, and their copy into col_idx is one contiguous stretch).  A row with more than kRowList
// distinct entries is built where its slots lie instead, and its block's rows all stay in their
// own slots (kBlockSpread in the block's total).  The total takes the place of the block's first
// two raw counts, which this block alone reads.
constexpr int kRowBlock = 128;
constexpr int kRowSlots = 32;  // a power of two
constexpr int kRowList = 28;   // distinct entries the table takes
constexpr int64_t kBlockSpread = (int64_t)1 << 62;

__device__ __forceinline__ int64_t* block_total(int32_t* raw, int64_t block) {
  return reinterpret_cast<int64_t*>(raw + block * kRowBlock);
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
__global__ void __launch_bounds__(kRowBlock) k_row_unique(int64_t n_nodes, int v, const int32_t* __restrict__ elems,
                                                          int cap, int32_t* __restrict__ slots,
                                                          int32_t* __restrict__ raw, int32_t* __restrict__ row_ptr,
                                                          CsrBuildFlags* flags) {
  __shared__ int32_t s_list[kRowSlots][kRowBlock];
  const bool vec = v == 4 && ((uintptr_t)elems & 15) == 0;
  const int t = threadIdx.x;
  const int64_t first = (int64_t)blockIdx.x * kRowBlock, i = first + t;
  int32_t* row = slots + i * cap;
  const int k = i < n_nodes ? max(0, min(raw[i], cap)) : 0;
  // the raw neighbours of slot entry x: up to 3 of an element's vertices, or x itself
  auto expand = [&](int32_t x, int32_t* nb) {
    int c = 0;
    if constexpr (WIDE) {
      nb[c++] = x;
    } else {
      int32_t vert[4];
      load_element(elems, v, vec, (int64_t)(uint32_t)x, vert);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        nb[q] = q < v && vert[q] != (int32_t)i ? vert[q] : -1;  // -1: none
      c = 4;
    }
    return c;
  };
  constexpr int E = WIDE ? 1 : 4;
  int u = 0, n_raw = 0;
  bool fits = true;
  static_assert(kRowSlots == 32 && kRowList < kRowSlots, "the hash keeps five bits and never fills the table");
#pragma unroll
  for (int h = 0; h < kRowSlots; ++h) s_list[h][t] = -1;
  for (int a0 = 0; a0 < k && fits; a0 += 4) {
    int32_t x[4], nb[4][E];
    if ((cap & 3) == 0) {  // the row starts on 16 bytes: one load for four entries
      const int4 r = *reinterpret_cast<const int4*>(row + a0);
      x[0] = r.x, x[1] = r.y, x[2] = r.z, x[3] = r.w;
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) x[q] = a0 + q < k ? row[a0 + q] : 0;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {  // four elements' loads in flight
#pragma unroll
      for (int r = 0; r < E; ++r) nb[q][r] = -1;
      if (a0 + q < k) expand(x[q], nb[q]);
    }
#pragma unroll
    for (int q = 0; q < 4 * E; ++q) {
      const int32_t y = nb[q / E][q % E];
      if (y < 0 || !fits) continue;
      ++n_raw;
      int h = (int)(((uint32_t)y * 0x9E3779B1u) >> 27);  // 5 bits: kRowSlots
      int32_t z = s_list[h][t];
      while (z != y && z >= 0) {  // kRowList < kRowSlots: an empty place is always met
        h = (h + 1) & (kRowSlots - 1);
        z = s_list[h][t];
      }
      if (z == y) continue;
      if (u == kRowList) {
        fits = false;
        continue;
      }
      s_list[h][t] = y;
      ++u;
    }
  }
  if (fits) {  // the distinct entries, sorted into the head of the column
    int w = 0;
    for (int h = 0; w < u; ++h) {
      const int32_t y = s_list[h][t];
      if (y < 0) continue;
      int b = w++;
      for (; b > 0 && s_list[b - 1][t] > y; --b) s_list[b][t] = s_list[b - 1][t];
      s_list[b][t] = y;
    }
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
      const int c = expand(row[base + a], nb), room = base + a + 1;
      for (int r = 0; r < c; ++r) {
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
  if (fits) {
    int32_t* dst = spread ? row : slots + first * cap + off;
    for (int a = 0; a < u; ++a) dst[a] = s_list[a][t];
  }
  if (t == 0) *block_total(raw, blockIdx.x) = total | (spread ? kBlockSpread : 0);
}

// Exclusive scan of the blocks' totals in place, by one block: each thread sums its share, the
// shares are scanned, and the totals are replaced by the blocks' starts.
constexpr int kSumThreads = 1024;

__global__ void __launch_bounds__(kSumThreads) k_scan_sums(int64_t nb, int64_t n_nodes, int32_t* __restrict__ raw,
                                                           int32_t* __restrict__ row_ptr, CsrBuildFlags* flags) {
  const int64_t per = (nb + kSumThreads - 1) / kSumThreads;
  const int64_t lo = min(nb, threadIdx.x * per), hi = min(nb, lo + per);
  int64_t sum = 0;
#pragma unroll 4
  for (int64_t b = lo; b < hi; ++b) sum += *block_total(raw, b) & ~kBlockSpread;
  int64_t total;
  int64_t run = block_scan<kSumThreads / 32>(sum, total) - sum;
  for (int64_t b = lo; b < hi; ++b) {
    const int64_t v = *block_total(raw, b);
    *block_total(raw, b) = run | (v & kBlockSpread);
    run += v & ~kBlockSpread;
  }
  if (threadIdx.x == 0) {
    flags->nnz = (unsigned long long)total;
    row_ptr[n_nodes] = (int32_t)total;
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
