// fem_assembly.cu -- global sparse assembly of the element matrices, the step
// after the element integration: A = sum_e P_e^T A_e P_e over the vertex graph
// of the mesh, as CSR for the scalar P1 forms or as BSR with d x d blocks for
// P1 elasticity (node-major unknowns v*d + c; block (c, c') of entry (v, w)
// gathers A_e[(c, i), (c', j)] with conn[e][i] = v, conn[e][j] = w).
//
// Built once per connectivity (fem_assembly_build):
//   incidences : vertex -> (element, local vertex) list in increasing element
//                order (the same counting / scan / fill / segment-sort steps as
//                the adjoint's record CSR)
//   pattern    : one warp per row v gathers the vertices of its incident
//                elements, sorts them in shared memory (bitonic), keeps the
//                distinct ones (the row's columns, increasing), and stores for
//                every incidence t and local vertex j the position of
//                conn[e][j] among them (colpos, one byte)
//   row blocks : (P1 forms and elasticity) rows that share elements, of like
//                length, in blocks of 32 / B^2 (16 for rows of 33 to 63
//                columns of the scalar forms); their incidences, padded to the
//                longest row of the block and interleaved, so that the lanes
//                of a warp read them coalesced.  Longer rows are listed.
// Assembly (fem_assemble), P1 forms and elasticity: one kernel, a warp per row
// block, a lane per row and block component (a few lanes per long row).  A lane
// walks its row's incidences in element order, reads the element row's NV entries of its
// component (16 bytes on tets) and adds them to its own column sums in shared
// memory.  No two lanes share a sum, so the order of every sum is the lane's
// program order:
//   scalar P1 forms: per 32-element tile the contributions in element order,
//                    then those tile sums in tile order (the build marks the
//                    first and the last contribution of every (tile, entry));
//   elasticity     : all contributions in element order.
// Every entry is therefore a fixed-order sum, bitwise reproducible.
#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/fem.h"
#include "fem_internal.h"
#include "fem_pipe.cuh"

namespace fem {

namespace {

constexpr int kRowCap = 512;    // candidate columns per row (incidences x (d+1))
constexpr int kMaxCols = 255;   // distinct columns per row (one-byte positions)
constexpr int kPatWarps = 4;

// Kinds of rows by the room that their sums take in a warp's shared memory:
// short ones, up to 32 columns, have a block of 32 / B^2 rows, a lane per
// component of a row's blocks; the wide rows of the scalar forms, 33 to 63
// columns, a block of 16; longer rows have no blocks (LongPlan).  Rows of more
// than 32 incidences go with the wide ones, which start first: among short rows
// they come late and hold a warp when the others are done (barycentric 40^3
// cube, vertices numbered at random, 95 -> 87 us).
enum : int { ROW_SHORT = 0, ROW_WIDE = 1, ROW_LONG = 2 };
constexpr int kWideRows = 16;
template <int B, int KIND>
struct BlockRows {
  static constexpr int rows = KIND == ROW_WIDE ? kWideRows : 32 / (B * B);
  static constexpr int cols = KIND == ROW_WIDE ? 63 : 32;  // and a column for padded slots, which add zeros to it
  static constexpr int shift = KIND == ROW_WIDE ? 6 : 7;   // log2 of the bytes between a lane's columns
  // a step's slots in units of blk_off
  static constexpr int unit = B == 1 ? 16 : rows, units = rows / unit;
  // Blocks and rows of a window, within which the build may order the rows by
  // their length: a prime number of blocks, so that the first blocks of the
  // windows, the longest ones, fall on different warps of the grid (with 32
  // blocks a window and 2432 warps the same 76 took them all: barycentric 40^3
  // cube, vertices numbered at random, 152 us against 122).
  static constexpr int win_blocks = B == 1 ? 31 : B == 2 ? 127 : 251, win_rows = win_blocks * rows;
};
constexpr uint32_t pad_word(int cols) { return uint32_t(cols) * 0x01010101u; }

// Marks in a byte of a slot's column word (scalar forms): the contribution is
// the first / the last one of its 32-element tile to its entry.
constexpr uint32_t kFirst = 0x40, kLast = 0x80;

enum : int { ASM_ROW_TOO_LONG = 1, ASM_BAD_VERTEX = 2, ASM_REPEATED_VERTEX = 4 };

__global__ void check_conn_kernel(const int32_t* __restrict__ conn, int64_t n, int64_t n_vert, int32_t* flag) {
  int bad = 0;
  for (int64_t k = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x)
    bad |= uint32_t(conn[k]) >= uint32_t(n_vert);
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, ASM_BAD_VERTEX);
}

__device__ __forceinline__ int next_pow2(int x) {
  int p = 32;
  while (p < x) p <<= 1;
  return p;
}

template <int NV, bool WRITE>
__global__ void __launch_bounds__(kPatWarps * 32)
    row_pattern_kernel(const int32_t* __restrict__ conn, const int32_t* __restrict__ inc_off,
                       const int32_t* __restrict__ inc, int64_t n_vert, int32_t* row_len,
                       const int32_t* __restrict__ row_ptr, int32_t* col_idx, uint8_t* colpos, int32_t* flag) {
  __shared__ uint32_t keys_s[kPatWarps][kRowCap];
  __shared__ uint32_t uniq_s[kPatWarps][kRowCap];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t* key = keys_s[warp];
  uint32_t* uniq = uniq_s[warp];
  const int64_t stride = int64_t(gridDim.x) * kPatWarps;
  for (int64_t v = int64_t(blockIdx.x) * kPatWarps + warp; v < n_vert; v += stride) {
    const int32_t b = inc_off[v];
    const int cnt = (inc_off[v + 1] - b) * NV;
    if (cnt > kRowCap) {  // warp-uniform
      if (lane == 0) {
        atomicOr(flag, ASM_ROW_TOO_LONG);
        if (!WRITE) row_len[v] = 0;
      }
      continue;
    }
    const int P = next_pow2(cnt);
    int bad = 0;
    for (int c = lane; c < P; c += 32) {
      uint32_t k = 0xFFFFFFFFu;
      if (c < cnt) {
        const int32_t s = inc[b + c / NV];  // e * NV + i
        const int32_t w = conn[int64_t(s / NV) * NV + c % NV];
        if (uint32_t(w) < uint32_t(n_vert))
          k = uint32_t(w);
        else
          bad = 1;
      }
      key[c] = k;
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(flag, ASM_BAD_VERTEX);
    __syncwarp();
    for (int k2 = 2; k2 <= P; k2 <<= 1)
      for (int jj = k2 >> 1; jj > 0; jj >>= 1) {
        for (int i = lane; i < P; i += 32) {
          const int ixj = i ^ jj;
          if (ixj > i) {
            const bool up = (i & k2) == 0;
            const uint32_t x = key[i], y = key[ixj];
            if ((x > y) == up) {
              key[i] = y;
              key[ixj] = x;
            }
          }
        }
        __syncwarp();
      }
    // distinct columns, in increasing order
    int nu = 0;
    for (int r = 0; r < cnt; r += 32) {
      const int i = r + lane;
      const bool head = i < cnt && key[i] != 0xFFFFFFFFu && (i == 0 || key[i] != key[i - 1]);
      const uint32_t bal = __ballot_sync(0xffffffffu, head);
      if (head) uniq[nu + __popc(bal & ((1u << lane) - 1u))] = key[i];
      nu += __popc(bal);
    }
    __syncwarp();
    if (nu > kMaxCols) {
      if (lane == 0) {
        atomicOr(flag, ASM_ROW_TOO_LONG);
        if (!WRITE) row_len[v] = 0;
      }
      continue;
    }
    if constexpr (!WRITE) {
      if (lane == 0) row_len[v] = nu;
    } else {
      const int32_t rp = row_ptr[v];
      for (int u = lane; u < nu; u += 32) col_idx[rp + u] = int32_t(uniq[u]);
      for (int c = lane; c < cnt; c += 32) {
        const int32_t s = inc[b + c / NV];
        const uint32_t w = uint32_t(conn[int64_t(s / NV) * NV + c % NV]);
        int lo = 0, hi = nu;  // first position with uniq >= w
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (uniq[mid] < w)
            lo = mid + 1;
          else
            hi = mid;
        }
        colpos[int64_t(b) * NV + c] = uint8_t(lo);
      }
    }
    __syncwarp();  // the buffers are refilled for the next row
  }
}

// ------------------------------------------------------------------ row blocks (P1 forms and elasticity)

// Most incidences of a row (row_pattern_kernel refuses more).
__host__ __device__ constexpr int max_incidences(int nv) { return kRowCap / nv; }

// An element of row v lists a vertex twice (its column positions coincide).
template <int NV>
__device__ __forceinline__ bool row_repeats(const int32_t* inc_off, const uint8_t* colpos, int64_t v) {
  for (int32_t t = inc_off[v]; t < inc_off[v + 1]; ++t)
#pragma unroll
    for (int i = 0; i < NV; ++i)
#pragma unroll
      for (int j = i + 1; j < NV; ++j)
        if (colpos[int64_t(t) * NV + i] == colpos[int64_t(t) * NV + j]) return true;
  return false;
}

// The order of the rows.  The rows of a warp should share elements, whose
// matrices they then read from the same lines; so the rows go by their number
// where rows numbered one after the other mostly are neighbours in the element
// list too, else by their first incidence.  (80^3 cube, vertices numbered at
// random: scalar 145 us by number, 100 by incidence, 87 numbered in order;
// elasticity 930, 444 and 437.)  Rows without elements drop out.  Long rows
// have no blocks, and neither have rows where an element repeats a vertex (the
// scalar forms refuse such elements).

// near[0], near[1]: the vertices v with elements that v + 1 has too, and those
// among them whose first incidences lie within kNear of each other.
constexpr int kNear = 512;

__global__ void row_near_kernel(const int32_t* __restrict__ inc_off, const int32_t* __restrict__ inc, int64_t n_vert,
                                int32_t* near) {
  int pairs = 0, close = 0;
  for (int64_t v = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; v + 1 < n_vert;
       v += int64_t(gridDim.x) * blockDim.x) {
    const int32_t a = inc_off[v], b = inc_off[v + 1];
    if (a == b || b == inc_off[v + 2]) continue;
    ++pairs;
    close += abs(inc[a] - inc[b]) <= kNear;
  }
  __syncwarp();
  pairs = __reduce_add_sync(0xffffffffu, pairs);
  close = __reduce_add_sync(0xffffffffu, close);
  if (pairs && (threadIdx.x & 31) == 0) {
    atomicAdd(near, pairs);
    atomicAdd(near + 1, close);
  }
}

// The place of row v among the rows: its number or its first incidence.
__device__ __forceinline__ int32_t row_key(const int32_t* inc_off, const int32_t* inc, int by_number, int64_t v) {
  return by_number ? int32_t(v) : inc[inc_off[v]];
}

template <int NV, int B>
__device__ __forceinline__ int row_kind(const int32_t* inc_off, const uint8_t* colpos, const int32_t* row_ptr,
                                        int repeats, int64_t v) {
  const int len = row_ptr[v + 1] - row_ptr[v];
  const bool room = len <= BlockRows<B, ROW_SHORT>::cols;
  if constexpr (B > 1) return room && !(repeats && row_repeats<NV>(inc_off, colpos, v)) ? ROW_SHORT : ROW_LONG;
  else if (len > BlockRows<B, ROW_WIDE>::cols) return ROW_LONG;
  return room && inc_off[v + 1] - inc_off[v] <= 32 ? ROW_SHORT : ROW_WIDE;
}

// flag[key] = 1 for every row of the kind.
template <int NV, int B, int KIND>
__global__ void row_flag_kernel(const int32_t* __restrict__ inc_off, const int32_t* __restrict__ inc,
                                const uint8_t* __restrict__ colpos, const int32_t* __restrict__ row_ptr,
                                int by_number, int repeats, int64_t n_vert, int32_t* __restrict__ flag) {
  for (int64_t v = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; v < n_vert; v += int64_t(gridDim.x) * blockDim.x)
    if (inc_off[v + 1] > inc_off[v] && row_kind<NV, B>(inc_off, colpos, row_ptr, repeats, v) == KIND)
      flag[row_key(inc_off, inc, by_number, v)] = 1;
}

// The flagged rows at the exclusive scan foff of their flags (long rows as ~v
// where an element repeats a vertex).
template <int NV, int B, int KIND>
__global__ void row_place_kernel(const int32_t* __restrict__ inc_off, const int32_t* __restrict__ inc,
                                 const uint8_t* __restrict__ colpos, const int32_t* __restrict__ foff,
                                 int by_number, int repeats, int64_t n_vert, int32_t* __restrict__ rows) {
  for (int64_t v = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; v < n_vert; v += int64_t(gridDim.x) * blockDim.x) {
    if (inc_off[v + 1] == inc_off[v]) continue;
    const int32_t s = row_key(inc_off, inc, by_number, v);
    if (foff[s + 1] > foff[s])
      rows[foff[s]] = int32_t(KIND == ROW_LONG && repeats && row_repeats<NV>(inc_off, colpos, v) ? ~v : v);
  }
}

// Rows of each kind, and where the blocks of the kinds begin: the wide ones first.
struct RowCounts {
  int32_t n_long, n_wide, n_short;
  __device__ int wide_blocks() const { return int((int64_t(n_wide) + kWideRows - 1) / kWideRows); }
  template <int B>
  __device__ int blocks() const {
    constexpr int G = BlockRows<B, ROW_SHORT>::rows;
    return wide_blocks() + int((int64_t(n_short) + G - 1) / G);
  }
};

// The blocks of a kind of rows, a CTA per window: the rows in their order where
// that pads the window's slots by no more than half, else by their incidence
// counts, the largest first (equal ones in their order).  order: the row, or -1
// behind the last one; steps: the incidences of each block's longest row, in
// units of slots.
//
// Sorted, a block's slots number at most the incidences of the block before
// it, so a window is padded by at most its rows' share of the largest count.
template <int NV, int B, int KIND>
__global__ void __launch_bounds__(256)
    block_order_kernel(const int32_t* __restrict__ inc_off, const int32_t* __restrict__ rows,
                       const RowCounts* __restrict__ counts, int32_t* __restrict__ order, int32_t* __restrict__ steps) {
  using K = BlockRows<B, KIND>;
  constexpr int G = K::rows, W = K::win_rows, P = 1024;
  static_assert(W <= P && W % G == 0 && max_incidences(NV) < 256, "keys: 255 - count, then the row");
  __shared__ uint32_t key[P];
  __shared__ int padded, total;
  const int tid = threadIdx.x;
  const int64_t n = KIND == ROW_WIDE ? counts->n_wide : counts->n_short;
  if (KIND == ROW_SHORT) {
    steps += counts->wide_blocks();
    order += int64_t(counts->wide_blocks()) * kWideRows;
  }
  for (int64_t r0 = int64_t(blockIdx.x) * W; r0 < n; r0 += int64_t(gridDim.x) * W) {
    if (tid == 0) padded = total = 0;
    for (int i = tid; i < P; i += 256) {
      const int64_t v = i < W && r0 + i < n ? rows[r0 + i] : -1;
      key[i] = (uint32_t(255 - (v < 0 ? 0 : inc_off[v + 1] - inc_off[v])) << 16) | uint32_t(i);
    }
    __syncthreads();
    for (int k = tid; k < W / G; k += 256) {
      int top = 0, sum = 0;
      for (int i = k * G; i < (k + 1) * G; ++i) {
        const int c = 255 - int(key[i] >> 16);
        top = c > top ? c : top;
        sum += c;
      }
      atomicAdd(&padded, G * top);
      atomicAdd(&total, sum);
    }
    __syncthreads();
    if (2 * padded > 3 * total)
      for (int k2 = 2; k2 <= P; k2 <<= 1)
        for (int jj = k2 >> 1; jj > 0; jj >>= 1) {
          for (int i = tid; i < P; i += 256) {
            const int ixj = i ^ jj;
            const uint32_t x = key[i], y = ixj > i ? key[ixj] : 0;
            if (ixj > i && (x > y) == ((i & k2) == 0)) {
              key[i] = y;
              key[ixj] = x;
            }
          }
          __syncthreads();
        }
    const int nb = int(((n - r0 < W ? n - r0 : W) + G - 1) / G);
    for (int i = tid; i < nb * G; i += 256) order[r0 + i] = r0 + i < n ? rows[r0 + int(key[i] & 0xFFFFu)] : -1;
    for (int k = tid; k < nb; k += 256) {
      int top = 0;
      for (int i = k * G; i < (k + 1) * G; ++i) top = max(top, 255 - int(key[i] >> 16));
      steps[r0 / G + k] = top * K::units;
    }
    __syncthreads();  // the keys are the next window's
  }
}

// The slots of every row: (element slot e * NV + i, one byte per local vertex
// j: the column position, for the scalar forms with the tile marks), padded
// with element slot -1 to the block's steps.  A tile's incidences of one row
// are neighbours (the list is in element order), so the marks come from a look
// at them.  first marks are counted, of the long rows too: one per (tile,
// entry), the tile records.
template <int NV, int B, int KIND>
__global__ void block_fill_kernel(const int32_t* __restrict__ inc_off, const int32_t* __restrict__ inc,
                                  const uint8_t* __restrict__ colpos, const int32_t* __restrict__ order,
                                  const int32_t* __restrict__ blk_off, const int32_t* __restrict__ long_rows,
                                  const RowCounts* __restrict__ counts, int2* __restrict__ slots, int32_t* n_records) {
  using K = BlockRows<B, KIND>;
  constexpr int G = K::rows;
  const int b0 = KIND == ROW_WIDE ? 0 : counts->wide_blocks();
  const int64_t at_end = int64_t(KIND == ROW_WIDE ? counts->wide_blocks() : counts->template blocks<B>() - b0) * G;
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  blk_off += b0;
  order += int64_t(b0) * kWideRows;
  int nrec = 0;
  // the word of incidence t of the row with incidences [t0, t1)
  auto word = [&](int32_t t, int32_t t0, int32_t t1) {
    uint32_t w = 0;
    const int32_t tile = (inc[t] / NV) >> 5;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const uint32_t c = colpos[int64_t(t) * NV + j];
      uint32_t m = c & 0x3Fu;  // long rows take no words
      if constexpr (B == 1) {
        bool first = true, last = true;
        for (int32_t u = t - 1; first && u >= t0 && (inc[u] / NV) >> 5 == tile; --u)
#pragma unroll
          for (int i = 0; i < NV; ++i) first &= colpos[int64_t(u) * NV + i] != c;
        for (int32_t u = t + 1; last && u < t1 && (inc[u] / NV) >> 5 == tile; ++u)
#pragma unroll
          for (int i = 0; i < NV; ++i) last &= colpos[int64_t(u) * NV + i] != c;
        m |= (first ? kFirst : 0u) | (last ? kLast : 0u);
        nrec += first;
      }
      w |= m << (8 * j);
    }
    return w;
  };
  for (int64_t at = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; at < at_end; at += stride) {
    const int64_t b = at / G, v = order[at];
    const int64_t s0 = int64_t(blk_off[b]) * K::unit;
    const int steps = (blk_off[b + 1] - blk_off[b]) / K::units;
    const int32_t t0 = v < 0 ? 0 : inc_off[v], t1 = v < 0 ? 0 : inc_off[v + 1];
    for (int k = 0; k < steps; ++k)
      slots[s0 + int64_t(k) * G + (at - b * G)] =
          k < t1 - t0 ? make_int2(inc[t0 + k], int(word(t0 + k, t0, t1))) : make_int2(-1, int(pad_word(K::cols)));
  }
  if constexpr (B == 1) {
    const int64_t n_long = KIND == ROW_SHORT ? counts->n_long : 0;
    for (int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; q < n_long; q += stride) {
      const int64_t v = long_rows[q];
      for (int32_t t = inc_off[v]; t < inc_off[v + 1]; ++t) word(t, inc_off[v], inc_off[v + 1]);
    }
    __syncwarp();
    nrec = __reduce_add_sync(0xffffffffu, nrec);
    if (nrec && (threadIdx.x & 31) == 0) atomicAdd(n_records, nrec);
  }
}

// Shared memory of a warp: [sums][open tile sums, scalar forms][stage].  The
// sum of column c of lane l lies at c * 32 + l, a lane's sums in its own bank.
// Padded slots add zeros to a column of their own, which keeps the loop free of
// branches.  (In a block of wide rows column c of lane l lies at c * 16 + l, and
// the upper lanes have padded slots only.)
//
// Scalar forms: the element rows come through a stage of two batches of two
// steps with 16-byte cp.async, which goes around L1.  A scattered load takes a
// 128-byte line of L1 for every 16 bytes in flight, and beside 200 KB of
// shared memory L1 has few: with register loads the kernel was bound by them
// (lanes 31.9 of 32 active, shared-memory pipe 53% busy, waiting on its queue;
// 96^3 cube 253 us against 134 us with the stage; batches of 1, 4 or 8 steps,
// or three and four batches, 136 to 160 us).  A lane copies and reads only its
// own pieces, so no barrier is needed.
// Blocks: neighbouring lanes read 48 contiguous bytes and half the sums'
// space, so register loads win (56^3 cube 149 us against 164 us staged); with
// 8 steps in flight and four CTAs per SM the rest of L1 keeps the sectors that
// a later row needs (four steps and eight CTAs: 162 us; on triangles the
// shorter rows prefer the latter, 42 against 46 us at 600 x 600).
template <int B>
struct BlockPlan {
  static constexpr bool staged = B == 1;
  static constexpr int warps = staged ? 1 : 4;
  static constexpr int min_ctas = staged ? 1 : B == 3 ? 4 : 8;
  static constexpr int batch = staged ? 2 : B == 3 ? 8 : 4;  // steps loaded together
  static constexpr int stages = staged ? 2 : 1;
  static constexpr size_t sums = size_t(BlockRows<B, ROW_SHORT>::cols + 1) * 128;
  static constexpr size_t stage_off = (B == 1 ? 2 : 1) * sums;
  static constexpr size_t per_warp = stage_off + (staged ? size_t(stages) * batch * 512 : 0);
  static constexpr size_t smem = warps * per_warp;
};

// Copies a lane's piece of an element row (NV floats) into its 16 stage bytes; zeros for a padded slot.
template <int NV>
__device__ __forceinline__ void copy_piece(void* dst, const float* A, int64_t off, bool real, int vec) {
  const float* src = real ? A + off : A;
  if (NV == 4 && vec) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)), "l"(src), "r"(real ? 16 : 0)
                 : "memory");
  } else {
#pragma unroll
    for (int j = 0; j < NV; ++j)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(smem_u32(static_cast<float*>(dst) + j)),
                   "l"(src + (real ? j : 0)), "r"(real ? 4 : 0)
                   : "memory");
  }
}

// Long rows (more than 63 columns, 32 of blocks): 32 / (NV B) of them per warp, a lane per column block component
// (c2, j), NV B neighbouring floats of an element row.  A lane walks the row's
// incidences in element order and adds its B values to the sums of its column
// in shared memory; the columns of an element differ, so a step has no
// conflicts.  The scalar forms keep, per column, the sum of the closed tiles,
// that of the open tile, and the open tile's number.  Rows of more columns
// than a warp has room for are walked once per range of columns; a row where
// an element repeats a vertex (~v in the list) is taken value by value.
template <int NV, int B>
struct LongPlan {
  static constexpr int lanes = NV * B, rows = 32 / lanes;
  static constexpr int words = int(BlockPlan<B>::per_warp / 4 / rows);  // of shared memory, per row
  static constexpr int per_col = B == 1 ? 3 : B * B;
  static constexpr int batch = B == 1 ? 8 : 4;  // incidences loaded together
  static constexpr int cols = (words / per_col - 1) | 1;  // an odd number of columns spreads the rows over the banks
  static_assert(B > 1 || cols < 128, "seven bits of a word");
};

template <int NV, int B>
__device__ __forceinline__ void assemble_long_rows(const int32_t* __restrict__ inc_off, const int32_t* __restrict__ inc,
                                                   const uint8_t* __restrict__ colpos,
                                                   const int32_t* __restrict__ row_ptr,
                                                   const int32_t* __restrict__ long_rows, int n_long, int64_t unit,
                                                   const float* __restrict__ A, float* __restrict__ val, float* sm,
                                                   int lane) {
  using LP = LongPlan<NV, B>;
  constexpr int BB = B * B, N = NV * B, L = LP::lanes, R = LP::rows, C = LP::cols, U = LP::batch;
  const int g = lane / L, l = lane % L, j = l % NV;
  const int64_t q = unit * R + g;
  const int32_t v = g < R && q < n_long ? __ldg(long_rows + q) : -1;
  const int32_t rb = v < 0 ? 0 : __ldg(row_ptr + v), len = v < 0 ? 0 : __ldg(row_ptr + v + 1) - rb;
  const int32_t t0 = v < 0 ? 0 : __ldg(inc_off + v), n = v < 0 ? 0 : __ldg(inc_off + v + 1) - t0;
  const int steps = __reduce_max_sync(0xffffffffu, n), maxlen = __reduce_max_sync(0xffffffffu, len);
  float* sum = sm + (g < R ? g : 0) * LP::words;  // [column][BB]; scalar forms: closed tiles, open tile, its number
  int* tile = reinterpret_cast<int*>(sum + 2 * C);
  for (int c0 = 0; c0 < maxlen; c0 += C) {
    const int here = len <= c0 ? 0 : len - c0 < C ? len - c0 : C;  // columns of this range
    for (int x = l; x < here * (B == 1 ? 1 : BB); x += L) {
      sum[x] = 0.f;
      if (B == 1) sum[C + x] = 0.f, tile[x] = -1;
    }
    __syncwarp();
    int32_t sl[U];  // slots and columns of the next batch
    int col[U];
    auto load = [&](int k0) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const bool on = k0 + u < n;
        sl[u] = on ? __ldg(inc + t0 + k0 + u) : 0;
        col[u] = on ? int(__ldg(colpos + (int64_t(t0) + k0 + u) * NV + j)) - c0 : -1;
      }
    };
    load(0);
    for (int k0 = 0; k0 < steps; k0 += U) {
      int32_t at[U];
      float a[U][B];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const bool in = col[u] >= 0 && col[u] < here;
        at[u] = in ? (B == 1 ? (((sl[u] / NV) >> 5) << 7) | col[u] : col[u]) : -1;  // the tile, the column
        const float* src = A + int64_t(sl[u] / NV) * (N * N) + (sl[u] % NV) * N + l;
#pragma unroll
        for (int c = 0; c < B; ++c) a[u][c] = in ? __ldg(src + c * NV * N) : 0.f;
      }
      load(k0 + U);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (at[u] >= 0) {
          if constexpr (B == 1) {
            const int c = at[u] & 127;
            float o = sum[C + c];
            if (tile[c] != at[u] >> 7) {
              sum[c] += o;
              tile[c] = at[u] >> 7;
              o = 0.f;
            }
            sum[C + c] = o + a[u][0];
          } else {
#pragma unroll
            for (int c = 0; c < B; ++c) sum[at[u] * BB + c * B + l / NV] += a[u][c];
          }
        }
        __syncwarp();
      }
    }
    for (int x = l; x < here * (B == 1 ? 1 : BB); x += L)
      __stcs(val + (int64_t(rb) + c0) * BB + x, B == 1 ? sum[x] + sum[C + x] : sum[x]);
    __syncwarp();  // the sums are the next range's
  }
  if constexpr (B > 1) {
    const int64_t q1 = (unit + 1) * R < n_long ? (unit + 1) * R : n_long;
    for (int64_t q2 = unit * R; q2 < q1; ++q2) {
      const int32_t r = ~__ldg(long_rows + q2);
      if (r < 0) continue;
      // a lane per value, every incidence of the row looked at
      const int32_t rp = __ldg(row_ptr + r), words = (__ldg(row_ptr + r + 1) - rp) * BB;
      for (int x = lane; x < words; x += 32) {
        const int c = x / BB, c1 = (x % BB) / B, c2 = x % B;
        float acc = 0.f;
        for (int32_t t = __ldg(inc_off + r); t < __ldg(inc_off + r + 1); ++t) {
          const int32_t s = __ldg(inc + t);
          const float* src = A + int64_t(s / NV) * (N * N) + (c1 * NV + s % NV) * N + c2 * NV;
#pragma unroll
          for (int i = 0; i < NV; ++i)
            if (__ldg(colpos + int64_t(t) * NV + i) == c) acc += __ldg(src + i);
        }
        val[int64_t(rp) * BB + x] = acc;
      }
    }
  }
}

struct BlockParams {
  const int32_t *inc_off, *inc;
  const uint8_t* colpos;
  const int32_t *row_ptr, *order, *blk_off;
  const int2* slots;
  const int32_t* long_rows;
  const RowCounts* counts;
  const float* A;
  float* val;
  int vec_A;
};

// The blocks block(0), block(1), .. below nblk of a kind that a warp serves;
// sm: its shared memory, whose sums are zero before and after.
template <int NV, int B, int KIND, class Blocks>
__device__ __forceinline__ void assemble_block_rows(const BlockParams& p, const Blocks& block, int64_t nblk,
                                                    unsigned char* sm, int lane) {
  using BP = BlockPlan<B>;
  using K = BlockRows<B, KIND>;
  constexpr int BB = B * B, G = K::rows, N = NV * B, U = BP::batch;
  constexpr uint32_t kPad = pad_word(K::cols), kCols = 0x3Fu << K::shift;
  constexpr int kPart = int(BP::sums);  // from a sum to the open tile sum
  char* mine = reinterpret_cast<char*>(sm) + 4 * lane;
  char* stage = reinterpret_cast<char*>(sm) + BP::stage_off + 16 * lane;
  const int g = lane / BB, q = lane % BB;  // row of the block, component (c, c2) = (q / B, q % B)
  // offset of the component's row and columns in A_e, without the element slot
  const float* Aq = p.A + (B == 1 ? 0 : (q / B) * NV * N + (q % B) * NV);
  const int32_t* order = p.order;  // of block 0 of the kind's numbering
  if (KIND == ROW_SHORT)
    order += int64_t(p.counts->wide_blocks()) * (kWideRows - G);
  // A block's first and last unit of slots and the lane's row in it; then that
  // row's bounds and the slots of the first batch.  Both are loaded ahead (two
  // blocks and one), for the latency of these loads is that of a short block's sums.
  struct Head {
    int32_t row, s0, s1;
  };
  auto load_head = [&](int64_t at) {
    Head h{-1, 0, 0};
    if (at < nblk) {
      h.s0 = __ldg(p.blk_off + at);
      h.s1 = __ldg(p.blk_off + at + 1);
      if (g < G) h.row = __ldg(order + at * G + g);
    }
    return h;
  };
  int2 ahead[U];  // slots of the next batch to load
  auto load_slots = [&](const Head& h, int k0) {
    const int2* sl = p.slots + int64_t(h.s0) * K::unit + g;
#pragma unroll
    for (int u = 0; u < U; ++u)
      ahead[u] = g < G && (k0 + u) * K::units < h.s1 - h.s0 ? __ldg(sl + int64_t(k0 + u) * G)
                                                            : make_int2(-1, int(kPad));
  };
  int32_t rb = 0, re = 0;
  auto load_row = [&](const Head& h) {
    rb = h.row >= 0 ? __ldg(p.row_ptr + h.row) : 0;
    re = h.row >= 0 ? __ldg(p.row_ptr + h.row + 1) : 0;
  };
  Head cur = load_head(block(0)), next = load_head(block(1));
  load_row(cur);
  load_slots(cur, 0);
  for (int i = 0; block(i) < nblk; ++i) {
    const Head next2 = load_head(block(i + 2));
    const int steps = (cur.s1 - cur.s0) / K::units;
    // row (c, i) of A_e, columns (c2, 0 .. NV-1): for tets 16 bytes at a multiple of 16
    auto piece = [&](int32_t s) {
      return B == 1 ? int64_t(s) * NV : int64_t(s / NV) * (N * N) + (s % NV) * N;
    };
    // adds a step's piece; its NV columns differ (or are all the pad column): read all, add, write all
    auto add_step = [&](const float(&a)[4], uint32_t w) {
      char* at[NV];
      float s[NV], o[NV];
#pragma unroll
      for (int j = 0; j < NV; ++j) at[j] = mine + ((j == 0 ? w << K::shift : w >> (8 * j - K::shift)) & kCols);
#pragma unroll
      for (int j = 0; j < NV; ++j) {
        s[j] = *reinterpret_cast<float*>(at[j]);
        if (B == 1) o[j] = *reinterpret_cast<float*>(at[j] + kPart);
      }
#pragma unroll
      for (int j = 0; j < NV; ++j) {
        if constexpr (B == 1) {
          const bool first = w & (kFirst << (8 * j)), last = w & (kLast << (8 * j));
          float r = (first ? 0.f : o[j]) + a[j];
          if (last) r = s[j] + r;
          *reinterpret_cast<float*>(at[j] + (last ? 0 : kPart)) = r;
        } else {
          *reinterpret_cast<float*>(at[j]) = s[j] + a[j];
        }
      }
    };
    if constexpr (BP::staged) {
      constexpr int T = BP::stages;
      uint32_t word[T][U];  // column words of the batches in flight
      auto copy_batch = [&](int st) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          copy_piece<NV>(stage + (st * U + u) * 512, Aq, piece(ahead[u].x), ahead[u].x >= 0, p.vec_A);
          word[st][u] = uint32_t(ahead[u].y);
        }
        cp_async_commit();
      };
#pragma unroll
      for (int st = 0; st < T - 1; ++st) {
        copy_batch(st);
        load_slots(cur, (st + 1) * U);
      }
      for (int k0 = 0; k0 < steps; k0 += T * U)
#pragma unroll
        for (int st = 0; st < T; ++st) {  // the batch at k0 + st * U, in stage st
          copy_batch(st == 0 ? T - 1 : st - 1);
          load_slots(cur, k0 + (st + T) * U);
          cp_async_wait<T - 1>();
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const float4 v = *reinterpret_cast<const float4*>(stage + (st * U + u) * 512);
            add_step({v.x, v.y, v.z, v.w}, word[st][u]);
          }
        }
      cp_async_wait<0>();
    } else {
      for (int k0 = 0; k0 < steps; k0 += U) {
        float a[U][4];
        uint32_t word[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const float* src = Aq + piece(ahead[u].x);
          word[u] = uint32_t(ahead[u].y);
#pragma unroll
          for (int j = 0; j < NV; ++j) a[u][j] = 0.f;
          if (ahead[u].x >= 0) {
            if (NV == 4 && p.vec_A) {
              const float4 v = __ldcg(reinterpret_cast<const float4*>(src));
              a[u][0] = v.x, a[u][1] = v.y, a[u][2] = v.z, a[u][3] = v.w;
            } else {
#pragma unroll
              for (int j = 0; j < NV; ++j) a[u][j] = __ldg(src + j);
            }
          }
        }
        load_slots(cur, k0 + U);
#pragma unroll
        for (int u = 0; u < U; ++u) add_step(a[u], word[u]);
      }
    }
    const int32_t row0 = rb;
    const int len = re - rb;
    load_row(next);
    load_slots(next, 0);
    const int maxlen = __reduce_max_sync(0xffffffffu, len);
    if constexpr (B == 1) {
      // pack the rows' values where the open tile sums were (all closed) and
      // store them coalesced: as one run where the rows are neighbours, else
      // row by row, two at a time where they are short
      int off = len;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, off, d);
        if (lane >= d) off += up;
      }
      const int total = __shfl_sync(0xffffffffu, off, 31);
      off -= len;
      __syncwarp();
      float* pack = reinterpret_cast<float*>(sm + kPart);
      for (int c = 0; c < maxlen; ++c)
        if (c < len) {
          float* w = reinterpret_cast<float*>(mine + (c << K::shift));
          pack[off + c] = *w;
          *w = 0.f;
        }
      __syncwarp();
      const int32_t run = __shfl_sync(0xffffffffu, row0, 0);  // every block has a first row
      if (__all_sync(0xffffffffu, len == 0 || row0 - off == run)) {
        for (int x = lane; x < total; x += 32) __stcs(p.val + int64_t(run) + x, pack[x]);
      } else {
        const int place = off << 6 | len;  // within the pack: at most 1024 values, 63 of a row
        auto store = [&](int row, int c) {
          const int32_t to = __shfl_sync(0xffffffffu, row0, row);
          const int from = __shfl_sync(0xffffffffu, place, row), m = from & 63;
          const float* src = pack + (from >> 6);
          if (c < m) __stcs(p.val + int64_t(to) + c, src[c]);
          if (KIND == ROW_WIDE && c + 32 < m) __stcs(p.val + int64_t(to) + c + 32, src[c + 32]);
        };
        if (KIND == ROW_SHORT && maxlen <= 16) {
#pragma unroll 4
          for (int h = 0; h < G; h += 2) store(h + (lane >> 4), lane & 15);
        } else {
#pragma unroll 4
          for (int h = 0; h < G; ++h) store(h, lane);
        }
      }
    } else {
      // a lane's values straight from its bank: 36 (16) contiguous bytes per row and column
      float* out = p.val + int64_t(row0) * BB + q;
      for (int c = 0; c < maxlen; ++c)
        if (c < len) {
          float* w = reinterpret_cast<float*>(mine + (c << K::shift));
          out[c * BB] = *w;
          *w = 0.f;
        }
    }
    __syncwarp();  // the sums are the next block's
    cur = next;
    next = next2;
  }
}

// One warp per row block: 32 rows of a scalar form, 8 of 2 x 2 blocks, 3 of
// 3 x 3 blocks; lane g * B^2 + q serves component q of row g.  A row kernel
// and not a tile pass with records per entry, because its traffic is one read
// of A, 8 bytes per incidence and the values (108 bytes per tet of a scalar
// form, against 197 with records), and because a lane's sums need neither
// atomics nor barriers.  Scalar forms, 96^3 cube: 241 us (tile pass 190 and
// entry pass 48) -> 124 us; elasticity, 56^3 cube: 517 us (a thread per row,
// 5.5 warps per SM) -> 146 us, 4.9 TB/s of the bytes it cannot do without.
// What bounds it: the L1 and shared-memory pipe (two or three conflict-free
// accesses a contribution, and a tag look-up per element row).
// The long rows come first, then the wide ones: they take longest.
template <int NV, int B>
__global__ void __launch_bounds__(BlockPlan<B>::warps * 32, BlockPlan<B>::min_ctas)
    assemble_blocks_kernel(const __grid_constant__ BlockParams p) {
  using BP = BlockPlan<B>;
  extern __shared__ __align__(128) unsigned char block_sm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char* sm = block_sm + size_t(warp) * BP::per_warp;
  const int64_t S = int64_t(gridDim.x) * BP::warps;
  int64_t b = int64_t(blockIdx.x) * BP::warps + warp;
  const RowCounts* counts = p.counts;
  grid_wait(b, counts);
  const int n_long = counts->n_long;
  const int64_t long_units = (int64_t(n_long) + LongPlan<NV, B>::rows - 1) / LongPlan<NV, B>::rows;
  for (; b < long_units; b += S)
    assemble_long_rows<NV, B>(p.inc_off, p.inc, p.colpos, p.row_ptr, p.long_rows, n_long, b, p.A, p.val,
                              reinterpret_cast<float*>(sm), lane);
  b -= long_units;
  // the sums are zero at the start of every block: zeroed here, and again as they are read out
  for (int x = lane; x < int(BP::stage_off / 4); x += 32) reinterpret_cast<float*>(sm)[x] = 0.f;
  __syncwarp();
  const int64_t nblk = counts->template blocks<B>(), wide = counts->wide_blocks();
  int64_t more = 0, lead = 0, mine = 0;
  if constexpr (B == 1) {
    if (wide > 0) {
      if (b < wide)
        assemble_block_rows<NV, B, ROW_WIDE>(p, [=](int i) { return b + i * S; }, wide, sm, lane);
      // Warps below more have taken a wide block more than the others, which
      // have a lead of as many short blocks as make up its steps.
      more = wide % S;
      const int64_t wide_units = p.blk_off[wide], n_short = nblk - wide;
      const int64_t fair = 2 * wide_units * n_short / (wide * (p.blk_off[nblk] - wide_units + 1));
      lead = more == 0 ? 0 : fair * (S - more) < n_short ? fair : n_short / (S - more);
      mine = b < more ? 0 : lead;
    }
  }
  auto block = [=](int i) {
    return i < mine ? wide + (b - more) + i * (S - more) : wide + lead * (S - more) + b + (i - mine) * S;
  };
  assemble_block_rows<NV, B, ROW_SHORT>(p, block, nblk, sm, lane);
}

struct AsmLayout {
  int32_t *inc_off, *inc, *row_ptr, *col_idx, *cursor, *partials;
  int32_t* flag;  // [0] build flags, [1] tile records (scalar forms), an element repeats a vertex (blocks)
  int32_t* near;    // row_near_kernel's counts
  RowCounts* counts;
  uint8_t* colpos;
  // row blocks (P1 forms and elasticity)
  int32_t* order;      // the rows of every block, the wide blocks first: the row, or -1
  int32_t* blk_off;    // [blocks + 1] first slot of each block, in units
  int2* slots;         // of every block, [steps][rows]: (element slot or -1, column word)
  int32_t* long_rows;  // [n_long]
  size_t bytes;
};

size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

AsmLayout asm_layout(int dim, int64_t n_elem, int64_t n_vert, void* base) {
  const int64_t nv = dim + 1;
  const int64_t cap = n_elem * nv * nv;  // contributions: bounds the entries
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = al256(off + bytes);
    return o;
  };
  AsmLayout L{};
  // Room for the padded slots of every mesh: a window in row order takes 1.5
  // times its incidences, a sorted one as many as its incidences and, for its
  // first block, the largest count for every row (block_order_kernel).  A
  // window of short rows and one of wide rows pad the same per row.
  const int64_t n_inc = n_elem * nv, n_rows = n_vert < n_inc ? n_vert : n_inc;
  const int64_t first_blocks = (n_rows / BlockRows<1, ROW_SHORT>::win_rows + 2) * max_incidences(int(nv));
  const int64_t slot_cap = n_inc + n_inc / 2 + 32 * (first_blocks < n_inc ? first_blocks : n_inc);
  // and, before the slots, for the flags, their scan and the rows (launch_row_blocks)
  const int64_t n_keys = n_vert > n_inc ? n_vert : n_inc;
  const size_t slot_bytes = sizeof(int2) * size_t(slot_cap);
  const size_t key_bytes = sizeof(int32_t) * size_t(2 * n_keys + 1 + n_rows);
  const size_t o_inc_off = take(sizeof(int32_t) * size_t(n_vert + 1));
  const size_t o_inc = take(sizeof(int32_t) * size_t(n_elem * nv));
  const size_t o_colpos = take(size_t(cap));
  const size_t o_row_ptr = take(sizeof(int32_t) * size_t(n_vert + 1));
  const size_t o_col = take(sizeof(int32_t) * size_t(cap));  // capacity: every entry distinct
  const size_t o_cursor = take(sizeof(int32_t) * size_t(n_vert + 4));
  const size_t o_part = take(sizeof(int32_t) * scan_partials_count(n_keys + 1));
  const size_t o_flag = take(sizeof(int32_t) * 8);
  const size_t o_order = take(sizeof(int32_t) * size_t(n_vert + 64));
  const size_t o_blk = take(sizeof(int32_t) * size_t(n_vert + 4));
  const size_t o_slots = take(slot_bytes > key_bytes ? slot_bytes : key_bytes);
  const size_t o_long = take(sizeof(int32_t) * size_t(n_vert));
  char* b = static_cast<char*>(base);
  L.inc_off = reinterpret_cast<int32_t*>(b + o_inc_off);
  L.inc = reinterpret_cast<int32_t*>(b + o_inc);
  L.colpos = reinterpret_cast<uint8_t*>(b + o_colpos);
  L.row_ptr = reinterpret_cast<int32_t*>(b + o_row_ptr);
  L.col_idx = reinterpret_cast<int32_t*>(b + o_col);
  L.cursor = reinterpret_cast<int32_t*>(b + o_cursor);
  L.partials = reinterpret_cast<int32_t*>(b + o_part);
  L.flag = reinterpret_cast<int32_t*>(b + o_flag);
  L.near = L.flag + 2;
  L.counts = reinterpret_cast<RowCounts*>(L.flag + 4);
  L.order = reinterpret_cast<int32_t*>(b + o_order);
  L.blk_off = reinterpret_cast<int32_t*>(b + o_blk);
  L.slots = reinterpret_cast<int2*>(b + o_slots);
  L.long_rows = reinterpret_cast<int32_t*>(b + o_long);
  L.bytes = off;
  return L;
}

unsigned grid_of(int64_t n, int per_block) {
  int64_t g = (n + per_block - 1) / per_block;
  const int64_t cap = int64_t(device_sm_count()) * 64;
  if (g > cap) g = cap;
  return unsigned(g < 1 ? 1 : g);
}

template <bool WRITE>
cudaError_t launch_pattern(int dim, const int32_t* conn, int64_t n_vert, const AsmLayout& L, cudaStream_t st) {
  const unsigned g = grid_of(n_vert, kPatWarps);
  if (dim == 2)
    row_pattern_kernel<3, WRITE><<<g, kPatWarps * 32, 0, st>>>(conn, L.inc_off, L.inc, n_vert, L.cursor, L.row_ptr,
                                                                L.col_idx, L.colpos, L.flag);
  else
    row_pattern_kernel<4, WRITE><<<g, kPatWarps * 32, 0, st>>>(conn, L.inc_off, L.inc, n_vert, L.cursor, L.row_ptr,
                                                                L.col_idx, L.colpos, L.flag);
  return cudaGetLastError();
}

// The rows of a kind in order, into rows, and their number.
template <int NV, int B, int KIND>
cudaError_t launch_rows_of(int64_t n_keys, int by_number, int repeats, int64_t n_vert, const AsmLayout& L,
                           int32_t* rows, int32_t* n_rows, cudaStream_t st) {
  // flags by key and their scan use the room of the slots
  int32_t* flag = reinterpret_cast<int32_t*>(L.slots);
  int32_t* foff = flag + n_keys;
  const unsigned gv = grid_of(n_vert, 256);
  cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(int32_t) * size_t(n_keys), st);
  if (e != cudaSuccess) return e;
  row_flag_kernel<NV, B, KIND><<<gv, 256, 0, st>>>(L.inc_off, L.inc, L.colpos, L.row_ptr, by_number, repeats, n_vert,
                                                flag);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = launch_exclusive_scan(flag, n_keys, L.partials, foff, st);
  if (e != cudaSuccess) return e;
  row_place_kernel<NV, B, KIND><<<gv, 256, 0, st>>>(L.inc_off, L.inc, L.colpos, foff, by_number, repeats, n_vert,
                                                 rows);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(n_rows, foff + n_keys, sizeof(int32_t), cudaMemcpyDeviceToDevice, st);
  return e;
}

// The row blocks of a built pattern (B = block size of the form), the rows by
// their number or by their first incidence.  Scalar forms also count their
// tile records into L.flag[1].
template <int NV, int B>
cudaError_t launch_row_blocks(int64_t n_elem, int64_t n_vert, int by_number, int repeats, const AsmLayout& L,
                              cudaStream_t st) {
  const int64_t n_keys = by_number ? n_vert : n_elem * NV;
  const int64_t cap = n_vert / BlockRows<B, ROW_SHORT>::unit + 2;  // blocks at most
  const unsigned gv = grid_of(n_vert, 256);
  int32_t* rows = reinterpret_cast<int32_t*>(L.slots) + 2 * n_keys + 1;  // behind the flags and their scan
  cudaError_t e = launch_rows_of<NV, B, ROW_LONG>(n_keys, by_number, repeats, n_vert, L, L.long_rows,
                                                  &L.counts->n_long, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(L.cursor, 0, sizeof(int32_t) * size_t(cap), st);
  if constexpr (B == 1) {
    if (e == cudaSuccess)
      e = launch_rows_of<NV, B, ROW_WIDE>(n_keys, by_number, 0, n_vert, L, rows, &L.counts->n_wide, st);
    if (e != cudaSuccess) return e;
    block_order_kernel<NV, B, ROW_WIDE><<<grid_of(n_vert, BlockRows<B, ROW_WIDE>::win_rows), 256, 0, st>>>(
        L.inc_off, rows, L.counts, L.order, L.cursor);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = launch_rows_of<NV, B, ROW_SHORT>(n_keys, by_number, repeats, n_vert, L, rows, &L.counts->n_short, st);
  if (e != cudaSuccess) return e;
  block_order_kernel<NV, B, ROW_SHORT><<<grid_of(n_vert, BlockRows<B, ROW_SHORT>::win_rows), 256, 0, st>>>(
      L.inc_off, rows, L.counts, L.order, L.cursor);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = launch_exclusive_scan(L.cursor, cap, L.partials, L.blk_off, st);
  if (e != cudaSuccess) return e;
  if constexpr (B == 1)
    block_fill_kernel<NV, B, ROW_WIDE><<<gv, 256, 0, st>>>(L.inc_off, L.inc, L.colpos, L.order, L.blk_off, L.long_rows,
                                                           L.counts, L.slots, L.flag + 1);
  block_fill_kernel<NV, B, ROW_SHORT><<<gv, 256, 0, st>>>(L.inc_off, L.inc, L.colpos, L.order, L.blk_off, L.long_rows,
                                                          L.counts, L.slots, L.flag + 1);
  return cudaGetLastError();
}

template <int NV, int B>
cudaError_t launch_assemble_t(const AsmLayout& L, const float* A, int64_t n_elem, int64_t n_vert, float* val,
                              cudaStream_t st) {
  auto kern = assemble_blocks_kernel<NV, B>;
  constexpr int warps = BlockPlan<B>::warps;
  constexpr size_t smem = BlockPlan<B>::smem;
  const cudaError_t e = ensure_smem(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  // blocks, and units of long rows: a row of more than cols columns has cols / (NV - 1) elements or more
  constexpr int cols = BlockRows<B, B == 1 ? ROW_WIDE : ROW_SHORT>::cols;
  const int64_t units = n_vert / BlockRows<B, ROW_SHORT>::rows + 2 +
                        n_elem * NV * (NV - 1) / cols / LongPlan<NV, B>::rows;
  // On triangles an element row's 12 bytes pass through L1, three copies to a
  // line that must stay until the third: 16 CTAs an SM leave L1 room for them,
  // the 19 that fit leave too little (barycentric 600^2 square 112 -> 80 us,
  // 900^2 square 60 -> 54, numbered at random 78 -> 68; 14 CTAs 82, 56, 68).
  constexpr int ctas = BlockPlan<B>::staged && NV == 3 ? 16 : 0;
  if (ctas > 0) {
    const cudaError_t c = cudaFuncSetAttribute(reinterpret_cast<const void*>(kern),
                                               cudaFuncAttributePreferredSharedMemoryCarveout,
                                               int((ctas * (smem + 1024) * 100 + 228 * 1024 - 1) / (228 * 1024)));
    if (c != cudaSuccess) cudaGetLastError();  // a preference only
  }
  const unsigned g = pipeline_grid(reinterpret_cast<const void*>(kern), warps, smem, units * 32, ctas);
  const BlockParams p{L.inc_off, L.inc, L.colpos, L.row_ptr, L.order, L.blk_off, L.slots, L.long_rows, L.counts, A, val,
                      int(reinterpret_cast<uintptr_t>(A) % 16 == 0)};
  return launch_chained(kern, g, unsigned(warps * 32), smem, st, p);
}

// ------------------------------------------------------------------ P2 unknowns (vertices, then edges)
//
// The P2 basis has one unknown per vertex and one per edge.  The edges are
// numbered from the vertex graph's pattern: row v's columns are sorted and
// contain v, so the edges with lower vertex v are its columns above v, and
// edge (v, w) gets V + eoff[v] + (position of w in row v) - (position of v) - 1
// with eoff the exclusive scan of those counts: the edges in increasing
// (lower vertex, higher vertex) order.  An element's unknowns (its vertices,
// then its edges in the local P2 order) form the connectivity of a second
// pattern, over the V + n_edges unknowns, which the row kernel assembles.

// The rows' incidences in chunks of four: row r holds chunks [choff[r],
// choff[r+1]).  They lie behind the column indices of the unknowns, over the
// entries that the pattern did not need and over the vertex graph, and take no
// room of their own (252 bytes an element on tets otherwise, a third of the
// workspace).  A mesh whose unknowns hardly share elements has no room there:
// its incidences are read as they are.
struct P2Plan {
  int32_t n_rows;  // V + n_edges
  int32_t at;      // of the chunks from g2.col_idx on, in 16 bytes
  int32_t n;       // chunks
  int32_t fits;
  // offsets of the element rows in A, (e * n + i) * n; -1 in the padding
  __device__ int4* slot4(int32_t* col_idx) const { return reinterpret_cast<int4*>(col_idx) + at; }
  // [chunk][n]: byte u = the column position of the element's unknown j for incidence u
  __device__ uint32_t* pos4(int32_t* col_idx) const { return reinterpret_cast<uint32_t*>(slot4(col_idx) + n); }
};

// Arrays of the P2 assembly: the vertex graph's incidences and pattern
// (positions per incidence), the edge offsets, the element unknowns, and the
// unknowns' incidences and pattern.
struct AsmP2Layout {
  AsmLayout g1;  // vertex graph (inc_off, inc, colpos, row_ptr, col_idx, cursor, partials, flag)
  AsmLayout g2;  // unknowns (same fields over up to V + E * n_edges rows)
  int32_t* eoff;   // [V + 1]
  int32_t* dofs;   // [E][n]
  P2Plan* plan;
  int32_t* choff() const { return g2.cursor; }  // [rows + 1]
  int64_t room;    // bytes from g2.col_idx to the end of g1 and eoff, which are dead once g2 is built
  int64_t rows_cap;
  size_t bytes;
};

AsmP2Layout asm_p2_layout(int dim, int64_t n_elem, int64_t n_vert, void* base) {
  const int64_t nv = dim + 1, ne = dim * (dim + 1) / 2, n = nv + ne;
  const int64_t rows_cap = n_vert + n_elem * ne;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = al256(off + bytes);
    return o;
  };
  char* b = static_cast<char*>(base);
  auto words = [&](int64_t n) { return reinterpret_cast<int32_t*>(b + take(sizeof(int32_t) * size_t(n))); };
  auto graph = [&](int64_t rows, int64_t per_elem, AsmLayout& G) {  // its columns, the last, are taken by the caller
    G.inc_off = words(rows + 1);
    G.inc = words(n_elem * per_elem);
    G.colpos = reinterpret_cast<uint8_t*>(b + take(size_t(n_elem * per_elem * per_elem)));
    G.row_ptr = words(rows + 1);
    G.cursor = words(rows + 1);
    G.partials = words(int64_t(scan_partials_count(rows + 1)));
  };
  AsmP2Layout L{};
  L.dofs = words(n_elem * n);
  L.g1.flag = words(8);
  L.g2.flag = L.g1.flag;
  L.plan = reinterpret_cast<P2Plan*>(L.g1.flag + 4);
  graph(rows_cap, n, L.g2);
  const size_t col = off;
  L.g2.col_idx = words(n_elem * n * n);
  graph(n_vert, nv, L.g1);
  L.g1.col_idx = words(n_elem * nv * nv);
  L.eoff = words(n_vert + 1);
  L.room = int64_t(off - col);
  L.rows_cap = rows_cap;
  L.bytes = off;
  return L;
}

// An element listing a vertex twice has no edge between the two: flagged.
template <int NV>
__global__ void check_repeat_kernel(const int32_t* __restrict__ conn, int64_t n_elem, int32_t* flag) {
  int bad = 0;
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < n_elem; e += int64_t(gridDim.x) * blockDim.x)
#pragma unroll
    for (int i = 0; i < NV; ++i)
#pragma unroll
      for (int j = i + 1; j < NV; ++j) bad |= conn[e * NV + i] == conn[e * NV + j];
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, ASM_REPEATED_VERTEX);
}

// Position of v in its own (sorted) row, or -1 for an empty row.
__device__ __forceinline__ int diag_pos(const int32_t* __restrict__ col, int32_t b, int32_t e, int32_t v) {
  int lo = b, hi = e;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (col[mid] < v)
      lo = mid + 1;
    else
      hi = mid;
  }
  return (lo < e && col[lo] == v) ? lo - b : -1;
}

// n_up[v] = the columns of row v above v: the edges whose lower vertex is v.
__global__ void edge_count_kernel(const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                                  int64_t n_vert, int32_t* n_up) {
  for (int64_t v = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; v < n_vert; v += int64_t(gridDim.x) * blockDim.x) {
    const int32_t b = row_ptr[v], e = row_ptr[v + 1];
    const int d = diag_pos(col, b, e, int32_t(v));
    n_up[v] = d < 0 ? 0 : (e - b) - d - 1;
  }
}

// Element unknowns in the local P2 order: each incidence (e, i) of row v
// writes dofs[e][i] = v and, for every vertex w = conn[e][j] > v, the number
// of edge (v, w) into the slot of local edge (min(i, j), max(i, j)): every
// element edge is written once, by its lower vertex.
template <int NV>
__global__ void edge_dof_kernel(const int32_t* __restrict__ conn, const int32_t* __restrict__ inc_off,
                                const int32_t* __restrict__ inc, const uint8_t* __restrict__ colpos,
                                const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                                const int32_t* __restrict__ eoff, int64_t n_vert, int32_t* __restrict__ dofs) {
  constexpr int NB = NV + NV * (NV - 1) / 2;
  for (int64_t v = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; v < n_vert; v += int64_t(gridDim.x) * blockDim.x) {
    const int d = diag_pos(col, row_ptr[v], row_ptr[v + 1], int32_t(v));
    const int64_t base = n_vert + eoff[v] - d - 1;
    for (int32_t t = inc_off[v]; t < inc_off[v + 1]; ++t) {
      const int32_t sl = inc[t];
      const int64_t el = sl / NV;
      const int i = sl % NV;
      dofs[el * NB + i] = int32_t(v);
#pragma unroll
      for (int j = 0; j < NV; ++j) {
        if (j == i || conn[el * NV + j] <= v) continue;
        const int a = i < j ? i : j, c = i < j ? j : i;
        const int q = a * (2 * NV - a - 1) / 2 + (c - a - 1);
        dofs[el * NB + NV + q] = int32_t(base + colpos[int64_t(t) * NV + j]);
      }
    }
  }
}

__global__ void store_rows_kernel(const int32_t* __restrict__ eoff, int64_t n_vert, P2Plan* plan) {
  if (blockIdx.x == 0 && threadIdx.x == 0) plan->n_rows = int32_t(n_vert + eoff[n_vert]);
}

// Where the chunks lie, and whether they fit (room: bytes from the column indices on).
__global__ void chunk_plan_kernel(const int32_t* row_ptr, const int32_t* choff, int nb, int64_t room, P2Plan* plan) {
  if (blockIdx.x || threadIdx.x) return;
  const int64_t at = (int64_t(row_ptr[plan->n_rows]) + 3) / 4, n = choff[plan->n_rows];
  plan->at = int32_t(at);
  plan->n = int32_t(n);
  plan->fits = 16 * at + n * (16 + 4 * nb) <= room;
}

// Chunks of four incidences per row.
__global__ void chunk_count_kernel(const int32_t* __restrict__ inc_off, int64_t n_rows, int32_t* cnt) {
  for (int64_t r = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; r < n_rows; r += int64_t(gridDim.x) * blockDim.x)
    cnt[r] = (inc_off[r + 1] - inc_off[r] + 3) / 4;
}

template <int NB>
__global__ void chunk_fill_kernel(const int32_t* __restrict__ inc_off, const int32_t* __restrict__ inc,
                                  const uint8_t* __restrict__ colpos, const int32_t* __restrict__ choff,
                                  const P2Plan* __restrict__ plan, int64_t n_rows, int32_t* col_idx) {
  if (!plan->fits) return;
  int4* slot4 = plan->slot4(col_idx);
  uint32_t* pos4 = plan->pos4(col_idx);
  for (int64_t r = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; r < n_rows; r += int64_t(gridDim.x) * blockDim.x) {
    const int32_t t0 = inc_off[r], n = inc_off[r + 1] - t0;
    for (int k = 0; k < n; k += 4) {
      const int64_t c = choff[r] + k / 4;
      int32_t s[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) s[u] = k + u < n ? inc[t0 + k + u] * NB : -1;  // fits: n_elem * NB^2 does
      slot4[c] = make_int4(s[0], s[1], s[2], s[3]);
      for (int j = 0; j < NB; ++j) {
        uint32_t w = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (k + u < n) w |= uint32_t(colpos[(int64_t(t0) + k + u) * NB + j]) << (8 * u);
        pos4[c * NB + j] = w;
      }
    }
  }
}

// The P2 build: vertex-graph pattern, edge numbers, element unknowns, then
// the unknowns' pattern.  Returns the unknown count and the flags (host).
template <int NV>
cudaError_t launch_p2_build(const int32_t* conn, int64_t n_elem, int64_t n_vert, const AsmP2Layout& L,
                            int32_t* rows_host, int32_t* flag_host, int32_t* nnz_host, cudaStream_t st) {
  constexpr int NB = NV + NV * (NV - 1) / 2;
  const AsmLayout& G1 = L.g1;
  const AsmLayout& G2 = L.g2;
  cudaError_t e = cudaMemsetAsync(G1.flag, 0, sizeof(int32_t) * 8, st);
  if (e == cudaSuccess && n_elem > 0) {
    check_conn_kernel<<<grid_of(n_elem * NV, 256), 256, 0, st>>>(conn, n_elem * NV, n_vert, G1.flag);
    check_repeat_kernel<NV><<<grid_of(n_elem, 256), 256, 0, st>>>(conn, n_elem, G1.flag);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(flag_host, G1.flag, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess || *flag_host) return e;
  const unsigned gv = grid_of(n_vert, kPatWarps);
  if (e == cudaSuccess) e = launch_key_csr(conn, n_elem * NV, n_vert, G1.inc_off, G1.inc, G1.cursor, G1.partials, st);
  if (e == cudaSuccess && n_vert > 0) {
    row_pattern_kernel<NV, false><<<gv, kPatWarps * 32, 0, st>>>(conn, G1.inc_off, G1.inc, n_vert, G1.cursor,
                                                                  G1.row_ptr, G1.col_idx, G1.colpos, G1.flag);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = launch_exclusive_scan(G1.cursor, n_vert, G1.partials, G1.row_ptr, st);
  if (e == cudaSuccess && n_vert > 0) {
    row_pattern_kernel<NV, true><<<gv, kPatWarps * 32, 0, st>>>(conn, G1.inc_off, G1.inc, n_vert, G1.cursor,
                                                                 G1.row_ptr, G1.col_idx, G1.colpos, G1.flag);
    edge_count_kernel<<<grid_of(n_vert, 256), 256, 0, st>>>(G1.row_ptr, G1.col_idx, n_vert, G1.cursor);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = launch_exclusive_scan(G1.cursor, n_vert, G1.partials, L.eoff, st);
  if (e == cudaSuccess && n_vert > 0) {
    edge_dof_kernel<NV><<<grid_of(n_vert, 256), 256, 0, st>>>(conn, G1.inc_off, G1.inc, G1.colpos, G1.row_ptr,
                                                               G1.col_idx, L.eoff, n_vert, L.dofs);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    store_rows_kernel<<<1, 32, 0, st>>>(L.eoff, n_vert, L.plan);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(rows_host, &L.plan->n_rows, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(flag_host, G1.flag, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess || *flag_host) return e;
  const int64_t R = *rows_host;
  const unsigned gr = grid_of(R, kPatWarps);
  e = launch_key_csr(L.dofs, n_elem * NB, R, G2.inc_off, G2.inc, G2.cursor, G2.partials, st);
  if (e == cudaSuccess && R > 0) {
    row_pattern_kernel<NB, false><<<gr, kPatWarps * 32, 0, st>>>(L.dofs, G2.inc_off, G2.inc, R, G2.cursor,
                                                                  G2.row_ptr, G2.col_idx, G2.colpos, G2.flag);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = launch_exclusive_scan(G2.cursor, R, G2.partials, G2.row_ptr, st);
  if (e == cudaSuccess && R > 0) {
    row_pattern_kernel<NB, true><<<gr, kPatWarps * 32, 0, st>>>(L.dofs, G2.inc_off, G2.inc, R, G2.cursor,
                                                                 G2.row_ptr, G2.col_idx, G2.colpos, G2.flag);
    e = cudaGetLastError();
  }
  // the counts take room of the vertex graph, which is dead, their scan that of the cursors
  int32_t* counts = G1.inc_off;
  if (e == cudaSuccess && R > 0) {
    chunk_count_kernel<<<grid_of(R, 256), 256, 0, st>>>(G2.inc_off, R, counts);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = launch_exclusive_scan(counts, R, G2.partials, L.choff(), st);
  if (e == cudaSuccess) {
    chunk_plan_kernel<<<1, 32, 0, st>>>(G2.row_ptr, L.choff(), NB, L.room, L.plan);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && R > 0) {
    chunk_fill_kernel<NB><<<grid_of(R, 256), 256, 0, st>>>(G2.inc_off, G2.inc, G2.colpos, L.choff(), L.plan, R,
                                                           G2.col_idx);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(nnz_host, G2.row_ptr + R, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(flag_host, G1.flag, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e;
}

// Rows of the P2 unknowns, 32 / NB of them per warp: lane group g (NB lanes)
// takes its own row, which accumulates in shared memory (at most kMaxCols
// columns).  For each incidence (e, i) of the row, in increasing element
// order, lane j of the group adds A_e[i][j] at the column position of the
// element's unknown j (distinct within an element); the warp then stores the
// rows, which lie side by side, and zeroes the buffers behind them.  Each
// entry is the sum of its contributions in element order.
//
// The incidences come in chunks of four: a lane takes their four slots with one
// 16-byte load and their four positions with one word, where a slot passed
// between lanes and a byte per incidence took two shuffles or loads for every
// addition, on the pipe that the additions use (shared-memory and load pipe
// 76% busy).  The next two chunks, of this row group or the next, are loaded
// under the additions.  61^3 cube: 312 -> 272 us; bound by instruction issue
// (60% active) and that pipe (74%), two accesses an addition, 2.6 wavefronts
// each over the random columns of three rows.  48 registers: ten warps on each
// quarter of an SM (40 registers spill: 330 us, 63 registers 309 us, without
// the loads ahead 314 us).  The rows' places in the output are formed after the
// additions: held across them they spilled 8 bytes on triangles (900^2 square
// 227 -> 218 us, numbered at random 262 -> 251).
//
// A mesh without room for the chunks, and a warp with a row of more than
// kRowCols columns, read the incidences as they are, four at a time, in a loop
// of their own (within the first it made that spill: 61^3 cube 329 us); such a
// warp takes the rows that its buffers hold at 256 columns each (two of three,
// three of five), then the others.  Buffers of 256 columns for every row cost
// triangles 8 to 28% (900^2 square 225 -> 244 us, numbered at random 255 ->
// 326: less room for L1).  40^3 cube of tets that share nothing: 685 us an
// incidence at a time, 311 us four at a time; 10000 fans of 60 triangles 218
// and 140 us.
constexpr int kRowWarps = 4;
constexpr int kRowCols = 160;
constexpr int kRowStride = kRowCols + 11;  // the rows of a warp start 11 banks apart
constexpr int kLongStride = 256;
static_assert(kLongStride > kMaxCols && 3 * kRowStride >= kLongStride, "a row of any length in the buffers");

template <int NB>
__global__ void __launch_bounds__(kRowWarps * 32, 10)
    assemble_rows_kernel(const int32_t* __restrict__ inc_off, const int32_t* __restrict__ inc,
                         const uint8_t* __restrict__ colpos, const int32_t* __restrict__ row_ptr,
                         const int32_t* __restrict__ choff, const P2Plan* plan,
                         const int32_t* __restrict__ col_idx, const float* __restrict__ A, float* __restrict__ val) {
  constexpr int G = 32 / NB;  // rows per warp
  constexpr int kWarpRows = G * kRowStride + 1;  // and a word for the lanes without a row
  __shared__ float acc_s[kRowWarps][kWarpRows];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane / NB, j = lane - g * NB;
  float* rows = acc_s[warp];
  float* acc = rows + g * kRowStride;
  // the row buffers are zero at the start of every row: zeroed once here, and
  // each column zeroed again as it is stored
  for (int c = lane; c < kWarpRows; c += 32) rows[c] = 0.f;
  __syncwarp();
  const float* Aj = A + j;
  int64_t first_row = (int64_t(blockIdx.x) * kRowWarps + warp) * G;
  grid_wait(first_row, plan);
  const uint32_t n_rows = plan->n_rows, S = gridDim.x * (kRowWarps * G);
  // words from col_idx on to lane j's position in chunk 0, chunks being counted from col_idx too
  const uint32_t chunk0 = plan->at, pos0 = 4 * (chunk0 + plan->n) - chunk0 * NB + j;
  uint32_t r0 = uint32_t(first_row);
  if (r0 >= n_rows) return;  // warp-uniform: no CTA-wide barrier
  // chunks [c0, c0 + nch) of the lane's row, its first value, the values of the warp's rows
  struct Rows {
    uint32_t c0;
    int32_t nch, rp, total;
  };
  auto load_rows = [&](uint32_t q0) {
    Rows m{0, 0, 0, 0};
    if (q0 >= n_rows) return m;
    const uint32_t r = q0 + g;
    const bool live = g < G && r < n_rows;
    const int32_t c = live ? __ldg(choff + r) : 0;
    m.c0 = chunk0 + c;
    m.nch = live ? __ldg(choff + r + 1) - c : 0;
    m.rp = __ldg(row_ptr + (r < n_rows ? r : n_rows));
    m.total = __ldg(row_ptr + (q0 + G < n_rows ? q0 + G : n_rows));  // minus the first row's rp
    return m;
  };
  int32_t sn[8];  // slots and positions of the next two chunks
  uint32_t pn[2];
  auto load_chunks = [&](const Rows& m, int k) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const bool on = k + h < m.nch;
      const uint32_t c = m.c0 + k + h;
      const int4 q = on ? __ldg(reinterpret_cast<const int4*>(col_idx) + c) : make_int4(-1, -1, -1, -1);
      sn[4 * h] = q.x, sn[4 * h + 1] = q.y, sn[4 * h + 2] = q.z, sn[4 * h + 3] = q.w;
      pn[h] = on ? __ldg(reinterpret_cast<const uint32_t*>(col_idx) + (pos0 + c * NB)) : 0u;  // below 2^32 words
    }
  };
  bool left = !plan->fits;  // rows for the second loop
  if (left) r0 = n_rows;
  Rows m = load_rows(r0);
  load_chunks(m, 0);
  for (; r0 < n_rows; r0 += S) {
    const Rows mn = load_rows(r0 + S);
    const int32_t end = __shfl_down_sync(0xffffffffu, m.rp, NB);  // of the lane's row
    if (__all_sync(0xffffffffu, g >= G || (g < G - 1 ? end : m.total) - m.rp <= kRowCols)) {
      const int steps = __reduce_max_sync(0xffffffffu, m.nch);
      if (steps == 0) load_chunks(mn, 0);
      // two chunks at a time: their eight element rows, the next two chunks'
      // slots and positions, then the additions in order
      for (int k = 0; k < steps; k += 2) {
        const uint32_t p[2] = {pn[0], pn[1]};
        float a[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) a[u] = sn[u] >= 0 ? __ldg(Aj + sn[u]) : 0.f;
        if (k + 2 < steps)
          load_chunks(m, k + 2);
        else
          load_chunks(mn, 0);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (k + h >= steps) break;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            // the padding adds a zero to column 0 (the lanes of a group alike)
            acc[(p[h] >> (8 * u)) & 0xFFu] += a[4 * h + u];
            __syncwarp();
          }
        }
      }
      const int32_t rp0 = __shfl_sync(0xffffffffu, m.rp, 0), total = m.total - rp0;
      int32_t first[G];  // of each row, within the warp's run of values
#pragma unroll
      for (int h = 1; h < G; ++h) first[h] = __shfl_sync(0xffffffffu, m.rp, h * NB) - rp0;
      for (int x = lane; x < total; x += 32) {
        int at = x;
#pragma unroll
        for (int h = 1; h < G; ++h)
          if (x >= first[h]) at = x - first[h] + h * kRowStride;
        __stcs(val + int64_t(rp0) + x, rows[at]);
        rows[at] = 0.f;
      }
      __syncwarp();  // the row buffers are refilled for the next rows
    } else {
      left = true;
      load_chunks(mn, 0);
    }
    m = mn;
  }
  if (!left) return;
  // the rows passed over, without chunks; their bounds one group of rows ahead
  struct Bounds {
    int32_t rp, re, tb, te;
  };
  auto load_bounds = [&](uint32_t q0) {
    const uint32_t r = q0 + g;
    Bounds v{0, 0, 0, 0};
    if (g < G && q0 < n_rows && r < n_rows)
      v = {__ldg(row_ptr + r), __ldg(row_ptr + r + 1), __ldg(inc_off + r), __ldg(inc_off + r + 1)};
    return v;
  };
  r0 = (blockIdx.x * kRowWarps + warp) * G;
  for (Bounds v = load_bounds(r0), vn; r0 < n_rows; r0 += S, v = vn) {
    vn = load_bounds(r0 + S);
    const int len = v.re - v.rp;
    const bool small = __all_sync(0xffffffffu, len <= kRowCols);
    if (small && plan->fits) continue;
    const int at_once = small ? G : kWarpRows / kLongStride, stride = small ? kRowStride : kLongStride;
    for (int h0 = 0; h0 < G; h0 += at_once) {
      const bool on = g >= h0 && g < h0 + at_once;
      float* row = rows + (on ? (g - h0) * stride : 0);
      const int n = on ? v.te - v.tb : 0;
      const int steps = __reduce_max_sync(0xffffffffu, n);
      for (int k0 = 0; k0 < steps; k0 += 4) {
        int pos[4];
        float a[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const bool in = k0 + u < n;
          pos[u] = in ? __ldg(colpos + int64_t(v.tb + k0 + u) * NB + j) : 0;
          a[u] = in ? __ldg(Aj + int64_t(__ldg(inc + v.tb + k0 + u)) * NB) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (k0 + u < n) row[pos[u]] += a[u];
          __syncwarp();
        }
      }
      for (int c = j; c < (on ? len : 0); c += NB) {
        __stcs(val + int64_t(v.rp) + c, row[c]);
        row[c] = 0.f;
      }
      __syncwarp();  // the buffers are refilled for the next rows
    }
  }
}

template <int NB>
cudaError_t launch_p2_assemble(const AsmP2Layout& L, const float* A, float* val, cudaStream_t st) {
  return launch_chained(assemble_rows_kernel<NB>, grid_of(L.rows_cap, kRowWarps * (32 / NB)), kRowWarps * 32, 0, st,
                        L.g2.inc_off, L.g2.inc, L.g2.colpos, L.g2.row_ptr, L.choff(), L.plan, L.g2.col_idx, A, val);
}

}  // namespace

}  // namespace fem

// ------------------------------------------------------------------ C ABI

namespace {

fem_status asm_fail(fem_status s, const char* msg) {
  fem::set_last_error("%s", msg);
  return s;
}

// Block size of the assembled matrix for a form: 1 (scalar forms), d (P1
// elasticity), 0 (not assembled: the coupling blocks are rectangular).
int asm_block(int form, int dim) {
  if (form == FEM_LAPLACE_P1 || form == FEM_LAPLACE_P1_W1 || form == FEM_LAPLACE_P1_ISO) return 1;
  if (form == FEM_LAPLACE_P2 || form == FEM_LAPLACE_P2_W1 || form == FEM_LAPLACE_P2_ISO) return 1;
  if (form == FEM_ELASTIC_P1) return dim;
  return 0;
}

// P2 forms: unknowns at the vertices and the edges.
bool asm_p2(int form) { return form == FEM_LAPLACE_P2 || form == FEM_LAPLACE_P2_W1 || form == FEM_LAPLACE_P2_ISO; }

fem_status asm_check(const fem_mesh* mesh, int form) {
  if (!mesh) return asm_fail(FEM_ERR_ARG, "mesh is NULL");
  if ((mesh->dim != 2 && mesh->dim != 3) || mesh->n_elem < 0 || mesh->n_vert < 0 || mesh->n_vert > INT32_MAX ||
      (mesh->n_elem > 0 && !mesh->conn))
    return asm_fail(FEM_ERR_ARG, "invalid mesh (dim 2/3, counts, conn)");
  if (form < FEM_LAPLACE_P1 || form > FEM_LAPLACE_P2_ISO) return asm_fail(FEM_ERR_ARG, "form out of range");
  if (asm_block(form, mesh->dim) == 0)
    return asm_fail(FEM_ERR_UNSUPPORTED, "assembly serves the square forms");
  const int64_t nodes = asm_p2(form) ? (mesh->dim + 1) * (mesh->dim + 2) / 2 : mesh->dim + 1;
  if (mesh->n_elem * nodes * nodes > INT32_MAX)
    return asm_fail(FEM_ERR_UNSUPPORTED, "n_elem * (nodes per element)^2 exceeds the int32 entry range");
  return FEM_OK;
}

// The P2 build (fem_assembly_build for the P2 forms).
fem_status p2_build(const fem_mesh* mesh, void* ws, size_t ws_bytes, int64_t* nnz, int64_t* n_records,
                    cudaStream_t st) {
  const fem::AsmP2Layout P = fem::asm_p2_layout(mesh->dim, mesh->n_elem, mesh->n_vert, ws);
  if (!ws || ws_bytes < P.bytes || reinterpret_cast<uintptr_t>(ws) % 256 != 0) {
    fem::set_last_error("assembly workspace needs %zu bytes, 256-byte aligned (got %zu)", P.bytes, ws_bytes);
    return FEM_ERR_WORKSPACE;
  }
  int32_t rows = 0, flag = 0, nz = 0;
  const cudaError_t e =
      mesh->dim == 2 ? fem::launch_p2_build<3>(mesh->conn, mesh->n_elem, mesh->n_vert, P, &rows, &flag, &nz, st)
                     : fem::launch_p2_build<4>(mesh->conn, mesh->n_elem, mesh->n_vert, P, &rows, &flag, &nz, st);
  if (e != cudaSuccess) {
    fem::set_last_error("fem_assembly_build: %s", cudaGetErrorString(e));
    return FEM_ERR_CUDA;
  }
  if (flag & fem::ASM_BAD_VERTEX) return asm_fail(FEM_ERR_ARG, "a connectivity entry is outside [0, n_vert)");
  if (flag & fem::ASM_REPEATED_VERTEX) return asm_fail(FEM_ERR_UNSUPPORTED, "an element repeats a vertex");
  if (flag & fem::ASM_ROW_TOO_LONG)
    return asm_fail(FEM_ERR_UNSUPPORTED, "an unknown has more than 255 neighbours or too many incident elements");
  if (nnz) *nnz = nz;
  if (n_records) *n_records = 0;
  return FEM_OK;
}

}  // namespace

extern "C" {

fem_status fem_assembly_workspace_size(const fem_mesh* mesh, int32_t form, size_t* bytes) {
  fem_status s = asm_check(mesh, form);
  if (s != FEM_OK) return s;
  if (!bytes) return asm_fail(FEM_ERR_ARG, "bytes is NULL");
  *bytes = asm_p2(form) ? fem::asm_p2_layout(mesh->dim, mesh->n_elem, mesh->n_vert, nullptr).bytes
                        : fem::asm_layout(mesh->dim, mesh->n_elem, mesh->n_vert, nullptr).bytes;
  return FEM_OK;
}

fem_status fem_assembly_build(const fem_mesh* mesh, int32_t form, void* ws, size_t ws_bytes, int64_t* nnz,
                              int64_t* n_records, void* stream) {
  fem_status s = asm_check(mesh, form);
  if (s != FEM_OK) return s;
  if (asm_p2(form)) return p2_build(mesh, ws, ws_bytes, nnz, n_records, static_cast<cudaStream_t>(stream));
  const fem::AsmLayout L = fem::asm_layout(mesh->dim, mesh->n_elem, mesh->n_vert, ws);
  if (!ws || ws_bytes < L.bytes || reinterpret_cast<uintptr_t>(ws) % 256 != 0) {
    fem::set_last_error("assembly workspace needs %zu bytes, 256-byte aligned (got %zu)", L.bytes, ws_bytes);
    return FEM_ERR_WORKSPACE;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int nv = mesh->dim + 1;
  const int64_t V = mesh->n_vert;
  cudaError_t e = cudaMemsetAsync(L.flag, 0, sizeof(int32_t) * 8, st);
  if (e == cudaSuccess && mesh->n_elem > 0) {
    fem::check_conn_kernel<<<fem::grid_of(mesh->n_elem * nv, 256), 256, 0, st>>>(mesh->conn, mesh->n_elem * nv, V,
                                                                                  L.flag);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = fem::launch_key_csr(mesh->conn, mesh->n_elem * nv, V, L.inc_off, L.inc, L.cursor, L.partials, st);
  if (e == cudaSuccess && V > 0) e = fem::launch_pattern<false>(mesh->dim, mesh->conn, V, L, st);
  if (e == cudaSuccess) e = fem::launch_exclusive_scan(L.cursor, V, L.partials, L.row_ptr, st);
  if (e == cudaSuccess && V > 0) e = fem::launch_pattern<true>(mesh->dim, mesh->conn, V, L, st);
  const int B = asm_block(form, mesh->dim);
  if (e == cudaSuccess && mesh->n_elem > 0) {  // the scalar forms refuse an element repeating a vertex
    const unsigned g = fem::grid_of(mesh->n_elem, 256);
    int32_t* flag = B == 1 ? L.flag : L.flag + 1;
    if (mesh->dim == 2)
      fem::check_repeat_kernel<3><<<g, 256, 0, st>>>(mesh->conn, mesh->n_elem, flag);
    else
      fem::check_repeat_kernel<4><<<g, 256, 0, st>>>(mesh->conn, mesh->n_elem, flag);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && V > 0) {
    fem::row_near_kernel<<<fem::grid_of(V, 256), 256, 0, st>>>(L.inc_off, L.inc, V, L.near);
    e = cudaGetLastError();
  }
  int32_t host[4] = {0, 0, 0, 0}, nz = 0, nrec = 0;  // build flags, repeated vertices (blocks), near
  if (e == cudaSuccess) e = cudaMemcpyAsync(host, L.flag, sizeof(host), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&nz, L.row_ptr + V, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess && host[0] == 0 && V > 0 && mesh->n_elem > 0) {
    const int by_number = 2 * int64_t(host[3]) >= host[2], repeats = host[1] != 0;
    if (mesh->dim == 2)
      e = B == 1 ? fem::launch_row_blocks<3, 1>(mesh->n_elem, V, by_number, repeats, L, st)
                 : fem::launch_row_blocks<3, 2>(mesh->n_elem, V, by_number, repeats, L, st);
    else
      e = B == 1 ? fem::launch_row_blocks<4, 1>(mesh->n_elem, V, by_number, repeats, L, st)
                 : fem::launch_row_blocks<4, 3>(mesh->n_elem, V, by_number, repeats, L, st);
    if (e == cudaSuccess && B == 1)
      e = cudaMemcpyAsync(&nrec, L.flag + 1, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  if (e != cudaSuccess) {
    fem::set_last_error("fem_assembly_build: %s", cudaGetErrorString(e));
    return FEM_ERR_CUDA;
  }
  if (host[0] & fem::ASM_BAD_VERTEX) return asm_fail(FEM_ERR_ARG, "a connectivity entry is outside [0, n_vert)");
  if (host[0] & fem::ASM_ROW_TOO_LONG)
    return asm_fail(FEM_ERR_UNSUPPORTED, "a vertex has more than 128 incident elements or 255 neighbours");
  if (host[0] & fem::ASM_REPEATED_VERTEX) return asm_fail(FEM_ERR_UNSUPPORTED, "an element repeats a vertex");
  if (nnz) *nnz = nz;
  if (n_records) *n_records = nrec;
  return FEM_OK;
}

fem_status fem_assembly_pattern(const fem_mesh* mesh, int32_t form, const void* ws, size_t ws_bytes,
                                const int32_t** row_ptr, const int32_t** col_idx) {
  fem_status s = asm_check(mesh, form);
  if (s != FEM_OK) return s;
  if (asm_p2(form)) {
    const fem::AsmP2Layout P = fem::asm_p2_layout(mesh->dim, mesh->n_elem, mesh->n_vert, const_cast<void*>(ws));
    if (!ws || ws_bytes < P.bytes) return asm_fail(FEM_ERR_WORKSPACE, "assembly workspace too small");
    if (row_ptr) *row_ptr = P.g2.row_ptr;
    if (col_idx) *col_idx = P.g2.col_idx;
    return FEM_OK;
  }
  const fem::AsmLayout L = fem::asm_layout(mesh->dim, mesh->n_elem, mesh->n_vert, const_cast<void*>(ws));
  if (!ws || ws_bytes < L.bytes) return asm_fail(FEM_ERR_WORKSPACE, "assembly workspace too small");
  if (row_ptr) *row_ptr = L.row_ptr;
  if (col_idx) *col_idx = L.col_idx;
  return FEM_OK;
}

fem_status fem_assembly_unknowns(const fem_mesh* mesh, int32_t form, const void* ws, size_t ws_bytes,
                                 int64_t* n_rows, const int32_t** dofs) {
  fem_status s = asm_check(mesh, form);
  if (s != FEM_OK) return s;
  if (!asm_p2(form)) {
    if (n_rows) *n_rows = mesh->n_vert;
    if (dofs) *dofs = mesh->conn;
    return FEM_OK;
  }
  const fem::AsmP2Layout P = fem::asm_p2_layout(mesh->dim, mesh->n_elem, mesh->n_vert, const_cast<void*>(ws));
  if (!ws || ws_bytes < P.bytes) return asm_fail(FEM_ERR_WORKSPACE, "assembly workspace too small");
  if (n_rows) {
    int32_t r = 0;
    const cudaError_t e = cudaMemcpy(&r, &P.plan->n_rows, sizeof(int32_t), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) {
      fem::set_last_error("fem_assembly_unknowns: %s", cudaGetErrorString(e));
      return FEM_ERR_CUDA;
    }
    *n_rows = r;
  }
  if (dofs) *dofs = P.dofs;
  return FEM_OK;
}

fem_status fem_assemble(const fem_mesh* mesh, int32_t form, const float* A, const void* ws, size_t ws_bytes,
                        float* values, void* stream) {
  fem_status s = asm_check(mesh, form);
  if (s != FEM_OK) return s;
  const fem::AsmLayout L = fem::asm_layout(mesh->dim, mesh->n_elem, mesh->n_vert, const_cast<void*>(ws));
  const size_t need = asm_p2(form) ? fem::asm_p2_layout(mesh->dim, mesh->n_elem, mesh->n_vert, nullptr).bytes : L.bytes;
  if (!ws || ws_bytes < need || reinterpret_cast<uintptr_t>(ws) % 256 != 0)
    return asm_fail(FEM_ERR_WORKSPACE, "assembly workspace too small or unaligned");
  if (mesh->n_vert == 0) return FEM_OK;
  // without elements every row is empty and nothing is written
  if (mesh->n_elem > 0 && (!values || !A)) return asm_fail(FEM_ERR_ARG, "A or values is NULL");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int B = asm_block(form, mesh->dim);
  cudaError_t e;
  if (asm_p2(form)) {  // the row kernel over the vertex and edge unknowns
    const fem::AsmP2Layout P = fem::asm_p2_layout(mesh->dim, mesh->n_elem, mesh->n_vert, const_cast<void*>(ws));
    e = mesh->dim == 2 ? fem::launch_p2_assemble<6>(P, A, values, st) : fem::launch_p2_assemble<10>(P, A, values, st);
  } else if (mesh->n_elem == 0) {
    return FEM_OK;
  } else if (mesh->dim == 2) {
    e = B == 1 ? fem::launch_assemble_t<3, 1>(L, A, mesh->n_elem, mesh->n_vert, values, st)
               : fem::launch_assemble_t<3, 2>(L, A, mesh->n_elem, mesh->n_vert, values, st);
  } else {
    e = B == 1 ? fem::launch_assemble_t<4, 1>(L, A, mesh->n_elem, mesh->n_vert, values, st)
               : fem::launch_assemble_t<4, 3>(L, A, mesh->n_elem, mesh->n_vert, values, st);
  }
  if (e != cudaSuccess) {
    fem::set_last_error("fem_assemble: %s", cudaGetErrorString(e));
    return FEM_ERR_CUDA;
  }
  return FEM_OK;
}

}  // extern "C"
