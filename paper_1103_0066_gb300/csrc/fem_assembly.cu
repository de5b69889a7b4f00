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
//   row blocks : (P1 forms and elasticity) the incidences of 32 / B^2
//                consecutive rows, padded to the longest row of the block and
//                interleaved, so that the lanes of a warp read them coalesced
// Assembly (fem_assemble), P1 forms and elasticity: one kernel, a warp per row
// block, a lane per row and block component.  A lane walks its row's
// incidences in element order, reads the element row's NV entries of its
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
constexpr int kFastCols = 32;   // columns of a row accumulated in shared memory
constexpr int kPadCol = kFastCols;  // the column of padded slots
constexpr int kPatWarps = 4;

// Rows of a row block: a row takes a lane per component of its blocks.
__host__ __device__ constexpr int block_rows(int B) { return 32 / (B * B); }
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

// Steps of each row block: the incidences of its longest row.  A row of more
// than kFastCols columns is scanned: among the 32 rows of a scalar block alone
// (it gets padding here), a block of three or eight rows as a whole (steps 0),
// like one where an element lists a vertex twice (its positions then coincide).
template <int NV, int B>
__global__ void block_steps_kernel(const int32_t* __restrict__ inc_off, const int32_t* __restrict__ row_ptr,
                                   const uint8_t* __restrict__ colpos, int64_t n_vert, int32_t* steps) {
  constexpr int G = block_rows(B);
  const int64_t nblk = (n_vert + G - 1) / G;
  for (int64_t b = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; b < nblk; b += int64_t(gridDim.x) * blockDim.x) {
    int n = 0;
    bool fast = true;
    for (int64_t v = b * G; v < (b + 1) * G && v < n_vert; ++v) {
      if (row_ptr[v + 1] - row_ptr[v] > kFastCols) {
        fast &= B == 1;
        continue;
      }
      const int c = inc_off[v + 1] - inc_off[v];
      n = c > n ? c : n;
      if constexpr (B > 1)  // the scalar forms refuse such elements
        for (int32_t t = inc_off[v]; fast && t < inc_off[v + 1]; ++t)
#pragma unroll
          for (int i = 0; i < NV; ++i)
#pragma unroll
            for (int j = i + 1; j < NV; ++j) fast &= colpos[int64_t(t) * NV + i] != colpos[int64_t(t) * NV + j];
    }
    steps[b] = fast ? n : 0;
  }
}

// The slots of every row: (element slot e * NV + i, one byte per local vertex
// j: the column position, for the scalar forms with the tile marks), padded
// with element slot -1 to the block's steps.  A tile's incidences of one row
// are neighbours (the list is in element order), so the marks come from a look
// at them.  first marks are counted: one per (tile, entry), the tile records.
template <int NV, int B>
__global__ void block_fill_kernel(const int32_t* __restrict__ inc_off, const int32_t* __restrict__ inc,
                                  const uint8_t* __restrict__ colpos, const int32_t* __restrict__ row_ptr,
                                  const int32_t* __restrict__ blk_off,
                                  int64_t n_vert, int64_t slot_cap, int2* __restrict__ slots, int32_t* n_records) {
  constexpr int G = block_rows(B);
  const int64_t nblk = (n_vert + G - 1) / G;
  const bool room = int64_t(blk_off[nblk]) * G <= slot_cap;
  int nrec = 0;
  for (int64_t v = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; v < n_vert; v += int64_t(gridDim.x) * blockDim.x) {
    const int64_t b = v / G;
    const int32_t s0 = blk_off[b], steps = blk_off[b + 1] - s0;
    const int32_t t0 = inc_off[v], n = inc_off[v + 1] - t0;
    const bool fits = row_ptr[v + 1] - row_ptr[v] <= kFastCols;
    for (int k = 0; k < (steps > n ? steps : n); ++k) {
      int2 q = make_int2(-1, kPadCol * 0x01010101);
      if (k < n) {
        const int32_t t = t0 + k;
        q.x = inc[t];
        uint32_t w = 0;
        const int32_t tile = (q.x / NV) >> 5;
#pragma unroll
        for (int j = 0; j < NV; ++j) {
          const uint32_t c = colpos[int64_t(t) * NV + j];
          uint32_t m = c & 0x3Fu;  // rows of more columns take the scanning path
          if constexpr (B == 1) {
            bool first = true, last = true;
            for (int32_t u = t - 1; first && u >= t0 && (inc[u] / NV) >> 5 == tile; --u)
#pragma unroll
              for (int i = 0; i < NV; ++i) first &= colpos[int64_t(u) * NV + i] != c;
            for (int32_t u = t + 1; last && u < t0 + n && (inc[u] / NV) >> 5 == tile; ++u)
#pragma unroll
              for (int i = 0; i < NV; ++i) last &= colpos[int64_t(u) * NV + i] != c;
            m |= (first ? kFirst : 0u) | (last ? kLast : 0u);
            nrec += first;
          }
          w |= m << (8 * j);
        }
        q.y = int(w);
      }
      if (room && k < steps)
        slots[(int64_t(s0) + k) * G + (v - b * G)] = fits ? q : make_int2(-1, kPadCol * 0x01010101);
    }
  }
  if constexpr (B == 1) {
    __syncwarp();
    nrec = __reduce_add_sync(0xffffffffu, nrec);
    if (nrec && (threadIdx.x & 31) == 0) atomicAdd(n_records, nrec);
  }
}

// Shared memory of a warp: [sums][open tile sums, scalar forms][stage].  The
// sum of column c of lane l lies at c * 32 + l, a lane's sums in its own bank.
// Padded slots add zeros to a column of their own (kPadCol), which keeps the
// loop free of branches.
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
  static constexpr size_t sums = size_t(kFastCols + 1) * 128;
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

// One warp per row block: 32 rows of a scalar form, 8 of 2 x 2 blocks, 3 of
// 3 x 3 blocks; lane g * B^2 + q serves component q of row g.  A row kernel
// and not a tile pass with records per entry, because its traffic is one read
// of A, 8 bytes per incidence and the values (108 bytes per tet of a scalar
// form, against 197 with records), and because a lane's sums need neither
// atomics nor barriers.  Scalar forms, 96^3 cube: 241 us (tile pass 190 and
// entry pass 48) -> 134 us; elasticity, 56^3 cube: 517 us (a thread per row,
// 5.5 warps per SM) -> 149 us, 4.8 TB/s of the bytes it cannot do without.
// What bounds it: the L1 and shared-memory pipe (two or three conflict-free
// accesses a contribution, and a tag look-up per element row).
template <int NV, int B>
__global__ void __launch_bounds__(BlockPlan<B>::warps * 32, BlockPlan<B>::min_ctas)
    assemble_blocks_kernel(const int32_t* __restrict__ inc_off, const int32_t* __restrict__ inc,
                           const uint8_t* __restrict__ colpos, const int32_t* __restrict__ row_ptr,
                           const int32_t* blk_off, const int2* __restrict__ slots, int64_t slot_cap,
                           const float* __restrict__ A, int64_t n_vert, float* __restrict__ val, int vec_A) {
  using BP = BlockPlan<B>;
  constexpr int BB = B * B, G = block_rows(B), N = NV * B, U = BP::batch;
  extern __shared__ __align__(128) unsigned char block_sm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char* wbase = block_sm + size_t(warp) * BP::per_warp;
  float* tot = reinterpret_cast<float*>(wbase);
  char* mine = reinterpret_cast<char*>(wbase) + 4 * lane;
  char* stage = reinterpret_cast<char*>(wbase) + BP::stage_off + 16 * lane;
  constexpr int kPart = int(BP::sums);     // from a sum to the open tile sum
  const int g = lane / BB, q = lane % BB;  // row of the block, component (c, c2) = (q / B, q % B)
  // offset of the component's row and columns in A_e, without the element slot
  const float* Aq = A + (B == 1 ? 0 : (q / B) * NV * N + (q % B) * NV);
  const int64_t nblk = (n_vert + G - 1) / G;
  int64_t b = int64_t(blockIdx.x) * BP::warps + warp;
  grid_wait(b, blk_off);
  const bool room = int64_t(blk_off[nblk]) * G <= slot_cap;
  // the sums are zero at the start of every block: zeroed here, and again as they are read out
  for (int c = 0; c <= kFastCols; ++c) *reinterpret_cast<float*>(mine + c * 128) = 0.f;
  // a lane per value, every incidence of the row looked at
  auto scan_row = [&](int64_t r) {
    const int32_t rp = __ldg(row_ptr + r), t0 = __ldg(inc_off + r), t1 = __ldg(inc_off + r + 1);
    const int words = (__ldg(row_ptr + r + 1) - rp) * BB;
    for (int x = lane; x < words; x += 32) {
      const int c = x / BB, c1 = (x % BB) / B, c2 = x % B;
      float sum = 0.f, part = 0.f;
      int tile = -1;
      for (int32_t t = t0; t < t1; ++t) {
        const int32_t s = __ldg(inc + t);
        const float* src = A + int64_t(s / NV) * (N * N) + (c1 * NV + s % NV) * N + c2 * NV;
        if (B == 1 && (s / NV) >> 5 != tile) {
          sum += part;
          part = 0.f;
          tile = (s / NV) >> 5;
        }
#pragma unroll
        for (int j = 0; j < NV; ++j)
          if (__ldg(colpos + int64_t(t) * NV + j) == c) (B == 1 ? part : sum) += __ldg(src + j);
      }
      val[int64_t(rp) * BB + x] = sum + part;
    }
  };
  for (; b < nblk; b += int64_t(gridDim.x) * BP::warps) {
    const int64_t r0 = b * G;
    const int nr = int(n_vert - r0 < G ? n_vert - r0 : G);
    const int32_t s0 = __ldg(blk_off + b), steps = __ldg(blk_off + b + 1) - s0;
    const int32_t rp0 = __ldg(row_ptr + r0), total = __ldg(row_ptr + r0 + nr) - rp0;
    if (total == 0) continue;
    if (room && steps > 0) {
      const bool live = g < nr;
      const int32_t rb = live ? __ldg(row_ptr + r0 + g) : 0;
      const int row_len = live ? __ldg(row_ptr + r0 + g + 1) - rb : 0;
      // scalar forms: a long row's slots are padding, it is scanned below
      const uint32_t long_lanes = B == 1 ? __ballot_sync(0xffffffffu, row_len > kFastCols) : 0u;
      const int len = B == 1 && row_len > kFastCols ? 0 : row_len;
      const int2* sl = slots + int64_t(s0) * G + g;
      int2 ahead[U];  // slots of the next batch to load
      auto load_slots = [&](int k0) {
#pragma unroll
        for (int u = 0; u < U; ++u)
          ahead[u] = live && k0 + u < steps ? __ldg(sl + (k0 + u) * G) : make_int2(-1, kPadCol * 0x01010101);
      };
      // row (c, i) of A_e, columns (c2, 0 .. NV-1): for tets 16 bytes at a multiple of 16
      auto piece = [&](int32_t s) {
        return B == 1 ? int64_t(s) * NV : int64_t(s / NV) * (N * N) + (s % NV) * N;
      };
      // adds a step's piece; its NV columns differ (or are all the pad column): read all, add, write all
      auto add_step = [&](const float(&a)[4], uint32_t w) {
        char* at[NV];
        float s[NV], o[NV];
#pragma unroll
        for (int j = 0; j < NV; ++j) at[j] = mine + ((j == 0 ? w << 7 : w >> (8 * j - 7)) & (0x3Fu << 7));
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
      load_slots(0);
      if constexpr (BP::staged) {
        constexpr int S = BP::stages;
        uint32_t word[S][U];  // column words of the batches in flight
        auto copy_batch = [&](int st) {
#pragma unroll
          for (int u = 0; u < U; ++u) {
            copy_piece<NV>(stage + (st * U + u) * 512, Aq, piece(ahead[u].x), ahead[u].x >= 0, vec_A);
            word[st][u] = uint32_t(ahead[u].y);
          }
          cp_async_commit();
        };
#pragma unroll
        for (int st = 0; st < S - 1; ++st) {
          copy_batch(st);
          load_slots((st + 1) * U);
        }
        for (int k0 = 0; k0 < steps; k0 += S * U)
#pragma unroll
          for (int st = 0; st < S; ++st) {  // the batch at k0 + st * U, in stage st
            copy_batch(st == 0 ? S - 1 : st - 1);
            load_slots(k0 + (st + S) * U);
            cp_async_wait<S - 1>();
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
              if (NV == 4 && vec_A) {
                const float4 v = __ldcg(reinterpret_cast<const float4*>(src));
                a[u][0] = v.x, a[u][1] = v.y, a[u][2] = v.z, a[u][3] = v.w;
              } else {
#pragma unroll
                for (int j = 0; j < NV; ++j) a[u][j] = __ldg(src + j);
              }
            }
          }
          load_slots(k0 + U);
#pragma unroll
          for (int u = 0; u < U; ++u) add_step(a[u], word[u]);
        }
      }
      const int maxlen = __reduce_max_sync(0xffffffffu, len);
      if (B == 1 && long_lanes == 0) {
        // pack the rows' values where the open tile sums were (all closed) and store them coalesced
        __syncwarp();
        float* pack = reinterpret_cast<float*>(wbase + kPart);
        for (int c = 0; c < maxlen; ++c)
          if (c < len) {
            float* w = reinterpret_cast<float*>(mine + c * 128);
            pack[rb - rp0 + c] = *w;
            *w = 0.f;
          }
        __syncwarp();
        for (int x = lane; x < total; x += 32) __stcs(val + int64_t(rp0) + x, pack[x]);
      } else {
        // a lane's values straight from its bank: 36 (16) contiguous bytes per row and column
        float* out = val + int64_t(rb) * BB + q;
        for (int c = 0; c < maxlen; ++c)
          if (c < len) {
            float* w = reinterpret_cast<float*>(mine + c * 128);
            out[c * BB] = *w;
            *w = 0.f;
          }
      }
      __syncwarp();  // the sums are the next block's
      if constexpr (B == 1)
        for (uint32_t left = long_lanes; left; left &= left - 1) scan_row(r0 + __ffs(left) - 1);
    } else {
      for (int h = 0; h < nr; ++h) scan_row(r0 + h);
    }
  }
}

struct AsmLayout {
  int32_t *inc_off, *inc, *row_ptr, *col_idx, *cursor, *partials;
  int32_t* flag;  // [0] build flags, [1] tile records (scalar forms)
  uint8_t* colpos;
  // row blocks (P1 forms and elasticity)
  int32_t* blk_off;  // [blocks + 1] first step of each block
  int2* slots;       // [steps][block_rows]: (element slot or -1, column word)
  int64_t slot_cap;
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
  // Room for padding the rows of a block to its longest one: twice the
  // incidences (a cube's rows need 1.1 times; a mesh that needs more than
  // twice takes the scanning path of the kernel, which reads no slots).
  L.slot_cap = 2 * n_elem * nv + 1024;
  const size_t o_inc_off = take(sizeof(int32_t) * size_t(n_vert + 1));
  const size_t o_inc = take(sizeof(int32_t) * size_t(n_elem * nv));
  const size_t o_colpos = take(size_t(cap));
  const size_t o_row_ptr = take(sizeof(int32_t) * size_t(n_vert + 1));
  const size_t o_col = take(sizeof(int32_t) * size_t(cap));  // capacity: every entry distinct
  const size_t o_cursor = take(sizeof(int32_t) * size_t(n_vert + 1));
  const size_t o_part = take(sizeof(int32_t) * scan_partials_count(n_vert + 1));
  const size_t o_flag = take(sizeof(int32_t) * 4);
  const size_t o_blk = take(sizeof(int32_t) * size_t(n_vert + 2));
  const size_t o_slots = take(sizeof(int2) * size_t(L.slot_cap));
  char* b = static_cast<char*>(base);
  L.inc_off = reinterpret_cast<int32_t*>(b + o_inc_off);
  L.inc = reinterpret_cast<int32_t*>(b + o_inc);
  L.colpos = reinterpret_cast<uint8_t*>(b + o_colpos);
  L.row_ptr = reinterpret_cast<int32_t*>(b + o_row_ptr);
  L.col_idx = reinterpret_cast<int32_t*>(b + o_col);
  L.cursor = reinterpret_cast<int32_t*>(b + o_cursor);
  L.partials = reinterpret_cast<int32_t*>(b + o_part);
  L.flag = reinterpret_cast<int32_t*>(b + o_flag);
  L.blk_off = reinterpret_cast<int32_t*>(b + o_blk);
  L.slots = reinterpret_cast<int2*>(b + o_slots);
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

// The row blocks of a built pattern (B = block size of the form).  Scalar
// forms also count their tile records into L.flag[1].
template <int NV, int B>
cudaError_t launch_row_blocks(int64_t n_vert, const AsmLayout& L, cudaStream_t st) {
  const int64_t nblk = (n_vert + block_rows(B) - 1) / block_rows(B);
  block_steps_kernel<NV, B><<<grid_of(nblk, 256), 256, 0, st>>>(L.inc_off, L.row_ptr, L.colpos, n_vert, L.cursor);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = launch_exclusive_scan(L.cursor, nblk, L.partials, L.blk_off, st);
  if (e != cudaSuccess) return e;
  block_fill_kernel<NV, B><<<grid_of(n_vert, 256), 256, 0, st>>>(L.inc_off, L.inc, L.colpos, L.row_ptr, L.blk_off,
                                                                 n_vert, L.slot_cap, L.slots, L.flag + 1);
  return cudaGetLastError();
}

template <int NV, int B>
cudaError_t launch_assemble_t(const AsmLayout& L, const float* A, int64_t n_vert, float* val, cudaStream_t st) {
  auto kern = assemble_blocks_kernel<NV, B>;
  constexpr int warps = BlockPlan<B>::warps;
  constexpr size_t smem = BlockPlan<B>::smem;
  const cudaError_t e = ensure_smem(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  const int64_t nblk = (n_vert + block_rows(B) - 1) / block_rows(B);
  const unsigned g = pipeline_grid(reinterpret_cast<const void*>(kern), warps, smem, nblk * 32, 0);
  return launch_chained(kern, g, unsigned(warps * 32), smem, st, L.inc_off, L.inc, L.colpos, L.row_ptr, L.blk_off,
                        L.slots, L.slot_cap, A, n_vert, val, int(reinterpret_cast<uintptr_t>(A) % 16 == 0));
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

// Arrays of the P2 assembly: the vertex graph's incidences and pattern
// (positions per incidence), the edge offsets, the element unknowns, and the
// unknowns' incidences and pattern.
struct AsmP2Layout {
  AsmLayout g1;  // vertex graph (inc_off, inc, colpos, row_ptr, col_idx, cursor, partials, flag)
  AsmLayout g2;  // unknowns (same fields over up to V + E * n_edges rows)
  int32_t* eoff;   // [V + 1]
  int32_t* dofs;   // [E][n]
  int32_t* n_rows; // one word: V + n_edges
  // the rows' incidences in chunks of four: row r holds chunks [choff[r], choff[r+1])
  int32_t* choff;   // [rows + 1]
  int4* slot4;      // offsets of the element rows in A, (e * n + i) * n; -1 in the padding
  uint32_t* pos4;   // [chunk][n]: byte u = the column position of the element's unknown j for incidence u
  int64_t chunk_cap;
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
  auto graph = [&](int64_t rows, int64_t per_elem, AsmLayout& G) {
    const int64_t cap = n_elem * per_elem * per_elem;
    const size_t o_inc_off = take(sizeof(int32_t) * size_t(rows + 1));
    const size_t o_inc = take(sizeof(int32_t) * size_t(n_elem * per_elem));
    const size_t o_colpos = take(size_t(cap));
    const size_t o_row_ptr = take(sizeof(int32_t) * size_t(rows + 1));
    const size_t o_col = take(sizeof(int32_t) * size_t(cap));
    const size_t o_cursor = take(sizeof(int32_t) * size_t(rows + 1));
    const size_t o_part = take(sizeof(int32_t) * scan_partials_count(rows + 1));
    G.inc_off = reinterpret_cast<int32_t*>(b + o_inc_off);
    G.inc = reinterpret_cast<int32_t*>(b + o_inc);
    G.colpos = reinterpret_cast<uint8_t*>(b + o_colpos);
    G.row_ptr = reinterpret_cast<int32_t*>(b + o_row_ptr);
    G.col_idx = reinterpret_cast<int32_t*>(b + o_col);
    G.cursor = reinterpret_cast<int32_t*>(b + o_cursor);
    G.partials = reinterpret_cast<int32_t*>(b + o_part);
  };
  AsmP2Layout L{};
  graph(n_vert, nv, L.g1);
  graph(rows_cap, n, L.g2);
  const size_t o_eoff = take(sizeof(int32_t) * size_t(n_vert + 1));
  const size_t o_dofs = take(sizeof(int32_t) * size_t(n_elem * n));
  const size_t o_flag = take(sizeof(int32_t) * 8);
  // 2.9 chunks per tet on a cube; a mesh that needs more room than this (many
  // unknowns with few elements each) reads the incidences one by one instead
  L.chunk_cap = n_elem * 9 / 2 + n_vert + 1024;
  const size_t o_choff = take(sizeof(int32_t) * size_t(rows_cap + 1));
  const size_t o_slot4 = take(sizeof(int4) * size_t(L.chunk_cap));
  const size_t o_pos4 = take(sizeof(uint32_t) * size_t(L.chunk_cap * n));
  L.choff = reinterpret_cast<int32_t*>(b + o_choff);
  L.slot4 = reinterpret_cast<int4*>(b + o_slot4);
  L.pos4 = reinterpret_cast<uint32_t*>(b + o_pos4);
  L.eoff = reinterpret_cast<int32_t*>(b + o_eoff);
  L.dofs = reinterpret_cast<int32_t*>(b + o_dofs);
  L.g1.flag = reinterpret_cast<int32_t*>(b + o_flag);
  L.g2.flag = L.g1.flag;
  L.n_rows = L.g1.flag + 4;
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

__global__ void store_rows_kernel(const int32_t* __restrict__ eoff, int64_t n_vert, int32_t* n_rows) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *n_rows = int32_t(n_vert + eoff[n_vert]);
}

// Chunks of four incidences per row.
__global__ void chunk_count_kernel(const int32_t* __restrict__ inc_off, int64_t n_rows, int32_t* cnt) {
  for (int64_t r = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; r < n_rows; r += int64_t(gridDim.x) * blockDim.x)
    cnt[r] = (inc_off[r + 1] - inc_off[r] + 3) / 4;
}

template <int NB>
__global__ void chunk_fill_kernel(const int32_t* __restrict__ inc_off, const int32_t* __restrict__ inc,
                                  const uint8_t* __restrict__ colpos, const int32_t* __restrict__ choff,
                                  int64_t n_rows, int64_t cap, int4* __restrict__ slot4, uint32_t* __restrict__ pos4) {
  if (choff[n_rows] > cap) return;  // no room: the rows are read one incidence at a time
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
    store_rows_kernel<<<1, 32, 0, st>>>(L.eoff, n_vert, L.n_rows);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(rows_host, L.n_rows, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
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
    chunk_count_kernel<<<grid_of(R, 256), 256, 0, st>>>(G2.inc_off, R, G2.cursor);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = launch_exclusive_scan(G2.cursor, R, G2.partials, L.choff, st);
  if (e == cudaSuccess && R > 0) {
    chunk_fill_kernel<NB><<<grid_of(R, 256), 256, 0, st>>>(G2.inc_off, G2.inc, G2.colpos, L.choff, R, L.chunk_cap,
                                                           L.slot4, L.pos4);
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
// under the additions.  61^3 cube: 312 -> 281 us; bound by instruction issue
// (68% active) and that pipe (70%), two accesses an addition, 2.6 wavefronts
// each over the random columns of three rows.  48 registers: five warps of
// these buffers per SM quarter and more (40 registers spill: 330 us, 63
// registers 309 us, without the loads ahead 314 us).
// A warp with a row of more than kRowCols columns, or a mesh without room for
// the chunks, takes its rows one after another, an incidence at a time.
constexpr int kRowWarps = 4;
constexpr int kRowCols = 160;
constexpr int kRowStride = kRowCols + 11;  // the rows of a warp start 11 banks apart
static_assert(3 * kRowStride >= kMaxCols, "one row of any length in the buffers of three");

template <int NB>
__global__ void __launch_bounds__(kRowWarps * 32, 10)
    assemble_rows_kernel(const int32_t* __restrict__ inc_off, const int32_t* __restrict__ inc,
                         const uint8_t* __restrict__ colpos, const int32_t* __restrict__ row_ptr,
                         const int32_t* __restrict__ choff, const int4* __restrict__ slot4,
                         const uint32_t* __restrict__ pos4, int64_t chunk_cap, const float* __restrict__ A,
                         const int32_t* n_rows_dev, float* __restrict__ val) {
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
  int64_t r0 = (int64_t(blockIdx.x) * kRowWarps + warp) * G;
  grid_wait(r0, n_rows_dev);
  const int64_t n_rows = *n_rows_dev;
  const bool chunked = choff[n_rows] <= chunk_cap;
  const int64_t S = int64_t(gridDim.x) * kRowWarps * G;
  if (r0 >= n_rows) return;  // warp-uniform: no CTA-wide barrier
  // chunks [c0, c0 + nch) of the lane's row, its first value, the values of the warp's rows
  struct Rows {
    int32_t c0, nch, rp, total;
  };
  auto load_rows = [&](int64_t q0) {
    Rows m{0, 0, 0, 0};
    if (q0 >= n_rows) return m;
    const int64_t r = q0 + g;
    const bool live = g < G && r < n_rows;
    m.c0 = live ? __ldg(choff + r) : 0;
    m.nch = live ? __ldg(choff + r + 1) - m.c0 : 0;
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
      const int64_t c = int64_t(m.c0) + k + h;
      const int4 q = on ? __ldg(slot4 + c) : make_int4(-1, -1, -1, -1);
      sn[4 * h] = q.x, sn[4 * h + 1] = q.y, sn[4 * h + 2] = q.z, sn[4 * h + 3] = q.w;
      pn[h] = on ? __ldg(pos4 + c * NB + j) : 0u;
    }
  };
  Rows m = load_rows(r0);
  if (chunked) load_chunks(m, 0);
  for (; r0 < n_rows; r0 += S) {
    const Rows mn = load_rows(r0 + S);
    const int32_t rp0 = __shfl_sync(0xffffffffu, m.rp, 0);
    int32_t first[G + 1];  // of each row, within the warp's run of values
#pragma unroll
    for (int h = 0; h < G; ++h) first[h] = __shfl_sync(0xffffffffu, m.rp, h * NB) - rp0;
    first[G] = m.total - rp0;
    bool fast = chunked;
#pragma unroll
    for (int h = 0; h < G; ++h) fast &= first[h + 1] - first[h] <= kRowCols;
    if (fast) {
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
      for (int x = lane; x < first[G]; x += 32) {
        int at = x;
#pragma unroll
        for (int h = 1; h < G; ++h)
          if (x >= first[h]) at = x - first[h] + h * kRowStride;
        __stcs(val + int64_t(rp0) + x, rows[at]);
        rows[at] = 0.f;
      }
      __syncwarp();  // the row buffers are refilled for the next rows
    } else {
      if (chunked) load_chunks(mn, 0);
      for (int h = 0; h < G && r0 + h < n_rows; ++h) {
        const int32_t tb = __ldg(inc_off + r0 + h), te = __ldg(inc_off + r0 + h + 1);
        for (int32_t t = tb; t < te; ++t) {
          if (lane < NB)
            rows[__ldg(colpos + int64_t(t) * NB + lane)] += __ldg(A + int64_t(__ldg(inc + t)) * NB + lane);
          __syncwarp();
        }
        const int32_t rp = __ldg(row_ptr + r0 + h), len = __ldg(row_ptr + r0 + h + 1) - rp;
        for (int x = lane; x < len; x += 32) {
          __stcs(val + int64_t(rp) + x, rows[x]);
          rows[x] = 0.f;
        }
        __syncwarp();
      }
    }
    m = mn;
  }
}

template <int NB>
cudaError_t launch_p2_assemble(const AsmP2Layout& L, const float* A, float* val, cudaStream_t st) {
  return launch_chained(assemble_rows_kernel<NB>, grid_of(L.rows_cap, kRowWarps * (32 / NB)), kRowWarps * 32, 0, st,
                        L.g2.inc_off, L.g2.inc, L.g2.colpos, L.g2.row_ptr, L.choff, L.slot4, L.pos4, L.chunk_cap, A,
                        L.n_rows, val);
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
  cudaError_t e = cudaMemsetAsync(L.flag, 0, sizeof(int32_t) * 4, st);
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
  if (e == cudaSuccess && B == 1 && mesh->n_elem > 0) {  // the scalar forms refuse an element repeating a vertex
    const unsigned g = fem::grid_of(mesh->n_elem, 256);
    if (mesh->dim == 2)
      fem::check_repeat_kernel<3><<<g, 256, 0, st>>>(mesh->conn, mesh->n_elem, L.flag);
    else
      fem::check_repeat_kernel<4><<<g, 256, 0, st>>>(mesh->conn, mesh->n_elem, L.flag);
    e = cudaGetLastError();
  }
  int32_t host[2] = {0, 0}, nrec = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&host[0], L.flag, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&host[1], L.row_ptr + V, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess && host[0] == 0 && V > 0) {
    if (mesh->dim == 2)
      e = B == 1 ? fem::launch_row_blocks<3, 1>(V, L, st) : fem::launch_row_blocks<3, 2>(V, L, st);
    else
      e = B == 1 ? fem::launch_row_blocks<4, 1>(V, L, st) : fem::launch_row_blocks<4, 3>(V, L, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&nrec, L.flag + 1, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
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
  if (nnz) *nnz = host[1];
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
    const cudaError_t e = cudaMemcpy(&r, P.n_rows, sizeof(int32_t), cudaMemcpyDeviceToHost);
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
    e = B == 1 ? fem::launch_assemble_t<3, 1>(L, A, mesh->n_vert, values, st)
               : fem::launch_assemble_t<3, 2>(L, A, mesh->n_vert, values, st);
  } else {
    e = B == 1 ? fem::launch_assemble_t<4, 1>(L, A, mesh->n_vert, values, st)
               : fem::launch_assemble_t<4, 3>(L, A, mesh->n_vert, values, st);
  }
  if (e != cudaSuccess) {
    fem::set_last_error("fem_assemble: %s", cudaGetErrorString(e));
    return FEM_ERR_CUDA;
  }
  return FEM_OK;
}

}  // extern "C"
