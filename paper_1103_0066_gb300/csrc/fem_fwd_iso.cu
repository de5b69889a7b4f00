// fem_fwd_iso.cu -- forward integration of the Laplacian on non-affine
// (quadratic-geometry) elements, Eqs. 16-19.
//
// Each element is given by its d+1 vertices (conn, coords) and the d(d+1)/2
// edge-midpoint nodes of its quadratic geometry map (mid, element by
// element).  Per lane (one element):
//   1. the nodes relative to vertex 0 (so the map's derivatives see small
//      differences, not absolute coordinates);
//   2. J at every vertex k from the derivatives of the quadratic geometry
//      basis there (small integers, compile time), its adjugate and det, and
//      J^{-1}_k = adj / det -- the values the projection of Eq. 17 interpolates;
//   3. |J| = |det J| at the centroid (Eq. 17 keeps |J| outside the integral);
//   4. A_ij = w |J| / DEN sum K^{ij}_{(k mu),(l nu)} J^{-1}_{mu a,k} J^{-1}_{nu a,l}
//      (Eq. 18) by the structure of K (fem_iso_mat.cuh): P2 tets take 2041
//      instructions a tile of 32 elements where the sum over the 78 folded
//      G entries took 3680, outgrew the instruction caches and was bound by
//      them (64^3 cube: 265 -> 162 us, 130 us with the bulk store); then the same tile
//      store as the affine kernel (Eq. 19).
// The Jacobian steps run in plain FP32: this path serves curved, non-sliver
// elements; an element with a singular J at a vertex or at the centroid is
// flagged degenerate and gets A = 0.
#include "fem_fwd.cuh"
#include "fem_iso_mat.cuh"

namespace fem {

namespace {

// acc = the upper triangle of A_e: the sums of fem_iso_mat.cuh times the
// common factor scale = w |J| / DEN.
template <int D, int FORM>
__device__ __forceinline__ void iso_accumulate(const float (&ji)[D + 1][D][D], float scale, float* acc) {
  if constexpr (FormTraits<D, FORM>::DEG == 1)
    iso_matrix_p1<D>(ji, acc);
  else
    iso_matrix_p2<D>(ji, acc);
#pragma unroll
  for (int t = 0; t < FormTraits<D, FORM>::NT; ++t) acc[t] *= scale;
}

template <int D, int FORM, class Sink, int... Ts>
__device__ __forceinline__ void put_all(Sink& sink, const float* acc, std::integer_sequence<int, Ts...>) {
  using FT = FormTraits<D, FORM>;
  (sink.template put<tri_row(Ts, FT::N), tri_col(Ts, FT::N)>(acc[Ts]), ...);
}

// CTA shape: warps never wait for one another, so the CTA size only sets how
// finely the register file is shared out.  On tets the P1 form runs one-warp
// CTAs with at least 20 resident per SM, which it reaches with 85 registers and
// without spills (24 or 32 CTAs spill and gain nothing); the P2 form with at
// least 16, which holds its 55 accumulators and four inverse Jacobians to 128
// registers (28 bytes spilled).
template <int D, int FORM>
struct IsoShape {
  static constexpr bool tight = (D == 3);
  static constexpr int threads = tight ? 32 : 128;
  static constexpr int min_ctas = tight ? (FORM == LAPLACE_P1_ISO ? 20 : 16) : 1;
};

// Per warp: [output stage][edge nodes of a tile][its coordinates].  The inputs
// are copied one tile ahead, except on P2 tets, where the 3.8 KB they take
// beside the 12.8 KB output stage cost more resident warps than the wait saved
// (64^3 cube, forward + adjoint 386 against 381 us; P1 tets 173 -> 168 us, P2
// triangles at 700 x 700 x 2 111 -> 100 us).
template <int D, int FORM, int ST>
struct IsoFwdPlan {
  using PL = FwdPlan<D, FORM, float, float>;
  static constexpr bool ahead = D == 2 || FORM == LAPLACE_P1_ISO;
  static constexpr size_t stage = PL::stage_of(ST);
  static constexpr size_t mid_bytes = align_up(size_t(32) * (D * D * (D + 1) / 2) * 4, 128);
  static constexpr size_t per_warp = stage + (ahead ? mid_bytes + 32 * (D + 1) * D * 4 : 0);
};

template <int D, int FORM, int ST>
__global__ void __launch_bounds__(IsoShape<D, FORM>::threads, IsoShape<D, FORM>::min_ctas)
    fem_fwd_iso_kernel(FwdParams<float, float> p, const float* __restrict__ mid) {
  using FT = FormTraits<D, FORM>;
  using PL = FwdPlan<D, FORM, float, float>;
  constexpr int NE = D * (D + 1) / 2;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  using IP = IsoFwdPlan<D, FORM, ST>;
  unsigned char* wbase = smem_raw + size_t(warp) * IP::per_warp;
  float* st = reinterpret_cast<float*>(wbase);
  float* ms = reinterpret_cast<float*>(wbase + IP::stage);                         // [32][NE * D]
  float* xs = reinterpret_cast<float*>(wbase + IP::stage + IP::mid_bytes) + lane;  // [(D + 1) * D][32]
  const int64_t ntiles = (p.n_elem + 31) / 32;
  const int64_t S = int64_t(gridDim.x) * nwarps;
  int64_t t = int64_t(blockIdx.x) * nwarps + warp;
  grid_wait(t);
  if (t >= ntiles) return;  // warp-uniform: the kernel has no CTA-wide barrier
  int err = 0, fnext = 0;
  int v[D + 1];
  load_conn<D>(p.conn, t * 32 + lane, p.n_elem, p.vec_conn, v);
  // copies tile's edge nodes and, by the vertex ids in v, its coordinates, then
  // loads the ids of the tile after it; the tile's gather flags
  auto copy_ahead = [&](int64_t tile) {
    int flags = 0;
    if (tile < ntiles) {
      const int cnt = int(p.n_elem - tile * 32 < 32 ? p.n_elem - tile * 32 : 32);
      tile_load_async(ms, mid + tile * 32 * (NE * D), cnt * (NE * D), lane);
      if (lane < cnt) {
        bool good = true;
#pragma unroll
        for (int k = 0; k <= D; ++k) good &= uint32_t(v[k]) < uint32_t(p.n_vert);
        flags = good ? GF_ELEM | GF_OK : GF_ELEM;
        if (good)
#pragma unroll
          for (int k = 0; k <= D; ++k)
#pragma unroll
            for (int a = 0; a < D; ++a) cp_async<4>(xs + (k * D + a) * 32, p.coords + uint32_t(v[k]) * uint64_t(D) + a);
      }
    }
    cp_async_commit();
    load_conn<D>(p.conn, (tile + S) * 32 + lane, p.n_elem, p.vec_conn, v);
    return flags;
  };
  if constexpr (IP::ahead) fnext = copy_ahead(t);
  for (; t < ntiles; t += S) {
    const int64_t e = t * 32 + lane;
    float X[D + 1][D];
    int flags = fnext;
    if constexpr (IP::ahead) {
      cp_async_wait<0>();
      __syncwarp();  // the tile's edge nodes were copied by other lanes
#pragma unroll
      for (int k = 0; k <= D; ++k)
#pragma unroll
        for (int a = 0; a < D; ++a) X[k][a] = xs[(k * D + a) * 32];
    } else {
      flags = gather_regs<D>(p.coords, p.n_vert, e, p.n_elem, v, X);
    }
    float ji[D + 1][D][D];
    float scale = 0.f;
    bool ok = false;
    if (flags & GF_OK) {
      const float w = (p.coef && e < p.n_elem) ? __ldg(p.coef + e) : 1.f;
      ok = iso_geometry<D, FORM, IP::ahead>(X, IP::ahead ? ms + lane * (NE * D) : mid + e * (NE * D), w, ji, scale);
      if (!ok) err |= DEVERR_DEGENERATE;
    } else if (flags & GF_ELEM) {
      err |= DEVERR_CONN;
    }
    if constexpr (IP::ahead) {
      __syncwarp();  // every lane has read its edge nodes: the next tile's may arrive
      fnext = copy_ahead(t + S);
    } else {
      load_conn<D>(p.conn, e + S * 32, p.n_elem, p.vec_conn, v);
    }
    fwd_fill_store<D, FORM, float, float, ST>(
        p, t, lane,
        [&](auto& sink) {
          float acc[FT::NT];
#pragma unroll
          for (int i = 0; i < FT::NT; ++i) acc[i] = 0.f;
          if (ok) iso_accumulate<D, FORM>(ji, scale, acc);
          put_all<D, FORM>(sink, acc, std::make_integer_sequence<int, FT::NT>{});
        },
        st, nullptr);
  }
  cp_async_wait<0>();
  if constexpr (ST == ST_BULK) bulk_wait<0>();  // the stage outlives every copy that reads it
  err = __reduce_or_sync(0xffffffffu, err);
  if (err && lane == 0 && p.dev_err) atomicOr(p.dev_err, err);
}

template <int D, int FORM>
cudaError_t launch_iso_t(const FwdLaunch& L, const float* mid) {
  FwdParams<float, float> p;
  p.conn = L.conn;
  p.coords = static_cast<const float*>(L.coords);
  p.coef = L.coef;
  p.A = static_cast<float*>(L.A);
  p.n_elem = L.n_elem;
  p.n_vert = L.n_vert;
  p.dev_err = L.dev_err;
  p.vec_conn = (D == 3) && (reinterpret_cast<uintptr_t>(L.conn) % 16 == 0);
  p.vec_store = (reinterpret_cast<uintptr_t>(L.A) % 16 == 0);
  using PL = FwdPlan<D, FORM, float, float>;
  constexpr int unaligned = PL::SCALAR ? ST_SCALAR : PL::plain_store;
  const bool wide = p.vec_store || !PL::SCALAR;
  auto kern = wide ? fem_fwd_iso_kernel<D, FORM, PL::plain_store> : fem_fwd_iso_kernel<D, FORM, unaligned>;
  const int warps = IsoShape<D, FORM>::threads / 32;
  const size_t per_warp =
      wide ? IsoFwdPlan<D, FORM, PL::plain_store>::per_warp : IsoFwdPlan<D, FORM, unaligned>::per_warp;
  const size_t smem = size_t(warps) * per_warp;
  cudaError_t st = ensure_smem(reinterpret_cast<const void*>(kern), smem);
  if (st != cudaSuccess) return st;
  const unsigned grid = pipeline_grid(reinterpret_cast<const void*>(kern), warps, smem, L.n_elem, L.ctas_per_sm);
  return launch_chained(kern, grid, unsigned(warps * 32), smem, L.stream, p, mid);
}

}  // namespace

cudaError_t launch_fwd_iso(const FwdLaunch& L, const float* mid) {
  if (L.dim == 2) {
    if (L.form == LAPLACE_P1_ISO) return launch_iso_t<2, LAPLACE_P1_ISO>(L, mid);
    if (L.form == LAPLACE_P2_ISO) return launch_iso_t<2, LAPLACE_P2_ISO>(L, mid);
  } else {
    if (L.form == LAPLACE_P1_ISO) return launch_iso_t<3, LAPLACE_P1_ISO>(L, mid);
    if (L.form == LAPLACE_P2_ISO) return launch_iso_t<3, LAPLACE_P2_ISO>(L, mid);
  }
  return cudaErrorInvalidValue;
}

}  // namespace fem
