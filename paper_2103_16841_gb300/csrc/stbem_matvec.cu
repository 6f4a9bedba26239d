// Products with the assembled operator over the block-banded storage.
//
// Storage (built by the quadrature epilogue): for the block of test column I
// and trial column J, every test row r of column I owns a band of W_IJ
// consecutive trial panels starting at rs[r]; the band values are stored
// column-major, value (r, w) at val[boff + w * R_I + r].
//
// Arithmetic choices, y = A x with x, y in FP64 at the boundary:
//   MV_FP64  FP64 accumulation of FP64 values (or of FP32 values when the
//            operator keeps FP32 values only) - residuals, FP64 solves;
//   MV_FP32  FP32 values, x rounded to FP32, FP32 accumulation - inner solves;
//   MV_TF32  tensor-core product (tcgen05, stbem_spmm_tc.cu): FP32 values
//            and x rounded to TF32 (10-bit mantissa), FP32 accumulation;
//   MV_BF16  the same on a BF16 copy of the values, x in BF16.
// The tensor-core path treats every block as a dense (rows of I) x K tile
// over the union of its rows' bands and multiplies it with the K x nrhs slab
// of x; each stored value is read from HBM once per 64 right-hand sides.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <numeric>
#include <type_traits>
#include <vector>

#include "stbem_internal.h"

namespace stbem {

// ---------------------------------------------------------------------------
// SpMV for one to a few right-hand sides (NR at a time, the matrix is read
// once per NR). A cluster of 1 to 8 CTAs per test column I. A thread owns VEC
// consecutive rows and reads VEC values (16 bytes where the column sizes allow
// it) at once; the cluster's threads form as many slots of a column's rows as
// fit, and slot s takes the trial columns s, s + slots, ...: columns of 24
// panels fill 252 of 256 threads, where a warp per column and a value per load
// left a quarter of the lanes idle and kept 48 bytes per thread in flight. The
// CTAs of a cluster give their sums to the first through its shared memory.
// FP32: bound by the latency of a block's chain (record, row start, values and
// x) and the HBM reads. FP64 accumulation: by the FP64 pipe (2 lanes per SM and
// cycle), so a thread takes one row (all lanes of a warp then share a block or
// two) and FP32 values widen in integer arithmetic.
// Level-3 sphere, 8 slabs (1.39 GB of FP32 values): one FP32 vector 803 ->
// 378 us (3.7 TB/s), four 1,789 -> 557 us; FP64 accumulation of one vector 3.38
// -> 1.56 ms, of five 11.7 -> 5.2 ms. Level-2 sphere, 15 slabs (columns of 45
// panels, one row per thread): 148 -> 97 us, FP64 of five 1.93 -> 0.82 ms.
// Icosahedron, 3 slabs, 64 FP32 vectors: 158 -> 18 us (one launch).
// ---------------------------------------------------------------------------
// CTAs per SM of the register budget, FP32, one right-hand side (level-3 sphere, 8 slabs:
// 572 us unbounded, 387 us with 5, 621 us with 6, which spills); four are best unbounded
constexpr int mv_ctas(int nr, int acc) { return acc == 4 && nr == 1 ? 5 : 0; }
constexpr int kMvThreads = 256;   // >= MAX_COL_TETS: at least one slot
static_assert(kMvThreads >= MAX_COL_TETS, "a column's rows fit the CTA");

template <typename V, int VEC>
struct alignas(sizeof(V) * VEC) Pack { V v[VEC]; };

// (double)f of a finite f; the conversion instruction takes the FP64 pipe as long as a fused multiply-add
__device__ __forceinline__ double widen(float f) {
  const uint32_t u = __float_as_uint(f), m = u & 0x7fffffffu;
  if (m - 1u < 0x007fffffu) return (double)f;   // denormal
  const uint32_t hi = (m >> 3) + 0x38000000u;
  return __hiloint2double((int)((u & 0x80000000u) | (m ? hi : 0u)), (int)(u << 29));
}
template <typename Acc, typename V>
__device__ __forceinline__ Acc value_as(V v) {
  if constexpr (sizeof(Acc) == 8 && sizeof(V) == 4) return widen(v);
  else return (Acc)v;
}

// x: [n][NR] when PACKED (one load serves the NR right-hand sides), else [NR][ld]
template <typename V, typename Acc, typename XT, int NR, int VEC, bool PACKED>
__device__ __forceinline__ void matvec_col(int64_t n_col, const int32_t* __restrict__ ctb,
                                           const int32_t* __restrict__ bw, const int64_t* __restrict__ boff,
                                           const int64_t* __restrict__ rsoff, const int32_t* __restrict__ rs,
                                           const V* __restrict__ val, const XT* __restrict__ x,
                                           double* __restrict__ y, int64_t ld, int nr, int64_t I, Acc* red) {
  namespace cg = cooperative_groups;
  auto cl = cg::this_cluster();
  const int part = (int)cl.block_rank(), parts = (int)cl.num_blocks();
  const int t0 = ctb[I], nt = ctb[I + 1] - t0, ntv = nt / VEC;
  const int slots = kMvThreads / ntv, slot = threadIdx.x / ntv, r = (threadIdx.x - slot * ntv) * VEC;
  const int first = part * slots + slot, step = parts * slots;
  Acc acc[VEC][NR];
#pragma unroll
  for (int v = 0; v < VEC; ++v)
#pragma unroll
    for (int k = 0; k < NR; ++k) acc[v][k] = Acc(0);
  if (slot < slots) {
    // block metadata of the slot's next J is fetched while the current block is summed
    int W_n = 0, je_n = 0;
    int64_t vo_n = 0, ro_n = 0;
    if (first < n_col) {
      const int64_t b = I * n_col + first;
      W_n = bw[b]; vo_n = boff[b]; ro_n = rsoff[b]; je_n = ctb[first + 1];
    }
    for (int64_t J = first; J < n_col; J += step) {
      const int W = W_n, je = je_n;
      const int64_t vo = vo_n, ro = ro_n;
      if (J + step < n_col) {
        const int64_t b = I * n_col + J + step;
        W_n = bw[b]; vo_n = boff[b]; ro_n = rsoff[b]; je_n = ctb[J + step + 1];
      }
      if (W == 0) continue;
      const Pack<int32_t, VEC> start = *reinterpret_cast<const Pack<int32_t, VEC>*>(rs + ro + r);
      const V* vp = val + vo + r;
      constexpr int CW = sizeof(Acc) == 4 || NR >= 4 ? 4 : 8;
      for (int w0 = 0; w0 < W; w0 += CW) {
        // the band values of a run are loaded together, then summed in order
        Pack<V, VEC> a[CW];
#pragma unroll
        for (int u = 0; u < CW; ++u)
          if (w0 + u < W) a[u] = *reinterpret_cast<const Pack<V, VEC>*>(vp + (int64_t)(w0 + u) * nt);
#pragma unroll
        for (int u = 0; u < CW; ++u)
#pragma unroll
          for (int v = 0; v < VEC; ++v) {
            const int j = start.v[v] + w0 + u;
            if (w0 + u < W && j < je) {   // (bands may reach past the column's end)
              const Acc av = value_as<Acc, V>(a[u].v[v]);
              if constexpr (PACKED) {
                const Pack<XT, NR> xv = *reinterpret_cast<const Pack<XT, NR>*>(x + (int64_t)j * NR);
#pragma unroll
                for (int k = 0; k < NR; ++k) acc[v][k] += av * (Acc)xv.v[k];
              } else {
#pragma unroll
                for (int k = 0; k < NR; ++k)
                  if (k < nr) acc[v][k] += av * (Acc)x[(int64_t)k * ld + j];
              }
            }
          }
      }
    }
#pragma unroll
    for (int v = 0; v < VEC; ++v)
#pragma unroll
      for (int k = 0; k < NR; ++k) red[(slot * nt + r + v) * NR + k] = acc[v][k];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < nt * nr; t += kMvThreads) {
    const int k = t / nt, row = t - k * nt;
    Acc sum = Acc(0);
    for (int q = 0; q < slots; ++q) sum += red[(q * nt + row) * NR + k];
    if (parts == 1) y[(int64_t)k * ld + t0 + row] = (double)sum;
    else red[row * NR + k] = sum;   // (slot 0's place, read by this thread alone)
  }
  if (parts > 1) {
    cl.sync();
    if (part == 0)
      for (int t = threadIdx.x; t < nt * nr; t += kMvThreads) {
        const int k = t / nt, row = t - k * nt;
        Acc sum = Acc(0);
        for (int q = 0; q < parts; ++q) sum += cl.map_shared_rank(red, q)[row * NR + k];
        y[(int64_t)k * ld + t0 + row] = (double)sum;
      }
    cl.sync();
  }
}

template <typename V, typename Acc, typename XT, int NR, int VEC, bool PACKED>
__global__ void __launch_bounds__(kMvThreads, mv_ctas(NR, sizeof(Acc))) k_matvec(int64_t n_col, const int32_t* __restrict__ ctb,
                         const int32_t* __restrict__ bw, const int64_t* __restrict__ boff,
                         const int64_t* __restrict__ rsoff, const int32_t* __restrict__ rs, const V* __restrict__ val,
                         const XT* __restrict__ x, double* __restrict__ y, int64_t n_tet, int nrhs) {
  extern __shared__ __align__(16) unsigned char red[];
  const int r0 = NR == 1 ? 0 : blockIdx.y * NR;   // (one vector is one group)
  matvec_col<V, Acc, XT, NR, VEC, PACKED>(n_col, ctb, bw, boff, rsoff, rs, val, x + r0 * n_tet, y + r0 * n_tet, n_tet,
                                          NR == 1 ? 1 : min(NR, nrhs - r0),
                                          blockIdx.x / cooperative_groups::this_cluster().num_blocks(),
                                          reinterpret_cast<Acc*>(red));
}

// The same over the block-diagonal operator of a batch: CTA k works on
// column cta_col[k] of segment cta_seg[k]; a segment's entries start at
// off within each of the vectors of length ld.
struct MvSeg {
  int64_t n_col, off;
  const int32_t* ctb;
  const int32_t* bw;
  const int64_t* boff;
  const int64_t* rsoff;
  const int32_t* rs;
  const void* val;
};

template <typename V, typename Acc, typename XT, int NR, int VEC, bool PACKED>
__global__ void __launch_bounds__(kMvThreads, mv_ctas(NR, sizeof(Acc))) k_matvec_batch(const MvSeg* __restrict__ segs,
                               const int32_t* __restrict__ cta_seg, const int32_t* __restrict__ cta_col,
                               const XT* __restrict__ x, double* __restrict__ y, int64_t ld, int nrhs) {
  extern __shared__ __align__(16) unsigned char red[];
  const unsigned col = blockIdx.x / cooperative_groups::this_cluster().num_blocks();
  const MvSeg sg = segs[cta_seg[col]];
  const int r0 = NR == 1 ? 0 : blockIdx.y * NR;   // (one vector is one group)
  matvec_col<V, Acc, XT, NR, VEC, PACKED>(sg.n_col, sg.ctb, sg.bw, sg.boff, sg.rsoff, sg.rs,
                                          static_cast<const V*>(sg.val), x + r0 * ld + (PACKED ? NR * sg.off : sg.off),
                                          y + r0 * ld + sg.off, ld, NR == 1 ? 1 : min(NR, nrhs - r0), cta_col[col],
                                          reinterpret_cast<Acc*>(red));
}

// out[g][j][k] = x[NR g + k][j] in FP32 (zero past the last vector)
template <int NR>
__global__ void k_pack_x(const double* __restrict__ x, float* __restrict__ out, int64_t n, int nrhs) {
  const int64_t total = n * ((nrhs + NR - 1) / NR);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t g = i / n, j = i - g * n;
    Pack<float, NR> v;
#pragma unroll
    for (int k = 0; k < NR; ++k) v.v[k] = NR * g + k < nrhs ? (float)x[(NR * g + k) * n + j] : 0.f;
    *reinterpret_cast<Pack<float, NR>*>(out + i * NR) = v;
  }
}

unsigned grid_for(int64_t n) { return (unsigned)std::min<int64_t>((n + 255) / 256, 152 * 16); }

bem_status ensure_ws(const bem_operator* op, int64_t floats) {
  if (op->ws_len >= floats) return BEM_OK;
  if (op->d_ws) cudaFree(op->d_ws);
  op->d_ws = nullptr;
  op->ws_len = 0;
  if (device_alloc((void**)&op->d_ws, sizeof(float) * floats) != cudaSuccess) {
    cudaGetLastError();
    set_error("out of device memory (matvec workspace)");
    return BEM_ERR_OUT_OF_MEMORY;
  }
  op->ws_len = floats;
  return BEM_OK;
}

// rows per thread: as many as divide every column and make 16 bytes; one where the FP64 pipe is the bound
template <typename V, typename Acc>
static int vec_width(int col_gcd) {
  if (sizeof(Acc) == 8) return 1;
  return col_gcd % 4 == 0 ? 4 : col_gcd % 2 == 0 ? 2 : 1;
}

// f(rows per thread, right-hand sides per pass) as compile-time constants
template <typename F>
static bem_status with_shape(int vec, int nr, F f) {
  auto g = [&](auto v) {
    return nr == 1 ? f(v, std::integral_constant<int, 1>()) : f(v, std::integral_constant<int, 4>());
  };
  if (vec == 4) return g(std::integral_constant<int, 4>());
  if (vec == 2) return g(std::integral_constant<int, 2>());
  return g(std::integral_constant<int, 1>());
}

// CTAs per test column: enough for five CTAs per SM (ten: level-2 sphere, 32
// slabs 341 us for 274 us), at most a portable cluster, and no more than have a
// trial column for each of their slots
static unsigned mv_cluster(int64_t n_ctas, int64_t n_col, int slots) {
  unsigned c = 1;
  while (c < 8 && (int64_t)c * n_ctas < 5 * 152 && (int64_t)c * slots < n_col) c *= 2;
  return c;
}

template <typename K, typename... Args>
static bem_status mv_launch(K kern, int64_t n_cols, unsigned groups, unsigned c, size_t smem, cudaStream_t s, Args... args) {
  const bem_status st = ensure_smem_attr((const void*)kern, smem);
  if (st != BEM_OK) return st;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n_cols * c), groups);
  cfg.blockDim = dim3(kMvThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = c;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  STBEM_CUDA(cudaLaunchKernelEx(&cfg, kern, args...));
  return BEM_OK;
}

// Right-hand sides [r0, r0 + k) in launches of at most as many groups of nr as a grid has layers
constexpr int kMaxLayers = 65535;
template <typename F>
static bem_status in_layers(int nr, int r0, int k, F launch) {
  for (const int end = r0 + k; r0 < end;) {
    const int n = std::min<int64_t>(end - r0, (int64_t)kMaxLayers * nr);
    const bem_status st = launch(r0, n);
    if (st != BEM_OK) return st;
    r0 += n;
  }
  return BEM_OK;
}

// A layer of the grid per group of NR right-hand sides; x packed [group][n][NR] (PACKED) or [nrhs][n].
template <typename V, typename Acc, typename XT, bool PACKED>
static bem_status spmv_launch(const bem_operator* op, const V* val, const XT* x, double* y, int nrhs, cudaStream_t s) {
  const bem_mesh* m = op->mesh;
  const int64_t n = m->n_tet;
  return with_shape(vec_width<V, Acc>(m->col_gcd), nrhs, [&](auto vec, auto nrc) -> bem_status {
    constexpr int VEC = sizeof(Acc) == 8 ? 1 : decltype(vec)::value, NR = decltype(nrc)::value;
    const unsigned c = mv_cluster(m->n_col, m->n_col, kMvThreads * VEC / m->max_col_tets);
    auto launch = [&](auto kern, int nr, int first, int count) {   // nr right-hand sides at a time
      return in_layers(nr, first, count, [&](int r0, int k) {
        return mv_launch(kern, m->n_col, (unsigned)((k + nr - 1) / nr), c, sizeof(Acc) * kMvThreads * VEC * nr, s, m->n_col,
                         (const int32_t*)m->d_col_tet_begin, (const int32_t*)op->d_bw, (const int64_t*)op->d_boff,
                         (const int64_t*)op->d_rsoff, (const int32_t*)op->d_rs, val, x + (int64_t)r0 * n,
                         y + (int64_t)r0 * n, n, k);
      });
    };
    // a last vector alone takes the kernel for one (where x is not packed)
    const int alone = !PACKED && NR > 1 && nrhs % NR == 1 ? 1 : 0;
    bem_status st = launch(k_matvec<V, Acc, XT, NR, VEC, PACKED>, NR, 0, nrhs - alone);
    if (st == BEM_OK && alone) st = launch(k_matvec<V, Acc, XT, 1, VEC, PACKED>, 1, nrhs - 1, 1);
    return st;
  });
}

static void pack_x(const double* x, float* out, int64_t n, int nrhs, cudaStream_t s) {
  if (nrhs == 1) k_pack_x<1><<<grid_for(n), 256, 0, s>>>(x, out, n, 1);
  else k_pack_x<4><<<grid_for(n * ((nrhs + 3) / 4)), 256, 0, s>>>(x, out, n, nrhs);
}

// FP32 numbers of the packed x of nrhs vectors of n entries
int64_t packed_len(int64_t n, int nrhs) { return nrhs == 1 ? n : n * ((nrhs + 3) / 4) * 4; }

bem_status op_matvec(const bem_operator* op, const double* x, double* y, int nrhs, int arith, cudaStream_t s) {
  // matrix-free operators: the operator's own precision, whatever `arith` asks
  if (op->opts.matrix_free) return op_matvec_free(op, x, y, nrhs, s);
  const bem_mesh* m = op->mesh;
  const int64_t n = m->n_tet;
  if (arith == MV_TF32 || arith == MV_BF16) {
    // passes of up to 64 right-hand sides
    for (int r0 = 0; r0 < nrhs; r0 += 64) {
      const int nr = std::min(64, nrhs - r0);
      const bem_status st = op_spmm_tc(op, x + (int64_t)r0 * n, y + (int64_t)r0 * n, nr, arith == MV_BF16, s);
      if (st != BEM_OK) return st;
    }
    return BEM_OK;
  }
  if (arith == MV_FP32) {
    if (!op->d_val32) {
      set_error("operator has no FP32 values (store_fp32 = 0)");
      return BEM_ERR_INVALID_ARG;
    }
    const bem_status st = ensure_ws(op, packed_len(n, nrhs));
    if (st != BEM_OK) return st;
    pack_x(x, op->d_ws, n, nrhs, s);
    return spmv_launch<float, float, float, true>(op, op->d_val32, op->d_ws, y, nrhs, s);
  }
  if (op->d_val) return spmv_launch<double, double, double, false>(op, op->d_val, x, y, nrhs, s);
  // mixed-precision operators keep FP32 values only
  return spmv_launch<float, double, double, false>(op, op->d_val32, x, y, nrhs, s);
}

bem_status BatchMatvec::init(const std::vector<bem_operator*>& o, cudaStream_t s) {
  ops = o;
  const int S = (int)ops.size();
  std::vector<MvSeg> segs(S);
  std::vector<int32_t> cseg, ccol;
  N = 0;
  col_gcd = 0;
  max_rows = 1;
  max_cols = 1;
  fp64_values = ops.empty() ? false : ops[0]->d_val != nullptr;
  for (int i = 0; i < S; ++i) {
    const bem_operator* op = ops[i];
    if ((op->d_val != nullptr) != fp64_values) {
      set_error("a batch takes one value precision");
      return BEM_ERR_INVALID_ARG;
    }
    segs[i].n_col = op->mesh->n_col;
    segs[i].off = N;
    segs[i].ctb = op->mesh->d_col_tet_begin;
    segs[i].bw = op->d_bw;
    segs[i].boff = op->d_boff;
    segs[i].rsoff = op->d_rsoff;
    segs[i].rs = op->d_rs;
    segs[i].val = fp64_values ? (const void*)op->d_val : (const void*)op->d_val32;
    for (int64_t I = 0; I < op->mesh->n_col; ++I) {
      cseg.push_back(i);
      ccol.push_back((int32_t)I);
    }
    col_gcd = std::gcd(col_gcd, op->mesh->col_gcd);
    max_rows = std::max(max_rows, op->mesh->max_col_tets);
    max_cols = std::max(max_cols, op->mesh->n_col);
    N += op->mesh->n_tet;
  }
  n_cta = (int64_t)cseg.size();
  if (device_alloc((void**)&d_segs, sizeof(MvSeg) * std::max(S, 1)) != cudaSuccess ||
      device_alloc((void**)&d_cseg, sizeof(int32_t) * std::max<int64_t>(n_cta, 1)) != cudaSuccess ||
      device_alloc((void**)&d_ccol, sizeof(int32_t) * std::max<int64_t>(n_cta, 1)) != cudaSuccess) {
    cudaGetLastError();
    set_error("out of device memory (batch matvec tables)");
    return BEM_ERR_OUT_OF_MEMORY;
  }
  STBEM_CUDA(cudaMemcpyAsync(d_segs, segs.data(), sizeof(MvSeg) * S, cudaMemcpyHostToDevice, s));
  STBEM_CUDA(cudaMemcpyAsync(d_cseg, cseg.data(), sizeof(int32_t) * n_cta, cudaMemcpyHostToDevice, s));
  STBEM_CUDA(cudaMemcpyAsync(d_ccol, ccol.data(), sizeof(int32_t) * n_cta, cudaMemcpyHostToDevice, s));
  STBEM_CUDA(cudaStreamSynchronize(s));
  return BEM_OK;
}

BatchMatvec::~BatchMatvec() {
  if (d_segs) cudaFree(d_segs);
  if (d_cseg) cudaFree(d_cseg);
  if (d_ccol) cudaFree(d_ccol);
  if (d_xf) cudaFree(d_xf);
}

bem_status BatchMatvec::apply(const double* x, double* y, int K, int arith, cudaStream_t s) {
  const MvSeg* sg = static_cast<const MvSeg*>(d_segs);
  auto run = [&](auto v0, auto a0, auto x0, auto packed, const auto* xin) -> bem_status {
    using V = decltype(v0);
    using Acc = decltype(a0);
    using XT = decltype(x0);
    return with_shape(vec_width<V, Acc>(col_gcd), K, [&](auto vec, auto nrc) -> bem_status {
      constexpr int VEC = sizeof(Acc) == 8 ? 1 : decltype(vec)::value, NR = decltype(nrc)::value;
      constexpr bool PACKED = decltype(packed)::value;
      const unsigned c = mv_cluster(n_cta, max_cols, kMvThreads * VEC / max_rows);
      auto launch = [&](auto kern, int nr, int first, int count) {
        return in_layers(nr, first, count, [&](int r0, int k) {
          return mv_launch(kern, n_cta, (unsigned)((k + nr - 1) / nr), c, sizeof(Acc) * kMvThreads * VEC * nr, s, sg,
                           (const int32_t*)d_cseg, (const int32_t*)d_ccol, xin + (int64_t)r0 * N, y + (int64_t)r0 * N, N, k);
        });
      };
      const int alone = !PACKED && NR > 1 && K % NR == 1 ? 1 : 0;
      bem_status st = launch(k_matvec_batch<V, Acc, XT, NR, VEC, PACKED>, NR, 0, K - alone);
      if (st == BEM_OK && alone) st = launch(k_matvec_batch<V, Acc, XT, 1, VEC, PACKED>, 1, K - 1, 1);
      return st;
    });
  };
  if (arith == MV_FP32 && !fp64_values) {
    if (xf_len < packed_len(N, K)) {
      if (d_xf) cudaFree(d_xf);
      d_xf = nullptr;
      xf_len = 0;
      if (device_alloc((void**)&d_xf, sizeof(float) * packed_len(N, K)) != cudaSuccess) {
        cudaGetLastError();
        set_error("out of device memory (batch matvec workspace)");
        return BEM_ERR_OUT_OF_MEMORY;
      }
      xf_len = packed_len(N, K);
    }
    pack_x(x, d_xf, N, K, s);
    return run(0.f, 0.f, 0.f, std::true_type(), d_xf);
  }
  if (arith == MV_FP64 || arith == MV_FP32)
    return fp64_values ? run(0.0, 0.0, 0.0, std::false_type(), x) : run(0.f, 0.0, 0.0, std::false_type(), x);
  set_error("batched products support FP64 and FP32 arithmetic");
  return BEM_ERR_UNSUPPORTED;
}

}  // namespace stbem
