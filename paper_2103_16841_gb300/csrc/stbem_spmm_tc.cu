// Tensor-core block product Y = A X for up to 64 right-hand sides per pass
// (the multi-right-hand-side product of the GMRES solves; A in TF32 or BF16,
// FP32 accumulation in tensor memory).
//
// Storage of A (eq. int_bform assembled into column blocks): block (I, J)
// holds, for every panel row r of spatial column I, a band of W values
// starting at trial panel rs[r]. Within a block the union of the rows' bands
// is a contiguous range of trial panels [cmin, cend), so block (I, J) is a
// dense (rows of I) x (cend - cmin) tile with the band filled in and zeros
// elsewhere: a dense contraction with the matching rows of X.
//
// Operand layout in shared memory (no swizzle): 16-byte chunks along K; chunk
// kc of row m at kc * (rows * 16) + m * 16, i.e. core matrices of 8 rows x
// 16 bytes, K-adjacent core matrices rows * 16 bytes apart (leading byte
// offset), M/N-adjacent ones 128 bytes apart (stride byte offset).
//   X is packed per pass as Xc[chunk][rhs][16 bytes]; one chunk is N x 16
//   contiguous bytes, and a TMA box of {256-byte rows, N / 16 rows, 2
//   chunks} (one K step) lands in exactly this layout.
//   The values are kept, for this product, in the same chunks: row r's band
//   re-cut at the 16-byte chunk boundaries of the trial panel index (slot j
//   of row r = the chunk starting at panel E * (floor(rs[r] / E) + j), zeros
//   outside the band), stored per block as [slot][row] (made once from the
//   assembled values, BF16 or TF32-rounded). Slots of a row group are padded
//   to the widest band of its columns: on spheres with 6 to 32 slabs they take
//   1.6-2.3 x the values' bytes in BF16 and 1.3-1.6 x in TF32, with 3 slabs (14
//   columns per group) 4.0 x and 2.9 x.
//   Building a block's A tile is then a copy of whole chunks.
//
// The MMA's 128 rows hold as many consecutive test columns as fit ("row
// groups": five columns of 24 panels), so "block" below is a row group against
// a trial column: its rows' row starts and chunk slots are kept in the group's
// order. Per block the pipeline costs about a microsecond whatever its size,
// and a column of 24 panels used a fifth of the tile. The blocks of a group are
// shared by PARTS CTAs, whose sums are added at the end, where groups are few.
// Level-3 sphere, 8 slabs: BF16 with 13 right-hand sides 2.26 -> 0.61 ms, TF32
// with 64 2.59 -> 1.01 ms; level-2 sphere, 32 slabs (a column per group, two
// parts), 64 right-hand sides: TF32 0.78 -> 0.64 ms, BF16 0.49 -> 0.41 ms.
//
// One CTA per (row group, part), six warps:
//   warps 0-3  build the A tile of each block (thread = row: its slots to
//              their chunk positions, the previous band's other chunks
//              cleared) in shared memory (k_spmm_tc) or in tensor memory with
//              tcgen05.st (k_spmm_tm; the MMA then reads A from tensor
//              memory, and shared memory holds only B, slots and row starts,
//              so more stages fit), then read the accumulator rows out of
//              tensor memory (thread = row) into y;
//   warp 4     (one lane) loads, per block, the X rows (TMA tensor copies),
//              the value slots and the row starts (bulk copies) and the
//              block's record, into one of up to 6 pipeline stages;
//   warp 5     owns the tensor-memory allocation; one lane issues
//              tcgen05.mma (M = 128 rows, N = right-hand sides rounded up to
//              16, K = 16 BF16 or 8 TF32 per instruction) accumulating every
//              block of the column into one tensor-memory tile, and commits
//              each stage back to the builders and the loader.
// Which kernel and how many stages (1-6) run is timed once per shape.
// Every mbarrier wait is bounded (kWaitBudget); a wait that runs out flags
// the operator, stops the CTA's pipeline and writes NaN to its rows.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "stbem_internal.h"
#include "stbem_tc.cuh"

namespace stbem {

// One non-empty block of a row group, in the order of its trial columns.
struct TcBlk {
  int32_t je;          // end of trial column J (internal panel index)
  int32_t W;           // widest band of its columns
  int32_t nt;          // rows (panels of the group's columns)
  int32_t cmin;        // union of the rows' bands [cmin, cend), clipped to J
  int32_t cend;
  int32_t t0;          // first row
  int64_t J;           // trial column
  int64_t ro;          // row-start offset (the groups' row order)
  int64_t vc[2];       // offset of the block's chunk slots (16-byte units): BF16, TF32
  int64_t pad2;
};
static_assert(sizeof(TcBlk) == 64, "TcBlk layout");

#define TRY_STATUS(x)                 \
  do {                                \
    const bem_status st_ = (x);       \
    if (st_ != BEM_OK) return st_;    \
  } while (0)

namespace {

constexpr long long kWaitBudget = 4000000000LL;   // clock cycles (about 2 s) per wait
constexpr int kThreads = 192;
constexpr int kMaxStages = 6;
// after the stages: 3 mbarriers per stage and one more, the tensor-memory
// address and the abort flag
constexpr size_t kTailBytes = 256;
static_assert(8 * (3 * kMaxStages + 1) + 8 <= kTailBytes, "stage tail");
constexpr uint32_t kRsBytes = 1024;   // per stage: row starts (<= 784 bytes) and the block record
constexpr uint32_t kMetaOff = 896;

// chunk slots of a row's band of width W (E values per chunk)
__host__ __device__ constexpr int tc_slots(int W, int E) { return (W + 2 * E - 2) / E; }

// Block records (warp per block) and the row starts in the groups' row order.
// Rows whose own column has no values in the block get an empty band at the
// block's first panel.
__global__ void k_tc_meta(int64_t nb, const int32_t* __restrict__ bG, const int32_t* __restrict__ bJ,
                          const int32_t* __restrict__ bW, const int64_t* __restrict__ ro_, const int64_t* __restrict__ vc16,
                          const int64_t* __restrict__ vc32, int64_t n_col, const int32_t* __restrict__ gtb,
                          const int32_t* __restrict__ ctb, const TetDev* __restrict__ tets, const int32_t* __restrict__ bw,
                          const int64_t* __restrict__ rsoff, const int32_t* __restrict__ rs, TcBlk* __restrict__ out,
                          int32_t* __restrict__ prs, int* __restrict__ span) {
  const int64_t k = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (k >= nb) return;
  const int64_t J = bJ[k], ro = ro_[k];
  const int t0 = gtb[bG[k]], nt = gtb[bG[k] + 1] - t0;
  int lo = INT_MAX, hi = INT_MIN;
  for (int r = lane; r < nt; r += 32) {
    const int I = tets[t0 + r].col;
    const int64_t b = I * n_col + J;
    const int W = bw[b];
    if (W <= 0) continue;
    const int s = rs[rsoff[b] + (t0 + r - ctb[I])];
    lo = min(lo, s);
    hi = max(hi, s + W);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  for (int r = lane; r < nt; r += 32) {
    const int I = tets[t0 + r].col;
    const int64_t b = I * n_col + J;
    prs[ro + r] = bw[b] > 0 ? rs[rsoff[b] + (t0 + r - ctb[I])] : lo;
  }
  if (lane == 0) {
    const int je = ctb[J + 1];
    hi = min(hi, je);
    TcBlk t;
    t.je = je;
    t.W = bW[k];
    t.nt = nt;
    t.cmin = lo;
    t.cend = hi;
    t.t0 = t0;
    t.J = J;
    t.ro = ro;
    t.vc[0] = vc16[k];
    t.vc[1] = vc32[k];
    t.pad2 = 0;
    out[k] = t;
    atomicMax(&span[0], hi - (lo & ~7));   // BF16: chunks of 8
    atomicMax(&span[1], hi - (lo & ~3));   // TF32: chunks of 4
  }
}

// The chunk slots of every block (warp per block): slot j of row r holds the
// values of trial panels E * (floor(rs[r] / E) + j) + [0, E) that lie in the
// row's band (and in column J), zeros elsewhere; BF16 or TF32-rounded FP32.
template <bool TF32, typename V>
__global__ void k_tc_pack_vals(int64_t nb, const TcBlk* __restrict__ blk, const V* __restrict__ val,
                               const int32_t* __restrict__ prs, int64_t n_col, const int32_t* __restrict__ ctb,
                               const TetDev* __restrict__ tets, const int32_t* __restrict__ bw,
                               const int64_t* __restrict__ boff, uint4* __restrict__ out) {
  constexpr int E = TF32 ? 4 : 8;
  const int lane = threadIdx.x & 31;
  for (int64_t k = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; k < nb;
       k += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const TcBlk b = blk[k];
    const int S = tc_slots(b.W, E), nt = b.nt;
    for (int idx = lane; idx < S * nt; idx += 32) {
      const int j = idx / nt, r = idx - j * nt;
      const int st = prs[b.ro + r];
      const int base = (st / E) * E + j * E;
      // the row's own column: its band width, values and rows
      const int I = tets[b.t0 + r].col;
      const int64_t ib = I * n_col + b.J;
      const int Wr = bw[ib], ntr = ctb[I + 1] - ctb[I];
      const V* vr = val + boff[ib] + (b.t0 + r - ctb[I]);
      auto at = [&](int col) {
        const int w = col - st;
        return (w >= 0 && w < Wr && col < b.je) ? (float)vr[(int64_t)w * ntr] : 0.f;
      };
      uint32_t wv[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        if (TF32) {
          uint32_t t;
          asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(t) : "f"(at(base + h)));
          wv[h] = t;
        } else {
          uint32_t p = 0;
#pragma unroll
          for (int e = 0; e < 2; ++e)
            p |= (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(at(base + 2 * h + e))) << (16 * e);
          wv[h] = p;
        }
      }
      out[b.vc[TF32 ? 1 : 0] + (int64_t)j * nt + r] = make_uint4(wv[0], wv[1], wv[2], wv[3]);
    }
  }
}

// Xc[c][n][e] = x[n][c E + e] (zero outside), BF16 or TF32-rounded FP32.
template <bool TF32>
__global__ void k_pack_xc(const double* __restrict__ x, int64_t n_tet, int nr, int N, int64_t nchunks,
                          void* __restrict__ Xc) {
  constexpr int E = TF32 ? 4 : 8;
  const int64_t total = nchunks * N * E;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = i / (N * E);
    const int rem = (int)(i % (N * E));
    const int n = rem / E, e = rem % E;
    const int64_t j = c * E + e;
    const float v = (n < nr && j < n_tet) ? (float)x[(int64_t)n * n_tet + j] : 0.f;
    if (TF32) {
      uint32_t t;
      asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(t) : "f"(v));
      static_cast<uint32_t*>(Xc)[i] = t;
    } else {
      static_cast<uint16_t*>(Xc)[i] = __bfloat16_as_ushort(__float2bfloat16_rn(v));
    }
  }
}

struct TcArgs {
  const int32_t* gtb;      // [groups + 1] first row of a group
  const int32_t* gptr;     // [groups + 1] into blk
  const TcBlk* blk;
  const uint4* vals;       // chunk slots of the product's type
  const int32_t* rs;       // row starts (16 bytes of tail room)
  const double* x;         // [nr][n_tet] (internal order)
  double* y;               // [parts][nr][n_tet] (internal order)
  int64_t n_tet;
  int nr, N;               // right-hand sides of the pass, MMA N (multiple of 16)
  int nkc;                 // chunk capacity of a stage's A and B tiles (even)
  uint32_t v_bytes;        // capacity of a stage's value buffer (multiple of 1024)
  int stages;
  uint32_t tmem_cols;
  int parts;               // CTAs that share a group's blocks
  int* err;                // set to 1 when a wait ran out of budget
};

template <bool TF32>
__device__ __forceinline__ float tc_rounded(float v) {
  if (!TF32) return __bfloat162float(__float2bfloat16_rn(v));
  uint32_t t;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(t) : "f"(v));
  return __uint_as_float(t);
}

// Row r's sum for right-hand side n in FP32 from the values that it has. The
// MMA multiplies a tile's zeros too, so one Inf or NaN in x makes NaN in all
// rows of a group with a block there; a sum that is not finite is formed again
// this way, and rows without a value at that panel keep theirs.
template <bool TF32>
__device__ float tc_row_sum(const TcBlk* __restrict__ blk, int nb, const uint4* __restrict__ vals,
                                         const int32_t* __restrict__ rs, const double* __restrict__ x, int nt, int r) {
  constexpr int E = TF32 ? 4 : 8;
  float acc = 0.f;
  for (int k = 0; k < nb; ++k) {
    const TcBlk& b = blk[k];
    const int base = rs[b.ro + r] / E * E, S = tc_slots(b.W, E);
    for (int j = 0; j < S; ++j) {
      const uint4 q = vals[b.vc[TF32 ? 1 : 0] + (int64_t)j * nt + r];
      const uint32_t w[4] = {q.x, q.y, q.z, q.w};
      for (int e = 0; e < E; ++e) {
        const float v = TF32 ? __uint_as_float(w[e]) : __uint_as_float(e & 1 ? w[e >> 1] & 0xffff0000u : w[e >> 1] << 16);
        if (v != 0.f) acc += v * tc_rounded<TF32>((float)x[base + j * E + e]);
      }
    }
  }
  return acc;
}

template <bool TF32>
__device__ __noinline__ void tc_again(const TcArgs& a, int b0, int nb, int t0, int nt, int r, int c, double* __restrict__ y) {
  for (int n = c; n < min(c + 16, a.nr); ++n) {
    double& o = y[(int64_t)n * a.n_tet + t0 + r];
    if (!isfinite(o)) o = tc_row_sum<TF32>(a.blk + b0, nb, a.vals, a.rs, a.x + (int64_t)n * a.n_tet, nt, r);
  }
}

// Per stage in shared memory: the A tile, the B tile (X rows), the block's
// value slots, its row starts (bulk copy from the 16-byte granule holding
// the first one) and its record (written by the loader).
template <bool TF32, int MT>
__global__ void __launch_bounds__(kThreads, 1) k_spmm_tc(const __grid_constant__ TcArgs a, const __grid_constant__ CUtensorMap tmx) {
  using namespace tc;
  constexpr int E = TF32 ? 4 : 8;         // elements per 16-byte chunk
  constexpr int ROWS = MT * 128;
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = blockIdx.x / a.parts, part = blockIdx.x - g * a.parts;
  const int t0 = a.gtb[g], nt = a.gtb[g + 1] - t0;
  const int nbg = a.gptr[g + 1] - a.gptr[g];
  const int b0 = a.gptr[g] + (int)((int64_t)nbg * part / a.parts);
  const int nb = a.gptr[g] + (int)((int64_t)nbg * (part + 1) / a.parts) - b0;
  double* y = a.y + (int64_t)part * a.nr * a.n_tet;
  const int ST = a.stages, N = a.N;
  const uint32_t a_bytes = (uint32_t)a.nkc * ROWS * 16, b_bytes = (uint32_t)a.nkc * N * 16;
  const uint32_t stage_bytes = a_bytes + b_bytes + a.v_bytes + kRsBytes;
  unsigned char* bar_base = smem + (size_t)ST * stage_bytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(bar_base);   // full_a[ST], full_b[ST], empty[ST], done
  uint32_t* slot = reinterpret_cast<uint32_t*>(bar_base + 8 * (3 * ST + 1));
  volatile int* abort_flag = reinterpret_cast<int*>(bar_base + 8 * (3 * ST + 1) + 4);
  auto full_a = [&](int s) { return smem_u32(&bars[s]); };
  auto full_b = [&](int s) { return smem_u32(&bars[ST + s]); };
  auto empty = [&](int s) { return smem_u32(&bars[2 * ST + s]); };
  const uint32_t done = smem_u32(&bars[3 * ST]);
  auto stage_a = [&](int s) { return smem + (size_t)s * stage_bytes; };
  auto stage_b = [&](int s) { return smem + (size_t)s * stage_bytes + a_bytes; };
  auto stage_v = [&](int s) { return smem + (size_t)s * stage_bytes + a_bytes + b_bytes; };
  auto stage_r = [&](int s) { return smem + (size_t)s * stage_bytes + a_bytes + b_bytes + a.v_bytes; };
  auto meta = [&](int s) { return reinterpret_cast<TcBlk*>(stage_r(s) + kMetaOff); };
  auto fail = [&]() {
    *abort_flag = 1;
    atomicExch(a.err, 1);
  };

  if (tid == 0) {
    for (int s = 0; s < ST; ++s) {
      mbar_init(full_a(s), 128);
      mbar_init(full_b(s), 1);
      mbar_init(empty(s), 1);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    fence_proxy_async();
  }
  if (warp == 5) tmem_alloc(smem_u32(slot), a.tmem_cols);
  // the A tiles start zero; afterwards each row rewrites or clears only the
  // chunks its previous band touched
  if (warp < 4)
    for (int s = 0; s < ST; ++s)
      for (int kc = 0; kc < a.nkc; ++kc)
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
          *reinterpret_cast<uint4*>(stage_a(s) + (size_t)kc * ROWS * 16 + (tid + 128 * mt) * 16) = make_uint4(0, 0, 0, 0);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;

  if (warp < 4) {
    // ---------------------------------------------------------------- builders
    int dirty_lo[kMaxStages][MT], dirty_hi[kMaxStages][MT];   // chunks of each stage's row band
#pragma unroll
    for (int q = 0; q < kMaxStages; ++q)
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) dirty_lo[q][mt] = dirty_hi[q][mt] = 0;
    for (int k = 0; k < nb; ++k) {
      const int s = k % ST, u = k / ST;
      if (u > 0 && !mbar_wait(empty(s), (u - 1) & 1, kWaitBudget)) { fail(); break; }
      if (!mbar_wait(full_b(s), u & 1, kWaitBudget)) { fail(); break; }   // record, values, row starts landed
      if (*abort_flag) break;
      const TcBlk* bm = meta(s);
      const int c0c = bm->cmin / E;                      // first chunk of the tile (trial panel index / E)
      const int nkk = 2 * ((bm->cend - c0c * E + 2 * E - 1) / (2 * E));   // chunks the MMAs read
      const int S = tc_slots(bm->W, E);
      const int32_t* R = reinterpret_cast<const int32_t*>(stage_r(s)) + (int)((bm->ro & 3));
      const uint4* V = reinterpret_cast<const uint4*>(stage_v(s));
      unsigned char* A = stage_a(s);
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
        const int r = tid + 128 * mt;
        unsigned char* row = A + r * 16;
        int lo_old = 0, hi_old = 0;
#pragma unroll
        for (int q = 0; q < kMaxStages; ++q)
          if (q == s) { lo_old = dirty_lo[q][mt]; hi_old = dirty_hi[q][mt]; }
        int lo_new = 0, hi_new = 0;
        if (r < nt) {
          lo_new = R[r] / E - c0c;
          hi_new = min(lo_new + S, nkk);
          for (int kc = lo_new; kc < hi_new; ++kc)
            *reinterpret_cast<uint4*>(row + (size_t)kc * ROWS * 16) = V[(kc - lo_new) * nt + r];
        }
        for (int kc = lo_old; kc < hi_old; ++kc)
          if (kc < lo_new || kc >= hi_new)
            *reinterpret_cast<uint4*>(row + (size_t)kc * ROWS * 16) = make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int q = 0; q < kMaxStages; ++q)
          if (q == s) { dirty_lo[q][mt] = lo_new; dirty_hi[q][mt] = hi_new; }
      }
      fence_proxy_async();
      mbar_arrive(full_a(s));
    }
    // ---------------------------------------------------------------- epilogue
    __syncwarp();
    const bool ok = mbar_wait(done, 0, kWaitBudget);
    if (!ok) fail();
    tc_fence_after();
    const bool bad = !ok || *abort_flag;
    __syncwarp();
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
      const int r = mt * 128 + warp * 32 + lane;
      for (int c = 0; c < N; c += 16) {
        float v[16];
        tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(mt * N + c), v);
        if (r < nt) {
          bool again = false;
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int n = c + j;
            if (n < a.nr) {
              const double o = nb == 0 ? 0.0 : bad ? __longlong_as_double(0x7ff8000000000000LL) : (double)v[j];
              y[(int64_t)n * a.n_tet + t0 + r] = o;
              again |= !isfinite(v[j]);
            }
          }
          if (again && nb > 0 && !bad) tc_again<TF32>(a, b0, nb, t0, nt, r, c, y);
        }
      }
    }
  } else if (warp == 4) {
    // ---------------------------------------------------------------- loader
    if (lane == 0) {
      prefetch_tensormap(&tmx);
      int issued = 0;
      TcBlk nxt = nb > 0 ? a.blk[b0] : TcBlk{};
      for (int k = 0; k < nb; ++k) {
        const int s = k % ST, u = k / ST;
        const TcBlk b = nxt;
        if (k + 1 < nb) nxt = a.blk[b0 + k + 1];          // the next record in flight meanwhile
        if (u > 0 && !mbar_wait(empty(s), (u - 1) & 1, kWaitBudget)) { fail(); break; }
        if (*abort_flag) break;
        *meta(s) = b;
        const int c0c = b.cmin / E;
        const int nk = (b.cend - c0c * E + 2 * E - 1) / (2 * E);
        const uint32_t v_bytes = (uint32_t)tc_slots(b.W, E) * nt * 16;
        const uint64_t rs_src = reinterpret_cast<uint64_t>(a.rs + (b.ro & ~(int64_t)3));
        const uint32_t rs_bytes = (uint32_t)(((b.ro & 3) + nt + 3) & ~3) * 4;
        mbar_arrive_expect_tx(full_b(s), (uint32_t)nk * 2 * N * 16 + v_bytes + rs_bytes);
        const uint32_t B = smem_u32(stage_b(s));
        for (int ks = 0; ks < nk; ++ks) tma_load_3d(B + (uint32_t)ks * 2 * N * 16, &tmx, 0, 0, c0c + 2 * ks, full_b(s));
        bulk_load(smem_u32(stage_v(s)), reinterpret_cast<uint64_t>(a.vals + b.vc[TF32 ? 1 : 0]), v_bytes, full_b(s));
        bulk_load(smem_u32(stage_r(s)), rs_src, rs_bytes, full_b(s));
        issued = k + 1;
      }
      // copies still in flight land before the CTA's shared memory is released
      for (int k = max(0, issued - ST); k < issued; ++k)
        if (!mbar_wait(full_b(k % ST), (k / ST) & 1, kWaitBudget)) fail();
    }
  } else {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      const uint32_t idesc = instr_desc(TF32 ? 2u : 1u, 128, N);
      for (int k = 0; k < nb; ++k) {
        const int s = k % ST, u = k / ST;
        if (!mbar_wait(full_a(s), u & 1, kWaitBudget) || !mbar_wait(full_b(s), u & 1, kWaitBudget)) {
          fail();
          break;
        }
        if (*abort_flag) break;
        tc_fence_after();
        const TcBlk* bm = meta(s);
        const int c0c = bm->cmin / E;
        const int nk = (bm->cend - c0c * E + 2 * E - 1) / (2 * E);
        const uint32_t A = smem_u32(stage_a(s)), B = smem_u32(stage_b(s));
        for (int ks = 0; ks < nk; ++ks) {
          const uint64_t bd = smem_desc(B + (uint32_t)ks * 2 * N * 16, (uint32_t)N * 16, 128);
#pragma unroll
          for (int mt = 0; mt < MT; ++mt) {
            const uint64_t ad = smem_desc(A + (uint32_t)ks * 2 * ROWS * 16 + mt * 128 * 16, ROWS * 16, 128);
            mma<TF32>(tmem + (uint32_t)(mt * N), ad, bd, idesc, (k > 0 || ks > 0) ? 1u : 0u);
          }
        }
        mma_commit(empty(s));
      }
      mma_commit(done);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 5) {
    tc_fence_after();
    tmem_dealloc(tmem, a.tmem_cols);
  }
}

// The same product with the A tiles in tensor memory: per stage MT x nkc
// chunks of 4 columns each (row m = lane m), written by the builder warps
// with tcgen05.st (warp w owns lanes 32w..32w+31, i.e. rows 32w + lane) and
// read by the MMA straight from tensor memory; shared memory then holds only
// the B tiles, value slots and row starts, so more stages fit.
template <bool TF32, int MT>
__global__ void __launch_bounds__(kThreads, 1) k_spmm_tm(const __grid_constant__ TcArgs a, const __grid_constant__ CUtensorMap tmx) {
  using namespace tc;
  constexpr int E = TF32 ? 4 : 8;         // elements per 16-byte chunk
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = blockIdx.x / a.parts, part = blockIdx.x - g * a.parts;
  const int t0 = a.gtb[g], nt = a.gtb[g + 1] - t0;
  const int nbg = a.gptr[g + 1] - a.gptr[g];
  const int b0 = a.gptr[g] + (int)((int64_t)nbg * part / a.parts);
  const int nb = a.gptr[g] + (int)((int64_t)nbg * (part + 1) / a.parts) - b0;
  double* y = a.y + (int64_t)part * a.nr * a.n_tet;
  const int ST = a.stages, N = a.N, NKC = a.nkc;
  const uint32_t b_bytes = (uint32_t)NKC * N * 16;
  const uint32_t stage_bytes = b_bytes + a.v_bytes + kRsBytes;
  unsigned char* bar_base = smem + (size_t)ST * stage_bytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(bar_base);   // full_a[ST], full_b[ST], empty[ST], done
  uint32_t* slot = reinterpret_cast<uint32_t*>(bar_base + 8 * (3 * ST + 1));
  volatile int* abort_flag = reinterpret_cast<int*>(bar_base + 8 * (3 * ST + 1) + 4);
  auto full_a = [&](int s) { return smem_u32(&bars[s]); };
  auto full_b = [&](int s) { return smem_u32(&bars[ST + s]); };
  auto empty = [&](int s) { return smem_u32(&bars[2 * ST + s]); };
  const uint32_t done = smem_u32(&bars[3 * ST]);
  auto stage_b = [&](int s) { return smem + (size_t)s * stage_bytes; };
  auto stage_v = [&](int s) { return smem + (size_t)s * stage_bytes + b_bytes; };
  auto stage_r = [&](int s) { return smem + (size_t)s * stage_bytes + b_bytes + a.v_bytes; };
  auto meta = [&](int s) { return reinterpret_cast<TcBlk*>(stage_r(s) + kMetaOff); };
  auto fail = [&]() {
    *abort_flag = 1;
    atomicExch(a.err, 1);
  };

  if (tid == 0) {
    for (int s = 0; s < ST; ++s) {
      mbar_init(full_a(s), 128);
      mbar_init(full_b(s), 1);
      mbar_init(empty(s), 1);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    fence_proxy_async();
  }
  if (warp == 5) tmem_alloc(smem_u32(slot), a.tmem_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  // column of chunk kc of M-tile mt in stage s (after the MT x N accumulator columns)
  auto a_col = [&](int s, int mt, int kc) { return (uint32_t)(MT * N + ((s * MT + mt) * NKC + kc) * 4); };

  if (warp < 4) {
    const uint32_t lanes = (uint32_t)(warp * 32) << 16;
    // the A tiles start zero
    for (int s = 0; s < ST; ++s)
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
        for (int kc = 0; kc < NKC; ++kc) tmem_st4(tmem + lanes + a_col(s, mt, kc), make_uint4(0, 0, 0, 0));
    tmem_st_wait();
    // ---------------------------------------------------------------- builders
    int dlo[kMaxStages][MT], dhi[kMaxStages][MT];   // chunks of each stage this warp left non-zero
#pragma unroll
    for (int q = 0; q < kMaxStages; ++q)
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) dlo[q][mt] = dhi[q][mt] = 0;
    for (int k = 0; k < nb; ++k) {
      const int s = k % ST, u = k / ST;
      if (u > 0 && !mbar_wait(empty(s), (u - 1) & 1, kWaitBudget)) { fail(); break; }
      if (!mbar_wait(full_b(s), u & 1, kWaitBudget)) { fail(); break; }   // record, values, row starts landed
      if (*abort_flag) break;
      const TcBlk* bm = meta(s);
      const int c0c = bm->cmin / E;
      const int nkk = 2 * ((bm->cend - c0c * E + 2 * E - 1) / (2 * E));   // chunks the MMAs read
      const int S = tc_slots(bm->W, E);
      const int32_t* R = reinterpret_cast<const int32_t*>(stage_r(s)) + (int)(bm->ro & 3);
      const uint4* V = reinterpret_cast<const uint4*>(stage_v(s));
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
        const int r = mt * 128 + warp * 32 + lane;
        int lo = 0, hi = 0;
        if (r < nt) {
          lo = R[r] / E - c0c;
          hi = min(lo + S, nkk);
        }
        // the warp's range: its rows' bands and what it left non-zero in this stage
        int wlo = hi > lo ? lo : INT_MAX, whi = hi > lo ? hi : 0;
#pragma unroll
        for (int o = 16; o; o >>= 1) {
          wlo = min(wlo, __shfl_xor_sync(0xffffffffu, wlo, o));
          whi = max(whi, __shfl_xor_sync(0xffffffffu, whi, o));
        }
        int olo = 0, ohi = 0;
#pragma unroll
        for (int q = 0; q < kMaxStages; ++q)
          if (q == s) { olo = dlo[q][mt]; ohi = dhi[q][mt]; }
        const int from = whi > 0 ? min(wlo, ohi > olo ? olo : wlo) : olo;
        const int to = max(whi, ohi);
        for (int kc = from; kc < to; ++kc) {
          const uint4 v = (kc >= lo && kc < hi) ? V[(kc - lo) * nt + r] : make_uint4(0, 0, 0, 0);
          tmem_st4(tmem + lanes + a_col(s, mt, kc), v);
        }
#pragma unroll
        for (int q = 0; q < kMaxStages; ++q)
          if (q == s) { dlo[q][mt] = whi > 0 ? wlo : 0; dhi[q][mt] = whi; }
      }
      tmem_st_wait();
      tc_fence_before();
      mbar_arrive(full_a(s));
    }
    // ---------------------------------------------------------------- epilogue
    __syncwarp();
    const bool ok = mbar_wait(done, 0, kWaitBudget);
    if (!ok) fail();
    tc_fence_after();
    const bool bad = !ok || *abort_flag;
    __syncwarp();
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
      const int r = mt * 128 + warp * 32 + lane;
      for (int c = 0; c < N; c += 16) {
        float v[16];
        tmem_ld16(tmem + lanes + (uint32_t)(mt * N + c), v);
        if (r < nt) {
          bool again = false;
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int n = c + j;
            if (n < a.nr) {
              const double o = nb == 0 ? 0.0 : bad ? __longlong_as_double(0x7ff8000000000000LL) : (double)v[j];
              y[(int64_t)n * a.n_tet + t0 + r] = o;
              again |= !isfinite(v[j]);
            }
          }
          if (again && nb > 0 && !bad) tc_again<TF32>(a, b0, nb, t0, nt, r, c, y);
        }
      }
    }
  } else if (warp == 4) {
    // ---------------------------------------------------------------- loader
    if (lane == 0) {
      prefetch_tensormap(&tmx);
      int issued = 0;
      TcBlk nxt = nb > 0 ? a.blk[b0] : TcBlk{};
      for (int k = 0; k < nb; ++k) {
        const int s = k % ST, u = k / ST;
        const TcBlk b = nxt;
        if (k + 1 < nb) nxt = a.blk[b0 + k + 1];          // the next record in flight meanwhile
        if (u > 0 && !mbar_wait(empty(s), (u - 1) & 1, kWaitBudget)) { fail(); break; }
        if (*abort_flag) break;
        *meta(s) = b;
        const int c0c = b.cmin / E;
        const int nk = (b.cend - c0c * E + 2 * E - 1) / (2 * E);
        const uint32_t v_bytes = (uint32_t)tc_slots(b.W, E) * nt * 16;
        const uint64_t rs_src = reinterpret_cast<uint64_t>(a.rs + (b.ro & ~(int64_t)3));
        const uint32_t rs_bytes = (uint32_t)(((b.ro & 3) + nt + 3) & ~3) * 4;
        mbar_arrive_expect_tx(full_b(s), (uint32_t)nk * 2 * N * 16 + v_bytes + rs_bytes);
        const uint32_t B = smem_u32(stage_b(s));
        for (int ks = 0; ks < nk; ++ks)
          tma_load_3d(B + (uint32_t)ks * 2 * N * 16, &tmx, 0, 0, c0c + 2 * ks, full_b(s));
        bulk_load(smem_u32(stage_v(s)), reinterpret_cast<uint64_t>(a.vals + b.vc[TF32 ? 1 : 0]), v_bytes, full_b(s));
        bulk_load(smem_u32(stage_r(s)), rs_src, rs_bytes, full_b(s));
        issued = k + 1;
      }
      // copies still in flight land before the CTA's shared memory is released
      for (int k = max(0, issued - ST); k < issued; ++k)
        if (!mbar_wait(full_b(k % ST), (k / ST) & 1, kWaitBudget)) fail();
    }
  } else {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      const uint32_t idesc = instr_desc(TF32 ? 2u : 1u, 128, N);
      for (int k = 0; k < nb; ++k) {
        const int s = k % ST, u = k / ST;
        if (!mbar_wait(full_a(s), u & 1, kWaitBudget) || !mbar_wait(full_b(s), u & 1, kWaitBudget)) {
          fail();
          break;
        }
        if (*abort_flag) break;
        tc_fence_after();
        const TcBlk* bm = meta(s);
        const int c0c = bm->cmin / E;
        const int nk = (bm->cend - c0c * E + 2 * E - 1) / (2 * E);
        const uint32_t B = smem_u32(stage_b(s));
        for (int ks = 0; ks < nk; ++ks) {
          const uint64_t bd = smem_desc(B + (uint32_t)ks * 2 * N * 16, (uint32_t)N * 16, 128);
#pragma unroll
          for (int mt = 0; mt < MT; ++mt)
            mma_ts<TF32>(tmem + (uint32_t)(mt * N), tmem + a_col(s, mt, 2 * ks), bd, idesc, (k > 0 || ks > 0) ? 1u : 0u);
        }
        mma_commit(empty(s));
      }
      mma_commit(done);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 5) {
    tc_fence_after();
    tmem_dealloc(tmem, a.tmem_cols);
  }
}

std::mutex g_tc_mu;
std::map<std::tuple<int64_t, int, int, int64_t, int, int, int>, std::pair<int, int>> g_tc_shape;   // shape -> (kind, stages)

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static std::once_flag once;
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// y = the sum of the parts, in order
__global__ void k_tc_sum(const double* __restrict__ part, double* __restrict__ y, int64_t n, int parts) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int p = 0; p < parts; ++p) s += part[p * n + i];
    y[i] = s;
  }
}

// Row groups of a mesh and their non-empty blocks, from the blocks' band widths
struct TcLayout {
  std::vector<int32_t> gcol{0}, gtb{0};   // [groups + 1] first column and row of a group
  std::vector<int32_t> ptr, bG, bJ, bW;   // blocks of a group; group, trial column and widest band of a block
  std::vector<int64_t> ro, vc16, vc32;    // its row starts and chunk slots (16 bytes each)
  int64_t nrows = 0, slots[2] = {0, 0}, cap[2] = {0, 0};   // in all, and most slot bytes of a block
  int max_rows = 0;
  int64_t groups() const { return (int64_t)gcol.size() - 1; }
};
TcLayout tc_layout(const bem_mesh* m, const int32_t* bw) {
  TcLayout L;
  const int64_t nc = m->n_col;
  // consecutive columns to at most 128 rows (one M tile); a taller column is a group of its own
  for (int64_t I = 0; I < nc;) {
    int64_t e = I + 1;
    while (e < nc && m->col_tet_begin[e + 1] - m->col_tet_begin[I] <= 128) ++e;
    L.max_rows = std::max(L.max_rows, m->col_tet_begin[e] - m->col_tet_begin[I]);
    L.gcol.push_back((int32_t)e);
    L.gtb.push_back(m->col_tet_begin[e]);
    I = e;
  }
  L.ptr.assign(L.groups() + 1, 0);
  std::vector<int32_t> wmax(nc);
  for (int64_t g = 0; g < L.groups(); ++g) {
    const int64_t nt = L.gtb[g + 1] - L.gtb[g];
    std::fill(wmax.begin(), wmax.end(), 0);
    for (int64_t I = L.gcol[g]; I < L.gcol[g + 1]; ++I)
      for (int64_t J = 0; J < nc; ++J) wmax[J] = std::max(wmax[J], bw[I * nc + J]);
    for (int64_t J = 0; J < nc; ++J) {
      const int W = wmax[J];
      if (W <= 0) continue;
      L.bG.push_back((int32_t)g);
      L.bJ.push_back((int32_t)J);
      L.bW.push_back(W);
      L.ro.push_back(L.nrows);
      L.vc16.push_back(L.slots[0]);
      L.vc32.push_back(L.slots[1]);
      L.nrows += nt;
      for (int t = 0; t < 2; ++t) {
        const int64_t n = tc_slots(W, t ? 4 : 8) * nt;
        L.slots[t] += n;
        L.cap[t] = std::max(L.cap[t], n * 16);
      }
    }
    L.ptr[g + 1] = (int32_t)L.bG.size();
  }
  return L;
}

// device arrays of the tables: group blocks, group rows, block records and row
// starts, which stay; the blocks' group, trial column, band, row starts and slots
// of both types, and the spans, which do not
constexpr int kTcArrays = 11;
void tc_array_bytes(int64_t groups, int64_t nblk, int64_t nrows, size_t* bytes) {
  const size_t nb = (size_t)std::max<int64_t>(nblk, 1), i4 = sizeof(int32_t), i8 = sizeof(int64_t);
  const size_t b[kTcArrays] = {i4 * (groups + 1), i4 * (groups + 1), sizeof(TcBlk) * nb,
                               i4 * (size_t)(nrows + 4) /* whole 16-byte granules are copied */, i4 * nb, i4 * nb, i4 * nb,
                               i8 * nb, i8 * nb, i8 * nb, sizeof(int) * 2};
  std::copy(b, b + kTcArrays, bytes);
}

// CTAs that share a group's blocks: some four CTAs per SM in all, of at least
// eight blocks each. The tensor cores' FP32 accumulation truncates, so a row's
// sum cut in parts comes out closer to the exact one, by an amount that grows
// with the row. Measured with two parts against none: level-3 sphere, 8 slabs
// (11,300 values per row) 1.2e-5 in BF16 and 1.9e-5 in TF32, level-2 sphere, 32
// slabs (5,300) 4e-6 and 6e-6. Long rows are cut in two at most, or left whole,
// which kept these two meshes within 1.3e-5 of the uncut sums; on others the
// difference is not bounded by that. More parts of long rows would be faster
// (level-3 sphere, BF16, 13 vectors: 522 us with 8 for 613) and more accurate.
int tc_parts(int64_t groups, int64_t nblk, int64_t per_row, bool bf16) {
  const int64_t per_group = nblk / std::max<int64_t>(groups, 1);
  const int most = per_row > 8000 ? (bf16 ? 2 : 1) : per_row > 3000 ? 2 : 8;
  int parts = 1;
  while (parts < most && groups * parts < 4 * 152 && per_group >= 16 * parts) parts *= 2;
  return parts;
}

// MMA N of a pass
int tc_n(int nrhs) { return std::max(16, (nrhs + 15) / 16 * 16); }
// FP32 numbers of the packed x (16 bytes per chunk and right-hand side) and of the parts' sums
int64_t tc_xc_len(int64_t n, int nrhs, bool bf16) {
  const int E = bf16 ? 8 : 4;
  return (n + E - 1) / E * tc_n(nrhs) * 4;
}
int64_t tc_ws_len(int64_t n, int nrhs, int parts, bool bf16) {
  return tc_xc_len(n, nrhs, bf16) + (parts > 1 ? 2 * parts * n * nrhs : 0);
}

// Row groups and block records of the operator (made once; an operator's
// sparsity structure never changes): the non-empty blocks of each group, their
// band unions, the offsets of their chunk slots in both types, and the row
// starts in the groups' row order.
bem_status ensure_tc_meta(const bem_operator* op, cudaStream_t s) {
  if (op->d_tc_blk) return BEM_OK;
  const bem_mesh* m = op->mesh;
  const int64_t nc = m->n_col;
  std::vector<int32_t> hbw(nc * nc);
  STBEM_CUDA(cudaMemcpyAsync(hbw.data(), op->d_bw, sizeof(int32_t) * nc * nc, cudaMemcpyDeviceToHost, s));
  STBEM_CUDA(cudaStreamSynchronize(s));
  const TcLayout L = tc_layout(m, hbw.data());
  const int64_t ng = L.groups(), nb = (int64_t)L.bG.size();
  struct Arrays {   // freed on every way out unless released
    void* p[kTcArrays] = {};
    ~Arrays() { for (void* q : p) cudaFree(q); }
  } A;
  size_t bytes[kTcArrays];
  tc_array_bytes(ng, nb, L.nrows, bytes);
  for (int k = 0; k < kTcArrays; ++k)
    if (device_alloc((void**)&A.p[k], bytes[k]) != cudaSuccess) {
      cudaGetLastError();
      A.p[k] = nullptr;
      set_error("out of device memory (tensor-core product tables)");
      return BEM_ERR_OUT_OF_MEMORY;
    }
  int hspan[2] = {0, 0};
  const void* src[kTcArrays] = {L.ptr.data(), L.gtb.data(), nullptr, nullptr, L.bG.data(), L.bJ.data(), L.bW.data(),
                                L.ro.data(), L.vc16.data(), L.vc32.data(), hspan};
  for (int k = 0; k < kTcArrays; ++k)
    if (src[k] && (nb > 0 || k < 2 || k == 10)) STBEM_CUDA(cudaMemcpyAsync(A.p[k], src[k], bytes[k], cudaMemcpyHostToDevice, s));
  if (nb > 0) {
    const int64_t threads = nb * 32;
    k_tc_meta<<<(unsigned)((threads + 255) / 256), 256, 0, s>>>(
        nb, (const int32_t*)A.p[4], (const int32_t*)A.p[5], (const int32_t*)A.p[6], (const int64_t*)A.p[7],
        (const int64_t*)A.p[8], (const int64_t*)A.p[9], nc, (const int32_t*)A.p[1], m->d_col_tet_begin, m->d_tet, op->d_bw,
        op->d_rsoff, op->d_rs, (TcBlk*)A.p[2], (int32_t*)A.p[3], (int*)A.p[10]);
    STBEM_CUDA(cudaGetLastError());
  }
  STBEM_CUDA(cudaMemcpyAsync(hspan, A.p[10], sizeof(hspan), cudaMemcpyDeviceToHost, s));
  STBEM_CUDA(cudaStreamSynchronize(s));
  if (!op->d_tc_err) {
    if (device_alloc((void**)&op->d_tc_err, sizeof(int)) != cudaSuccess) {
      cudaGetLastError();
      op->d_tc_err = nullptr;
      set_error("out of device memory (tensor-core product flag)");
      return BEM_ERR_OUT_OF_MEMORY;
    }
    STBEM_CUDA(cudaMemsetAsync(op->d_tc_err, 0, sizeof(int), s));
  }
  op->d_tc_gptr = (int32_t*)A.p[0];
  op->d_tc_gtb = (int32_t*)A.p[1];
  op->d_tc_blk = A.p[2];
  op->d_tc_rs = (int32_t*)A.p[3];
  for (int k = 0; k < 4; ++k) A.p[k] = nullptr;
  op->tc_groups = ng;
  op->tc_rows = L.max_rows;
  op->tc_nrows = L.nrows;
  op->tc_nblk = nb;
  op->tc_span[0] = hspan[0];
  op->tc_span[1] = hspan[1];
  for (int t = 0; t < 2; ++t) {
    op->tcv_len[t] = L.slots[t];
    op->tcv_cap[t] = L.cap[t];
  }
  return BEM_OK;
}

// the chunk slots of the product's type, made on first use and after a reassembly
bem_status ensure_tc_vals(const bem_operator* op, bool tf32, cudaStream_t s) {
  const int t = tf32 ? 1 : 0;
  if (op->d_tcv[t] && !op->tcv_stale[t]) return BEM_OK;
  if (!op->d_tcv[t] &&
      device_alloc((void**)&op->d_tcv[t], sizeof(uint4) * (size_t)std::max<int64_t>(op->tcv_len[t], 1)) != cudaSuccess) {
    cudaGetLastError();
    op->d_tcv[t] = nullptr;
    set_error("out of device memory (tensor-core product values)");
    return BEM_ERR_OUT_OF_MEMORY;
  }
  op->tcv_stale[t] = false;
  if (op->tc_nblk == 0) return BEM_OK;
  const TcBlk* blk = static_cast<const TcBlk*>(op->d_tc_blk);
  uint4* out = static_cast<uint4*>(op->d_tcv[t]);
  const unsigned grid = (unsigned)std::min<int64_t>((op->tc_nblk * 32 + 255) / 256, 152 * 32);
  const bem_mesh* m = op->mesh;
  auto pack = [&](auto kern, auto* val) {
    kern<<<grid, 256, 0, s>>>(op->tc_nblk, blk, val, op->d_tc_rs, m->n_col, m->d_col_tet_begin, m->d_tet, op->d_bw, op->d_boff,
                              out);
  };
  if (tf32) pack(k_tc_pack_vals<true, float>, op->d_val32);
  else if (op->d_val32) pack(k_tc_pack_vals<false, float>, op->d_val32);
  else pack(k_tc_pack_vals<false, double>, op->d_val);
  STBEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

// kind 0: A tiles in shared memory (k_spmm_tc); kind 1: in tensor memory (k_spmm_tm)
template <bool TF32, int MT>
bem_status launch_tc(int kind, const TcArgs& a, const CUtensorMap& map, size_t smem, int64_t n_cta, cudaStream_t s) {
  const void* kern = kind ? (const void*)k_spmm_tm<TF32, MT> : (const void*)k_spmm_tc<TF32, MT>;
  TRY_STATUS(ensure_smem_attr(kern, smem));
  if (kind) k_spmm_tm<TF32, MT><<<(unsigned)n_cta, kThreads, smem, s>>>(a, map);
  else k_spmm_tc<TF32, MT><<<(unsigned)n_cta, kThreads, smem, s>>>(a, map);
  STBEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

}  // namespace

int64_t tc_bytes(const bem_operator* op, const int32_t* bw, bool bf16) {
  if (!op->tc_plan.groups) {
    const TcLayout L = tc_layout(op->mesh, bw);
    op->tc_plan = {L.groups(), (int64_t)L.bG.size(), L.nrows, {L.slots[0], L.slots[1]}};
  }
  size_t a[kTcArrays];
  tc_array_bytes(op->tc_plan.groups, op->tc_plan.nblk, op->tc_plan.nrows, a);
  int64_t b = sizeof(int) + 16 * std::max<int64_t>(op->tc_plan.slots[bf16 ? 0 : 1], 1);
  for (size_t x : a) b += (int64_t)x;
  return b;
}

int64_t matvec_ws_bytes(const bem_operator* op, int arith, int nrhs) {
  const int64_t n = op->mesh->n_tet;
  if (arith == MV_FP32) return 4 * packed_len(n, nrhs);
  if (arith != MV_TF32 && arith != MV_BF16) return 0;
  const bool bf16 = arith == MV_BF16;
  return 4 * tc_ws_len(n, std::min(nrhs, 64), tc_parts(op->tc_plan.groups, op->tc_plan.nblk, op->nstored / n, bf16), bf16);
}

int64_t tc_table_bytes(const bem_operator* op) {
  int64_t b = op->d_tc_blk ? op->tc_nblk * (int64_t)sizeof(TcBlk) + (op->tc_groups + 1) * 8 + op->tc_nrows * 4 : 0;
  for (int t = 0; t < 2; ++t)
    if (op->d_tcv[t]) b += op->tcv_len[t] * 16;
  return b;
}

bem_status op_spmm_tc(const bem_operator* op, const double* x, double* y, int nrhs, bool bf16, cudaStream_t s) {
  const bem_mesh* m = op->mesh;
  const int64_t n = m->n_tet;
  if (nrhs < 1 || nrhs > 64) {
    set_error("tensor-core product: 1..64 right-hand sides per pass");
    return BEM_ERR_INVALID_ARG;
  }
  if (!bf16 && !op->d_val32) {
    set_error("TF32 products need FP32 values (store_fp32 = 1)");
    return BEM_ERR_INVALID_ARG;
  }
  TRY_STATUS(ensure_tc_meta(op, s));
  TRY_STATUS(ensure_tc_vals(op, !bf16, s));
  auto enc = encode_fn();
  if (!enc) {
    set_error("tensor-core product: cuTensorMapEncodeTiled is not available");
    return BEM_ERR_UNSUPPORTED;
  }
  const int E = bf16 ? 8 : 4;
  const int N = tc_n(nrhs);
  const int64_t nchunks = (n + E - 1) / E;
  const int parts = tc_parts(op->tc_groups, op->tc_nblk, op->nstored / n, bf16);
  const int64_t xc_len = tc_xc_len(n, nrhs, bf16);
  TRY_STATUS(ensure_ws(op, tc_ws_len(n, nrhs, parts, bf16)));
  void* Xc = op->d_ws;
  if (bf16) k_pack_xc<false><<<grid_for(nchunks * N * E), 256, 0, s>>>(x, n, nrhs, N, nchunks, Xc);
  else k_pack_xc<true><<<grid_for(nchunks * N * E), 256, 0, s>>>(x, n, nrhs, N, nchunks, Xc);
  STBEM_CUDA(cudaGetLastError());

  // Xc as rows of 256 bytes: {256-byte row, N / 16 rows per chunk, chunks};
  // a box of {256 bytes, N / 16, 2 chunks} is one K step of the B tile
  CUtensorMap map;
  const int inner = 256 / (bf16 ? 2 : 4);
  cuuint64_t dims[3] = {(cuuint64_t)inner, (cuuint64_t)(N / 16), (cuuint64_t)nchunks};
  cuuint64_t strides[2] = {256, (cuuint64_t)N * 16};
  cuuint32_t box[3] = {(cuuint32_t)inner, (cuuint32_t)(N / 16), 2};
  cuuint32_t es[3] = {1, 1, 1};
  const CUresult r = enc(&map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, Xc, dims,
                         strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("tensor-core product: tensor map rejected (" + std::to_string((int)r) + ")");
    return BEM_ERR_CUDA;
  }
  const int MT = op->tc_rows > 128 ? 2 : 1;
  const int span = std::max(op->tc_span[bf16 ? 0 : 1], 1);
  const int nkc = 2 * ((span + 2 * E - 1) / (2 * E));
  // value slots of the largest block; a multiple of 1024 bytes keeps every
  // stage's TMA tiles aligned
  const size_t v_bytes = ((size_t)op->tcv_cap[bf16 ? 0 : 1] + 1023) & ~(size_t)1023;
  // shared memory per stage: A tile (kind 0 only), B tile, value slots, row starts
  const size_t stage_b = (size_t)nkc * N * 16 + v_bytes + kRsBytes;
  const size_t stage_a = (size_t)nkc * MT * 128 * 16;
  const size_t tail = kTailBytes;
  size_t smem_max = 0;
  {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    smem_max = (size_t)v;
  }
  TcArgs a;
  a.gtb = op->d_tc_gtb;
  a.gptr = op->d_tc_gptr;
  a.blk = static_cast<const TcBlk*>(op->d_tc_blk);
  a.vals = static_cast<const uint4*>(op->d_tcv[bf16 ? 0 : 1]);
  a.rs = op->d_tc_rs;
  a.parts = parts;
  a.x = x;
  a.y = parts > 1 ? reinterpret_cast<double*>(op->d_ws + xc_len) : y;
  a.n_tet = n;
  a.nr = nrhs;
  a.N = N;
  a.nkc = nkc;
  a.v_bytes = (uint32_t)v_bytes;
  a.err = op->d_tc_err;
  auto pow2 = [](int c) {
    uint32_t v = 32;
    while (v < (uint32_t)c) v <<= 1;
    return v;
  };
  // tensor-memory columns: the accumulator, and for kind 1 the A tiles of every stage
  auto cols_of = [&](int kind, int st) { return kind ? MT * N + st * MT * nkc * 4 : MT * N; };
  auto fits = [&](int kind, int st) {
    const size_t smem = st * (stage_b + (kind ? 0 : stage_a)) + tail;
    return smem <= smem_max && cols_of(kind, st) <= 512;
  };
  auto launch = [&](int kind, int st) -> bem_status {
    a.stages = st;
    a.tmem_cols = pow2(cols_of(kind, st));
    const size_t smem = st * (stage_b + (kind ? 0 : stage_a)) + tail;
    const int64_t n_cta = op->tc_groups * parts;
    if (bf16)
      return MT == 1 ? launch_tc<false, 1>(kind, a, map, smem, n_cta, s) : launch_tc<false, 2>(kind, a, map, smem, n_cta, s);
    return MT == 1 ? launch_tc<true, 1>(kind, a, map, smem, n_cta, s) : launch_tc<true, 2>(kind, a, map, smem, n_cta, s);
  };
  // the product with a shape, and the sum of its parts
  auto product = [&](int kind, int st) -> bem_status {
    TRY_STATUS(launch(kind, st));
    if (parts > 1) k_tc_sum<<<grid_for(n * nrhs), 256, 0, s>>>(a.y, y, n * nrhs, parts);
    STBEM_CUDA(cudaGetLastError());
    return BEM_OK;
  };
  // launch shape: where the A tiles live and the pipeline depth (1 to 6
  // stages; with the stage size they fix the CTAs per SM), timed once per
  // shape in the process, then kept. Neither changes the arithmetic (every
  // CTA sums its blocks in order), so the candidates give the same bits.
  std::vector<std::pair<int, int>> cand;
  for (int kind = 0; kind < 2; ++kind)
    for (int st = 1; st <= kMaxStages; ++st)
      if (fits(kind, st)) cand.emplace_back(kind, st);
  if (cand.empty()) {
    set_error("tensor-core product: the widest block does not fit in shared or tensor memory");
    return BEM_ERR_UNSUPPORTED;
  }
  const auto key = std::make_tuple(op->tc_groups * 16 + parts, op->tc_rows, op->tc_span[bf16 ? 0 : 1], op->tcv_cap[bf16 ? 0 : 1], N,
                                   (int)bf16, op->ctx->device);
  {
    std::lock_guard<std::mutex> lk(g_tc_mu);
    auto it = g_tc_shape.find(key);
    if (it != g_tc_shape.end()) return product(it->second.first, it->second.second);
  }
  cudaEvent_t e0, e1;
  STBEM_CUDA(cudaEventCreate(&e0));
  STBEM_CUDA(cudaEventCreate(&e1));
  float best = 1e30f;
  std::pair<int, int> best_c = cand.back();
  bem_status st = BEM_OK;
  for (const auto& c : cand) {
    if ((st = launch(c.first, c.second)) != BEM_OK) break;   // warm-up
    cudaEventRecord(e0, s);
    if ((st = launch(c.first, c.second)) != BEM_OK) break;
    cudaEventRecord(e1, s);
    if (cudaEventSynchronize(e1) != cudaSuccess) {
      st = BEM_ERR_CUDA;
      set_error("tensor-core product: tuning launch failed");
      break;
    }
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (ms < best) {
      best = ms;
      best_c = c;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st != BEM_OK) return st;
  {
    std::lock_guard<std::mutex> lk(g_tc_mu);
    g_tc_shape[key] = best_c;
  }
  return product(best_c.first, best_c.second);
}

namespace {
// One thread waits, with the product's bounded wait, on an mbarrier that
// nothing arrives on; it records whether the wait gave up and after how many
// cycles.
__global__ void k_wait_selftest(long long budget, int* gave_up, long long* cycles) {
  __shared__ uint64_t bar;
  const uint32_t b = tc::smem_u32(&bar);
  tc::mbar_init(b, 1);
  tc::fence_proxy_async();
  const long long t0 = clock64();
  const bool ok = tc::mbar_wait(b, 0, budget);
  *cycles = clock64() - t0;
  *gave_up = ok ? 0 : 1;
}
}  // namespace

bem_status op_tc_error(const bem_operator* op, int* flag) {
  *flag = 0;
  if (!op->d_tc_err) return BEM_OK;
  STBEM_CUDA(cudaMemcpy(flag, op->d_tc_err, sizeof(int), cudaMemcpyDeviceToHost));
  return BEM_OK;
}

}  // namespace stbem

using namespace stbem;

extern "C" bem_status bem_selftest_bounded_wait(bem_context* ctx, double* waited_ms) {
  if (!ctx) {
    set_error("bem_selftest_bounded_wait: null context");
    return BEM_ERR_INVALID_ARG;
  }
  STBEM_CUDA(cudaSetDevice(ctx->device));
  int* d_flag = nullptr;
  long long* d_cyc = nullptr;
  if (device_alloc((void**)&d_flag, sizeof(int)) != cudaSuccess || device_alloc((void**)&d_cyc, sizeof(long long)) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(d_flag);
    set_error("out of device memory");
    return BEM_ERR_OUT_OF_MEMORY;
  }
  int dev_clock_khz = 0;
  cudaDeviceGetAttribute(&dev_clock_khz, cudaDevAttrClockRate, ctx->device);
  const long long budget = 2000000;   // clock cycles: about a millisecond
  k_wait_selftest<<<1, 1, 0, ctx->stream>>>(budget, d_flag, d_cyc);
  int flag = 0;
  long long cyc = 0;
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(&flag, d_flag, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&cyc, d_cyc, sizeof(long long), cudaMemcpyDeviceToHost, ctx->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  cudaFree(d_flag);
  cudaFree(d_cyc);
  if (e != cudaSuccess) {
    set_error(std::string("bem_selftest_bounded_wait: ") + cudaGetErrorString(e));
    return BEM_ERR_CUDA;
  }
  if (waited_ms) *waited_ms = dev_clock_khz > 0 ? (double)cyc / dev_clock_khz : 0.0;
  if (flag) {
    set_error("bounded wait gave up (expected: nothing arrives on the self-test barrier)");
    return BEM_ERR_DEVICE_TIMEOUT;
  }
  return BEM_OK;
}
