// Work on one block (I, J) of the matrix: panels over spatial triangle
// ("column") I against panels over column J. Shared by the pattern pass and
// the quadrature: the context of an operator, the FP32 image of a column and
// the sparsity bits of a block, found by a whole CTA.
#pragma once
#include "stbem_internal.h"

namespace stbem {

// FP32 image of a panel for the sparsity filter (48 bytes)
struct PanelF {
  float vt[4];        // vertex times as in TetDev
  float ball[5];
  float tmin, pmax;
  uint8_t lo, hi;     // surfaces, relative to the column's first
  uint8_t dup, pad;
};
static_assert(sizeof(PanelF) == 48, "PanelF layout");

// FP32 image of a column: corners, frame and centroid ball
struct ColF {
  float Xh[3][3];
  ColR<float> R;
  float ctr[3], rad;
};
static_assert(sizeof(FaceF) == 48, "FaceF is copied in 16-byte pieces");

struct BlockCtx {
  int64_t n_col;
  int mq, nq, n_theta, prec;
  ArcRule rule;
  float margin;
  double S;
  const ColGeom* cols;
  const ColF* colf;
  const int32_t* col_tet_begin;
  const int32_t* col_surf_begin;
  const SurfDev* surf;
  const FaceF* facef;
  const TetDev* tets;
  const PanelF* panf;
  const double* pts;
  const float4* ptsf;          // outer points (t, x, y, z) rounded to FP32
  const double* trange;
  int32_t* bw;
  int64_t* bnnz;
  const int64_t* boff;
  const int64_t* rsoff;
  int32_t* rs;
  double* val;
  float* val32;
  int max_surf, max_tet;
  unsigned long long* counter;
  unsigned long long* inner;   // pattern pass: inner integrals m_Q^2 x (test face, trial panel) (null: not counted)
  uint2* gran;                 // pattern pass: (apexes, potentials) of each run of GRAN blocks (null: not counted)
  // matrix-free product: when mf_y is set the entries are not stored but
  // y[k][i] += A_ij x[k][j] is accumulated (x, y: [mf_nrhs][mf_ld], internal order)
  const double* mf_x;
  double* mf_y;
  int mf_nrhs;
  int64_t mf_ld;
};

// the quadrature takes its scratch by runs of GRAN consecutive blocks
constexpr int GRAN = 8;

// shared-memory image of a block: the trial column's panels, the distances of
// the test column's outer points to the trial corners, the faces' windows
struct BlockSm {
  int64_t I, J;
  int tetI, ntI, surfI, nsI;   // test column
  int tetJ, ntJ, surfJ, nsJ;   // trial column
  float Dmax, Dmin, rmax;
  int wmax;                    // widest trial window of a face
  float X[3][3];               // trial corners
};

__host__ __device__ inline int bit_words(int max_tet) { return (max_tet + 31) / 32; }
__host__ __device__ inline size_t bits_smem(int max_tet, int max_surf, int nq) {
  size_t s = sizeof(PanelF) * max_tet;                                            // panels
  s += sizeof(float) * (((size_t)3 * max_surf * nq + 3) / 4 * 4);                 // corner distances
  s += sizeof(uint32_t) * (((size_t)max_surf * bit_words(max_tet) + 3) / 4 * 4);  // bits
  s += sizeof(uint32_t) * ((max_surf + 3) / 4 * 4);                               // windows
  return s;
}

#ifdef __CUDACC__
__device__ __forceinline__ double dist3x(const double* a, const double* b) {
  double dx = __dsub_rn(a[0], b[0]), dy = __dsub_rn(a[1], b[1]), dz = __dsub_rn(a[2], b[2]);
  return __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)));
}
// (IEEE square roots here whatever the unit's FP32 flags: the filter's margin
// is set against the correctly rounded operations)
__device__ __forceinline__ float dist3f(float x, float y, float z, const float* b) {
  float dx = x - b[0], dy = y - b[1], dz = z - b[2];
  return __fsqrt_rn(dx * dx + dy * dy + dz * dz);
}

// ---------------------------------------------------------------------------
// Sparsity predicate for one outer point and one panel (the contract):
//   C1  tau_min(j) < t_q
//   C2  max_b |x_q - y_b| - (t_q - tau_b) >= 0
//   C3  not (phi_Xi(x_q - c_j) - d_r(|x_q - c_j|) > 0)     (Theorem phi_xi_sphere)
// FP64 values with the contract's operation order decide; an FP32 estimate
// with a rigorous error margin settles the clear cases first.
// ---------------------------------------------------------------------------
static __device__ __noinline__ bool c2_exact(const double* x, const TetDev& T, const ColGeom& G) {
  double mx = -INFINITY;
  for (int b = 0; b < 4; ++b) {
    int k = b < 3 ? b : T.dup;
    double v = __dsub_rn(dist3x(x + 1, G.X[k]), __dsub_rn(x[0], T.vt[b]));
    if (v > mx) mx = v;
  }
  return mx >= 0.0;
}
static __device__ __noinline__ bool c3_fail_exact(const double* x, const TetDev& T) {
  double al = dist3x(x + 1, T.ball + 1);
  double phi = __dsub_rn(al, __dsub_rn(x[0], T.ball[0]));
  double rj = T.ball[4];
  double s2 = __dsqrt_rn(2.0);
  double dr = (al < __ddiv_rn(rj, s2)) ? __dadd_rn(al, __dsqrt_rn(__dsub_rn(__dmul_rn(rj, rj), __dmul_rn(al, al))))
                                       : __dmul_rn(rj, s2);
  return __dsub_rn(phi, dr) > 0.0;
}

// x: the point in FP64, xf: rounded to FP32, r: its FP32 distances to the
// column's corners, T: the panel in FP32, D: in FP64
__device__ __forceinline__ bool point_sees(const double* x, const float4& xf, const float* r, const PanelF& T,
                                           const TetDev& D, const ColGeom& G, float margin) {
  // C1: rounding is monotone, so only equal FP32 times need the FP64 ones
  if (T.tmin > xf.x) return false;
  if (T.tmin == xf.x && !(D.tmin < x[0])) return false;
  // C2
  {
    const float v0 = r[0] - (xf.x - T.vt[0]), v1 = r[1] - (xf.x - T.vt[1]), v2 = r[2] - (xf.x - T.vt[2]);
    const float v3 = r[T.dup] - (xf.x - T.vt[3]);
    const float mx = fmaxf(fmaxf(v0, v1), fmaxf(v2, v3));
    if (!(mx > margin)) {
      if (mx < -margin) return false;
      if (!c2_exact(x, D, G)) return false;
    }
  }
  // C3
  {
    const float al = dist3f(xf.y, xf.z, xf.w, T.ball + 1);
    const float phi = al - (xf.x - T.ball[0]);
    const float rj = T.ball[4];
    const float dr = (al < rj * 0.70710678f) ? al + __fsqrt_rn(fmaxf(rj * rj - al * al, 0.f)) : rj * 1.41421356f;
    const float v = phi - dr;
    if (v > margin) return false;
    if (!(v < -margin) && c3_fail_exact(x, D)) return false;
  }
  return true;
}

struct BlockPtr {      // the regions of bits_smem
  PanelF* pan;
  float* r;            // [face][point][3]
  uint32_t* bits;      // [face][words]
  uint32_t* win;       // [face]: first panel | panels << 16
};
__device__ __forceinline__ BlockPtr block_ptr(unsigned char* smem, int max_tet, int max_surf, int nq) {
  BlockPtr p;
  p.pan = reinterpret_cast<PanelF*>(smem);
  p.r = reinterpret_cast<float*>(p.pan + max_tet);
  p.bits = reinterpret_cast<uint32_t*>(p.r + ((size_t)3 * max_surf * nq + 3) / 4 * 4);
  p.win = p.bits + (max_surf * bit_words(max_tet) + 3) / 4 * 4;
  return p;
}

// Trial column J into shared memory (all threads; ends with a barrier).
__device__ __forceinline__ void load_trial(const BlockCtx& B, int64_t J, BlockSm& C, PanelF* pan) {
  const int tet0 = B.col_tet_begin[J], nt = B.col_tet_begin[J + 1] - tet0;
  if (threadIdx.x == 0) {
    C.J = J;
    C.tetJ = tet0;
    C.ntJ = nt;
    C.surfJ = B.col_surf_begin[J];
    C.nsJ = B.col_surf_begin[J + 1] - C.surfJ;
    C.rmax = 0.f;
  }
  if (threadIdx.x < 9) C.X[threadIdx.x / 3][threadIdx.x % 3] = B.colf[J].Xh[threadIdx.x / 3][threadIdx.x % 3];
  __syncthreads();
  const uint4* src = reinterpret_cast<const uint4*>(B.panf + tet0);
  uint4* dst = reinterpret_cast<uint4*>(pan);
  for (int k = threadIdx.x; k < 3 * nt; k += blockDim.x) {
    const uint4 v = src[k];
    dst[k] = v;
    if (k % 3 == 2) atomicMax(reinterpret_cast<int*>(&C.rmax), (int)v.x);   // ball radius (>= 0: orders as an integer)
  }
  __syncthreads();
}

// Test column I: its ranges and the bounds of the distance between the columns.
__device__ __forceinline__ void load_test(const BlockCtx& B, int64_t I, BlockSm& C) {
  if (threadIdx.x < 32) {
    const ColF& GI = B.colf[I];
    const ColF& GJ = B.colf[C.J];
    const int l = threadIdx.x;
    float v = 0.f;
    if (l < 9) {
      const int a = l / 3, b = l - 3 * a;
      const float dx = GI.Xh[a][0] - GJ.Xh[b][0], dy = GI.Xh[a][1] - GJ.Xh[b][1], dz = GI.Xh[a][2] - GJ.Xh[b][2];
      v = sqrtf(dx * dx + dy * dy + dz * dz);
    }
#pragma unroll
    for (int o = 8; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (l == 0) {
      const float dx = GI.ctr[0] - GJ.ctr[0], dy = GI.ctr[1] - GJ.ctr[1], dz = GI.ctr[2] - GJ.ctr[2];
      C.Dmax = v;
      C.Dmin = fmaxf(0.f, sqrtf(dx * dx + dy * dy + dz * dz) - GI.rad - GJ.rad);
      C.I = I;
      C.tetI = B.col_tet_begin[I];
      C.ntI = B.col_tet_begin[I + 1] - C.tetI;
      C.surfI = B.col_surf_begin[I];
      C.nsI = B.col_surf_begin[I + 1] - C.surfI;
      C.wmax = 0;
    }
  }
  __syncthreads();
}

// Pattern bits of every face of column I against the panels of column J
// (load_trial and load_test done; all threads; ends with a barrier). Bound by
// FP32 issue and latency. A face's trial window (panels the column distances
// do not exclude) is found by one thread; the distances of the outer points
// to the trial corners are shared by the panels of the column; then one
// thread per (face, panel of its window) over the whole CTA, which keeps the
// lanes busy where a warp per face left half of them idle (windows are 6-20
// panels wide). The windows are FP32 with slack: they only skip panels that
// are certainly outside the pattern, the predicate decides.
__device__ __forceinline__ void block_bits(const BlockCtx& B, BlockSm& C, const BlockPtr& P) {
  const int ns = C.nsI, nq = B.nq, words = bit_words(B.max_tet);
  const float slack = 8e-6f * (float)B.S;
  for (int f = threadIdx.x; f < ns; f += blockDim.x) {
    const float tlo = (float)B.trange[2 * (int64_t)(C.surfI + f)], thi = (float)B.trange[2 * (int64_t)(C.surfI + f) + 1];
    const float lim1 = tlo - C.Dmax - slack;
    int a = 0, b = C.ntJ;  // first j with pmax >= lim1
    while (a < b) { const int m = (a + b) >> 1; if (P.pan[m].pmax < lim1) a = m + 1; else b = m; }
    const int jlo = a;
    const float lim2 = thi + fminf(0.f, C.rmax * 1.4142137f - C.Dmin) + slack;
    b = C.ntJ;             // first j with tmin >= lim2
    while (a < b) { const int m = (a + b) >> 1; if (P.pan[m].tmin < lim2) a = m + 1; else b = m; }
    P.win[f] = (uint32_t)jlo | ((uint32_t)(a - jlo) << 16);
    if (a > jlo) atomicMax(&C.wmax, a - jlo);
  }
  for (int k = threadIdx.x; k < ns * words; k += blockDim.x) P.bits[k] = 0u;
  __syncthreads();
  const int wmax = C.wmax;
  if (wmax == 0) return;
  const float4* pf = B.ptsf + (int64_t)C.surfI * nq;
  for (int k = threadIdx.x; k < ns * nq; k += blockDim.x) {
    const float4 x = pf[k];
#pragma unroll
    for (int c = 0; c < 3; ++c) P.r[3 * k + c] = dist3f(x.y, x.z, x.w, C.X[c]);
  }
  __syncthreads();
  const double* pd = B.pts + (int64_t)C.surfI * nq * 4;
  const TetDev* td = B.tets + C.tetJ;
  const ColGeom& G = B.cols[C.J];
  for (int it = threadIdx.x; it < ns * wmax; it += blockDim.x) {
    const int f = it / wmax, o = it - f * wmax;
    const uint32_t w = P.win[f];
    if (o >= (int)(w >> 16)) continue;
    const int j = (int)(w & 0xffffu) + o;
    const PanelF T = P.pan[j];
    bool hit = false;
    for (int q = f * nq; q < (f + 1) * nq && !hit; ++q)
      hit = point_sees(pd + 4 * (int64_t)q, pf[q], P.r + 3 * q, T, td[j], G, B.margin);
    if (hit) atomicOr(&P.bits[f * words + (j >> 5)], 1u << (j & 31));
  }
  __syncthreads();
}

// segment of global work item g: prefix[seg] <= g < prefix[seg + 1]
__device__ inline int find_seg(const int64_t* prefix, int S, int64_t g) {
  int lo = 0, hi = S;
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (prefix[mid] <= g) lo = mid;
    else hi = mid;
  }
  return lo;
}

// surfaces of the panels in a face's bits: first and count (0: none)
__device__ __forceinline__ void bits_surfaces(const uint32_t* fb, int words, const PanelF* pan, int& slo, int& n) {
  int lo = 1 << 30, hi = -1;
  for (int w = 0; w < words; ++w) {
    uint32_t m = fb[w];
    while (m) {
      const int j = 32 * w + __ffs(m) - 1;
      m &= m - 1;
      const int a = pan[j].lo, b = pan[j].hi;
      lo = min(lo, min(a, b));
      hi = max(hi, max(a, b));
    }
  }
  slo = hi < 0 ? 0 : lo;
  n = hi < 0 ? 0 : hi - lo + 1;
}
#endif

// quadrature in stages (stbem_stage.cu)
int stage_apex_per_sm(bool fp32, int max_tet, int max_surf, int nq);
void stage_scratch(bool fp32, int max_tet, int max_surf, int sms, const std::vector<const std::vector<uint2>*>& gran,
                   int64_t* least, int64_t* wanted);
bem_status stage_run(const BlockCtx& one, const BlockCtx* many, const int64_t* prefix, int S, bool fp32, int sms,
                     const std::vector<const std::vector<uint2>*>& gran, const std::vector<int64_t>& blocks, int64_t end,
                     void* scratch, int64_t bytes, int per_sm, cudaStream_t side, cudaStream_t s);

}  // namespace stbem
