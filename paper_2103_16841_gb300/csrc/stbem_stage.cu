// Quadrature and assembly of the matrix in stages (eq. int_bform).
//
// For every face F with nu_{F,t} != 0 over test column I and every outer
// point x_q on F (composite midpoint rule, Fig. int_tri_mid) the potentials W
// of the faces over trial column J are evaluated,
//     U[F][j] = sum_q V 1_{sigma_j}(x_q) = sum_q (W_lo(j)(x_q) - W_hi(j)(x_q)),
// and A_ij = |K_I| / m_Q^2 * (U[F_lo(i)][j] - U[F_hi(i)][j]) (eq. int_bform
// with nu_{F,t}|F| = -|K| on the lower face, +|K| on the upper).
//
// The blocks (I, J) are taken in chunks whose intermediate data fit the
// operator's scratch. Per chunk:
//   k_apex       a CTA per block: the block's pattern bits; one thread per
//                (face, outer point): its geometry against column J and the
//                class of every face of its window (dark: W = 0, fully lit:
//                the whole triangle's W, cut: queued)
//   k_cut_far    one thread per queued pair in the far field: the edge pieces
//                and the conic arc of the cut face
//   k_cut_any    pairs in the near field and arcs the far form refuses
//   k_cut_fp64   near-singular faces of the mixed path, in FP64
//   k_assemble   a CTA per block: U and the entries (or their product with x)
// The FP64 operator takes the same stages in FP64, with one queue.
//
// Why stages: the cut faces are about a third of the pairs and cost ten times
// a dark or lit one. In one kernel with a warp per face, 14 of 32 lanes were
// active, every warp held the registers and shared memory of the largest
// phase (8 to 16 warps per SM), and the phases' code did not fit the
// instruction caches. Queues fill the lanes, and each stage has its own
// register budget and occupancy. The intermediate data are about 170 bytes
// per (face, outer point), written and read once.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "stbem_block.cuh"
#include "stbem_internal.h"

namespace stbem {

bem_status upload_gauss_stage(const double* x, const double* w, const float* xf, const float* wf, size_t n) {
  STBEM_CUDA(cudaMemcpyToSymbol(c_gl_x, x, n * sizeof(double)));
  STBEM_CUDA(cudaMemcpyToSymbol(c_gl_w, w, n * sizeof(double)));
  STBEM_CUDA(cudaMemcpyToSymbol(c_gl_xf, xf, n * sizeof(float)));
  STBEM_CUDA(cudaMemcpyToSymbol(c_gl_wf, wf, n * sizeof(float)));
  return BEM_OK;
}

namespace {

// One apex (face, outer point) against a trial column, as the cut stages need it.
struct alignas(16) ApexF {
  float xb[2], d, far_rho;
  float rs[3], E[3];             // corner distances, whole-edge integrals
  float rho_hi[3], rho_lo[3], nt_hi, nt_lo;
  int far;
  uint32_t slot0;                // potential of the window's first face
  int32_t surf0;                 // and that face
  int32_t col, pt, seg;
  double xb64[2], d64;           // where the conic's size cancels (d0_cancels)
};
static_assert(sizeof(ApexF) == 128, "ApexF layout");
struct alignas(16) ApexD {
  double t, d, xb[2], rs[3], E[3];
  uint32_t slot0;
  int32_t surf0, col, seg;
};
static_assert(sizeof(ApexD) == 96, "ApexD layout");

template <typename R> struct Types;
template <> struct Types<float> { typedef ApexF Apex; typedef FaceF Face; };
template <> struct Types<double> { typedef ApexD Apex; typedef FaceGeom Face; };

enum { CNT_APEX, CNT_ASM, CNT_SLOT, CNT_RAY, CNT_FAR, CNT_ANY, CNT_COP, CNT_F64, CNT_N };

struct StageArgs {
  BlockCtx one;                  // the operator (S <= 1), or the sizes all operators of a batch share
  const BlockCtx* many;
  const int64_t* prefix;
  int S;
  int64_t g0, g1;                // blocks of the chunk (dense order, operators one after the other)
  void* apex;
  void* W;                       // potentials; a queued one holds its apex's index until it is computed
  uint32_t *q_far, *q_any;
  uint32_t *q_64, *q_64_last;    // FP64 faces: coplanar apexes from the front, the others from the back
  uint2* fmeta;                  // per block and face: first potential, window (first face | faces << 16)
  uint32_t* bits;                // per block and face
  unsigned* cnt;
  void* uslab;                   // per CTA of k_assemble: U where shared memory does not hold it
  int ucap;                      // entries of U that shared memory holds
};

constexpr int kApexThreads = 256;   // >= MAX_COL_SURF: one thread per face in the window scan
static_assert(kApexThreads >= MAX_COL_SURF, "one thread per face");
constexpr int kCutThreads = 128;
constexpr int k64Threads = 128;     // (a warp per CTA: level-3 sphere, 8 slabs 239 ms, four warps 214)
// scratch of an assembly: 256 MiB / 512 MiB / 1 GiB / 2 GiB gave 308 / 238 / 239 / 236 ms
// on the level-3 sphere with 8 slabs, 52 / 49 / 45 / 43 ms on the level-2 sphere with 15
constexpr size_t kScratch = (size_t)1 << 30;
constexpr int kAsmThreads = 128;

// exclusive sum over the CTA (kApexThreads threads); *total = the sum
__device__ __forceinline__ unsigned cta_scan(unsigned v, unsigned* s_w, unsigned* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned u = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += u;
  }
  if (lane == 31) s_w[warp] = inc;
  __syncthreads();
  unsigned off = 0, sum = 0;
#pragma unroll
  for (int w = 0; w < kApexThreads / 32; ++w) {
    const unsigned x = s_w[w];
    if (w < warp) off += x;
    sum += x;
  }
  *total = sum;
  __syncthreads();
  return off + inc - v;
}

// appends v to a queue (dir: upwards or downwards); the active lanes take their places with one atomic
__device__ __forceinline__ void push(uint32_t* q, int dir, unsigned* n, uint32_t v) {
  const unsigned m = __activemask(), lane = threadIdx.x & 31;
  const int leader = __ffs(m) - 1;
  unsigned base = 0;
  if ((int)lane == leader) base = atomicAdd(n, (unsigned)__popc(m));
  base = __shfl_sync(m, base, leader);
  q[dir * (int)(base + __popc(m & ((1u << lane) - 1u)))] = v;
}

// ---- geometry of an apex against the trial column ----------------------

__device__ __forceinline__ void frame_points(PtR<float>& T, const ColR<float>& R) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    T.q[k][0] = R.Q[k][0] - T.xb[0];
    T.q[k][1] = R.Q[k][1] - T.xb[1];
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    T.ps[k] = T.q[k][0] * R.U[k][1] - T.q[k][1] * R.U[k][0];
    T.ws[k] = T.q[k][0] * R.U[k][0] + T.q[k][1] * R.U[k][1];
  }
}

// A function of its own: inlined, its products were contracted with those of
// the geometry around it, and the near edges came out an ulp apart from the
// same edges integrated elsewhere.
__device__ __noinline__ float whole_edge(const PtR<float>& T, const ColR<float>& R, int k) {
  return edge_full_mixed(T, R, k);
}

// Positions of a test column against a trial column, mixed path: what the
// outer points of all its faces share, since a point's position depends on its
// node alone (only its time depends on the face). Relative position, height,
// foot point and corner distances are formed in FP64: they carry the
// cancellation between |x - y| and t - tau, and their FP32 roundings decide
// between forms of a face's integral that differ by 1e-6 (formed in FP32 pairs,
// some 50 of 30 million entries of the level-2 sphere with 15 slabs came out
// by up to 1e-6 apart). One array per quantity, [nq] each. k_apex on the
// level-3 sphere with 8 slabs: 70.5 ms of launches with pairs per face, 66.0 so.
struct Positions {
  double *r[3], *rlo, *xb64[2], *d64;
  float *xb[2], *d, *far_rho, *rs[3], *E[3];
  int* far;
};
constexpr size_t kPosBytes = 7 * sizeof(double) + 10 * sizeof(float) + sizeof(int);
__device__ __forceinline__ Positions positions(unsigned char* smem, int nq) {
  Positions P;
  double* d = reinterpret_cast<double*>(smem);
  auto next64 = [&] { double* p = d; d += nq; return p; };
  for (int k = 0; k < 3; ++k) P.r[k] = next64();
  P.rlo = next64();
  P.xb64[0] = next64(); P.xb64[1] = next64(); P.d64 = next64();
  float* f = reinterpret_cast<float*>(d);
  auto next32 = [&] { float* p = f; f += nq; return p; };
  P.xb[0] = next32(); P.xb[1] = next32(); P.d = next32(); P.far_rho = next32();
  for (int k = 0; k < 3; ++k) P.rs[k] = next32();
  for (int k = 0; k < 3; ++k) P.E[k] = next32();
  P.far = reinterpret_cast<int*>(f);
  return P;
}
// position q in registers (T.far, T.ps and T.ws are not set)
__device__ __forceinline__ void take_position(const Positions& P, int q, const ColR<float>& R, PtR<float>& T) {
  T.d = P.d[q];
  T.xb[0] = P.xb[0][q];
  T.xb[1] = P.xb[1][q];
  for (int k = 0; k < 3; ++k) {
    T.rs[k] = P.rs[k][q];
    T.q[k][0] = R.Q[k][0] - T.xb[0];
    T.q[k][1] = R.Q[k][1] - T.xb[1];
  }
  T.C = T.rs[0];
}

// x: [nq] outer points of a face of the test column (all threads; ends with a barrier)
__device__ __forceinline__ void column_positions(const double* x, int nq, const ColGeom& G, const ColR<float>& R,
                                                 const Positions& P) {
  // a warp takes the frames or the distances, not both
  const int frames = (nq + 31) / 32 * 32;
  for (int it = threadIdx.x; it < frames + 3 * nq; it += blockDim.x) {
    if (it < frames) {
      if (it >= nq) continue;
      const double* y = x + 4 * it;
      const double rel[3] = {y[1] - G.c0[0], y[2] - G.c0[1], y[3] - G.c0[2]};
      double d = rel[0] * G.n[0] + rel[1] * G.n[1] + rel[2] * G.n[2];
      if (fabs(d) < 1e-13 * G.diam) d = 0.0;
      const double xb0 = rel[0] * G.e1[0] + rel[1] * G.e1[1] + rel[2] * G.e1[2];
      const double xb1 = rel[0] * G.e2[0] + rel[1] * G.e2[1] + rel[2] * G.e2[2];
      PtR<float> T;
      T.xb[0] = (float)xb0;
      T.xb[1] = (float)xb1;
      frame_points(T, R);
      float out = 0.f;
#pragma unroll
      for (int k = 0; k < 3; ++k) out = fmaxf(out, -T.ps[k]);
      P.d64[it] = d;
      P.xb64[0][it] = xb0;
      P.xb64[1][it] = xb1;
      P.rlo[it] = sqrt(d * d + (double)out * (double)out);
      P.d[it] = (float)d;
      P.xb[0][it] = T.xb[0];
      P.xb[1][it] = T.xb[1];
      P.far_rho[it] = out;
      P.far[it] = out >= FAR_RHO * R.diam;
    } else {
      const int q = (it - frames) / 3, k = (it - frames) - 3 * q;
      const double* y = x + 4 * q;
      const double dx = y[1] - G.X[k][0], dy = y[2] - G.X[k][1], dz = y[3] - G.X[k][2];
      const double r = sqrt(dx * dx + dy * dy + dz * dz);
      P.r[k][q] = r;
      P.rs[k][q] = (float)r;
    }
  }
  __syncthreads();
  for (int it = threadIdx.x; it < 3 * nq; it += blockDim.x) {
    const int q = it / 3, k = it - 3 * q;
    PtR<float> T;
    take_position(P, q, R, T);
    frame_points(T, R);
    T.far = P.far[q];
    T.far_rho = P.far_rho[q];
    P.E[k][q] = whole_edge(T, R, k);
  }
  __syncthreads();
}

// ---- k_apex ------------------------------------------------------------

template <typename R>
size_t apex_smem(int max_tet, int max_surf, int nq) {
  size_t s = bits_smem(max_tet, max_surf, nq);
  s = (s + 15) / 16 * 16 + sizeof(typename Types<R>::Face) * max_surf;
  if (sizeof(R) == 4) s += (kPosBytes * nq + 7) / 8 * 8;
  return s + sizeof(uint2) * max_surf + sizeof(uint16_t) * ((max_surf + 7) / 8 * 8);
}

template <typename R>
__global__ void __launch_bounds__(kApexThreads, sizeof(R) == 4 ? 4 : 2) k_apex(const StageArgs a) {
  constexpr bool FP32 = sizeof(R) == 4;
  typedef typename Types<R>::Face Face;
  typedef typename Types<R>::Apex Apex;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ BlockSm C;
  __shared__ BlockCtx B;
  __shared__ __align__(16) ColR<float> G;
  __shared__ unsigned s_w[kApexThreads / 32], s_base[4];
  __shared__ int s_seg;
  const int tid = threadIdx.x, nq = a.one.nq, max_surf = a.one.max_surf, words = bit_words(a.one.max_tet);
  const BlockPtr P = block_ptr(smem, a.one.max_tet, max_surf, nq);
  Face* Fs = reinterpret_cast<Face*>(smem + (bits_smem(a.one.max_tet, max_surf, nq) + 15) / 16 * 16);
  unsigned char* after = reinterpret_cast<unsigned char*>(Fs + max_surf);
  const Positions X = positions(after, nq);
  uint2* fm = reinterpret_cast<uint2*>(after + (FP32 ? (kPosBytes * nq + 7) / 8 * 8 : 0));
  uint16_t* act = reinterpret_cast<uint16_t*>(fm + max_surf);
  if (tid == 0 && a.S <= 1) B = a.one;
  int cur = a.S > 1 ? -1 : 0;
  for (;;) {
    if (tid == 0) s_base[3] = atomicAdd(&a.cnt[CNT_APEX], 1u);
    __syncthreads();
    const int64_t g = a.g0 + s_base[3];
    if (g >= a.g1) break;
    int64_t b = g;
    if (a.S > 1) {
      if (tid == 0) s_seg = find_seg(a.prefix, a.S, g);
      __syncthreads();
      if (s_seg != cur && tid == 0) B = a.many[s_seg];
      cur = s_seg;
      b -= a.prefix[cur];
    }
    __syncthreads();
    if (B.bw[b] == 0) continue;
    const int64_t I = b / B.n_col, J = b % B.n_col;
    load_trial(B, J, C, P.pan);
    load_test(B, I, C);
    block_bits(B, C, P);
    // trial faces and column frame
    if constexpr (FP32) {
      const uint4* src = reinterpret_cast<const uint4*>(B.facef + C.surfJ);
      for (int k = tid; k < 3 * C.nsJ; k += kApexThreads) reinterpret_cast<uint4*>(Fs)[k] = src[k];
      const float* cs = reinterpret_cast<const float*>(&B.colf[J].R);
      for (int k = tid; k < (int)(sizeof(G) / 4); k += kApexThreads) reinterpret_cast<float*>(&G)[k] = cs[k];
      __syncthreads();
      column_positions(B.pts + 4 * (int64_t)C.surfI * nq, nq, B.cols[J], G, X);
    } else {
      for (int k = tid; k < C.nsJ; k += kApexThreads) Fs[k] = B.surf[C.surfJ + k].f;
    }
    // windows of the faces, their places among the chunk's potentials
    int slo = 0, nsw = 0;
    if (tid < C.nsI) bits_surfaces(P.bits + tid * words, words, P.pan, slo, nsw);
    unsigned total;
    const unsigned ex = cta_scan((unsigned)(nsw * nq) | (nsw ? 1u << 24 : 0u), s_w, &total);
    const int nact = (int)(total >> 24);
    if (tid == 0) {
      s_base[0] = atomicAdd(&a.cnt[CNT_SLOT], total & 0xffffffu);
      s_base[1] = atomicAdd(&a.cnt[CNT_RAY], (unsigned)(nact * nq));
    }
    __syncthreads();
    const unsigned ray0 = s_base[1];
    if (tid < C.nsI) {
      const uint2 m = make_uint2(s_base[0] + (ex & 0xffffffu), (unsigned)slo | ((unsigned)nsw << 16));
      fm[tid] = m;
      a.fmeta[(g - a.g0) * max_surf + tid] = m;
      if (nsw) act[ex >> 24] = (uint16_t)tid;
    }
    for (int k = tid; k < C.nsI * words; k += kApexThreads) a.bits[(g - a.g0) * max_surf * words + k] = P.bits[k];
    __syncthreads();
    const int nr = nact * nq, lane = tid & 31;
    R* W = static_cast<R*>(a.W);
    for (int r = tid; r - lane < nr; r += kApexThreads) {   // (whole warps)
      const bool on = r < nr;
      int n = 0, first = 0;
      uint32_t slot0 = 0;
      int pt = 0, q = 0;
      double t = 0.0;
      typename std::conditional<FP32, PtR<float>, PointCol>::type T;
      ConeM M;
      R Wst = R(0);
      bool far = true;
      if (on) {
        const int k = r / nq, f = act[k];
        q = r - k * nq;
        const uint2 m = fm[f];
        first = (int)(m.y & 0xffffu);
        n = (int)(m.y >> 16);
        slot0 = m.x + q;
        pt = (C.surfI + f) * nq + q;
        if constexpr (FP32) {
          take_position(X, q, G, T);
          t = B.pts[4 * (int64_t)pt];
          for (int c = 0; c < 3; ++c) split2(X.r[c][q] - t, M.rho_hi[c], M.rho_lo[c]);
          split2(X.rlo[q] - t, M.rlot_hi, M.rlot_lo);
          Wst = (X.E[0][q] + X.E[1][q]) + X.E[2][q];
          far = X.far[q];
        } else {
          point_col(B.pts + 4 * (int64_t)pt, B.cols[J], T, false);
          Wst = T.Wst;
        }
      }
      bool any = false;
      const int wmax = __reduce_max_sync(0xffffffffu, n);
      for (int s0 = 0; s0 < wmax; s0 += 64) {
        unsigned long long mask = 0;
        const int s1 = min(n, s0 + 64);
        for (int s = s0; s < s1; ++s) {
          int cls;
          R F[3];
          if constexpr (FP32) {
            // one FP32 sum settles what is far from the cone: the pairs' sums differ from
            // it by less than the filter's margin
            const FaceF& Fc = Fs[first + s];
            const float mx = fmaxf(fmaxf(Fc.p_hi[0] + M.rho_hi[0], Fc.p_hi[1] + M.rho_hi[1]), Fc.p_hi[2] + M.rho_hi[2]);
            cls = mx < -B.margin ? (int)FACE_LIT : Fc.pmin_hi + M.rlot_hi > B.margin ? (int)FACE_DARK
                                                                                    : face_class_mixed(T, M, Fc, F);
          } else {
            double c;
            cls = face_class(B.cols[J], T, Fs[first + s], F, c);
          }
          if (cls == FACE_CUT) mask |= 1ull << (s - s0);
          else W[slot0 + s * nq] = cls == FACE_LIT ? Wst : R(0);
        }
        any |= mask != 0;
        // places in the queues: a scan over the warp and one atomic per queue
        const unsigned cnt = (unsigned)__popcll(mask);
        const unsigned mine = far ? cnt : cnt << 16;
        unsigned at = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned u = __shfl_up_sync(0xffffffffu, at, o);
          if (lane >= o) at += u;
        }
        unsigned base_far = 0, base_any = 0;
        if (lane == 31) {
          if (at & 0xffffu) base_far = atomicAdd(&a.cnt[CNT_FAR], at & 0xffffu);
          if (at >> 16) base_any = atomicAdd(&a.cnt[CNT_ANY], at >> 16);
        }
        base_far = __shfl_sync(0xffffffffu, base_far, 31);
        base_any = __shfl_sync(0xffffffffu, base_any, 31);
        at -= mine;
        uint32_t* to = far ? a.q_far + base_far + (at & 0xffffu) : a.q_any + base_any + (at >> 16);
        while (mask) {
          const int s = s0 + __ffsll((long long)mask) - 1;
          mask &= mask - 1;
          const uint32_t slot = slot0 + s * nq;
          *to++ = slot;
          if constexpr (FP32) W[slot] = __uint_as_float(ray0 + r);
          else W[slot] = __hiloint2double(0, (int)(ray0 + r));
        }
      }
      if (any) {
        Apex Y;
        if constexpr (FP32) {
          for (int i = 0; i < 2; ++i) { Y.xb[i] = T.xb[i]; Y.xb64[i] = X.xb64[i][q]; }
          Y.d = T.d; Y.d64 = X.d64[q]; Y.far_rho = X.far_rho[q]; Y.far = far;
          for (int k = 0; k < 3; ++k) {
            Y.rs[k] = T.rs[k]; Y.E[k] = X.E[k][q]; Y.rho_hi[k] = M.rho_hi[k]; Y.rho_lo[k] = M.rho_lo[k];
          }
          split2(-t, Y.nt_hi, Y.nt_lo);
          Y.pt = pt;
        } else {
          Y.t = T.t; Y.d = T.D.d; Y.xb[0] = T.D.xb[0]; Y.xb[1] = T.D.xb[1];
          for (int k = 0; k < 3; ++k) { Y.rs[k] = T.D.rs[k]; Y.E[k] = T.D.Efull[k]; }
        }
        Y.slot0 = slot0; Y.surf0 = C.surfJ + first; Y.col = (int32_t)J; Y.seg = cur;
        static_cast<Apex*>(a.apex)[ray0 + r] = Y;
      }
    }
    __syncthreads();
  }
}

// ---- cut faces ---------------------------------------------------------

// a queued pair of the mixed path: its apex, face and column; false: near-singular
struct CutF {
  PtR<float> T;
  ColR<float> R;
  FaceCutIn<float> in;
};
__device__ __forceinline__ bool load_cut(const StageArgs& a, uint32_t slot, uint32_t ray, CutF& c) {
  const ApexF& Y = static_cast<const ApexF*>(a.apex)[ray];
  const BlockCtx& B = a.S > 1 ? a.many[Y.seg] : a.one;
  const int surf = Y.surf0 + (int)(slot - Y.slot0) / a.one.nq;
  const FaceF Fc = B.facef[surf];
  c.R = B.colf[Y.col].R;
  PtR<float>& T = c.T;
  ConeM M;
  T.d = Y.d;
  T.xb[0] = Y.xb[0]; T.xb[1] = Y.xb[1];
  T.far = Y.far;
  T.far_rho = Y.far_rho;
  for (int k = 0; k < 3; ++k) {
    T.rs[k] = Y.rs[k]; T.Efull[k] = Y.E[k]; M.rho_hi[k] = Y.rho_hi[k]; M.rho_lo[k] = Y.rho_lo[k];
  }
  T.C = T.rs[0];
  M.nt_hi = Y.nt_hi; M.nt_lo = Y.nt_lo;
  frame_points(T, c.R);
  float F[3];
  for (int k = 0; k < 3; ++k) F[k] = add2(Fc.p_hi[k], Fc.p_lo[k], M.rho_hi[k], M.rho_lo[k]);
  const float cc = face_c_mixed(T, M, Fc, c.R.diam);
  if (near_singular_mixed(cc, T.d, c.R.diam)) return false;
  cut_in_mixed(T, M, Fc, F, cc, c.in);
  if (d0_cancels(c.in)) c.in.D0 = d0_fp64(B.pts[4 * (int64_t)Y.pt], Y.xb64, Y.d64, B.surf[surf].f);
  return true;
}

// The crossings of the conic with edge k (as in face_cut): the lit part [la, lb]
// of the edge and which ends are crossings; false: no lit part.
__device__ __forceinline__ bool edge_lit(const CutF& c, int k, float& la, float& lb, bool& la_root, bool& lb_root) {
  const int k1 = (k + 1) % 3;
  const float Fa = c.in.F[k], Fb = c.in.F[k1];
  la = 0.f;
  lb = 1.f;
  la_root = lb_root = false;
  if (Fa < 0.f && Fb < 0.f) return true;
  const float a0 = c.in.a0[k], a1 = c.in.a1[k], L = c.R.L[k];
  const float Ex = c.R.U[k][0] * L, Ey = c.R.U[k][1] * L;
  const float A2 = L * L - a1 * a1;
  const float B2 = 2.f * ((c.T.q[k][0] * Ex + c.T.q[k][1] * Ey) + a0 * a1);
  const float C2 = Fa * (c.T.rs[k] + a0);
  // both roots, or one where the edge is parallel to the cone (r1 then fails every test below)
  float r0 = 2.f, r1 = 2.f;
  if (fabsf(A2) <= 1e-6f * (L * L + a1 * a1)) {
    if (B2 != 0.f) r0 = -C2 / B2;
  } else {
    const float disc = B2 * B2 - 4.f * A2 * C2;
    if (disc >= 0.f) {
      const float sq = sqrtf(disc);
      const float qq = -0.5f * (B2 + (B2 >= 0.f ? sq : -sq));
      if (qq != 0.f) { r0 = qq / A2; r1 = C2 / qq; }
      else r0 = 0.f;
    }
  }
  const float slack = 1e-5f;
  const bool ok0 = a0 - a1 * r0 > 0.f && r0 >= -slack && r0 <= 1.f + slack;
  const bool ok1 = a0 - a1 * r1 > 0.f && r1 >= -slack && r1 <= 1.f + slack;
  r0 = fminf(1.f, fmaxf(0.f, r0));
  r1 = fminf(1.f, fmaxf(0.f, r1));
  const float lo = ok0 ? (ok1 ? fminf(r0, r1) : r0) : r1, hi = ok0 ? (ok1 ? fmaxf(r0, r1) : r0) : r1;
  if (Fa < 0.f) {           // exit on this edge
    if (ok0 || ok1) { lb = hi; lb_root = true; }
    return true;
  }
  if (Fb < 0.f) {           // entry on this edge
    if (ok0 || ok1) { la = lo; la_root = true; }
    return true;
  }
  if (ok0 && ok1 && hi > lo) {
    la = lo; lb = hi; la_root = lb_root = true;
    return true;
  }
  return false;
}

// (a function of its own for the same reason as whole_edge)
__device__ __noinline__ bool chord_arc(const float* xb, float d, float C, float far_rho, const float* g, const float* A,
                                       const float* D, const ArcRule& rule, float& out) {
  return arc_far<float>(xb, d, C, far_rho, g, A, D, rule, out);
}

// The far field's cut faces (nine tenths of them on a fine sphere): a lit set
// with one exit and one entry, so one arc and at most two edges with a crossing,
// taken in registers; the edges' Gauss rules run in two converged turns (first
// and second crossed edge) instead of three divergent ones. What has other
// events, or an arc the chord form refuses, goes on to the other queue. The
// arithmetic is face_cut's and arc_far's. Bound by issue and the latency of
// the gathers: level-3 sphere, 8 slabs 193 -> 149 ms of quadrature against the
// general code in this kernel (with the warp-wide queue places of k_apex), level-2
// sphere, 32 slabs 106 -> 87 ms.
__global__ void __launch_bounds__(kCutThreads, 6) k_cut_far(const StageArgs a) {
  float* W = static_cast<float*>(a.W);
  const unsigned n = a.cnt[CNT_FAR];
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t slot = a.q_far[i];
    CutF c;
    if (!load_cut(a, slot, __float_as_uint(W[slot]), c)) {
      if (c.T.d == 0.f) push(a.q_64, 1, &a.cnt[CNT_COP], slot);
      else push(a.q_64_last, -1, &a.cnt[CNT_F64], slot);
      continue;
    }
    float t[3] = {0.f, 0.f, 0.f}, h2[2] = {0.f, 0.f};   // edge terms; the crossed edges' lit ranges
    float l2[2] = {0.f, 0.f};
    int k2[2] = {-1, -1}, n_exit = 0, n_entry = 0;
    float A[2] = {0.f, 0.f}, E[2] = {0.f, 0.f};          // exit and entry, column coordinates
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      float la, lb;
      bool ra, rb;
      if (!edge_lit(c, k, la, lb, ra, rb)) continue;
      if (!ra && !rb) {
        t[k] = c.T.Efull[k];
        continue;
      }
      const int z = k2[0] < 0 ? 0 : 1;   // (a third crossed edge has other events: not taken here)
      if (z == 0) { k2[0] = k; l2[0] = la; h2[0] = lb; }
      else { k2[1] = k; l2[1] = la; h2[1] = lb; }
      const float Ux = c.R.U[k][0], Uy = c.R.U[k][1], L = c.R.L[k];
      if (ra) { ++n_entry; E[0] = c.R.Q[k][0] + la * Ux * L; E[1] = c.R.Q[k][1] + la * Uy * L; }
      if (rb) { ++n_exit; A[0] = c.R.Q[k][0] + lb * Ux * L; A[1] = c.R.Q[k][1] + lb * Uy * L; }
    }
    if (n_exit + n_entry == 0) {
      const float G2 = c.in.g[0] * c.in.g[0] + c.in.g[1] * c.in.g[1];
      if (!(G2 < 1.f && c.in.c > 0.f && c.in.D0 > 0.f)) W[slot] = 0.f;   // no closed ellipse: nothing lit
      else push(a.q_any, 1, &a.cnt[CNT_ANY], slot);
      continue;
    }
    if (n_exit != 1 || n_entry != 1) {
      push(a.q_any, 1, &a.cnt[CNT_ANY], slot);
      continue;
    }
    // the crossed edges
    float m2[2], hh[2];
#pragma unroll 1
    for (int z = 0; z < 2; ++z) {
      const int k = k2[z];
      m2[z] = hh[z] = 0.f;
      if (k < 0) continue;
      const float la = l2[z], lb = h2[z];
      const float h = 0.5f * (lb - la);
      if (!(h > 0.f)) continue;
      const float mid = 0.5f * (la + lb);
      const float L = k == 0 ? c.R.L[0] : k == 1 ? c.R.L[1] : c.R.L[2];
      const float ps = k == 0 ? c.T.ps[0] : k == 1 ? c.T.ps[1] : c.T.ps[2];
      const float ws = k == 0 ? c.T.ws[0] : k == 1 ? c.T.ws[1] : c.T.ws[2];
      const float Ux = k == 0 ? c.R.U[0][0] : k == 1 ? c.R.U[1][0] : c.R.U[2][0];
      const float Uy = k == 0 ? c.R.U[0][1] : k == 1 ? c.R.U[1][1] : c.R.U[2][1];
      const float Qx = k == 0 ? c.R.Q[0][0] : k == 1 ? c.R.Q[1][0] : c.R.Q[2][0];
      const float Qy = k == 0 ? c.R.Q[0][1] : k == 1 ? c.R.Q[1][1] : c.R.Q[2][1];
      const float q0x = -c.T.xb[0], q0y = -c.T.xb[1];
      const int nn = gauss_order<float>((-ws / L - mid) / h, fabsf(ps) / (L * h), a.one.rule.ltol_f, 3, 10);
      const float* X = gl_nodes<float>(nn);
      const float* Wt = gl_weights<float>(nn);
      const float ex = Ux * L, ey = Uy * L, d2 = c.T.d * c.T.d;
      float acc = 0.f;
      for (int g = 0; g < nn; ++g) {
        const float lam = mid + h * X[g];
        const float ux = Qx + lam * ex, uy = Qy + lam * ey;
        const float qx = q0x + ux, qy = q0y + uy, q2 = qx * qx + qy * qy;
        const float r = sqrtf(q2 + d2);
        const float del = (ux * (2.f * q0x + ux) + uy * (2.f * q0y + uy)) / (r + c.T.C);
        acc += Wt[g] * del / q2;
      }
      m2[z] = acc * ps * L;
      hh[z] = h;
    }
    float v = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (k == k2[0]) v = __fadd_rn(v, __fmul_rn(m2[0], hh[0]));
      else if (k == k2[1]) v = __fadd_rn(v, __fmul_rn(m2[1], hh[1]));
      else v += t[k];
    }
    const float D[2] = {E[0] - A[0], E[1] - A[1]};
    float arc = 0.f;
    if (!chord_arc(c.T.xb, c.T.d, c.T.C, c.T.far_rho, c.in.g, A, D, a.one.rule, arc)) {
      push(a.q_any, 1, &a.cnt[CNT_ANY], slot);
      continue;
    }
    v += arc;
    if (!isfinite(v)) push(a.q_64_last, -1, &a.cnt[CNT_F64], slot);
    else W[slot] = v;
  }
}

// The other cut faces: near apexes, several arcs, whole ellipses. A value that
// is not finite is recomputed in FP64. Bound by issue with about half of the
// lanes at work; 80 registers (6 CTAs per SM).
__global__ void __launch_bounds__(kCutThreads, 6) k_cut_any(const StageArgs a) {
  float* W = static_cast<float*>(a.W);
  const unsigned n = a.cnt[CNT_ANY];
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t slot = a.q_any[i];
    CutF c;
    if (!load_cut(a, slot, __float_as_uint(W[slot]), c)) {
      if (c.T.d == 0.f) push(a.q_64, 1, &a.cnt[CNT_COP], slot);
      else push(a.q_64_last, -1, &a.cnt[CNT_F64], slot);
      continue;
    }
    ArcRec<float> arc[3];
    int na = 0;
    float v = (float)face_cut<float>(c.R, c.T, c.in, a.one.rule, arc, &na);
    for (int k = 0; k < na; ++k) v += arc_value<float>(arc[k], a.one.rule);
    if (!isfinite(v)) push(a.q_64_last, -1, &a.cnt[CNT_F64], slot);
    else W[slot] = v;
  }
}

// Bound by the FP64 pipe (a warp instruction takes it for 19 cycles) and, where
// a chunk has few, by their serial chain. Coplanar apexes (closed form, about
// a fifth of the work of the others' mapped Gauss nodes) have warps of their
// own.
__global__ void __launch_bounds__(k64Threads) k_cut_fp64(const StageArgs a) {
  float* W = static_cast<float*>(a.W);
  const unsigned n1 = a.cnt[CNT_F64], n1w = (n1 + 31) / 32 * 32, n = n1w + a.cnt[CNT_COP];
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    if (i >= n1 && i < n1w) continue;
    const uint32_t slot = i < n1 ? *(a.q_64_last - i) : a.q_64[i - n1w];
    const ApexF& Y = static_cast<const ApexF*>(a.apex)[__float_as_uint(W[slot])];
    const BlockCtx& B = a.S > 1 ? a.many[Y.seg] : a.one;
    W[slot] = (float)face_W_fp64(B.pts + 4 * (int64_t)Y.pt, B.cols[Y.col],
                                 B.surf[Y.surf0 + (int)(slot - Y.slot0) / a.one.nq].f, a.one.n_theta);
  }
}

// the FP64 operator's cut faces
__global__ void __launch_bounds__(kCutThreads) k_cut_d(const StageArgs a) {
  double* W = static_cast<double*>(a.W);
  const unsigned n = a.cnt[CNT_FAR];
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t slot = a.q_far[i];
    const ApexD Y = static_cast<const ApexD*>(a.apex)[(uint32_t)__double2loint(W[slot])];
    const BlockCtx& B = a.S > 1 ? a.many[Y.seg] : a.one;
    const ColGeom& G = B.cols[Y.col];
    ColR<double> R;
    make_colr<double>(G, R);
    PointCol P;
    P.t = Y.t;
    P.rlo = 0.0;                    // the class is known: the pair is cut
    P.D.d = Y.d; P.D.xb[0] = Y.xb[0]; P.D.xb[1] = Y.xb[1];
    P.D.far = 0; P.D.C = 0.0; P.D.far_rho = 0.0;
    for (int k = 0; k < 3; ++k) {
      P.r[k] = P.D.rs[k] = Y.rs[k];
      P.D.Efull[k] = Y.E[k];
      P.D.q[k][0] = R.Q[k][0] - Y.xb[0];
      P.D.q[k][1] = R.Q[k][1] - Y.xb[1];
    }
    for (int k = 0; k < 3; ++k) {
      P.D.ps[k] = P.D.q[k][0] * R.U[k][1] - P.D.q[k][1] * R.U[k][0];
      P.D.ws[k] = P.D.q[k][0] * R.U[k][0] + P.D.q[k][1] * R.U[k][1];
    }
    const FaceGeom Fc = B.surf[Y.surf0 + (int)(slot - Y.slot0) / a.one.nq].f;
    double F[3], c;
    for (int k = 0; k < 3; ++k) F[k] = (Fc.p[k] - P.t) + P.r[k];
    c = P.t - (Fc.p[0] + Fc.g[0] * P.D.xb[0] + Fc.g[1] * P.D.xb[1]);
    if (fabs(c) < 1e-13 * G.diam) c = 0.0;
    FaceCutIn<double> in;
    cut_in_fp64(P, Fc, F, c, in);
    W[slot] = face_cut<double>(R, P.D, in, a.one.rule);
  }
}

// ---- k_assemble --------------------------------------------------------

constexpr size_t kUBytes = 24576;   // shared memory for U

template <typename R>
size_t asm_smem(int max_tet, int max_surf) {
  const int words = bit_words(max_tet);
  return kUBytes + sizeof(uint32_t) * ((size_t)max_surf * words + 3 * max_surf + 2 * max_tet + 16);
}

// Bound by latency and L1 traffic: the entries are written once, coalesced;
// the potentials are read twice (as the lower and the upper face of a panel).
template <typename R>
__global__ void __launch_bounds__(kAsmThreads) k_assemble(const StageArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ BlockCtx B;
  __shared__ int s_seg, s_wU;
  __shared__ unsigned s_g;
  __shared__ R s_scale;
  const int tid = threadIdx.x, nq = a.one.nq, max_surf = a.one.max_surf, max_tet = a.one.max_tet;
  const int words = bit_words(max_tet);
  R* Us = reinterpret_cast<R*>(smem);
  uint32_t* bits = reinterpret_cast<uint32_t*>(smem + kUBytes);
  uint2* fm = reinterpret_cast<uint2*>(bits + (max_surf * words + 1) / 2 * 2);
  int* jf = reinterpret_cast<int*>(fm + max_surf);                        // first panel of a face's bits
  uint32_t* lohi = reinterpret_cast<uint32_t*>(jf + max_surf);            // faces of the trial panels
  uint32_t* row = lohi + max_tet;                                         // first panel | lo << 16 | hi << 24 of a row
  const R* W = static_cast<const R*>(a.W);
  if (tid == 0 && a.S <= 1) B = a.one;
  int cur = a.S > 1 ? -1 : 0;
  for (;;) {
    if (tid == 0) {
      s_g = atomicAdd(&a.cnt[CNT_ASM], 1u);
      s_wU = 0;
    }
    __syncthreads();
    const int64_t g = a.g0 + s_g;
    if (g >= a.g1) break;
    int64_t b = g;
    if (a.S > 1) {
      if (tid == 0) s_seg = find_seg(a.prefix, a.S, g);
      __syncthreads();
      if (s_seg != cur && tid == 0) B = a.many[s_seg];
      cur = s_seg;
      b -= a.prefix[cur];
      __syncthreads();
    }
    const int Wd = B.bw[b];
    __syncthreads();
    if (Wd == 0) continue;
    const int64_t I = b / B.n_col, J = b % B.n_col;
    const int t0 = B.col_tet_begin[I], nt = B.col_tet_begin[I + 1] - t0;
    const int tJ = B.col_tet_begin[J], ntJ = B.col_tet_begin[J + 1] - tJ;
    const int ns = B.col_surf_begin[I + 1] - B.col_surf_begin[I];
    if (tid == 0) s_scale = (R)(B.cols[I].area / (4.0 * STBEM_PI * nq));
    for (int f = tid; f < ns; f += kAsmThreads) {
      fm[f] = a.fmeta[(g - a.g0) * max_surf + f];
      int lo = -1, hi = -1;
      for (int w = 0; w < words; ++w) {
        const uint32_t m = a.bits[((g - a.g0) * max_surf + f) * words + w];
        bits[f * words + w] = m;
        if (m) {
          if (lo < 0) lo = 32 * w + __ffs(m) - 1;
          hi = 32 * w + 31 - __clz(m);
        }
      }
      jf[f] = max(lo, 0);
      if (lo >= 0) atomicMax(&s_wU, hi - lo + 1);
    }
    for (int j = tid; j < ntJ; j += kAsmThreads) {
      const PanelF& D = B.panf[tJ + j];
      lohi[j] = (uint32_t)D.lo | ((uint32_t)D.hi << 16);
    }
    __syncthreads();
    const int wU = s_wU;
    R* U = ns * wU <= a.ucap ? Us : static_cast<R*>(a.uslab) + (size_t)blockIdx.x * max_surf * max_tet;
    for (int it = tid; it < ns * wU; it += kAsmThreads) {
      const int f = it / wU, j = jf[f] + it - f * wU;
      R u = R(0);
      if (j < ntJ && ((bits[f * words + (j >> 5)] >> (j & 31)) & 1u)) {
        const uint2 m = fm[f];
        const uint32_t lh = lohi[j];
        const int slo = (int)(m.y & 0xffffu);
        const R* lo = W + m.x + ((int)(lh & 0xffffu) - slo) * nq;
        const R* hi = W + m.x + ((int)(lh >> 16) - slo) * nq;
        for (int q = 0; q < nq; ++q) u += lo[q] - hi[q];
      }
      U[it] = u;
    }
    for (int r = tid; r < nt; r += kAsmThreads) {
      const PanelF& D = B.panf[t0 + r];
      int first = -1;
      for (int w = 0; w < words && first < 0; ++w) {
        const uint32_t m = bits[D.lo * words + w] | bits[D.hi * words + w];
        if (m) first = 32 * w + __ffs(m) - 1;
      }
      row[r] = (uint32_t)max(first, 0) | ((uint32_t)D.lo << 16) | ((uint32_t)D.hi << 24);
    }
    __syncthreads();
    const R scale = s_scale;
    auto entry = [&](uint32_t rw, int j) {
      const int lo = (int)((rw >> 16) & 0xffu), hi = (int)(rw >> 24);
      const int ol = j - jf[lo], oh = j - jf[hi];
      const R ul = (unsigned)ol < (unsigned)wU ? U[lo * wU + ol] : R(0);
      const R uh = (unsigned)oh < (unsigned)wU ? U[hi * wU + oh] : R(0);
      return scale * (ul - uh);
    };
    if (B.mf_y) {
      // fused product: the row's band times x, one atomic add per right-hand side
      for (int it = tid; it < nt * B.mf_nrhs; it += kAsmThreads) {
        const int k = it / nt, r = it - k * nt;
        const uint32_t rw = row[r];
        const int first = (int)(rw & 0xffffu);
        const double* xk = B.mf_x + (int64_t)k * B.mf_ld + tJ;
        double sacc = 0.0;
        for (int j = first; j < min(first + Wd, ntJ); ++j) sacc += (double)entry(rw, j) * xk[j];
        atomicAdd(B.mf_y + (int64_t)k * B.mf_ld + t0 + r, sacc);
      }
    } else {
      const int64_t voff = B.boff[b], roff = B.rsoff[b];
      for (int r = tid; r < nt; r += kAsmThreads) B.rs[roff + r] = tJ + (int)(row[r] & 0xffffu);
      for (int e = tid; e < nt * Wd; e += kAsmThreads) {
        const int w = e / nt, r = e - w * nt;
        const uint32_t rw = row[r];
        const int j = (int)(rw & 0xffffu) + w;
        const R v = j < ntJ ? entry(rw, j) : R(0);
        if (B.val) B.val[voff + e] = (double)v;
        if (B.val32) B.val32[voff + e] = (float)v;
      }
    }
    __syncthreads();
  }
}

size_t up256(size_t n) { return (n + 255) / 256 * 256; }

int occupancy(const void* kern, int threads, size_t smem) {
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, smem) != cudaSuccess) cudaGetLastError();
  return std::max(per, 1);
}

size_t slot_bytes(bool fp32) { return fp32 ? 4 + 3 * 4 : 8 + 4; }
size_t apex_bytes(bool fp32) { return fp32 ? sizeof(ApexF) : sizeof(ApexD); }
// scratch of `blocks` blocks with `rays` apexes and `slots` potentials (with the regions' alignment)
size_t chunk_bytes(bool fp32, int max_tet, int max_surf, int64_t blocks, int64_t rays, int64_t slots) {
  return 8 * 256 + rays * apex_bytes(fp32) + slots * slot_bytes(fp32) +
         (size_t)blocks * max_surf * (sizeof(uint2) + sizeof(uint32_t) * bit_words(max_tet));
}
// fixed part: counters, and U of every CTA of k_assemble where shared memory does not hold it
size_t fixed_bytes(bool fp32, int max_tet, int max_surf, int sms) {
  const size_t u = (size_t)max_tet * max_surf * (fp32 ? 4 : 8);
  return 256 + (u > kUBytes ? up256(u * sms * 4) : 0);
}

// Intermediate data of a chunk where the scratch holds two of them, of `all` bytes:
// at least four chunks on the mixed path, whose side stream has other work than the
// first (FP64 stages all wait for one pipe), but not below 256 MiB: every chunk pays
// the serial chain of its FP64 faces. Reassembly of the level-0 sphere with 2 slabs
// 945 -> 343 us (625 before the stages), level-1, 5 slabs 2.9 -> 2.0 ms (64 and 128
// MiB: 2.7 and 2.5); nothing changes where the whole takes 1 GiB and more.
int64_t chunk_part(bool fp32, int64_t all) {
  const int64_t small = (int64_t)256 << 20;
  return fp32 ? std::max(all / 4, std::min(all, small)) : all;
}

}  // namespace

int stage_apex_per_sm(bool fp32, int max_tet, int max_surf, int nq) {
  const size_t smem = fp32 ? apex_smem<float>(max_tet, max_surf, nq) : apex_smem<double>(max_tet, max_surf, nq);
  const void* kern = fp32 ? (const void*)k_apex<float> : (const void*)k_apex<double>;
  ensure_smem_attr(kern, smem);
  return std::min(occupancy(kern, kApexThreads, smem), 4);
}

// Scratch of a quadrature over the blocks counted in `gran`: at least the
// largest run of GRAN blocks, at most kScratch bytes.
void stage_scratch(bool fp32, int max_tet, int max_surf, int sms, const std::vector<const std::vector<uint2>*>& gran,
                   int64_t* least, int64_t* wanted) {
  size_t big = 0, all = 0;
  for (const auto* v : gran)
    for (const uint2& c : *v) {
      const size_t n = chunk_bytes(fp32, max_tet, max_surf, GRAN, c.x, c.y);
      big = std::max(big, n);
      all += n;
    }
  const size_t fixed = fixed_bytes(fp32, max_tet, max_surf, sms);
  *least = (int64_t)up256(fixed + big);
  // two chunks, or all of it in one pass
  const size_t room = 2 * fixed + std::max<size_t>(all, fp32 ? 2 * chunk_part(fp32, (int64_t)all) : 0);
  *wanted = (int64_t)up256(std::max(fixed + big, std::min(room + 512, kScratch)));
}

// All stages over the blocks [0, end) of the concatenated operators. The
// chunks alternate between two halves of the scratch: the FP64 faces (some
// thousand per chunk, each a serial chain of most of a millisecond) and the
// entries of one chunk run on the side stream (where there is one) while the
// caller's stream takes the next chunk's apexes and FP32 faces. Large chunks
// pay: each kernel of a chunk costs about 10 us of ramp and tail. Level-2
// sphere, 15 slabs: 94 ms one chunk after the other, 45 ms so; level-3 sphere,
// 8 slabs: 263 and 214 ms. On every way out the caller's stream waits for the
// side stream.
bem_status stage_run(const BlockCtx& one, const BlockCtx* many, const int64_t* prefix, int S, bool fp32, int sms,
                     const std::vector<const std::vector<uint2>*>& gran, const std::vector<int64_t>& blocks, int64_t end,
                     void* scratch, int64_t bytes, int per_sm, cudaStream_t side, cudaStream_t s) {
  const int mt = one.max_tet, ms = one.max_surf, nq = one.nq;
  const size_t fixed = fixed_bytes(fp32, mt, ms, sms);
  unsigned char* base = static_cast<unsigned char*>(scratch);
  // two halves where the scratch holds the largest run of blocks twice
  size_t least = 0, all = 0;
  for (const auto* v : gran)
    for (const uint2& c : *v) {
      const size_t n = chunk_bytes(fp32, mt, ms, GRAN, c.x, c.y);
      least = std::max(least, n);
      all += n;
    }
  const int halves = !side || bytes / 2 / 256 * 256 < (int64_t)(fixed + least) ? 1 : 2;
  const int64_t half_bytes = bytes / halves / 256 * 256;
  StageArgs a;
  a.one = one;
  a.many = many;
  a.prefix = prefix;
  a.S = S;
  a.ucap = (int)(kUBytes / (fp32 ? 4 : 8));
  const size_t sm_apex = fp32 ? apex_smem<float>(mt, ms, nq) : apex_smem<double>(mt, ms, nq);
  const size_t sm_asm = fp32 ? asm_smem<float>(mt, ms) : asm_smem<double>(mt, ms);
  const void* k_asm = fp32 ? (const void*)k_assemble<float> : (const void*)k_assemble<double>;
  bem_status st = ensure_smem_attr(k_asm, sm_asm);
  if (st != BEM_OK) return st;
  const int n_apex = sms * std::max(1, std::min(per_sm, stage_apex_per_sm(fp32, mt, ms, nq)));
  int n_asm = sms * occupancy(k_asm, kAsmThreads, sm_asm);
  if (fixed > 256) n_asm = std::min(n_asm, sms * 4);   // one slab per CTA
  const int n_far = sms * occupancy((const void*)(fp32 ? (const void*)k_cut_far : (const void*)k_cut_d), kCutThreads, 0);
  const int n_any = sms * occupancy((const void*)k_cut_any, kCutThreads, 0);
  const int n_64 = sms * occupancy((const void*)k_cut_fp64, k64Threads, 0);

  struct Events {   // apex and FP32 faces done, entries done, per half
    cudaEvent_t e[4] = {};
    ~Events() { for (auto x : e) if (x) cudaEventDestroy(x); }
  } ev;
  if (halves == 2)
    for (auto& x : ev.e) STBEM_CUDA(cudaEventCreateWithFlags(&x, cudaEventDisableTiming));

  int64_t n_chunk = 0;
  bool forked = false;   // the side stream has work of this run
  auto flush = [&](int64_t g0, int64_t g1, int64_t rays, int64_t slots) -> bem_status {
    if (rays == 0) return BEM_OK;
    const int64_t nb = g1 - g0;
    const int h = (int)(n_chunk % halves);
    unsigned char* p = base + h * half_bytes;
    const cudaStream_t t = halves == 2 ? side : s;   // FP64 faces and entries
    if (n_chunk >= 2 && halves == 2) STBEM_CUDA(cudaStreamWaitEvent(s, ev.e[2 + h], 0));
    a.cnt = reinterpret_cast<unsigned*>(p);
    a.uslab = p + 256;
    p += fixed;
    auto take = [&](size_t n) { unsigned char* r = p; p += up256(n); return r; };
    a.g0 = g0;
    a.g1 = g1;
    a.apex = take(rays * apex_bytes(fp32));
    a.W = take(slots * (fp32 ? 4 : 8));
    a.q_far = reinterpret_cast<uint32_t*>(take(slots * 4));
    a.q_any = a.q_64 = a.q_64_last = nullptr;
    if (fp32) {
      a.q_any = reinterpret_cast<uint32_t*>(take(slots * 4));
      a.q_64 = reinterpret_cast<uint32_t*>(take(slots * 4));
      a.q_64_last = a.q_64 + slots - 1;
    }
    a.fmeta = reinterpret_cast<uint2*>(take(nb * ms * sizeof(uint2)));
    a.bits = reinterpret_cast<uint32_t*>(take(nb * ms * sizeof(uint32_t) * bit_words(mt)));
    if (p - base > (h + 1) * half_bytes) {
      set_error("quadrature scratch too small");
      return BEM_ERR_INTERNAL;
    }
    STBEM_CUDA(cudaMemsetAsync(a.cnt, 0, sizeof(unsigned) * CNT_N, s));
    auto hand_over = [&]() -> bem_status {
      if (halves == 1) return BEM_OK;
      STBEM_CUDA(cudaEventRecord(ev.e[h], s));
      STBEM_CUDA(cudaStreamWaitEvent(side, ev.e[h], 0));
      forked = true;
      return BEM_OK;
    };
    if (fp32) {
      k_apex<float><<<n_apex, kApexThreads, sm_apex, s>>>(a);
      k_cut_far<<<n_far, kCutThreads, 0, s>>>(a);
      k_cut_any<<<n_any, kCutThreads, 0, s>>>(a);
      st = hand_over();
      if (st != BEM_OK) return st;
      k_cut_fp64<<<n_64, k64Threads, 0, t>>>(a);
      k_assemble<float><<<n_asm, kAsmThreads, sm_asm, t>>>(a);
    } else {
      k_apex<double><<<n_apex, kApexThreads, sm_apex, s>>>(a);
      st = hand_over();
      if (st != BEM_OK) return st;
      k_cut_d<<<n_far, kCutThreads, 0, t>>>(a);
      k_assemble<double><<<n_asm, kAsmThreads, sm_asm, t>>>(a);
    }
    STBEM_CUDA(cudaGetLastError());
    if (halves == 2) STBEM_CUDA(cudaEventRecord(ev.e[2 + h], side));
    ++n_chunk;
    return BEM_OK;
  };
  // chunks: runs of granules that fit a half
  const int64_t chunk = std::min<int64_t>(half_bytes, fixed + std::max<int64_t>(least, chunk_part(fp32, all)));
  int64_t g0 = 0, g1 = 0, rays = 0, slots = 0, off = 0;
  for (size_t o = 0; o < gran.size(); ++o) {
    const int64_t nb = std::min(blocks[o], end - off);
    for (int64_t k = 0; k * GRAN < nb; ++k) {
      const uint2 c = (*gran[o])[k];
      const int64_t h0 = off + k * GRAN, h1 = off + std::min<int64_t>(nb, (k + 1) * GRAN);
      if (h1 > g0 && g1 > g0 &&
          (int64_t)(fixed + chunk_bytes(fp32, mt, ms, h1 - g0, rays + c.x, slots + c.y)) > chunk) {
        st = flush(g0, g1, rays, slots);
        if (st != BEM_OK) break;
        g0 = h0;
        rays = slots = 0;
      }
      g1 = h1;
      rays += c.x;
      slots += c.y;
    }
    if (st != BEM_OK) break;
    off += blocks[o];
  }
  if (st == BEM_OK) st = flush(g0, g1, rays, slots);
  // the caller's stream goes on when the side stream is done
  if (forked) {
    STBEM_CUDA(cudaEventRecord(ev.e[2], side));
    STBEM_CUDA(cudaStreamWaitEvent(s, ev.e[2], 0));
  }
  return st;
}

}  // namespace stbem
