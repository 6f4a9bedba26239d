// Mesh geometry, outer points, the sparsity pattern pass, right-hand sides and
// look-ups of the light-cone-clipped single-layer Galerkin matrix. The matrix
// is cut into blocks (I, J) of panels over spatial triangle ("column") I
// times panels over column J; persistent grids pop blocks from a device
// counter. The quadrature itself is in stbem_stage.cu.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <vector>

#include "stbem_block.cuh"
#include "stbem_internal.h"

namespace stbem {

static double __longlong_as_double_host(long long b) {
  double d;
  std::memcpy(&d, &b, sizeof(d));
  return d;
}

bem_status upload_exp_table();

bem_status upload_gauss_tables() {
  std::vector<double> X(MAX_NTHETA * (MAX_NTHETA + 1) / 2), W(X.size());
  for (int n = 1; n <= MAX_NTHETA; ++n) {
    int off = n * (n - 1) / 2;
    for (int i = 0; i < n; ++i) {
      double z = std::cos(STBEM_PI * (i + 0.75) / (n + 0.5)), dp = 1.0;
      for (int it = 0; it < 100; ++it) {
        double p0 = 1.0, p1 = z;
        for (int k = 2; k <= n; ++k) {
          double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
          p0 = p1;
          p1 = p2;
        }
        if (n == 1) { p1 = z; p0 = 1.0; }
        dp = n * (z * p1 - p0) / (z * z - 1.0);
        double dz = p1 / dp;
        z -= dz;
        if (std::fabs(dz) < 1e-16) break;
      }
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= n; ++k) {
        double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      if (n == 1) { p1 = z; p0 = 1.0; }
      dp = n * (z * p1 - p0) / (z * z - 1.0);
      X[off + i] = z;
      W[off + i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
  }
  std::copy(X.begin(), X.end(), h_gl_x);
  std::copy(W.begin(), W.end(), h_gl_w);
  std::vector<float> Xf(X.begin(), X.end()), Wf(W.begin(), W.end());
  std::copy(Xf.begin(), Xf.end(), h_gl_xf);
  std::copy(Wf.begin(), Wf.end(), h_gl_wf);
  STBEM_CUDA(cudaMemcpyToSymbol(c_gl_x, X.data(), X.size() * sizeof(double)));
  STBEM_CUDA(cudaMemcpyToSymbol(c_gl_w, W.data(), W.size() * sizeof(double)));
  STBEM_CUDA(cudaMemcpyToSymbol(c_gl_xf, Xf.data(), Xf.size() * sizeof(float)));
  STBEM_CUDA(cudaMemcpyToSymbol(c_gl_wf, Wf.data(), Wf.size() * sizeof(float)));
  const bem_status st = upload_exp_table();
  return st != BEM_OK ? st : upload_gauss_stage(X.data(), W.data(), Xf.data(), Wf.data(), X.size());
}

// ---------------------------------------------------------------------------
// Staging: column frames, face gradients, panel balls, and their FP32 images
// (in the same kernels and one allocation: mesh creation is some launches long)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void col_f32(const ColGeom& G, ColF& F) {
  for (int k = 0; k < 3; ++k)
    for (int i = 0; i < 3; ++i) F.Xh[k][i] = (float)G.X[k][i];
  make_colr<float>(G, F.R);
  for (int i = 0; i < 3; ++i) F.ctr[i] = (float)G.ctr[i];
  F.rad = (float)G.rad;
}
__device__ __forceinline__ void panel_f32(const TetDev& D, int s0, PanelF& F) {
  for (int k = 0; k < 4; ++k) F.vt[k] = (float)D.vt[k];
  for (int k = 0; k < 5; ++k) F.ball[k] = (float)D.ball[k];
  F.tmin = (float)D.tmin;
  F.pmax = (float)D.pmax;
  F.lo = (uint8_t)(D.lo - s0);
  F.hi = (uint8_t)(D.hi - s0);
  F.dup = (uint8_t)D.dup;
  F.pad = 0;
}

__global__ void k_col_geom(int64_t n_col, const double* sv_xyz, const int32_t* corner_sv, ColGeom* out, ColF* outf) {
  int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= n_col) return;
  const int32_t* s = corner_sv + 3 * c;
  make_colgeom(sv_xyz + 3 * s[0], sv_xyz + 3 * s[1], sv_xyz + 3 * s[2], out[c]);
  col_f32(out[c], outf[c]);
}

// surf_p [n_surf][3] corner times; surf_col [n_surf]
__global__ void k_surf_geom(int64_t n_surf, const ColGeom* cols, const double* surf_p, const int32_t* surf_col,
                            SurfDev* out, FaceF* outf) {
  int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (s >= n_surf) return;
  SurfDev S;
  S.col = surf_col[s];
  S.pad = 0;
  for (int k = 0; k < 3; ++k) S.f.p[k] = surf_p[3 * s + k];
  face_gradient(cols[S.col], S.f);
  out[s] = S;
  make_facef(S.f, outf[s]);
}

// tet_vx [n_tet][4][4]: the panel's vertices (t,x,y,z) in the caller's order;
// the 4D ball is formed in that order with the fixed operation order of the
// sparsity contract: centre (((X0+X1)+X2)+X3)/4, radius max_v |X_v - c|.
__global__ void k_tet_ball(int64_t n_tet, const double* tet_vx, TetDev* tets, const int32_t* col_surf_begin, PanelF* outf) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n_tet) return;
  const double* X = tet_vx + 16 * i;
  double c[4];
  for (int d = 0; d < 4; ++d)
    c[d] = __ddiv_rn(__dadd_rn(__dadd_rn(__dadd_rn(X[d], X[4 + d]), X[8 + d]), X[12 + d]), 4.0);
  double mx = 0.0;
  for (int v = 0; v < 4; ++v) {
    double a = __dsub_rn(X[4 * v + 0], c[0]), b = __dsub_rn(X[4 * v + 1], c[1]);
    double e = __dsub_rn(X[4 * v + 2], c[2]), f = __dsub_rn(X[4 * v + 3], c[3]);
    double l = __dsqrt_rn(__dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(a, a), __dmul_rn(b, b)), __dmul_rn(e, e)),
                                    __dmul_rn(f, f)));
    if (l > mx) mx = l;
  }
  for (int d = 0; d < 4; ++d) tets[i].ball[d] = c[d];
  tets[i].ball[4] = mx;
  panel_f32(tets[i], col_surf_begin[tets[i].col], outf[i]);
}

bem_status mesh_device_geometry(bem_mesh* m, const double* d_sv_xyz, const int32_t* d_col_corner_sv,
                                const double* d_tet_vx, const int32_t* d_surf_col, const double* d_surf_p) {
  cudaStream_t s = m->ctx->stream;
  int th = 128;
  auto up = [](size_t n) { return (n + 255) / 256 * 256; };
  const size_t nc = up(sizeof(ColF) * m->n_col), nf = up(sizeof(FaceF) * m->n_surf), np = sizeof(PanelF) * m->n_tet;
  STBEM_CUDA(device_alloc(&m->d_images, nc + nf + np));
  m->d_colf = m->d_images;
  m->d_facef = static_cast<unsigned char*>(m->d_images) + nc;
  m->d_panf = static_cast<unsigned char*>(m->d_images) + nc + nf;
  k_col_geom<<<(unsigned)((m->n_col + th - 1) / th), th, 0, s>>>(m->n_col, d_sv_xyz, d_col_corner_sv, m->d_col,
                                                                 static_cast<ColF*>(m->d_colf));
  k_surf_geom<<<(unsigned)((m->n_surf + th - 1) / th), th, 0, s>>>(m->n_surf, m->d_col, d_surf_p, d_surf_col,
                                                                   m->d_surf, static_cast<FaceF*>(m->d_facef));
  k_tet_ball<<<(unsigned)((m->n_tet + th - 1) / th), th, 0, s>>>(m->n_tet, d_tet_vx, m->d_tet, m->d_col_surf_begin,
                                                                 static_cast<PanelF*>(m->d_panf));
  STBEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

// ---------------------------------------------------------------------------
// Outer points (Fig. int_tri_mid): canonical corner order (ascending spatial
// id) and x = (A + xi1 (B - A)) + xi2 (C - A) without fused operations.
// ---------------------------------------------------------------------------
__global__ void k_outer_points(int64_t n_surf, int mq, const ColGeom* cols, const SurfDev* surf, double* pts,
                               float* ptsf, double* trange) {
  int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (s >= n_surf) return;
  const SurfDev S = surf[s];
  const ColGeom& G = cols[S.col];
  double A[4] = {S.f.p[0], G.X[0][0], G.X[0][1], G.X[0][2]};
  double B[4] = {S.f.p[1], G.X[1][0], G.X[1][1], G.X[1][2]};
  double C[4] = {S.f.p[2], G.X[2][0], G.X[2][1], G.X[2][2]};
  int nq = mq * mq;
  double* out = pts + (int64_t)s * nq * 4;
  double tlo = 1e300, thi = -1e300;
  int n = 0;
  for (int pass = 0; pass < 2; ++pass) {
    double off = pass == 0 ? 1.0 / 3.0 : 2.0 / 3.0;
    for (int i = 0; i < mq; ++i)
      for (int j = 0; i + j <= mq - 1 - pass; ++j) {
        double x1 = __ddiv_rn(__dadd_rn((double)i, off), (double)mq);
        double x2 = __ddiv_rn(__dadd_rn((double)j, off), (double)mq);
        for (int d = 0; d < 4; ++d) {
          double p = __dadd_rn(A[d], __dmul_rn(x1, __dsub_rn(B[d], A[d])));
          out[4 * n + d] = __dadd_rn(p, __dmul_rn(x2, __dsub_rn(C[d], A[d])));
          ptsf[(int64_t)s * nq * 4 + 4 * n + d] = (float)out[4 * n + d];
        }
        tlo = fmin(tlo, out[4 * n]);
        thi = fmax(thi, out[4 * n]);
        ++n;
      }
  }
  trange[2 * s] = tlo;
  trange[2 * s + 1] = thi;
}

bem_status op_outer_points(bem_operator* op, cudaStream_t s) {
  const bem_mesh* m = op->mesh;
  int th = 128;
  k_outer_points<<<(unsigned)((m->n_surf + th - 1) / th), th, 0, s>>>(m->n_surf, op->mq, m->d_col, m->d_surf,
                                                                      op->d_pts, op->d_ptsf, op->d_pts_trange);
  STBEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

__device__ inline int64_t pop_block(unsigned long long* counter) {
  __shared__ unsigned long long s_b;
  if (threadIdx.x == 0) s_b = atomicAdd(counter, 1ull);
  __syncthreads();
  int64_t b = (int64_t)s_b;
  __syncthreads();
  return b;
}

// Pass 1: band width and pattern count of block (I, J), from the bits of its
// faces (block_bits). One row per thread, then one face per thread.
__device__ __forceinline__ void pattern_block(const BlockCtx& B, const BlockSm& C, const BlockPtr& P, int* s_w,
                                              unsigned long long* s_n) {
  const int words = bit_words(B.max_tet);
  const int64_t b = C.I * B.n_col + C.J;
  int wmax = 0;
  unsigned int cnt = 0;
  if (C.wmax > 0)
    for (int r = threadIdx.x; r < C.ntI; r += blockDim.x) {
      const PanelF& D = B.panf[C.tetI + r];
      const uint32_t* lo = P.bits + D.lo * words;
      const uint32_t* hi = P.bits + D.hi * words;
      int first = -1, last = -1;
      for (int w = 0; w < words; ++w) {
        const uint32_t m = lo[w] | hi[w];
        cnt += __popc(m);
        if (m) {
          if (first < 0) first = 32 * w + __ffs(m) - 1;
          last = 32 * w + 31 - __clz(m);
        }
      }
      if (first >= 0) wmax = max(wmax, last - first + 1);
    }
  wmax = __reduce_max_sync(0xffffffffu, wmax);
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if ((threadIdx.x & 31) == 0) { s_w[threadIdx.x >> 5] = wmax; s_n[threadIdx.x >> 5] = cnt; }
  __syncthreads();
  if (threadIdx.x == 0) {
    int w = 0;
    unsigned long long n = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) { w = max(w, s_w[i]); n += s_n[i]; }
    B.bw[b] = w;
    B.bnnz[b] = (int64_t)n;
  }
  if (B.gran && C.wmax > 0) {
    // apexes and potentials of the quadrature (k_apex)
    unsigned rays = 0, slots = 0;
    for (int f = threadIdx.x; f < C.nsI; f += blockDim.x) {
      int slo, n;
      bits_surfaces(P.bits + f * words, words, P.pan, slo, n);
      if (n) rays += B.nq;
      slots += n * B.nq;
    }
    rays = __reduce_add_sync(0xffffffffu, rays);
    slots = __reduce_add_sync(0xffffffffu, slots);
    if ((threadIdx.x & 31) == 0 && rays) {
      atomicAdd(&B.gran[b / GRAN].x, rays);
      atomicAdd(&B.gran[b / GRAN].y, slots);
    }
  }
  if (B.inner && C.wmax > 0) {
    // inner integrals of the block: every outer point of a test face against
    // every trial panel the face's pattern bits admit
    unsigned int m = 0;
    for (int k = threadIdx.x; k < C.nsI * words; k += blockDim.x) m += __popc(P.bits[k]);
    m = __reduce_add_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0 && m) atomicAdd(B.inner, (unsigned long long)m * (unsigned long long)B.nq);
  }
  __syncthreads();
}

// Bound by issue and latency (FP32 filter, shared memory): the level-3
// sphere with 8 slabs takes 18.6 ms (a warp per face: 125.9), the level-2 sphere
// with 32 slabs 6.8 ms (24.0).
// Work items are runs of kPatternRun test columns against one trial column,
// whose image is then loaded once; short runs on small meshes keep every SM
// busy. The grid takes the items of all operators of a batch (S > 1; the
// contexts share the largest column sizes, so the shared layout is uniform),
// prefix counting items; one operator comes as the kernel argument.
constexpr int kPatternThreads = 128;

__global__ void __launch_bounds__(kPatternThreads) k_pattern(const BlockCtx one, const BlockCtx* __restrict__ many,
                                                             const int64_t* __restrict__ prefix, int S, int run,
                                                             int64_t items, unsigned long long* counter) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ BlockSm C;
  __shared__ int s_w[kPatternThreads / 32];
  __shared__ unsigned long long s_n[kPatternThreads / 32];
  __shared__ BlockCtx B;
  __shared__ int s_seg;
  if (threadIdx.x == 0 && S <= 1) B = one;
  int cur = S > 1 ? -1 : 0;
  const BlockPtr P = block_ptr(smem, one.max_tet, one.max_surf, one.nq);
  for (;;) {
    int64_t g = pop_block(counter);
    if (g >= items) break;
    if (S > 1) {
      if (threadIdx.x == 0) s_seg = find_seg(prefix, S, g);
      __syncthreads();
      const int seg = s_seg;
      if (seg != cur && threadIdx.x == 0) B = many[seg];
      cur = seg;
      g -= prefix[seg];
      __syncthreads();
    }
    const int64_t I0 = g / B.n_col * run, J = g % B.n_col;
    load_trial(B, J, C, P.pan);
    for (int64_t I = I0; I < min(I0 + run, B.n_col); ++I) {
      load_test(B, I, C);
      block_bits(B, C, P);
      pattern_block(B, C, P, s_w, s_n);
    }
  }
}

// test columns per work item of the pattern pass
static int pattern_run(int64_t n_blocks) { return (int)std::max<int64_t>(1, std::min<int64_t>(8, n_blocks / 16384)); }

// The dynamic shared-memory limit of a kernel is state of the device shared by
// every host thread: operators of different sizes launching the same kernel
// concurrently (server slots) must never lower it under another's launch, so
// it only grows, under a lock.
bem_status ensure_smem_attr(const void* kern, size_t bytes) {
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, size_t> set_to;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lk(mu);
  size_t& cur = set_to[std::make_pair(dev, kern)];
  if (bytes <= cur) return BEM_OK;
  STBEM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  cur = bytes;
  return BEM_OK;
}

static int persistent_grid(const void* kern, size_t smem, int threads) {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, smem);
  if (per < 1) per = 1;
  return sms * per;
}

static BlockCtx make_ctx(const bem_operator* op) {
  const bem_mesh* m = op->mesh;
  BlockCtx B;
  B.n_col = m->n_col;
  B.mq = op->mq; B.nq = op->nq; B.n_theta = op->n_theta; B.prec = op->opts.precision;
  B.rule = make_rule(op->opts.precision, op->n_theta);
  B.S = m->coord_scale;
  B.margin = (float)(1.6e-5 * m->coord_scale);  // > 4x the FP32 error bound of C2 and C3
  B.cols = m->d_col; B.colf = static_cast<const ColF*>(m->d_colf); B.panf = static_cast<const PanelF*>(m->d_panf);
  B.facef = static_cast<const FaceF*>(m->d_facef);
  B.col_tet_begin = m->d_col_tet_begin; B.col_surf_begin = m->d_col_surf_begin;
  B.surf = m->d_surf; B.tets = m->d_tet; B.pts = op->d_pts; B.ptsf = reinterpret_cast<const float4*>(op->d_ptsf);
  B.trange = op->d_pts_trange;
  B.bw = op->d_bw; B.bnnz = op->d_bnnz; B.boff = op->d_boff; B.rsoff = op->d_rsoff; B.rs = op->d_rs;
  B.val = op->d_val; B.val32 = op->d_val32;
  B.max_surf = m->max_col_surf; B.max_tet = m->max_col_tets;
  B.counter = nullptr;
  B.inner = nullptr;
  B.gran = op->d_gran;
  B.mf_x = nullptr; B.mf_y = nullptr; B.mf_nrhs = 0; B.mf_ld = m->n_tet;
  return B;
}

static bem_status get_counter(const bem_operator* op, unsigned long long** out, cudaStream_t s) {
  STBEM_CUDA(cudaMemsetAsync(op->d_counter, 0, sizeof(unsigned long long), s));
  *out = op->d_counter;
  return BEM_OK;
}

static bem_status launch_pattern(const BlockCtx& one, const BlockCtx* many, const int64_t* prefix, int S, int run,
                                 int64_t items, unsigned long long* counter, cudaStream_t s) {
  const size_t smem = bits_smem(one.max_tet, one.max_surf, one.nq);
  const bem_status st = ensure_smem_attr((const void*)k_pattern, smem);
  if (st != BEM_OK) return st;
  const int64_t grid = std::min<int64_t>(persistent_grid((const void*)k_pattern, smem, kPatternThreads), items);
  k_pattern<<<(unsigned)grid, kPatternThreads, smem, s>>>(one, many, prefix, S, run, items, counter);
  STBEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

bem_status op_pattern(bem_operator* op, cudaStream_t s) {
  BlockCtx B = make_ctx(op);
  bem_status st = get_counter(op, &B.counter, s);
  if (st != BEM_OK) return st;
  STBEM_CUDA(cudaMemsetAsync(op->d_counter + 1, 0, sizeof(unsigned long long), s));
  B.inner = op->d_counter + 1;
  STBEM_CUDA(cudaMemsetAsync(op->d_gran, 0, sizeof(uint2) * op->n_gran(), s));
  const int64_t nc = op->mesh->n_col;
  const int run = pattern_run(nc * nc);
  return launch_pattern(B, nullptr, nullptr, 1, run, nc * ((nc + run - 1) / run), B.counter, s);
}

int quad_max_per_sm(const bem_operator* op) {
  return stage_apex_per_sm(op->opts.precision == BEM_PREC_MIXED, op->mesh->max_col_tets, op->mesh->max_col_surf, op->nq);
}

void quad_scratch(const bem_operator* op, int64_t* least, int64_t* wanted) {
  stage_scratch(op->opts.precision == BEM_PREC_MIXED, op->mesh->max_col_tets, op->mesh->max_col_surf,
                (int)op->ctx->sm_count, {&op->h_gran}, least, wanted);
}

bem_status quad_launch(const bem_operator* op, int per_sm, int64_t end, const double* mf_x, double* mf_y, int nrhs,
                       void* scratch, int64_t bytes, cudaStream_t side, cudaStream_t s) {
  BlockCtx B = make_ctx(op);
  const int64_t nb = op->mesh->n_col * op->mesh->n_col;
  B.mf_x = mf_x;
  B.mf_y = mf_y;
  B.mf_nrhs = nrhs;
  return stage_run(B, nullptr, nullptr, 1, op->opts.precision == BEM_PREC_MIXED, (int)op->ctx->sm_count,
                   {&op->h_gran}, {nb}, std::min(end, nb), scratch, bytes, per_sm, side, s);
}

// takes the context's second stream and, with `memory`, its scratch (true if there is that
// much), unless they are held, or in use by unfinished work of another stream
bool ScratchHold::claim(Scratch& c, bool memory, int64_t wanted) {
  // queries and allocations here concern no stream under capture, so another thread's
  // capture (global mode) is none of their business
  struct Relaxed {
    cudaStreamCaptureMode m = cudaStreamCaptureModeRelaxed;
    Relaxed() { cudaThreadExchangeStreamCaptureMode(&m); }
    ~Relaxed() { cudaThreadExchangeStreamCaptureMode(&m); }
  } relaxed;
  std::lock_guard<std::mutex> lk(c.mu);
  if (c.busy) return false;
  if (!c.done && cudaEventCreateWithFlags(&c.done, cudaEventDisableTiming) != cudaSuccess) {
    cudaGetLastError();
    c.done = nullptr;
    return false;
  }
  if (c.last != s && cudaEventQuery(c.done) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  c.busy = true;
  from = &c;
  side = c.side;
  if (!memory) return false;
  if (c.bytes < wanted) {
    cudaFree(c.p);   // (waits for the work on it)
    c.p = nullptr;
    c.bytes = 0;
    if (cudaMalloc(&c.p, wanted) == cudaSuccess) {
      c.bytes = wanted;
    } else {
      cudaGetLastError();
      c.p = nullptr;
    }
  }
  if (!c.p || cudaStreamWaitEvent(s, c.done, 0) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  p = c.p;
  bytes = c.bytes;
  return true;
}

bool ScratchHold::take_idle(Scratch& c, int64_t wanted, cudaStream_t stream) {
  s = stream;
  if (claim(c, true, wanted)) return true;
  release();
  return false;
}

bem_status ScratchHold::take(Scratch& c, bool own_block, int64_t least, int64_t wanted, cudaStream_t stream) {
  s = stream;
  if (claim(c, !own_block, wanted)) return BEM_OK;
  own = true;
  for (int64_t n = wanted;; n = std::max(least, n / 4)) {
    if (device_alloc_async(&p, n, s) == cudaSuccess) {
      bytes = n;
      return BEM_OK;
    }
    cudaGetLastError();
    p = nullptr;
    if (n <= least) break;
  }
  set_error("out of device memory (quadrature scratch)");
  return BEM_ERR_OUT_OF_MEMORY;
}

void ScratchHold::release() {
  if (own && p) cudaFreeAsync(p, s);
  if (from) {
    std::lock_guard<std::mutex> lk(from->mu);
    cudaEventRecord(from->done, s);
    from->last = s;
    from->busy = false;
  }
  from = nullptr;
  p = nullptr;
  side = nullptr;
}

void scratch_trim(Scratch& c) {
  std::lock_guard<std::mutex> lk(c.mu);
  if (c.busy) return;
  cudaFree(c.p);
  c.p = nullptr;
  c.bytes = 0;
}

namespace {
std::mutex g_contexts_mu;
std::vector<bem_context*> g_contexts;

// gives back the idle scratch of the current device's contexts; false: there was none
bool trim_idle() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  bool some = false;
  std::lock_guard<std::mutex> lk(g_contexts_mu);
  for (bem_context* c : g_contexts) {
    if (c->device != dev) continue;
    {
      std::lock_guard<std::mutex> l2(c->scratch.mu);
      some = some || (c->scratch.p && !c->scratch.busy);
    }
    scratch_trim(c->scratch);
  }
  return some;
}

template <typename F>
cudaError_t with_room(F alloc) {
  cudaError_t e = alloc();
  if (e == cudaSuccess) return e;
  cudaGetLastError();   // (a later launch's check must not see it)
  if (e != cudaErrorMemoryAllocation || !trim_idle()) return e;
  e = alloc();
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}
}  // namespace

void contexts_add(bem_context* c) {
  std::lock_guard<std::mutex> lk(g_contexts_mu);
  g_contexts.push_back(c);
}
void contexts_remove(bem_context* c) {
  std::lock_guard<std::mutex> lk(g_contexts_mu);
  g_contexts.erase(std::remove(g_contexts.begin(), g_contexts.end(), c), g_contexts.end());
}
cudaError_t device_alloc(void** p, size_t bytes) {
  return with_room([&] { return cudaMalloc(p, bytes); });
}
cudaError_t device_alloc_async(void** p, size_t bytes, cudaStream_t s) {
  return with_room([&] { return cudaMallocAsync(p, bytes, s); });
}

bem_status op_quadrature(bem_operator* op, cudaStream_t s) {
  int64_t least = 0, wanted = 0;
  quad_scratch(op, &least, &wanted);
  const bool capped = op->scratch_cap >= 0;
  if (capped) wanted = std::max(least, std::min(wanted, op->reserve_bytes + op->scratch_cap));
  ScratchHold h;
  bem_status st = h.take(op->ctx->scratch, capped, least, wanted, s);
  if (st != BEM_OK) return st;
  st = choose_quad_shape(op, h.p, h.bytes, h.side, s);
  if (st != BEM_OK) return st;
  return quad_launch(op, op->quad_per_sm, op->mesh->n_col * op->mesh->n_col, nullptr, nullptr, 0, h.p, h.bytes, h.side, s);
}

FreeScratch::FreeScratch(const bem_operator* o, cudaStream_t s) {
  if (!o->opts.matrix_free || o->held) return;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return;
  }
  int64_t least = 0, wanted = 0;
  quad_scratch(o, &least, &wanted);
  if (wanted <= o->tmp_bytes || !h.take_idle(o->ctx->scratch, wanted, s)) return;
  op = o;
  op->held = &h;
}

// Matrix-free product y = A x (internal order, [nrhs][n_tet]): the quadrature
// pass with the entries summed against x instead of stored. An operator's own
// scratch (op_layout) is for captured products and calls beside another holder of
// the context's: level-3 sphere, 8 slabs 149 ms with the context's 1 GiB, 806
// with its own 87 MB; level-2 sphere, 15 slabs 33 ms and 144 with 64 MiB.
bem_status op_matvec_free(const bem_operator* op, const double* x, double* y, int nrhs, cudaStream_t s) {
  STBEM_CUDA(cudaMemsetAsync(y, 0, sizeof(double) * op->mesh->n_tet * nrhs, s));
  const int per_sm = op->quad_per_sm > 0 ? op->quad_per_sm : quad_max_per_sm(op);
  const int64_t nb = op->mesh->n_col * op->mesh->n_col;
  if (op->held) return quad_launch(op, per_sm, nb, x, y, nrhs, op->held->p, op->held->bytes, op->held->side, s);
  return quad_launch(op, per_sm, nb, x, y, nrhs, op->d_tmp, op->tmp_bytes, op->side, s);
}

// ---------------------------------------------------------------------------
// Batched passes over the blocks of several operators. All contexts take the
// largest column sizes of the batch, so the shared memory layout is the same
// for every block, and the quadrature scratch is shared.
// ---------------------------------------------------------------------------
bem_status op_outer_points_all(const std::vector<bem_operator*>& ops, cudaStream_t s) {
  for (bem_operator* op : ops) {
    bem_status st = op_outer_points(op, s);
    if (st != BEM_OK) return st;
  }
  return BEM_OK;
}

static void batch_dims(const std::vector<bem_operator*>& ops, int& max_tet, int& max_surf) {
  max_tet = 1;
  max_surf = 1;
  for (const bem_operator* op : ops) {
    max_tet = std::max(max_tet, op->mesh->max_col_tets);
    max_surf = std::max(max_surf, op->mesh->max_col_surf);
  }
}

// run > 0: the prefix counts the pattern pass's work items, else blocks
static bem_status upload_batch(const std::vector<bem_operator*>& ops, BatchDev& dev, int max_tet, int max_surf,
                               int run, int64_t* total, BlockCtx* first, cudaStream_t s) {
  const int S = (int)ops.size();
  std::vector<BlockCtx> ctx(S);
  std::vector<int64_t> prefix(S + 1, 0);
  for (int i = 0; i < S; ++i) {
    ctx[i] = make_ctx(ops[i]);
    ctx[i].max_tet = max_tet;
    ctx[i].max_surf = max_surf;
    ctx[i].counter = dev.d_counter;
    const int64_t nc = ops[i]->mesh->n_col;
    prefix[i + 1] = prefix[i] + nc * (run > 0 ? (nc + run - 1) / run : nc);
  }
  *total = prefix[S];
  *first = ctx[0];
  STBEM_CUDA(cudaMemcpyAsync(dev.d_ctx, ctx.data(), sizeof(BlockCtx) * S, cudaMemcpyHostToDevice, s));
  STBEM_CUDA(cudaMemcpyAsync(dev.d_prefix, prefix.data(), sizeof(int64_t) * (S + 1), cudaMemcpyHostToDevice, s));
  STBEM_CUDA(cudaMemsetAsync(dev.d_counter, 0, sizeof(unsigned long long), s));
  STBEM_CUDA(cudaStreamSynchronize(s));   // the host arrays above go out of scope
  return BEM_OK;
}

bem_status op_pattern_batch(const std::vector<bem_operator*>& ops, BatchDev& dev, cudaStream_t s) {
  if (ops.empty()) return BEM_OK;
  int mt, ms;
  batch_dims(ops, mt, ms);
  int64_t blocks = 0, items = 0;
  for (const bem_operator* op : ops) blocks += op->mesh->n_col * op->mesh->n_col;
  const int run = pattern_run(blocks);
  BlockCtx first;
  for (bem_operator* op : ops) STBEM_CUDA(cudaMemsetAsync(op->d_gran, 0, sizeof(uint2) * op->n_gran(), s));
  bem_status st = upload_batch(ops, dev, mt, ms, run, &items, &first, s);
  if (st != BEM_OK) return st;
  return launch_pattern(first, static_cast<const BlockCtx*>(dev.d_ctx), dev.d_prefix, (int)ops.size(), run, items,
                        dev.d_counter, s);
}

static void batch_grans(const std::vector<bem_operator*>& ops, std::vector<const std::vector<uint2>*>& gran,
                        std::vector<int64_t>& blocks) {
  for (const bem_operator* op : ops) {
    gran.push_back(&op->h_gran);
    blocks.push_back(op->mesh->n_col * op->mesh->n_col);
  }
}

bem_status op_quadrature_batch(const std::vector<bem_operator*>& ops, BatchDev& dev, cudaStream_t s) {
  if (ops.empty()) return BEM_OK;
  for (const bem_operator* op : ops)
    if (op->opts.precision != ops[0]->opts.precision || op->nq != ops[0]->nq || op->n_theta != ops[0]->n_theta) {
      set_error("a batch takes one precision, m_Q and n_theta");
      return BEM_ERR_INVALID_ARG;
    }
  int mt, ms;
  batch_dims(ops, mt, ms);
  int64_t total = 0;
  BlockCtx first;
  bem_status st = upload_batch(ops, dev, mt, ms, 0, &total, &first, s);
  if (st != BEM_OK) return st;
  const bool fp32 = ops[0]->opts.precision == BEM_PREC_MIXED;
  const int sms = (int)ops[0]->ctx->sm_count;
  const int occ = stage_apex_per_sm(fp32, mt, ms, ops[0]->nq);
  std::vector<const std::vector<uint2>*> gran;
  std::vector<int64_t> blocks;
  batch_grans(ops, gran, blocks);
  int64_t least = 0, wanted = 0;
  stage_scratch(fp32, mt, ms, sms, gran, &least, &wanted);
  ScratchHold h;
  st = h.take(ops[0]->ctx->scratch, false, least, wanted, s);
  if (st != BEM_OK) return st;
  auto launch = [&](int per, int64_t end) {
    return stage_run(first, static_cast<const BlockCtx*>(dev.d_ctx), dev.d_prefix, (int)ops.size(), fp32, sms, gran,
                     blocks, end, h.p, h.bytes, per, h.side, s);
  };
  int per = occ, how = 0;
  if (ops[0]->ctx->tune_mode) {
    // the batch's own shape class; sample: 1/32 of the block queue
    const std::string key = batch_shape_class(ops[0]->ctx, ops[0]->opts.precision, ops[0]->nq, ops[0]->n_theta, mt,
                                              ms, (int64_t)ops.size(), total);
    std::vector<int> codes;
    for (int p = std::max(1, occ - 2); p <= occ; ++p) codes.push_back(p);
    st = tune_launch_shape(ops[0]->ctx, key, codes, std::max<int64_t>(total / 32, 1), launch, s, &per, &how, nullptr);
    if (st != BEM_OK) return st;
  }
  return launch(per, total);
}

size_t block_ctx_size() { return sizeof(BlockCtx); }

// ---------------------------------------------------------------------------
// Value scan: non-finite count and largest magnitude
// ---------------------------------------------------------------------------
template <typename V>
__global__ void k_value_scan(const V* v, int64_t n, unsigned long long* bad, unsigned long long* maxbits) {
  unsigned long long nb = 0;
  double mx = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double x = (double)v[i];
    if (!isfinite(x)) ++nb;
    else mx = fmax(mx, fabs(x));
  }
  for (int o = 16; o > 0; o >>= 1) {
    nb += __shfl_xor_sync(0xffffffffu, nb, o);
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if ((threadIdx.x & 31) == 0) {
    if (nb) atomicAdd(bad, nb);
    atomicMax(maxbits, (unsigned long long)__double_as_longlong(mx));  // non-negative doubles order as integers
  }
}

bem_status op_value_scan(const bem_operator* op, int64_t* nbad, double* maxabs, cudaStream_t s) {
  unsigned long long* d;
  STBEM_CUDA(device_alloc((void**)&d, 2 * sizeof(unsigned long long)));
  STBEM_CUDA(cudaMemsetAsync(d, 0, 2 * sizeof(unsigned long long), s));
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (op->nstored > 0) {
    if (op->d_val) k_value_scan<double><<<sms * 8, 256, 0, s>>>(op->d_val, op->nstored, d, d + 1);
    else k_value_scan<float><<<sms * 8, 256, 0, s>>>(op->d_val32, op->nstored, d, d + 1);
  }
  unsigned long long h[2];
  cudaError_t e = cudaMemcpyAsync(h, d, sizeof(h), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(d);
  if (e != cudaSuccess) { set_error(cudaGetErrorString(e)); return BEM_ERR_CUDA; }
  *nbad = (int64_t)h[0];
  long long bits = (long long)h[1];
  *maxabs = __longlong_as_double_host(bits);
  return BEM_OK;
}

// ---------------------------------------------------------------------------
// Entry lookup (internal indices) and pattern CSR export
// ---------------------------------------------------------------------------
__global__ void k_entries(int64_t n, const int32_t* ij, const float* val32, const TetDev* tets, int64_t n_col,
                          const int32_t* col_tet_begin, const int32_t* bw, const int64_t* boff, const int64_t* rsoff,
                          const int32_t* rs, const double* val, double* out) {
  int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= n) return;
  int i = ij[2 * k], j = ij[2 * k + 1];
  int I = tets[i].col, J = tets[j].col;
  int64_t b = (int64_t)I * n_col + J;
  int W = bw[b];
  double v = 0.0;
  if (W > 0) {
    int r = i - col_tet_begin[I];
    int nt = col_tet_begin[I + 1] - col_tet_begin[I];
    int start = rs[rsoff[b] + r];
    int w = j - start;
    if (w >= 0 && w < W) v = val ? val[boff[b] + (int64_t)w * nt + r] : (double)val32[boff[b] + (int64_t)w * nt + r];
  }
  out[k] = v;
}

bem_status op_entries(const bem_operator* op, int64_t n, const int32_t* d_ij, double* d_out, cudaStream_t s) {
  const bem_mesh* m = op->mesh;
  if (n == 0) return BEM_OK;
  k_entries<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, d_ij, op->d_val32, m->d_tet, m->n_col, m->d_col_tet_begin,
                                                       op->d_bw, op->d_boff, op->d_rsoff, op->d_rs, op->d_val, d_out);
  STBEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

// Pattern rows (internal numbering): count pass, then fill pass (columns are
// written in internal order; the caller permutes and sorts).
__global__ void __launch_bounds__(kPatternThreads) k_pattern_rows(BlockCtx B, int64_t* rowcount, const int64_t* rowptr,
                                                                  int32_t* cols, int fill, int64_t I_only) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ BlockSm C;
  const BlockPtr P = block_ptr(smem, B.max_tet, B.max_surf, B.nq);
  const uint32_t* bits = P.bits;
  const int words = bit_words(B.max_tet);
  const int64_t nblk = I_only >= 0 ? B.n_col : B.n_col * B.n_col;
  for (;;) {
    int64_t b = pop_block(B.counter);
    if (b >= nblk) break;
    if (I_only >= 0) b += I_only * B.n_col;
    if (B.bw[b] == 0) continue;
    load_trial(B, b % B.n_col, C, P.pan);
    load_test(B, b / B.n_col, C);
    block_bits(B, C, P);
    const int t0 = C.tetI, nt = C.ntI, s0 = C.surfI;
    for (int r = threadIdx.x; r < nt; r += blockDim.x) {
      const TetDev& D = B.tets[t0 + r];
      int lo = D.lo - s0, hi = D.hi - s0;
      int cnt = 0;
      for (int w = 0; w < words; ++w) cnt += __popc(bits[lo * words + w] | bits[hi * words + w]);
      if (!cnt) continue;
      unsigned long long pos = atomicAdd((unsigned long long*)&rowcount[t0 + r], (unsigned long long)cnt);
      if (fill) {
        for (int w = 0; w < words; ++w) {
          uint32_t m = bits[lo * words + w] | bits[hi * words + w];
          while (m) {
            int l = __ffs(m) - 1;
            m &= m - 1;
            cols[rowptr[t0 + r] + (int64_t)pos++] = C.tetJ + 32 * w + l;
          }
        }
      }
    }
    __syncthreads();
  }
}

bem_status op_pattern_csr(const bem_operator* op, int64_t* d_rowcount, int64_t* d_rowptr, int32_t* d_cols, bool fill,
                          cudaStream_t s, int64_t I_only) {
  BlockCtx B = make_ctx(op);
  bem_status st = get_counter(op, &B.counter, s);
  if (st != BEM_OK) return st;
  const size_t smem = bits_smem(B.max_tet, B.max_surf, B.nq);
  {
    bem_status sa = ensure_smem_attr((const void*)k_pattern_rows, smem);
    if (sa != BEM_OK) return sa;
  }
  int grid = persistent_grid((const void*)k_pattern_rows, smem, kPatternThreads);
  k_pattern_rows<<<grid, kPatternThreads, smem, s>>>(B, d_rowcount, d_rowptr, d_cols, fill ? 1 : 0, I_only);
  STBEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

// ---------------------------------------------------------------------------
// Right-hand side: b_i = int_K [g(P_lo(y), y) - g(P_hi(y), y)] dA
// (= -sum_F nu_{F,t} int_F g dS, eq. int_bform with A = Id) = S_lo - S_hi, S_F
// the integral of the data over face F's graph. K is split into 4^k congruent
// sub-triangles, k chosen so that a sub-triangle spans at most half the
// data's length scale (pulse width, or 0.5 for the sin^2 data), and each gets
// a Duffy-collapsed 8 x 8 Gauss-Legendre rule.
// ---------------------------------------------------------------------------

// exp(z), z <= 0, by the table-driven method of P. T. P. Tang (ACM TOMS 15,
// 1989): z = (128 n + j) ln 2 / 128 + r, exp(z) = 2^n 2^(j/128) (1 + p(r)) with
// the Taylor polynomial of degree 5 (|r| <= 0.0028: r^6 / 720 < 1e-18), about
// an ulp. Eleven FP64 instructions where the general function takes some
// twenty, and the FP64 pipe is what the right-hand side is bound by. Below
// -708 (denormal results) and for NaN the general function answers.
__device__ __forceinline__ double exp_neg(double z, const double* __restrict__ tab) {
  if (!(z > -708.0)) return exp(z);
  const double magic = 6755399441055744.0;   // 1.5 * 2^52: the sum's low bits are the rounded integer
  const double kd = __fma_rn(z, 128.0 / 0.693147180559945309417, magic);
  const int k = __double2loint(kd);
  const double kf = __dsub_rn(kd, magic);
  // ln 2 / 128 in two parts, the first with 32 trailing zero bits
  double r = __fma_rn(kf, -0x1.62e42feep-8, z);
  r = __fma_rn(kf, -0x1.a39ef35793c76p-40, r);
  double p = __fma_rn(r, 1.0 / 120.0, 1.0 / 24.0);
  p = __fma_rn(p, r, 1.0 / 6.0);
  p = __fma_rn(p, r, 0.5);
  p = __fma_rn(r * r, p, r);
  const double t = tab[k & 127];
  const double v = __fma_rn(t, p, t);
  return __hiloint2double(__double2hiint(v) + ((k >> 7) << 20), __double2loint(v));
}

__device__ __constant__ double c_exp2_tab[128];   // 2^(j/128)

bem_status upload_exp_table() {
  double t[128];
  for (int j = 0; j < 128; ++j) t[j] = std::exp2(j / 128.0);
  STBEM_CUDA(cudaMemcpyToSymbol(c_exp2_tab, t, sizeof(t)));
  return BEM_OK;
}

constexpr int kRhsThreads = 128;

// S[r][F] by a warp per (face, right-hand side): the 64 nodes of a
// sub-triangle on the lanes, two each, and a loop over the sub-triangles. The
// data's argument (t - <y, d> - c) / w, and t, are linear on K: a node costs
// two FMAs, and S_F serves the panel below and the panel above (a thread per
// panel formed both its faces at every node from coordinates and left a mesh
// of 1,920 panels to 15 CTAs). FP64-bound: 64
// pulses on 30,720 panels 444 -> 72 ms (2.0e9 nodes of 15 FP64 instructions: 58 ms).
template <int KIND>
__global__ void __launch_bounds__(kRhsThreads) k_rhs_faces(int64_t n_surf, const SurfDev* __restrict__ surf,
                                                           const ColGeom* __restrict__ cols, int nrhs,
                                                           const double* __restrict__ params, double2* __restrict__ S) {
  __shared__ double tab[128];
  for (int k = threadIdx.x; k < 128; k += kRhsThreads) tab[k] = c_exp2_tab[k];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  // this lane's nodes: (a, c) = (lane / 8, lane % 8) and (lane / 8 + 4, lane % 8)
  const double* X = gl_x() + 8 * 7 / 2;
  const double* Wt = gl_w() + 8 * 7 / 2;
  double m1[2], m2[2], wn[2];
  const double v = 0.5 * (X[lane & 7] + 1.0), wv = 0.5 * Wt[lane & 7];
  for (int h = 0; h < 2; ++h) {
    const double u = 0.5 * (X[(lane >> 3) + 4 * h] + 1.0), wu = 0.5 * Wt[(lane >> 3) + 4 * h];
    m1[h] = u * (1.0 - v);
    m2[h] = u * v;           // Duffy: Jacobian 2 |sub| u
    wn[h] = wu * wv * u;
  }
  const int64_t n = n_surf * nrhs, step = (int64_t)gridDim.x * (kRhsThreads / 32);
  for (int64_t it = (int64_t)blockIdx.x * (kRhsThreads / 32) + (threadIdx.x >> 5); it < n; it += step) {
    const int64_t r = it / n_surf, f = it - r * n_surf;
    const SurfDev& F = surf[f];
    const ColGeom& G = cols[F.col];
    const double* prm = KIND == BEM_DATA_PULSE ? params + 5 * r : nullptr;
    double a[3];   // the argument at the corners
    for (int k = 0; k < 3; ++k) {
      a[k] = F.f.p[k];   // (fused: a corner's rounding is common to all nodes of the face)
      if (KIND == BEM_DATA_PULSE)
        a[k] = __fma_rn(-G.X[k][0], prm[0], __fma_rn(-G.X[k][1], prm[1], __fma_rn(-G.X[k][2], prm[2], a[k] - prm[3]))) / prm[4];
    }
    const double scale = KIND == BEM_DATA_PULSE ? 0.5 * prm[4] : 0.5;
    int lev = 0;
    while (lev < 4 && G.diam / (double)(1 << lev) > scale) ++lev;
    const int m = 1 << lev;
    const double e1 = (a[1] - a[0]) / m, e2 = (a[2] - a[0]) / m;
    double acc = 0.0;
    auto add = [&](double base, double d1, double d2) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const double x = base + m1[h] * d1 + m2[h] * d2;
        double g;
        if (KIND == BEM_DATA_PULSE) {
          g = exp_neg(-x * x, tab);
        } else {
          g = 0.0;
          if (x > 0.0 && x < 2.0) {
            const double sn = sin(0.5 * STBEM_PI * x);
            g = sn * sn;
          }
        }
        acc += wn[h] * g;
      }
    };
    for (int p = 0; p < m; ++p)
      for (int q = 0; p + q < m; ++q) {
        add(a[0] + p * e1 + q * e2, e1, e2);
        if (p + q + 2 <= m) add(a[0] + (p + 1) * e1 + q * e2, e2, e2 - e1);
      }
    // the sum and its rounding error (Knuth's two-sum): b is a small difference of two S
    double lost = 0.0;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const double x = __shfl_xor_sync(0xffffffffu, acc, o);
      lost += __shfl_xor_sync(0xffffffffu, lost, o);
      const double t = __dadd_rn(acc, x), z = __dsub_rn(t, acc);
      lost += __dadd_rn(__dsub_rn(acc, __dsub_rn(t, z)), __dsub_rn(x, z));
      acc = t;
    }
    // each sub-triangle has area |K| / m^2; Duffy Jacobian 2 |sub| u
    if (lane == 0) {
      const double sc = 2.0 * G.area / ((double)m * m), h = __dmul_rn(sc, acc);
      S[it] = make_double2(h, __fma_rn(sc, acc, -h) + sc * lost);
    }
  }
}

// b[r][i] = S[r][lo(i)] - S[r][hi(i)] (internal panel order)
__global__ void k_rhs_panels(int64_t n_tet, int64_t n_surf, int nrhs, const TetDev* tets, const double2* S, double* b) {
  int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (tid >= n_tet * nrhs) return;
  const int64_t r = tid / n_tet, i = tid - r * n_tet;
  const TetDev& D = tets[i];
  const double2 lo = S[r * n_surf + D.lo], hi = S[r * n_surf + D.hi];
  b[tid] = (lo.x - hi.x) + (lo.y - hi.y);
}

// Points and weights of the right-hand side rule for arbitrary data: per
// surface (a face tau = P(y) over K), K split into 4^level congruent
// triangles in the order of k_rhs_faces (row p, then q; upright, then inverted),
// each with a Duffy-collapsed ng x ng Gauss-Legendre rule. One thread per
// (surface, sub-triangle); pts may be null (weights only).
__global__ void k_rhs_points(int64_t n_surf, const SurfDev* surf, const ColGeom* cols, int level, int ng,
                             double* pts, double* wts) {
  const int m = 1 << level, nsub = m * m;
  int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (tid >= n_surf * nsub) return;
  const int64_t sidx = tid / nsub;
  const int k = (int)(tid - sidx * nsub);
  // sub-triangle k -> corners (barycentric)
  double a0[3], a1[3], a2[3];
  int cnt = 0;
  bool found = false;
  for (int p = 0; p < m && !found; ++p)
    for (int q = 0; p + q < m && !found; ++q) {
      double u0[3] = {1.0 - (double)(p + q) / m, (double)p / m, (double)q / m};
      double u1[3] = {1.0 - (double)(p + q + 1) / m, (double)(p + 1) / m, (double)q / m};
      double u2[3] = {1.0 - (double)(p + q + 1) / m, (double)p / m, (double)(q + 1) / m};
      if (cnt++ == k) {
        for (int c = 0; c < 3; ++c) { a0[c] = u0[c]; a1[c] = u1[c]; a2[c] = u2[c]; }
        found = true;
      } else if (p + q + 2 <= m) {
        if (cnt++ == k) {
          double v0[3] = {1.0 - (double)(p + q + 2) / m, (double)(p + 1) / m, (double)(q + 1) / m};
          for (int c = 0; c < 3; ++c) { a0[c] = u1[c]; a1[c] = v0[c]; a2[c] = u2[c]; }
          found = true;
        }
      }
    }
  const SurfDev S = surf[sidx];
  const ColGeom& G = cols[S.col];
  const double* X = gl_x() + ng * (ng - 1) / 2;
  const double* Wt = gl_w() + ng * (ng - 1) / 2;
  const double jac = 2.0 * G.area / (double)nsub;   // Duffy: 2 |sub| u
  int64_t o = (sidx * nsub + k) * (int64_t)ng * ng;
  for (int a = 0; a < ng; ++a) {
    const double u = 0.5 * (X[a] + 1.0), wu = 0.5 * Wt[a];
    for (int c = 0; c < ng; ++c, ++o) {
      const double v = 0.5 * (X[c] + 1.0), wv = 0.5 * Wt[c];
      const double m0 = 1.0 - u, m1 = u * (1.0 - v), m2 = u * v;
      double l[3];
      for (int e = 0; e < 3; ++e) l[e] = m0 * a0[e] + m1 * a1[e] + m2 * a2[e];
      wts[o] = jac * wu * wv * u;
      if (pts) {
        pts[4 * o] = l[0] * S.f.p[0] + l[1] * S.f.p[1] + l[2] * S.f.p[2];
        for (int e = 0; e < 3; ++e) pts[4 * o + 1 + e] = l[0] * G.X[0][e] + l[1] * G.X[1][e] + l[2] * G.X[2][e];
      }
    }
  }
}

// S[r][s] = sum_q w_q g[r][s * npps + q] in ascending q (one thread per (r, s))
__global__ void k_rhs_face_sums(int64_t n_surf, int64_t npps, int nrhs, const double* wts, const double* g,
                                double* S) {
  int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (tid >= n_surf * nrhs) return;
  const int64_t r = tid / n_surf, sidx = tid - r * n_surf;
  const double* gw = g + r * n_surf * npps + sidx * npps;
  const double* ww = wts + sidx * npps;
  double acc = 0.0;
  for (int64_t q = 0; q < npps; ++q) acc += ww[q] * gw[q];
  S[tid] = acc;
}

// b[r][i] = S[r][lo(i)] - S[r][hi(i)] (internal panel order)
__global__ void k_rhs_combine(int64_t n_tet, int64_t n_surf, int nrhs, const TetDev* tets, const double* S, double* b) {
  int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (tid >= n_tet * nrhs) return;
  const int64_t r = tid / n_tet, i = tid - r * n_tet;
  const TetDev& D = tets[i];
  b[tid] = S[r * n_surf + D.lo] - S[r * n_surf + D.hi];
}

// The face integrals of as many right-hand sides as 64 MiB hold at a time: the
// workspace stays small beside b, and four million (face, right-hand side) pairs
// fill the device many times over.
bem_status op_rhs(const bem_operator* op, int kind, int nrhs, const double* d_params, double* d_b, cudaStream_t s) {
  const bem_mesh* m = op->mesh;
  const int64_t room = ((int64_t)64 << 20) / (sizeof(double2) * std::max<int64_t>(m->n_surf, 1));
  const int most = (int)std::min<int64_t>(nrhs, std::max<int64_t>(room, 1));
  double2* S = nullptr;
  cudaError_t e = device_alloc_async((void**)&S, sizeof(double2) * std::max<int64_t>(m->n_surf * most, 1), s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    set_error(std::string("cudaMallocAsync: ") + cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? BEM_ERR_OUT_OF_MEMORY : BEM_ERR_CUDA;
  }
  for (int r0 = 0; r0 < nrhs; r0 += most) {
    const int k = std::min(most, nrhs - r0);
    const int64_t nb = m->n_tet * k;
    const unsigned grid = (unsigned)std::min<int64_t>((m->n_surf * k + 3) / 4, 152 * 64);
    const double* prm = d_params ? d_params + 5 * (int64_t)r0 : nullptr;
    if (kind == BEM_DATA_PULSE)
      k_rhs_faces<BEM_DATA_PULSE><<<grid, kRhsThreads, 0, s>>>(m->n_surf, m->d_surf, m->d_col, k, prm, S);
    else
      k_rhs_faces<BEM_DATA_SIN2_UNIFORM><<<grid, kRhsThreads, 0, s>>>(m->n_surf, m->d_surf, m->d_col, k, prm, S);
    k_rhs_panels<<<(unsigned)((nb + 127) / 128), 128, 0, s>>>(m->n_tet, m->n_surf, k, m->d_tet, S, d_b + r0 * m->n_tet);
  }
  e = cudaGetLastError();
  cudaFreeAsync(S, s);
  STBEM_CUDA(e);
  return BEM_OK;
}

bem_status op_rhs_points(const bem_operator* op, int level, int ng, double* d_pts, double* d_wts, cudaStream_t s) {
  const bem_mesh* m = op->mesh;
  const int64_t n = m->n_surf * ((int64_t)1 << (2 * level));
  if (n == 0) return BEM_OK;
  k_rhs_points<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(m->n_surf, m->d_surf, m->d_col, level, ng, d_pts, d_wts);
  STBEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

bem_status op_rhs_samples(const bem_operator* op, int level, int ng, const double* d_wts, const double* d_g, int nrhs,
                          double* d_S, double* d_b, cudaStream_t s) {
  const bem_mesh* m = op->mesh;
  const int64_t npps = ((int64_t)1 << (2 * level)) * ng * ng;
  const int64_t ns = m->n_surf * nrhs, nb = m->n_tet * nrhs;
  if (ns > 0)
    k_rhs_face_sums<<<(unsigned)((ns + 127) / 128), 128, 0, s>>>(m->n_surf, npps, nrhs, d_wts, d_g, d_S);
  if (nb > 0)
    k_rhs_combine<<<(unsigned)((nb + 127) / 128), 128, 0, s>>>(m->n_tet, m->n_surf, nrhs, m->d_tet, d_S, d_b);
  STBEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

// ---------------------------------------------------------------------------
// Kernel-level inner potentials for arbitrary (point, panel) pairs
// ---------------------------------------------------------------------------
template <bool FP32>
__global__ void k_inner(int64_t n, const double* x4, const double* tv, const int32_t* sv, int n_theta, double* out) {
  int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= n) return;
  const double* X = tv + 16 * k;
  const int32_t* s = sv + 4 * k;
  // corners: distinct spatial ids ascending; lower / upper times per corner
  int ids[3], nid = 0;
  for (int v = 0; v < 4; ++v) {
    bool dup = false;
    for (int q = 0; q < nid; ++q) dup |= ids[q] == s[v];
    if (!dup && nid < 3) ids[nid++] = s[v];
  }
  if (nid != 3) { out[k] = nan(""); return; }
  for (int a = 1; a < 3; ++a)
    for (int b = a; b > 0 && ids[b - 1] > ids[b]; --b) { int t = ids[b]; ids[b] = ids[b - 1]; ids[b - 1] = t; }
  double cx[3][3];
  FaceGeom Flo, Fhi;
  for (int c = 0; c < 3; ++c) {
    double lo = 1e300, hi = -1e300;
    for (int v = 0; v < 4; ++v)
      if (s[v] == ids[c]) {
        for (int i = 0; i < 3; ++i) cx[c][i] = X[4 * v + 1 + i];
        lo = fmin(lo, X[4 * v]);
        hi = fmax(hi, X[4 * v]);
      }
    Flo.p[c] = lo;
    Fhi.p[c] = hi;
  }
  ColGeom G;
  make_colgeom(cx[0], cx[1], cx[2], G);
  face_gradient(G, Flo);
  face_gradient(G, Fhi);
  PointCol P;
  point_col(x4 + 4 * k, G, P, FP32);
  const ArcRule rule = make_rule(FP32 ? BEM_PREC_MIXED : BEM_PREC_FP64, n_theta);
  double wl = face_W<FP32>(G, P, Flo, rule), wh = face_W<FP32>(G, P, Fhi, rule);
  if (FP32 && !isfinite(wl)) wl = face_W_fp64(x4 + 4 * k, G, Flo, n_theta);
  if (FP32 && !isfinite(wh)) wh = face_W_fp64(x4 + 4 * k, G, Fhi, n_theta);
  out[k] = (wl - wh) / (4.0 * STBEM_PI);
}

bem_status inner_potentials(int64_t n, const double* d_x4, const double* d_tets, const int32_t* d_sv, int prec,
                            int n_theta, double* d_out, cudaStream_t s) {
  if (n == 0) return BEM_OK;
  unsigned g = (unsigned)((n + 127) / 128);
  if (prec == BEM_PREC_MIXED) k_inner<true><<<g, 128, 0, s>>>(n, d_x4, d_tets, d_sv, n_theta, d_out);
  else k_inner<false><<<g, 128, 0, s>>>(n, d_x4, d_tets, d_sv, n_theta, d_out);
  STBEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

// ---------------------------------------------------------------------------
// Permutations between caller and internal panel order
// ---------------------------------------------------------------------------
__global__ void k_permute(const int32_t* perm, const double* in, double* out, int64_t n, int nrhs, int to_internal) {
  int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= n * nrhs) return;
  int64_t r = k / n, i = k % n;
  int64_t p = perm[i];  // internal i -> caller p
  if (to_internal) out[r * n + i] = in[r * n + p];
  else out[r * n + p] = in[r * n + i];
}

bem_status permute(const int32_t* d_perm, const double* in, double* out, int64_t n, int nrhs, bool to_internal,
                   cudaStream_t s) {
  int64_t tot = n * nrhs;
  if (tot == 0) return BEM_OK;
  k_permute<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(d_perm, in, out, n, nrhs, to_internal ? 1 : 0);
  STBEM_CUDA(cudaGetLastError());
  return BEM_OK;
}

}  // namespace stbem
