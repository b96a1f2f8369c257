// fwi_internal.h -- shared declarations between the C-ABI host code (fwi_api.cu)
// and the CUDA kernels (fwi_kernels.cu). Not part of the public ABI.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace fwi {

constexpr int kFields = 27;  // 3 levels x (3 displacement + 6 stress components)
constexpr int kLevelFields = 9;

// Mesh geometry and per-node coefficient sources, passed by value to kernels.
// ---- bounds-checked build (-DFWI_BOUNDS_CHECK)
// Every node number read from a list (shell, face, source and receiver points, snapshot
// and sweep lists) and every node a structured kernel derives from its tile is checked
// before any access: a failed check records (site << 48) | (index & (2^48 - 1)) in the
// context's error word (the first one wins) and the thread skips that node, so nothing out
// of range is read or written; the call then returns FWI_E_BOUNDS. In the normal build
// guard() is the constant true and the checks compile away.
enum BoundsSite {
  kSiteShell = 1, kSiteFace = 2, kSitePml = 3, kSiteInterior = 4, kSitePoint = 5,
  kSiteGradient = 7, kSiteSnapshot = 8, kSitePersist = 9
};
#ifdef FWI_BOUNDS_CHECK
__device__ __forceinline__ bool guard(unsigned long long *err, int site, long long idx, long long n) {
  if (idx >= 0 && idx < n) return true;
  if (err) atomicCAS(err, 0ull, ((unsigned long long)site << 48) | ((unsigned long long)idx & 0xffffffffffffull));
  return false;
}
#else
__device__ __forceinline__ bool guard(unsigned long long *, int, long long, long long) { return true; }
#endif

struct Geo {
  int n[3];         // nodes per axis (NI, NJ, NK)
  int px;           // row pitch: node (i, j, k) is at (k * NJ + j) * px + i; px = NI rounded up to 4
  int lo[3], hi[3]; // interior element range per axis, [lo, hi)
  int m[3];         // material-grid nodes per axis (2nx+1, 2ny+1, 2nz+1)
  int top_dir;      // 1: displacement fixed on k = 0 (top PML)
  int box_lo[3], box_hi[3];  // inclusive node box whose elements are all interior (no fixed faces)
  int64_t stride;   // floats per state field (>= node count, padded)
  int64_t nnode, nmat;
  float inv_h;      // 1 / h
  float rho;
  float inv_rho_h;  // 1 / (rho h)
  float wdetj;      // (h/2)^3
  const float *alpha[3];  // stretch alpha_s at each node coordinate, per axis
  const float *ialpha[3]; // 1 / alpha_s (rounded from FP64)
  const float *beta[3];   // stretch beta_s, 1/s
  const float *lam, *mu;  // interior material grid [k][j][i]
  const float *lam_n, *mu_n;  // lambda, mu at every node in the state layout (PML: clamped interface value)
  const int *shell;       // node numbers of the interface shell (see shell_kernel)
  int nshell;
  const int *face;        // node numbers of the PML nodes on the grid's outer faces
  int nface;
  unsigned long long *oob;  // error word of the bounds-checked build (else null)
  // bounded waits of interior_kernel on its plane copies: after wait_cycles clock cycles a
  // wait gives up, sets *status to FWI_E_TIMEOUT (6) and the block returns; copy_extra > 0
  // makes every plane barrier expect that many bytes more than the copy delivers (tests of
  // the timeout path only)
  int *status;
  long long wait_cycles;
  int copy_extra;
  // launch shapes (fwi_tune_tiles; they change no node's arithmetic)
  int int_kc;             // most planes per block of interior_kernel (see chunk_planes)
  int pml_seg;            // an x segment of pml_kernel is up to 4 pml_seg node pairs wide (see Region there)
};

// One RK4 stage over every node (see fwi_kernels.cu).
//  stage 0: out = rate(Y)                   (fwi_rhs)
//  stage 1..3: out = X + cdt * rate(Y)   (stage 1: X must be Y; the kernels read Y only)
//  stage 4: out = (-X + Y2 + 2 Y3 + Y)/3 + cdt * rate(Y)   (out may alias X)
struct StageArgs {
  const float *Y;    // stage input
  const float *X;    // step start
  const float *Y2, *Y3;
  float *out;
  float cdt;
  int stage;
  float *hist;       // stage 4: interior displacement written here as [3][nmat], or null
  // a batch of nshot shots: shot b's buffers start sstride floats (history: hstride)
  // after shot b-1's; one launch of each stage kernel advances every shot of the batch
  int nshot;
  int64_t sstride, hstride;
};

// Point loads on the rate-level displacement of a stage's output and receiver samples of its
// value level. fused: the thread that writes a node applies them (kernels of few blocks, where
// a launch of their own would be a good part of the stage: 16x16x8, 4 % of a gradient; only
// planes k0 .. k1 have any, none when k1 < k0, so the other planes pay one comparison), except
// on launch_pml's nodes, where a point is rare and the check would cost registers. Else, and
// there, points_kernel does, after the stage's kernels (in the kernels of a 96x96x48 mesh the
// check's code and registers cost 3 % of the interior and 2 % of the shell kernel).
//  load 1 (sources): + cdt table[i0] src_vec[3 b + c] at src_node[b] of shot b;
//  load 2 (receiver residuals): + cdt e rec_vec[3 r + c] at receiver r, e = table[i0][r][c], or
//    the mean with table[i1] when i1 >= 0 (shot b's table at + b tstride);
//  traces: [nrec][3] of shot b at + b tstride, or null.
struct Points {
  bool fused;
  int load, i0, i1, nrec;
  int k0, k1;
  const int64_t *src_node;
  const float *src_vec, *rec_vec, *table;
  const int *rec_of;  // of the nodes rec0 .. rec0 + rec_n - 1 (the receivers' planes): receiver, or -1
  int64_t rec0, rec_n;
  float *traces;
  int64_t tstride;
};

// Planes per block of a kernel whose blocks march along z: the power of two up to `most` that
// takes the fewest plane steps, ceil(blocks / slots) (k + start), for `tiles` (x, y) tiles of
// all shots, `planes` planes and `slots` blocks resident on the GPU; `start` is the cost of
// filling a block's ring, in planes. Long chunks save ring fills on large grids; on small
// ones they leave the SMs idle (16x16x8 elements: 8 blocks of 8 planes took 36 us where 64
// blocks of one plane take 12 us).
inline int chunk_planes(int64_t tiles, int planes, int slots, int most, double start) {
  int best = 1;
  double cost = -1.0;
  for (int k = 1; k <= most; k *= 2) {
    const int64_t blocks = tiles * ((planes + k - 1) / k);
    const double c = (double)((blocks + slots - 1) / slots) * (k + start);
    if (cost < 0.0 || c <= cost) {
      cost = c;
      best = k;
    }
  }
  return best;
}
constexpr int kSms = 152;  // SMs of the GPU

// the buffers of shot `shot` of the batch
__host__ __device__ inline StageArgs shot_args(StageArgs a, int shot) {
  const int64_t o = (int64_t)shot * a.sstride;
  a.Y += o;
  if (a.X) a.X += o;
  if (a.Y2) a.Y2 += o;
  if (a.Y3) a.Y3 += o;
  a.out += o;
  if (a.hist) a.hist += (int64_t)shot * a.hstride;
  return a;
}

__device__ __forceinline__ bool has_points(const Points &q, int K) { return K >= q.k0 && K <= q.k1; }

// RK4 stage update of one variable's three levels at a node, for the list kernels: the step-start
// values are loaded together and before any of the node's stores (a.out may be a.X, so a load
// after a store waits its own latency: nine in a row for a node's three variables made up much of
// those kernels' time). The levels of variable f are the fields f, 9 + f, 18 + f. The fused
// multiply-adds are written out: a node's value must not depend on which variant of a kernel
// (warps per block, points) a launch's size picks, and the compiler contracts a sum of two
// products either way.
//
// Stage 4: s / 3 + cdt rate (the PML kernel's stage2 does the same). The FP32 constant 1/3 is 3e-8 too
// large: multiplied by it alone, the third fused or rounded by itself, the state grows by that
// share every step. So the product is corrected by its exact remainder s - 3 q. 2000 steps
// forward and adjoint on 16x16x8 elements against FP64: traces 1.8e-6 off with the product alone,
// 1.0e-6 so, J 3.8e-6 and 5e-8, the gradient for lambda 8.5e-6 and 2.6e-7. The constant in two
// parts (two FMAs behind the rate's product) is as exact and as fast; the remainder added to the
// rate's term, one rounding in all, is 0.5 to 1 % slower on the smallest meshes.
__device__ __forceinline__ float stage4(float s, float cdt, float rate) {
  const float q = __fmul_rn(s, 1.f / 3.f);
  return __fmaf_rn(cdt, rate, __fmaf_rn(__fmaf_rn(-3.f, q, s), 1.f / 3.f, q));
}
struct StepStart {
  float v[3];
};
__device__ __forceinline__ StepStart load_start(const StageArgs &a, int64_t i0, int64_t nine) {
  StepStart x{{0.f, 0.f, 0.f}};
  if (a.stage >= 2) {  // in stage 1 X is the stage input
#pragma unroll
    for (int l = 0; l < 3; l++) x.v[l] = __ldcs(a.X + i0 + l * nine);
  }
  if (a.stage == 4) {
#pragma unroll
    for (int l = 0; l < 3; l++) x.v[l] = __fmaf_rn(2.f, __ldcs(a.Y3 + i0 + l * nine), __ldcs(a.Y2 + i0 + l * nine) - x.v[l]);
  }
  return x;
}
__device__ __forceinline__ float stage_value(const StageArgs &a, float x, float yv, float rate) {
  if (a.stage == 0) return rate;
  if (a.stage == 1) return __fmaf_rn(a.cdt, rate, yv);
  if (a.stage < 4) return __fmaf_rn(a.cdt, rate, x);
  return stage4(x + yv, a.cdt, rate);
}

// receiver at a node, or -1
__device__ __forceinline__ int rec_at(const Points &q, int64_t node) {
  const int64_t m = node - q.rec0;
  return m >= 0 && m < q.rec_n ? __ldg(q.rec_of + m) : -1;
}

// a node of a plane with points, after this thread wrote its components c0 .. c1 - 1: adds the
// point load and takes the sample. It reads the values back (by the thread that wrote them), so
// that the rest of a kernel holds nothing for it.
__device__ __forceinline__ void node_points(const Points &q, const StageArgs &a, int64_t b, int64_t S, int64_t node, int c0,
                                            int c1, unsigned long long *oob) {
  const int r = q.load == 2 || q.traces ? rec_at(q, node) : -1;
  const bool rec = r >= 0 && guard(oob, kSitePoint, r, q.nrec), src = q.load == 1 && node == __ldg(q.src_node + b);
  if (!rec && !src) return;
#pragma unroll 1
  for (int c = c0; c < c1; c++) {
    if (src) {
      a.out[(18 + c) * S + node] += a.cdt * __ldg(q.table + q.i0) * __ldg(q.src_vec + 3 * b + c);
    } else if (q.load == 2) {
      const float *t = q.table + b * q.tstride + 3 * (int64_t)r + c;
      float e = __ldg(t + (int64_t)q.i0 * q.nrec * 3);
      if (q.i1 >= 0) e = 0.5f * (e + __ldg(t + (int64_t)q.i1 * q.nrec * 3));
      a.out[(18 + c) * S + node] += a.cdt * e * __ldg(q.rec_vec + 3 * (int64_t)r + c);
    }
    if (q.traces && rec) q.traces[b * q.tstride + (int64_t)r * 3 + c] = a.out[(9 + c) * S + node];
  }
}

// a node number of the state layout: inside the grid and not in a row's padding
__device__ __forceinline__ bool node_ok(const Geo &g, int site, long long node) {
  return guard(g.oob, site, node, (long long)g.px * g.n[1] * g.n[2]) && guard(g.oob, site, node % g.px, g.n[0]);
}

// One RK4 stage is four kernels writing disjoint node sets; they read the same
// input and may run concurrently on different streams. Each launcher returns the
// number of kernels it launched:
//  launch_interior: nodes all of whose elements are interior (fwi_interior.cu), with the tensor
//                   map of the stage input from plane_map. plane_map is false when it could not
//                   be encoded (Y not 16-byte aligned, or the driver entry point missing): the
//                   one way a stage can be refused, so it comes before the first launch;
//  launch_pml:      nodes all of whose elements are PML, off the outer faces (fwi_pml.cu);
//  launch_shell:    the interface shell (fwi_stage.cu);
//  launch_pml_face: the PML nodes on the outer faces of the grid (fwi_pml.cu).
// launch_points: points_kernel over the sources and receivers (only those on launch_pml's
// nodes when q.fused), after the stage's kernels.
struct alignas(128) PlaneMap {  // a CUtensorMap
  unsigned char bytes[128];
};
bool plane_map(const Geo &g, const StageArgs &a, PlaneMap *tm);
int launch_interior(const Geo &g, const StageArgs &a, const Points &q, const PlaneMap &tm, cudaStream_t s);
int launch_pml(const Geo &g, const StageArgs &a, bool adjoint, cudaStream_t s);
void launch_points(const Geo &g, const StageArgs &a, const Points &q, const int64_t *rec_node, cudaStream_t s);
int launch_pml_face(const Geo &g, const StageArgs &a, const Points &q, bool adjoint, cudaStream_t s);
int launch_shell(const Geo &g, const StageArgs &a, const Points &q, bool adjoint, cudaStream_t s);
// raises the interior kernel's shared-memory limit on the current device
cudaError_t prepare_interior();

// A whole forward sweep (steps n0 .. n1 - 1) of nshot shots in one cooperative launch
// (fwi_stage.cu): every node takes the general per-node formulas of the shell kernel, the
// four stages of a step are separated by grid-wide barriers, and the source loads, the
// receiver samples and the displacement history are written by the threads that own the
// nodes. Each barrier's spin gives up after wait_cycles clock cycles and sets *status to
// FWI_E_TIMEOUT; the kernel then returns. A barrier waits for gridDim.x + extra arrivals
// (extra > 0 only to exercise that path).
struct PersistArgs {
  float *st[4];               // X, Y2, Y3, Y4 of the batch's first shot (shot b at + b sstride)
  int nshot;
  int64_t sstride;
  int n0, n1;                 // steps t_n -> t_{n+1} of the sweep
  float dt;
  const int *nodes;           // every node of the grid, (k, j, i) order
  int nall;
  Points pts;                 // the sources, and the receivers' samples of level 0 (load 1)
  float *hist;                // displacement history, level n at hist + n hstep (shot b at + b hstride), or null
  int64_t hstep, hstride;
  unsigned *bar;              // [2]: arrival count and generation, zero before the launch
  int extra;
  long long wait_cycles;
  int *status;
};
cudaError_t launch_persistent_forward(const Geo &g, const PersistArgs &p, cudaStream_t s);

// rec_of[node[r] - rec0] = r for the nrec receivers, -1 at the other of its rec_n entries
void launch_rec_map(const int64_t *node, int nrec, int *rec_of, int64_t rec0, int64_t rec_n, cudaStream_t s);

// Gradient integrand of (C.1f)/(C.1g) at one time level, accumulated in FP64:
// gl[i] -= wdt * sum_e W detJ (div w)(div u), gm[i] -= wdt * sum_e W detJ 2 eps(w):eps(u),
// for the shots b = 0 .. nshot - 1 in order (adjoint state at w_state + b sstride, history
// level at u_hist + b hstride).
void launch_gradient(const Geo &g, const float *w_state, const float *u_hist, double wdt, double *gl,
                     double *gm, cudaStream_t s, int nshot = 1, int64_t sstride = 0, int64_t hstride = 0);

// resid = traces - observed (n values); partial sums of w_n dt e^2 / 2 per block into part;
// flag set to 1 on a non-finite trace value.
int misfit_blocks(int64_t n);
void launch_residual(const float *traces, const float *observed, float *resid, int64_t n,
                     int64_t per_step, int nsteps, double dt, double *part, int *flag, cudaStream_t s);
void launch_sum(const double *part, int nblocks, double *out, cudaStream_t s);

// Compact snapshot of nshot RK4 state sets (shot b at state + b sstride) into snap (shot b
// at snap + b snap_stride), or back (pack = false): u and udot (fields 9-11, 18-20) over
// all `stride` entries, then the other 21 fields at the npml PML nodes of `list`, each in
// a slot of npad >= npml floats (npad a multiple of 64). The restored state's other
// entries of those 21 fields must already be zero (no stage kernel writes them).
void launch_snapshot(float *state, float *snap, const int *list, int64_t npml, int64_t npad, int64_t stride,
                     int nshot, int64_t sstride, int64_t snap_stride, bool pack, cudaStream_t s,
                     unsigned long long *oob = nullptr);

// flag = 1 if any value of x (n doubles) is not finite.
void launch_check_finite(const double *x, int64_t n, int *flag, cudaStream_t s);
// g.lam_n / g.mu_n from the material grid (run whenever lam or mu change)
void launch_extend_material(const Geo &g, float *lam_n, float *mu_n, cudaStream_t s);

// reduced-space update helpers (fwi_opt.cu); vectors hold (lambda, mu) halves of nmat values
void opt_wdot(const double *a, const double *b, const double *w, int64_t nmat, double *part, double *out,
              cudaStream_t s);
void opt_axpby(double *y, double a, const double *x, double b, int64_t n, cudaStream_t s);
void opt_riesz(const double *gl, const double *gm, const double *mt, double *g, int64_t nmat, int mask,
               cudaStream_t s);
// plain dot product of n values (fixed-order reduction), part: >= 1024 doubles
void opt_dot(const double *a, const double *b, int64_t n, double *part, double *out, cudaStream_t s);
// regularisation term (8)/(9) of a field on the material grid (m nodes per axis):
// gradient (C.1b)-(C.1e) into g, functional into *value (device), part: >= 1024 doubles
void opt_regularization(const float *f, const int m[3], double h, bool tv, double eps, double *g, double *part,
                        double *value, cudaStream_t s);
void opt_trial(const double *m, const double *d, double alpha, float *lam, float *mu, int64_t nmat, unsigned *flags,
               cudaStream_t s);
void opt_pack(const float *lam, const float *mu, double *m, int64_t nmat, cudaStream_t s);
void opt_absmax(const double *x, int64_t n, unsigned long long *out, cudaStream_t s);

}  // namespace fwi
