// gmg.cu -- geometric-multigrid preconditioned CG (pb_pcg_solve with
// PB_PRECOND_GMG).  The paper lists geometric multigrid among the classical PB
// solvers (Sec. 2) and names multigrid solvers tailored to the PB problem as
// the way to further gains (Sec. 4); the scheme below is the one the oracle
// (oracle/gmg.py) states:
//
//   levels     vertex-centred: coarse node I sits on fine node 2I, coarse size
//              (n + 1) / 2 per axis, down to 3 nodes on the shortest axis;
//   operator   the h^2-scaled seven-point operator rediscretised at spacing
//              2h: a coarse edge's eps is the series combination
//              2 / (1/e_a + 1/e_b) of the two fine edges it spans on the fine
//              line through the coarse nodes, lambda the fine node's, and
//              kbar^2 (2h)^2 replaces kbar^2 h^2;
//   transfer   trilinear prolongation P (coarse ghosts zero), restriction
//              P^T r / 2;
//   V-cycle    NU damped-Jacobi sweeps (weight OMEGA) from zero, coarse
//              correction, NU sweeps; COARSE_SWEEPS sweeps on the coarsest
//              level: a symmetric positive definite preconditioner;
//   outer      preconditioned CG (Sec. 2.2) in FP64 with z = V(r); the V-cycle
//              runs in FP32 on FP32 copies of each level's operator.
//
// The FP64 edges from which the hierarchy is coarsened are dense: ex (nz, ny,
// nx+1), ey (nz, ny+1, nx), ez (nz+1, ny, nx), edge entry e of a line being the
// edge between nodes e-1 and e.  Vectors and FP32 coefficients have rows of P
// elements, nx rounded up to a multiple of four (pads zero), so that a thread
// works on four nodes of a row with 16-byte accesses; an FP32 coefficient array
// holds the edge below each node, and the edge above is the next node's (on the
// last node it multiplies the zero ghost).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "pb.h"
#include "pb_host.h"
#include "pb_internal.cuh"
#include "solve.cuh"

namespace pb {

constexpr float MG_OMEGA = 0.8f;
constexpr int MG_NU = 2, MG_COARSEST = 3, MG_COARSE_SWEEPS = 20, MG_NT = 256;

struct MgDims {
  int nx, ny, nz;
  __host__ __device__ int pitch() const { return (nx + 3) / 4 * 4; }
  __host__ __device__ size_t padded() const { return (size_t)pitch() * ny * nz; }
  __host__ __device__ size_t nodes() const { return (size_t)nx * ny * nz; }
  __host__ __device__ size_t nex() const { return (size_t)(nx + 1) * ny * nz; }
  __host__ __device__ size_t ney() const { return (size_t)nx * (ny + 1) * nz; }
  __host__ __device__ size_t nez() const { return (size_t)nx * ny * (nz + 1); }
};

static int mg_blocks(size_t n) {
  const size_t b = (n + MG_NT - 1) / MG_NT;
  return (int)(b < 152 * 32 ? (b ? b : 1) : 152 * 32);
}
#define MG_LOOP(t, n) \
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < (n); t += (size_t)gridDim.x * blockDim.x)

// Level 0 FP64 edges and lambda from the grid: its FP64 edge arrays (row
// pitch px) when it has them, else the code bits.
__global__ void k_mg_level0(MgDims d, int px, const uint8_t *code, const double *ex64, const double *ey64,
                            const double *ez64, double ein, double eout, double *ex, double *ey,
                            double *ez, uint8_t *lam) {
  MG_LOOP(t, d.nex()) {  // x-edges: entry i of row (j, k) is the edge (i-1, i)
    const size_t i = t % (d.nx + 1), row = t / (d.nx + 1);
    if (ex64) {
      ex[t] = ex64[row * px + i];
    } else {
      const bool first = i == 0;
      const uint8_t c = code[row * px + (first ? 0 : i - 1)];
      ex[t] = (first ? (c & 1u) : (c & 2u)) ? ein : eout;
    }
  }
  MG_LOOP(t, d.ney()) {  // y-edges: row j of plane k is the edge (j-1, j)
    const size_t i = t % d.nx, j = (t / d.nx) % (d.ny + 1), k = t / ((size_t)d.nx * (d.ny + 1));
    if (ey64) {
      ey[t] = ey64[(k * (d.ny + 1) + j) * px + i];
    } else {
      const bool first = j == 0;
      const uint8_t c = code[(k * d.ny + (first ? 0 : j - 1)) * px + i];
      ey[t] = (first ? (c & 4u) : (c & 8u)) ? ein : eout;
    }
  }
  MG_LOOP(t, d.nez()) {  // z-edges: plane k is the edge (k-1, k)
    const size_t i = t % d.nx, j = (t / d.nx) % d.ny, k = t / ((size_t)d.nx * d.ny);
    if (ez64) {
      ez[t] = ez64[(k * d.ny + j) * px + i];
    } else {
      const bool first = k == 0;
      const uint8_t c = code[((first ? 0 : k - 1) * d.ny + j) * px + i];
      ez[t] = (first ? (c & 16u) : (c & 32u)) ? ein : eout;
    }
  }
  MG_LOOP(t, d.nodes()) {
    const size_t i = t % d.nx, row = t / d.nx;
    lam[t] = (code[row * px + i] & 64u) ? 0 : 1;
  }
}

__device__ __forceinline__ double mg_series(double a, double b) {
  return __ddiv_rn(2.0, __dadd_rn(__ddiv_rn(1.0, a), __ddiv_rn(1.0, b)));
}

// Coarse FP64 edges and lambda of level l+1 from level l.
__global__ void k_mg_coarsen(MgDims f, MgDims c, const double *fex, const double *fey, const double *fez,
                             const uint8_t *flam, double *cex, double *cey, double *cez, uint8_t *clam) {
  MG_LOOP(t, c.nex()) {
    const size_t I = t % (c.nx + 1), J = (t / (c.nx + 1)) % c.ny, K = t / ((size_t)(c.nx + 1) * c.ny);
    const size_t row = ((2 * K) * f.ny + 2 * J) * (f.nx + 1);
    const long a = min(max(2 * (long)I - 1, 0L), (long)f.nx), b = min(2 * (long)I, (long)f.nx);
    cex[t] = mg_series(fex[row + a], fex[row + b]);
  }
  MG_LOOP(t, c.ney()) {
    const size_t I = t % c.nx, J = (t / c.nx) % (c.ny + 1), K = t / ((size_t)c.nx * (c.ny + 1));
    const long a = min(max(2 * (long)J - 1, 0L), (long)f.ny), b = min(2 * (long)J, (long)f.ny);
    const size_t base = (2 * K) * (f.ny + 1) * (size_t)f.nx + 2 * I;
    cey[t] = mg_series(fey[base + a * f.nx], fey[base + b * f.nx]);
  }
  MG_LOOP(t, c.nez()) {
    const size_t I = t % c.nx, J = (t / c.nx) % c.ny, K = t / ((size_t)c.nx * c.ny);
    const long a = min(max(2 * (long)K - 1, 0L), (long)f.nz), b = min(2 * (long)K, (long)f.nz);
    const size_t base = (2 * J) * (size_t)f.nx + 2 * I, pl = (size_t)f.nx * f.ny;
    cez[t] = mg_series(fez[a * pl + base], fez[b * pl + base]);
  }
  MG_LOOP(t, c.nodes()) {
    const size_t I = t % c.nx, J = (t / c.nx) % c.ny, K = t / ((size_t)c.nx * c.ny);
    clam[t] = flam[((2 * K) * f.ny + 2 * J) * f.nx + 2 * I];
  }
}

// FP32 copies of a level's edges, its diagonal (six edges in the order x-, x+,
// y-, y+, z-, z+, then + kbh2 lambda, summed in FP64) and its reciprocal.  Row
// pads: 0.
__global__ void k_mg_finish(MgDims d, double kbh2, const double *ex, const double *ey, const double *ez,
                            const uint8_t *lam, float *cx, float *cy, float *cz, float *fdiag, float *frd) {
  const size_t P = d.pitch();
  MG_LOOP(e, d.padded()) {
    const size_t row = e / P, i = e - row * P, k = row / d.ny;
    if (i >= (size_t)d.nx) {
      cx[e] = cy[e] = cz[e] = fdiag[e] = frd[e] = 0.f;
      continue;
    }
    const size_t t = row * d.nx + i, pl = (size_t)d.nx * d.ny, xr = t + row, yr = t + k * d.nx;
    double s = __dadd_rn(ex[xr], ex[xr + 1]);
    s = __dadd_rn(s, ey[yr]);
    s = __dadd_rn(s, ey[yr + d.nx]);
    s = __dadd_rn(s, ez[t]);
    s = __dadd_rn(s, ez[t + pl]);
    s = __dadd_rn(s, __dmul_rn(kbh2, (double)lam[t]));
    cx[e] = (float)ex[xr];
    cy[e] = (float)ey[yr];
    cz[e] = (float)ez[t];
    fdiag[e] = (float)s;
    frd[e] = __frcp_rn((float)s);
  }
}

// ---------------------------------------------------------------------------
// The operator of one level in FP32: explicit arrays, or (level 0 of a grid
// with packed codes) the grid's code bytes and a table by code byte, one byte
// a node instead of 16.

struct MgOp {
  MgDims d;
  const float *cx, *cy, *cz, *diag, *rd;   // rd = 1 / diag
  const uint8_t *code;                     // packed: [nz][ny][px]
  int px;
  float ein, eout, dt[NDTAB], rt[NDTAB];   // packed: diag and 1 / diag by dtab_index
};

// Scalars of the outer CG on the device, so that a graph of several iterations
// runs without host round trips: rz = r.z, rr = r.r; done stops the iterations
// (convergence when rr < stop2 = (tol ||b||)^2, the iteration cap, or
// breakdown), it counts those taken; ctas counts the CTAs that have finished a
// kernel whose last one forms the scalars.
struct MgScal {
  double rz, rr, alpha, beta, stop2;
  int it, done, status, max_iter;
  unsigned ctas;
};

// Programmatic dependent launch: the kernels of an iteration are short, so each
// starts while its predecessor drains and waits here for its results.
__device__ __forceinline__ void mg_pdl() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// A thread's column: a group of four x nodes of row j, planes k0 .. k1 - 1.
// Consecutive threads are consecutive groups whatever nx is, on to the next run of
// planes at a plane's end (a plane of 3x3 nodes has three groups: with CTAs that end
// at a plane's end, 3x3x20000 nodes took 2,551 us a solve, so 689), and two
// divisions serve the column.
struct Column {
  uint32_t o;      // offset of the group in a plane
  int i, j, k0, k1;
  bool in;
  uint32_t mask;   // bit u: node i + u is in the grid
};
__device__ __forceinline__ Column mg_column(const MgDims &d, int zc) {
  Column c;
  const uint32_t gpr = (uint32_t)d.pitch() / 4, groups = gpr * (uint32_t)d.ny, all = blockIdx.x * MG_NT + threadIdx.x;
  const uint32_t run = all / groups, t = all - run * groups;
  c.j = (int)(t / gpr);
  c.i = 4 * (int)(t - (uint32_t)c.j * gpr);
  c.o = (uint32_t)c.j * (uint32_t)d.pitch() + (uint32_t)c.i;
  c.in = run < (uint32_t)(d.nz + zc - 1) / (uint32_t)zc;
  c.k0 = (int)run * zc;
  c.k1 = min(c.k0 + zc, d.nz);
  c.mask = c.i + 4 <= d.nx ? 0xFu : (1u << (d.nx - c.i)) - 1u;
  return c;
}
// The launch of a column kernel over a level: planes of a column, and the grid.
struct MgLaunch {
  int zc;
  unsigned ctas;
};
// One wave of resident CTAs (a second, partly empty one costs as much as the
// first: the FP64 operator at 129^3 in 1.2 waves took 44 us, in one 34), or
// fewer on levels too small for one.
template <typename F>
static MgLaunch mg_plan(F *kernel, const MgDims &d, int num_sms) {
  int per_sm = 1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, MG_NT, 0) != cudaSuccess || per_sm < 1) per_sm = 1;
  const size_t groups = (size_t)d.pitch() / 4 * d.ny;
  const int runs = std::max(1, (int)std::min((size_t)d.nz, (size_t)num_sms * per_sm * MG_NT / groups));
  const int zc = (d.nz + runs - 1) / runs;
  return MgLaunch{zc, (unsigned)((groups * ((d.nz + zc - 1) / zc) + MG_NT - 1) / MG_NT)};
}

template <typename T> struct V4 { T v[4]; };
__device__ __forceinline__ V4<float> ld4(const float *p) {
  const float4 a = *(const float4 *)p;
  return V4<float>{{a.x, a.y, a.z, a.w}};
}
__device__ __forceinline__ V4<double> ld4(const double *p) {
  const double2 a = ((const double2 *)p)[0], b = ((const double2 *)p)[1];
  return V4<double>{{a.x, a.y, b.x, b.y}};
}
__device__ __forceinline__ void st4(float *p, const V4<float> &a) {
  *(float4 *)p = make_float4(a.v[0], a.v[1], a.v[2], a.v[3]);
}
__device__ __forceinline__ void st4(double *p, const V4<double> &a) {
  ((double2 *)p)[0] = make_double2(a.v[0], a.v[1]);
  ((double2 *)p)[1] = make_double2(a.v[2], a.v[3]);
}
template <typename T> __device__ __forceinline__ V4<T> ld4_if(bool in, const T *p) {
  return in ? ld4(p) : V4<T>{};
}
// A float as a double without the FP64 pipe (a conversion takes it as long as
// a multiplication): bits moved; a subnormal float is first scaled by 2^32, exactly.
__device__ __forceinline__ double widen(float f) {
  const bool small = fabsf(f) < 1.17549435e-38f;
  const uint32_t u = __float_as_uint(small ? f * 4294967296.f : f);
  uint32_t hi = ((u & 0x7FFFFFFFu) >> 3) + 0x38000000u + ((u & 0x7F800000u) == 0x7F800000u ? 0x38000000u : 0u);
  hi -= small ? 32u << 20 : 0u;
  hi = (u & 0x7FFFFFFFu) ? hi : 0u;
  return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(u << 29));
}

// {diag, 1 / diag} of the packed operator by code byte.
__device__ __forceinline__ void mg_table(const MgOp &A, float2 *tab) {
  for (int t = threadIdx.x; t < 128; t += blockDim.x) {
    const int k = dtab_index(t);
    tab[t] = make_float2(A.dt[k], A.rt[k]);
  }
  __syncthreads();
}

// a / b, correctly rounded, from rb = 1 / b correctly rounded: Markstein's
// correction of a quotient by its exact remainder.  A remainder, or a quotient, that
// a normal float cannot hold takes the division.
__device__ __forceinline__ float mg_div(float a, float b, float rb) {
  const float q = a * rb;
  if (fminf(fabsf(a) * 0x1p-24f, fabsf(q)) < 0x1p-125f && a != 0.f) return __fdiv_rn(a, b);
  return fmaf(fmaf(-q, b, a), rb, q);
}
// One damped-Jacobi step of a node: u + (omega (r - A u)) / diag, s the sum of
// eps u_nb.  (Every operation of the V-cycle rounds as it did when each sweep
// was a kernel with one node a thread: in FP32 another order of operations
// moves a solution to 1e-6 by 2e-8, the size of its rounding noise.)
__device__ __forceinline__ float mg_step(float u, float r, float s, float diag, float rd) {
  const float res = __fsub_rn(r, fmaf(diag, u, -s));
  return __fadd_rn(u, mg_div(__fmul_rn(MG_OMEGA, res), diag, rd));
}
// sum over the six edges of eps u_nb at the group of column c in plane k; um, uc,
// up: u of the group on the planes below, at and above (0 outside).  diag, rd:
// of the nodes (0 at row pads).
template <bool PACKED, bool RECIP>
__device__ __forceinline__ V4<float> mg_neighbours(const MgOp &A, const float2 *tab, const float *u, const Column &c,
                                                   int k, const V4<float> &um, const V4<float> &uc,
                                                   const V4<float> &up, V4<float> &diag, V4<float> &rd) {
  const int P = A.d.pitch();
  const size_t pl = (size_t)P * A.d.ny, e = k * pl + c.o;
  const V4<float> ym = ld4_if(c.j > 0, u + e - P), yp = ld4_if(c.j + 1 < A.d.ny, u + e + P);
  const float xl = c.i > 0 ? u[e - 1] : 0.f, xr = c.i + 4 < A.d.nx ? u[e + 4] : 0.f;
  V4<float> s;
  if constexpr (PACKED) {
    const uint32_t codes = *(const uint32_t *)(A.code + ((size_t)k * A.d.ny + c.j) * A.px + c.i);
    const float ei = A.ein, eo = A.eout;
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const uint32_t b = codes >> (8 * q);
      const float2 t = tab[b & 127u];
      diag.v[q] = t.x;
      rd.v[q] = t.y;
      float a = __fmul_rn((b & 1u) ? ei : eo, q ? uc.v[q - 1] : xl);
      a = fmaf((b & 2u) ? ei : eo, q < 3 ? uc.v[q + 1] : xr, a);
      a = fmaf((b & 4u) ? ei : eo, ym.v[q], a);
      a = fmaf((b & 8u) ? ei : eo, yp.v[q], a);
      a = fmaf((b & 16u) ? ei : eo, um.v[q], a);
      a = fmaf((b & 32u) ? ei : eo, up.v[q], a);
      s.v[q] = a;
    }
  } else {
    const V4<float> x = ld4(A.cx + e), y0 = ld4(A.cy + e), y1 = ld4_if(c.j + 1 < A.d.ny, A.cy + e + P);
    const V4<float> z0 = ld4(A.cz + e), z1 = ld4_if(k + 1 < A.d.nz, A.cz + e + pl);
    const float x4 = c.i + 4 < A.d.nx ? A.cx[e + 4] : 0.f;
    diag = ld4(A.diag + e);
    if (RECIP) rd = ld4(A.rd + e);
#pragma unroll
    for (int q = 0; q < 4; q++) {
      float a = __fmul_rn(x.v[q], q ? uc.v[q - 1] : xl);
      a = fmaf(q < 3 ? x.v[q + 1] : x4, q < 3 ? uc.v[q + 1] : xr, a);
      a = fmaf(y0.v[q], ym.v[q], a);
      a = fmaf(y1.v[q], yp.v[q], a);
      a = fmaf(z0.v[q], um.v[q], a);
      a = fmaf(z1.v[q], up.v[q], a);
      s.v[q] = a;
    }
  }
  return s;
}
__device__ __forceinline__ void keep(V4<float> &a, uint32_t mask) {
#pragma unroll
  for (int q = 0; q < 4; q++)
    if (!(mask >> q & 1u)) a.v[q] = 0.f;
}

// Dot products of the outer CG, and the scalars that follow from them: 256 CTAs
// take a contiguous share of the nodes each (in the order of a dense array), a
// thread every 256th of it; partial sums by halves; the last CTA to finish adds
// the 256 partials by halves.  A pass of its own, although the kernels that
// produce the vectors could add up their products: V-cycles in FP32 turn a last
// bit of a scalar into 1e-8 of the solution to 1e-6 (the FP32 copy of r rounds
// differently, and so on), so the order of these sums is part of the result.
enum : int { DOT_ALPHA, DOT_STOP, DOT_BETA, DOT_RR };
// Loads in flight a thread: half of the 33 nodes it has at 129^3, so two trips to
// memory (with 8, five: an iteration 239 us for 218); a larger grid takes more trips.
constexpr int MG_DOT_CTAS = 256, MG_DOT_BATCH = 17;
__device__ __forceinline__ double mg_wide(double v) { return v; }
__device__ __forceinline__ double mg_wide(float v) { return widen(v); }
template <int WHAT, typename B>
__global__ void __launch_bounds__(MG_NT) k_mg_dot(MgDims d, MgScal *S, const double *a, const B *b, double *part) {
  __shared__ double red[MG_NT];
  __shared__ int last;
  mg_pdl();
  if (WHAT != DOT_RR && S->done) return;
  const uint32_t n = (uint32_t)d.nodes(), per = (n + MG_DOT_CTAS - 1) / MG_DOT_CTAS, nx = d.nx, P = d.pitch();
  const uint32_t lo = blockIdx.x * per, hi = min(lo + per, n);
  uint32_t t = lo + threadIdx.x;
  uint32_t row = t / nx, i = t - row * nx;
  const uint32_t rows = MG_NT / nx, rest = MG_NT - rows * nx;  // MG_NT nodes on
  double s = 0.0;
  while (t < hi) {
    double u[MG_DOT_BATCH];
    B v[MG_DOT_BATCH];
    int m = 0;
#pragma unroll
    for (int q = 0; q < MG_DOT_BATCH; q++) {  // loads first
      if (t < hi) {
        const size_t e = (size_t)row * P + i;
        u[q] = a[e];
        v[q] = b[e];
        m++;
      }
      t += MG_NT;
      i += rest;
      row += rows;
      if (i >= nx) {
        i -= nx;
        row++;
      }
    }
#pragma unroll
    for (int q = 0; q < MG_DOT_BATCH; q++)
      if (q < m) s = fma(u[q], mg_wide(v[q]), s);
  }
  red[threadIdx.x] = s;
  __syncthreads();
  auto halves = [&]() {
    for (int w = MG_NT / 2; w > 0; w >>= 1) {
      if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
      __syncthreads();
    }
  };
  halves();
  if (threadIdx.x == 0) {
    part[blockIdx.x] = red[0];
    __threadfence();
    last = atomicAdd(&S->ctas, 1u) == MG_DOT_CTAS - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  static_assert(MG_DOT_CTAS == MG_NT, "a partial a thread");
  red[threadIdx.x] = __ldcg(part + threadIdx.x);
  __syncthreads();
  halves();
  if (threadIdx.x != 0) return;
  S->ctas = 0;
  const double sum = red[0];
  if (WHAT == DOT_ALPHA) {  // p.Ap: alpha = r.z / p.Ap, or breakdown
    const double alpha = S->rz / sum;
    if (!(sum > 0.0) || !isfinite(alpha)) {
      S->status = PB_ERR_BREAKDOWN;
      S->done = 1;
      S->alpha = 0.0;
    } else {
      S->alpha = alpha;
    }
  } else if (WHAT == DOT_STOP) {  // r.r after an update: the stop test
    S->rr = sum;
    S->it++;
    if (sum < S->stop2) {
      S->status = PB_OK;
      S->done = 1;
    } else if (S->it >= S->max_iter) {
      S->done = 1;
    }
  } else if (WHAT == DOT_BETA) {  // r.z
    S->beta = sum / S->rz;
    S->rz = sum;
  } else {
    S->rr = sum;
  }
}

// One damped-Jacobi sweep: out = u + omega (r - A u) / diag.  (The first of a
// level, from zero, is (omega r) / diag: the kernels that make a level's
// right-hand side write it too.)
template <bool PACKED>
__global__ void __launch_bounds__(MG_NT) k_mg_sweep(const __grid_constant__ MgOp A, int zc, const MgScal *S,
                                                    const float *u, const float *r, float *out) {
  __shared__ float2 tab[PACKED ? 128 : 1];
  if (PACKED) mg_table(A, tab);
  mg_pdl();
  if (S->done) return;
  const Column c = mg_column(A.d, zc);
  if (!c.in) return;
  const size_t pl = (size_t)A.d.pitch() * A.d.ny;
  V4<float> um = ld4_if(c.k0 > 0, u + (c.k0 - 1) * pl + c.o), uc = ld4(u + c.k0 * pl + c.o);
  for (int k = c.k0; k < c.k1; k++) {
    const size_t e = k * pl + c.o;
    const V4<float> up = ld4_if(k + 1 < A.d.nz, u + e + pl), rv = ld4(r + e);
    V4<float> diag, rd, z;
    const V4<float> s = mg_neighbours<PACKED, true>(A, tab, u, c, k, um, uc, up, diag, rd);
#pragma unroll
    for (int q = 0; q < 4; q++) z.v[q] = mg_step(uc.v[q], rv.v[q], s.v[q], diag.v[q], rd.v[q]);
    keep(z, c.mask);
    st4(out + e, z);
    um = uc;
    uc = up;
  }
}

// res = r - A z.
template <bool PACKED>
__global__ void __launch_bounds__(MG_NT) k_mg_residual(const __grid_constant__ MgOp A, int zc, const MgScal *S,
                                                       const float *z, const float *r, float *res) {
  __shared__ float2 tab[PACKED ? 128 : 1];
  if (PACKED) mg_table(A, tab);
  mg_pdl();
  if (S->done) return;
  const Column c = mg_column(A.d, zc);
  if (!c.in) return;
  const size_t pl = (size_t)A.d.pitch() * A.d.ny;
  V4<float> um = ld4_if(c.k0 > 0, z + (c.k0 - 1) * pl + c.o), uc = ld4(z + c.k0 * pl + c.o);
  for (int k = c.k0; k < c.k1; k++) {
    const size_t e = k * pl + c.o;
    const V4<float> up = ld4_if(k + 1 < A.d.nz, z + e + pl), rv = ld4(r + e);
    V4<float> diag, rd, out;
    const V4<float> s = mg_neighbours<PACKED, false>(A, tab, z, c, k, um, uc, up, diag, rd);
#pragma unroll
    for (int q = 0; q < 4; q++) out.v[q] = __fsub_rn(rv.v[q], fmaf(diag.v[q], uc.v[q], -s.v[q]));
    keep(out, c.mask);
    st4(res + e, out);
    um = uc;
    uc = up;
  }
}

// Coarse right-hand side P^T res / 2 (coarse node I takes fine nodes 2I and 2I
// +- 1 with weights 1 and 1/2 per axis, plane by plane, row by row), and the
// first sweep y = (omega r) / diag.  A thread makes four coarse nodes of a
// row: fine nodes 2I - 1 .. 2I + 7.
__device__ __forceinline__ void mg_plane_sum(const MgDims &f, const float *res, int I, int J, int k, float wk,
                                             V4<float> &s) {
  if (k < 0 || k >= f.nz) return;
  const int P = f.pitch();
#pragma unroll
  for (int dj = -1; dj <= 1; dj++) {
    const int j = 2 * J + dj;
    if (j < 0 || j >= f.ny) continue;
    const float *row = res + ((size_t)k * f.ny + j) * P + 2 * I;
    const V4<float> a = ld4(row), b = ld4_if(2 * I + 4 < P, row + 4);  // (pads are 0)
    const float v[9] = {I > 0 ? row[-1] : 0.f, a.v[0], a.v[1], a.v[2], a.v[3], b.v[0], b.v[1], b.v[2], b.v[3]};
    const float w = (dj ? 0.5f : 1.f) * wk;
#pragma unroll
    for (int q = 0; q < 4; q++) {
      s.v[q] = fmaf(0.5f * w, v[2 * q], s.v[q]);
      s.v[q] = fmaf(w, v[2 * q + 1], s.v[q]);
      s.v[q] = fmaf(0.5f * w, v[2 * q + 2], s.v[q]);
    }
  }
}
__global__ void __launch_bounds__(MG_NT) k_mg_restrict(MgDims d, int zc, MgDims f, const MgScal *S, const float *res,
                                                       const float *diag, const float *rd, float *rc, float *yc) {
  mg_pdl();
  if (S->done) return;
  const Column c = mg_column(d, zc);
  if (!c.in) return;
  const size_t pl = (size_t)d.pitch() * d.ny;
  for (int k = c.k0; k < c.k1; k++) {
    const size_t e = k * pl + c.o;
    const V4<float> dg = ld4(diag + e), rv = ld4(rd + e);
    V4<float> v = {}, y;
    mg_plane_sum(f, res, c.i, c.j, 2 * k - 1, 0.5f, v);
    mg_plane_sum(f, res, c.i, c.j, 2 * k, 1.f, v);
    mg_plane_sum(f, res, c.i, c.j, 2 * k + 1, 0.5f, v);
#pragma unroll
    for (int q = 0; q < 4; q++) v.v[q] *= 0.5f;
    keep(v, c.mask);
#pragma unroll
    for (int q = 0; q < 4; q++) y.v[q] = mg_div(__fmul_rn(MG_OMEGA, v.v[q]), dg.v[q], rv.v[q]);
    st4(rc + e, v);
    st4(yc + e, y);
  }
}

// z += P e: fine node i takes coarse i/2 (even) or the mean of (i-1)/2 and
// (i+1)/2 (odd), per axis; coarse indices past the end are the zero ghost (and
// row pads).  Adds coarse row J of plane K, weight w, to the four nodes' sums.
__device__ __forceinline__ void mg_row_add(const MgDims &c, const float *e, int I, int J, int K, float w,
                                           V4<float> &s) {
  if (J >= c.ny || K >= c.nz) return;
  const int P = c.pitch();
  const float *row = e + ((size_t)K * c.ny + J) * P + I;  // I is even: I and I + 1 are in the row or its pads
  const float a0 = row[0], a1 = row[1], a2 = I + 2 < P ? row[2] : 0.f;
  const float h = 0.5f * w;
  s.v[0] = fmaf(w, a0, s.v[0]);
  s.v[1] = fmaf(h, a1, fmaf(h, a0, s.v[1]));
  s.v[2] = fmaf(w, a1, s.v[2]);
  s.v[3] = fmaf(h, a2, fmaf(h, a1, s.v[3]));
}
__device__ __forceinline__ void mg_plane_add(const MgDims &c, const float *e, int i, int j, int K, float wk,
                                             V4<float> &s) {
  const float w = j & 1 ? 0.5f * wk : wk;
  mg_row_add(c, e, i / 2, j / 2, K, w, s);
  if (j & 1) mg_row_add(c, e, i / 2, j / 2 + 1, K, w, s);
}
__global__ void __launch_bounds__(MG_NT) k_mg_prolong_add(MgDims f, int zc, MgDims d, const MgScal *S, const float *e,
                                                          float *z) {
  mg_pdl();
  if (S->done) return;
  const Column c = mg_column(f, zc);
  if (!c.in) return;
  const size_t pl = (size_t)f.pitch() * f.ny;
  for (int k = c.k0; k < c.k1; k++) {
    V4<float> v = {};
    mg_plane_add(d, e, c.i, c.j, k / 2, k & 1 ? 0.5f : 1.f, v);
    if (k & 1) mg_plane_add(d, e, c.i, c.j, k / 2 + 1, 0.5f, v);
    keep(v, c.mask);
    V4<float> u = ld4(z + k * pl + c.o);
#pragma unroll
    for (int q = 0; q < 4; q++) u.v[q] = __fadd_rn(u.v[q], v.v[q]);
    st4(z + k * pl + c.o, u);
  }
}

// ---------------------------------------------------------------------------
// The coarse end of the V-cycle in one CTA: every level from the first whose
// operators and vectors (with those below it) fit the CTA's shared memory.
// Kernels of a few hundred nodes cost a launch each (2 us, and there were
// about 45 of them an iteration); here a sweep costs a barrier: 17^3 and below
// in 27 us.

constexpr int MG_TAIL_NT = 1024, MG_TAIL_MAX = 8, MG_TAIL_BATCH = 4;
// Arrays of one level, dense, in shared memory (offsets in floats).  cx[t],
// cy[t], cz[t]: the coefficient of the edge below node t on each axis, 0 on the
// boundary, so that the edge above is the next node's (row's, plane's) entry
// and a sweep needs neither indices nor tests: neighbours outside the grid are
// multiplied by 0.  The arrays that are read past their ends have a plane of
// zeros there.  The coefficients of all levels come first: one block that a
// solve's first kernel lays out in global memory and every V-cycle copies.
struct TailLevel {
  MgDims d;
  int n, cx, cy, cz, diag, rd, r, z0, z1, res;
};
struct MgTail {
  int n;                       // levels
  int coef, all;               // floats of the coefficient block, of everything
  TailLevel lv[MG_TAIL_MAX];
  const float *block;          // the coefficients in global memory
  const float *r, *y;          // right-hand side of its first level, and its first sweep
  float *z;                    // the result
};
// Offsets for the levels given; the sizes.
static void mg_tail_layout(MgTail &T) {
  int p = 0;
  auto take = [&](int &o, int n, int before, int after) {
    p += before;
    o = p;
    p += n + after;
  };
  for (int l = 0; l < T.n; l++) {
    TailLevel &L = T.lv[l];
    L.n = (int)L.d.nodes();
    const int pad = L.d.nx * L.d.ny;
    take(L.cx, L.n, 0, pad);
    take(L.cy, L.n, 0, pad);
    take(L.cz, L.n, 0, pad);
    take(L.diag, L.n, 0, 0);
    take(L.rd, L.n, 0, 0);
  }
  p = round_up(p, 4);
  T.coef = p;
  for (int l = 0; l < T.n; l++) {
    TailLevel &L = T.lv[l];
    const int pad = L.d.nx * L.d.ny;
    take(L.z0, L.n, pad, pad);
    take(L.z1, L.n, pad, pad);
    take(L.r, L.n, 0, 0);
    take(L.res, L.n, 0, 0);
  }
  T.all = p;
}
__device__ __forceinline__ void tail_ijk(const MgDims &d, int t, int &i, int &j, int &k) {
  const uint32_t row = (uint32_t)t / (uint32_t)d.nx;
  i = (int)((uint32_t)t - row * d.nx);
  k = (int)(row / (uint32_t)d.ny);
  j = (int)(row - (uint32_t)k * d.ny);
}
// The block's part of one level, from the level's arrays (rows of P).
__global__ void k_mg_tail_pack(TailLevel L, const float *cx, const float *cy, const float *cz, const float *diag,
                               const float *rd, float *block) {
  const int pad = L.d.nx * L.d.ny, P = L.d.pitch();
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < L.n + pad; t += gridDim.x * blockDim.x) {
    int i, j, k;
    tail_ijk(L.d, t, i, j, k);
    const bool in = t < L.n;
    const size_t e = ((size_t)k * L.d.ny + j) * P + i;
    block[L.cx + t] = in && i > 0 ? cx[e] : 0.f;
    block[L.cy + t] = in && j > 0 ? cy[e] : 0.f;
    block[L.cz + t] = in && k > 0 ? cz[e] : 0.f;
    if (in) {
      block[L.diag + t] = diag[e];
      block[L.rd + t] = rd[e];
    }
  }
}
__device__ __forceinline__ float tail_neighbours(const float *sm, const TailLevel &L, const float *u, int t) {
  const int nx = L.d.nx, pl = nx * L.d.ny;
  const float *cx = sm + L.cx + t, *cy = sm + L.cy + t, *cz = sm + L.cz + t;
  float s = __fmul_rn(cx[0], u[t - 1]);
  s = fmaf(cx[1], u[t + 1], s);
  s = fmaf(cy[0], u[t - nx], s);
  s = fmaf(cy[nx], u[t + nx], s);
  s = fmaf(cz[0], u[t - pl], s);
  return fmaf(cz[pl], u[t + pl], s);
}
// f(t) of MG_TAIL_BATCH nodes a thread, then their stores (which would
// otherwise hold the next node's loads back).
template <typename F>
__device__ __forceinline__ void tail_each(int n, float *out, F f) {
  for (int t0 = threadIdx.x; t0 < n; t0 += MG_TAIL_BATCH * MG_TAIL_NT) {
    float v[MG_TAIL_BATCH];
#pragma unroll
    for (int b = 0; b < MG_TAIL_BATCH; b++)
      if (t0 + b * MG_TAIL_NT < n) v[b] = f(t0 + b * MG_TAIL_NT);
#pragma unroll
    for (int b = 0; b < MG_TAIL_BATCH; b++)
      if (t0 + b * MG_TAIL_NT < n) out[t0 + b * MG_TAIL_NT] = v[b];
  }
  __syncthreads();
}
__device__ __forceinline__ void tail_sweep(float *sm, const TailLevel &L, const float *u, float *out) {
  const float *diag = sm + L.diag, *rd = sm + L.rd, *r = sm + L.r;
  tail_each(L.n, out, [&](int t) { return mg_step(u[t], r[t], tail_neighbours(sm, L, u, t), diag[t], rd[t]); });
}
__global__ void __launch_bounds__(MG_TAIL_NT) k_mg_tail(const __grid_constant__ MgTail T, const MgScal *S) {
  extern __shared__ __align__(16) float sm[];
  // coefficients: constant through a solve, copied before the wait
#pragma unroll 8
  for (int t = threadIdx.x; t < T.coef / 4; t += MG_TAIL_NT) ((float4 *)sm)[t] = ((const float4 *)T.block)[t];
  for (int t = T.coef + threadIdx.x; t < T.all; t += MG_TAIL_NT) sm[t] = 0.f;
  __syncthreads();
  mg_pdl();
  if (S->done) return;
  {
    const TailLevel &L = T.lv[0];
    const int P = L.d.pitch();
    auto at = [&](int t) { const uint32_t row = (uint32_t)t / (uint32_t)L.d.nx; return row * (uint32_t)P + (t - row * L.d.nx); };
    tail_each(L.n, sm + L.r, [&](int t) { return T.r[at(t)]; });
    tail_each(L.n, sm + L.z0, [&](int t) { return T.y[at(t)]; });
  }
  for (int l = 0; l + 1 < T.n; l++) {  // down: two sweeps from zero (z0: the first), residual, restriction
    const TailLevel &L = T.lv[l], &C = T.lv[l + 1];
    float *z0 = sm + L.z0, *z1 = sm + L.z1, *res = sm + L.res, *r = sm + L.r;
    tail_sweep(sm, L, z0, z1);
    tail_each(L.n, res,
              [&](int t) { return __fsub_rn(r[t], fmaf(sm[L.diag + t], z1[t], -tail_neighbours(sm, L, z1, t))); });
    for (int t = threadIdx.x; t < C.n; t += MG_TAIL_NT) {
      int I, J, K;
      tail_ijk(C.d, t, I, J, K);
      const int nx = L.d.nx, ny = L.d.ny, nz = L.d.nz;
      float v = 0.f;
#pragma unroll
      for (int dk = -1; dk <= 1; dk++) {
        const int k = 2 * K + dk;
        if (k < 0 || k >= nz) continue;
#pragma unroll
        for (int dj = -1; dj <= 1; dj++) {
          const int j = 2 * J + dj;
          if (j < 0 || j >= ny) continue;
          const float *row = res + (k * ny + j) * nx + 2 * I;
          const float xm = I > 0 ? row[-1] : 0.f, xp = 2 * I + 1 < nx ? row[1] : 0.f;
          const float w = (dk ? 0.5f : 1.f) * (dj ? 0.5f : 1.f);
          v = fmaf(0.5f * w, xp, fmaf(w, row[0], fmaf(0.5f * w, xm, v)));
        }
      }
      v *= 0.5f;
      sm[C.r + t] = v;
      sm[C.z0 + t] = mg_div(__fmul_rn(MG_OMEGA, v), sm[C.diag + t], sm[C.rd + t]);
    }
    __syncthreads();
  }
  {  // coarsest: z0 is the first sweep; an odd number more leaves the result in z1
    static_assert(MG_COARSE_SWEEPS % 2 == 0, "the last sweep ends in z1");
    const TailLevel &L = T.lv[T.n - 1];
    float *z0 = sm + L.z0, *z1 = sm + L.z1;
    if (L.n <= 32) {  // one warp, a node a lane
      if (threadIdx.x < 32) {
        const int t = threadIdx.x;
        for (int s = 1; s < MG_COARSE_SWEEPS; s++) {
          const float *u = s & 1 ? z0 : z1;
          if (t < L.n)
            (s & 1 ? z1 : z0)[t] =
                mg_step(u[t], sm[L.r + t], tail_neighbours(sm, L, u, t), sm[L.diag + t], sm[L.rd + t]);
          __syncwarp();
        }
      }
      __syncthreads();
    } else {
      for (int s = 1; s < MG_COARSE_SWEEPS; s++) tail_sweep(sm, L, s & 1 ? z0 : z1, s & 1 ? z1 : z0);
    }
  }
  for (int l = T.n - 2; l >= 0; l--) {  // up: correction, two sweeps
    const TailLevel &L = T.lv[l], &C = T.lv[l + 1];
    float *z0 = sm + L.z0, *z1 = sm + L.z1;
    const float *e = sm + C.z1;
    const int cx = C.d.nx, cy = C.d.ny;
    auto row_add = [&](int i, int J, int K, float w, float v) -> float {
      if (J >= cy || K >= C.d.nz) return v;
      const float *row = e + (K * cy + J) * cx + i / 2;
      if (!(i & 1)) return fmaf(w, row[0], v);
      return fmaf(0.5f * w, i / 2 + 1 < cx ? row[1] : 0.f, fmaf(0.5f * w, row[0], v));
    };
    tail_each(L.n, z1, [&](int t) {
      int i, j, k;
      tail_ijk(L.d, t, i, j, k);
      const float w = (k & 1 ? 0.5f : 1.f) * (j & 1 ? 0.5f : 1.f);
      float v = 0.f;
      for (int K = k / 2; K <= (k + 1) / 2; K++)
        for (int J = j / 2; J <= (j + 1) / 2; J++) v = row_add(i, J, K, w, v);
      return __fadd_rn(z1[t], v);
    });
    tail_sweep(sm, L, z1, z0);
    tail_sweep(sm, L, z0, z1);
  }
  const TailLevel &L = T.lv[0];
  const int P = L.d.pitch();
  for (int t = threadIdx.x; t < L.n; t += MG_TAIL_NT) {
    const uint32_t row = (uint32_t)t / (uint32_t)L.d.nx;
    T.z[row * (uint32_t)P + (t - row * L.d.nx)] = sm[L.z1 + t];
  }
}

// ---------------------------------------------------------------------------
// Outer CG, FP64.

// A of level 0 in FP64: the grid's code bytes, or its FP64 edges and diagonal
// (row pitch px).  Bound by its FP64 arithmetic (7 operations a node).
struct MgOp64 {
  MgDims d;
  int px;
  const uint8_t *code;
  const double *ex, *ey, *ez, *diag;
  double ein, eout, dt[NDTAB];
};
template <bool PACKED>
__device__ __forceinline__ V4<double> mg_apply64(const MgOp64 &A, const double *tab, const double *u, const Column &c,
                                                 int k, const V4<double> &um, const V4<double> &uc,
                                                 const V4<double> &up) {
  const int P = A.d.pitch();
  const size_t pl = (size_t)P * A.d.ny, e = k * pl + c.o;
  const V4<double> ym = ld4_if(c.j > 0, u + e - P), yp = ld4_if(c.j + 1 < A.d.ny, u + e + P);
  const double xl = c.i > 0 ? u[e - 1] : 0.0, xr = c.i + 4 < A.d.nx ? u[e + 4] : 0.0;
  const size_t q0 = ((size_t)k * A.d.ny + c.j) * A.px + c.i;
  V4<double> a;
  if constexpr (PACKED) {
    // (one form for every node: a warp that met both the uniform and the
    // general one would pay for both)
    const uint32_t codes = *(const uint32_t *)(A.code + q0);
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const uint32_t b = codes >> (8 * q);
      double s = __dmul_rn((b & 1u) ? A.ein : A.eout, q ? uc.v[q - 1] : xl);
      s = fma((b & 2u) ? A.ein : A.eout, q < 3 ? uc.v[q + 1] : xr, s);
      s = fma((b & 4u) ? A.ein : A.eout, ym.v[q], s);
      s = fma((b & 8u) ? A.ein : A.eout, yp.v[q], s);
      s = fma((b & 16u) ? A.ein : A.eout, um.v[q], s);
      s = fma((b & 32u) ? A.ein : A.eout, up.v[q], s);
      a.v[q] = fma(tab[b & 127u], uc.v[q], -s);
    }
  } else {
    const size_t y0 = q0 + (size_t)k * A.px;
    const V4<double> ex = ld4(A.ex + q0), eym = ld4(A.ey + y0), eyp = ld4(A.ey + y0 + A.px);
    const V4<double> ezm = ld4(A.ez + q0), ezp = ld4(A.ez + q0 + (size_t)A.px * A.d.ny), dg = ld4(A.diag + q0);
    const double ex4 = c.mask & 8u ? A.ex[q0 + 4] : 0.0;  // (past the row if its last node is not in the grid)
#pragma unroll
    for (int q = 0; q < 4; q++) {
      double s = __dmul_rn(ex.v[q], q ? uc.v[q - 1] : xl);
      s = fma(q < 3 ? ex.v[q + 1] : ex4, q < 3 ? uc.v[q + 1] : xr, s);
      s = fma(eym.v[q], ym.v[q], s);
      s = fma(eyp.v[q], yp.v[q], s);
      s = fma(ezm.v[q], um.v[q], s);
      s = fma(ezp.v[q], up.v[q], s);
      a.v[q] = fma(dg.v[q], uc.v[q], -s);
    }
  }
#pragma unroll
  for (int q = 0; q < 4; q++)
    if (!(c.mask >> q & 1u)) a.v[q] = 0.0;
  return a;
}
template <bool PACKED>
__device__ __forceinline__ void mg_table64(const MgOp64 &A, double *tab) {
  if constexpr (PACKED) {
    for (int t = threadIdx.x; t < 128; t += blockDim.x) tab[t] = A.dt[dtab_index(t)];
    __syncthreads();
  }
}
// ap = A p
template <bool PACKED>
__global__ void __launch_bounds__(MG_NT) k_mg_apply(const __grid_constant__ MgOp64 A, int zc, const MgScal *S,
                                                    const double *p, double *ap) {
  __shared__ double tab[PACKED ? 128 : 1];
  mg_table64<PACKED>(A, tab);
  mg_pdl();
  if (S->done) return;
  const Column c = mg_column(A.d, zc);
  if (!c.in) return;
  const size_t pl = (size_t)A.d.pitch() * A.d.ny;
  V4<double> um = ld4_if(c.k0 > 0, p + (c.k0 - 1) * pl + c.o), uc = ld4(p + c.k0 * pl + c.o);
  for (int k = c.k0; k < c.k1; k++) {
    const size_t e = k * pl + c.o;
    const V4<double> up = ld4_if(k + 1 < A.d.nz, p + e + pl);
    st4(ap + e, mg_apply64<PACKED>(A, tab, p, c, k, um, uc, up));
    um = uc;
    uc = up;
  }
}
// The V-cycle's right-hand side of a group, from the residual, and its first
// sweep y = (omega r) / diag.
template <bool PACKED>
__device__ __forceinline__ void mg_rhs(const MgOp &F, const float2 *tab, const Column &c, int k, size_t e,
                                       const V4<double> &v, float *r32, float *y) {
  V4<float> f, w;
#pragma unroll
  for (int q = 0; q < 4; q++) f.v[q] = (float)v.v[q];
  if constexpr (PACKED) {
    const uint32_t codes = *(const uint32_t *)(F.code + ((size_t)k * F.d.ny + c.j) * F.px + c.i);
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const float2 t = tab[codes >> (8 * q) & 127u];
      w.v[q] = mg_div(__fmul_rn(MG_OMEGA, f.v[q]), t.x, t.y);
    }
  } else {
    const V4<float> dg = ld4(F.diag + e), rd = ld4(F.rd + e);
#pragma unroll
    for (int q = 0; q < 4; q++) w.v[q] = mg_div(__fmul_rn(MG_OMEGA, f.v[q]), dg.v[q], rd.v[q]);
  }
  st4(r32 + e, f);
  st4(y + e, w);
}
// r = b - A x (b in the padded layout); r32, y: the V-cycle's right-hand side
// (r32 NULL: not wanted)
template <bool PACKED>
__global__ void __launch_bounds__(MG_NT) k_mg_true_residual(const __grid_constant__ MgOp64 A, int zc,
                                                            const __grid_constant__ MgOp F, const double *x,
                                                            const double *b, double *r, float *r32, float *y) {
  __shared__ double tab[PACKED ? 128 : 1];
  __shared__ float2 tab32[PACKED ? 128 : 1];
  mg_table64<PACKED>(A, tab);
  if (PACKED) mg_table(F, tab32);
  mg_pdl();
  const Column c = mg_column(A.d, zc);
  if (!c.in) return;
  const size_t pl = (size_t)A.d.pitch() * A.d.ny;
  V4<double> um = ld4_if(c.k0 > 0, x + (c.k0 - 1) * pl + c.o), uc = ld4(x + c.k0 * pl + c.o);
  for (int k = c.k0; k < c.k1; k++) {
    const size_t e = k * pl + c.o;
    const V4<double> up = ld4_if(k + 1 < A.d.nz, x + e + pl);
    const V4<double> a = mg_apply64<PACKED>(A, tab, x, c, k, um, uc, up);
    V4<double> v = ld4(b + ((size_t)k * A.d.ny + c.j) * A.px + c.i);  // pads are 0
#pragma unroll
    for (int q = 0; q < 4; q++) v.v[q] = __dsub_rn(v.v[q], a.v[q]);
    st4(r + e, v);
    if (r32) mg_rhs<PACKED>(F, tab32, c, k, e, v, r32, y);
    um = uc;
    uc = up;
  }
}
// x += alpha p, r -= alpha Ap, the V-cycle's right-hand side
template <bool PACKED>
__global__ void __launch_bounds__(MG_NT) k_mg_update(const __grid_constant__ MgOp F, int zc, const MgScal *S,
                                                     const double *p, const double *ap, double *x, double *r,
                                                     float *r32, float *y) {
  __shared__ float2 tab[PACKED ? 128 : 1];
  if (PACKED) mg_table(F, tab);
  mg_pdl();
  if (S->done) return;
  const Column c = mg_column(F.d, zc);
  if (!c.in) return;
  const size_t pl = (size_t)F.d.pitch() * F.d.ny;
  const double alpha = S->alpha;
  for (int k = c.k0; k < c.k1; k++) {
    const size_t e = k * pl + c.o;
    const V4<double> pv = ld4(p + e), av = ld4(ap + e);
    V4<double> xv = ld4(x + e), v = ld4(r + e);
#pragma unroll
    for (int q = 0; q < 4; q++) {
      xv.v[q] = fma(alpha, pv.v[q], xv.v[q]);
      v.v[q] = fma(-alpha, av.v[q], v.v[q]);
    }
    st4(x + e, xv);
    st4(r + e, v);
    mg_rhs<PACKED>(F, tab, c, k, e, v, r32, y);
  }
}
// p = z + beta p; first: p = z (no direction before).  n4: groups of four
__global__ void __launch_bounds__(MG_NT) k_mg_direction(size_t n4, const MgScal *S, int first, const float *z,
                                                        double *p) {
  mg_pdl();
  if (S->done) return;
  const double beta = S->beta;
  MG_LOOP(t, n4) {
    const V4<float> zv = ld4(z + 4 * t);
    V4<double> pv = {};
    if (!first) pv = ld4(p + 4 * t);
#pragma unroll
    for (int q = 0; q < 4; q++) pv.v[q] = fma(beta, pv.v[q], widen(zv.v[q]));
    st4(p + 4 * t, pv);
  }
}

}  // namespace pb

using namespace pb;

// ---------------------------------------------------------------------------
// Host side: the hierarchy of a grid, built on the first GMG solve.

struct pb_mg {
  int num_sms = 1;
  struct Level {
    MgDims d;
    double kbh2;
    double *ex64 = nullptr, *ey64 = nullptr, *ez64 = nullptr;
    uint8_t *lam = nullptr;
    float *cx = nullptr, *cy = nullptr, *cz = nullptr, *diag = nullptr, *rd = nullptr;
    float *z0 = nullptr, *z1 = nullptr, *r = nullptr, *res = nullptr;
    MgOp op;
  };
  std::vector<Level> lv;
  bool packed = false;      // level 0 from the grid's codes
  MgOp64 op64;              // level 0 in FP64
  size_t tail = 0;          // first level of the one-CTA kernel (lv.size(): none)
  MgTail T;                 // its levels
  float *block = nullptr;   // ... and coefficients
  void *slab = nullptr;     // every array above and below
  double *x = nullptr, *r = nullptr, *p = nullptr, *ap = nullptr, *part = nullptr;
  MgScal *S = nullptr;      // device scalars of the outer CG
  MgScal *hS = nullptr;     // pinned host copy
  // graph of MG_GRAPH_ITERS outer iterations (captured on the first solve)
  cudaGraphExec_t graph = nullptr;
  unsigned long long graph_launches = 0;  // kernels per graph launch
};

void pb_mg_release(pb_mg *m) {
  if (!m) return;
  if (m->graph) cudaGraphExecDestroy(m->graph);
  if (m->hS) cudaFreeHost(m->hS);
  if (m->slab) cudaFree(m->slab);
  delete m;
}

// Launch with programmatic stream serialization (mg_pdl in the kernels).
template <typename... Params, typename... Args>
static void mg_launch(void (*k)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k, Params(args)...);
}

static pb_status mg_build(pb_grid *g, pb_mg **out) {
  cudaStream_t s = g->ctx->stream;
  pb_mg *m = new pb_mg();
  m->num_sms = g->ctx->num_sms;
  auto fail = [&](pb_status st) {
    pb_mg_release(m);
    return st;
  };
  MgDims d{g->d.nx, g->d.ny, g->d.nz};
  double kbh2 = g->kbh2;
  while (true) {
    pb_mg::Level L;
    L.d = d;
    L.kbh2 = kbh2;
    m->lv.push_back(L);
    if (std::min(d.nx, std::min(d.ny, d.nz)) <= MG_COARSEST) break;
    d = MgDims{(d.nx + 1) / 2, (d.ny + 1) / 2, (d.nz + 1) / 2};
    kbh2 *= 4.0;  // kbar^2 (2h)^2
  }
  m->packed = g->d.eps_model == PB_EPS_MIDPOINT;  // the codes are the operator
  // the one-CTA end of the V-cycle: as many of the last levels as its shared
  // memory holds (never level 0, whose last sweep forms r.z)
  m->tail = m->lv.size();
  while (m->tail > 1 && m->lv.size() - m->tail < (size_t)MG_TAIL_MAX) {
    MgTail T = {};
    T.n = (int)(m->lv.size() - (m->tail - 1));
    size_t nodes = 0;
    for (int t = 0; t < T.n; t++) {
      T.lv[t].d = m->lv[m->tail - 1 + t].d;
      nodes += T.lv[t].d.nodes();
    }
    if (nodes > 20000) break;  // (more than any shared memory holds; keeps the offsets small)
    mg_tail_layout(T);
    if ((size_t)T.all * 4 > (size_t)g->ctx->max_smem) break;
    m->tail--;
    m->T = T;
  }
  if (m->tail < m->lv.size() && allow_all_smem(k_mg_tail) != cudaSuccess) {
    cudaGetLastError();
    m->tail = m->lv.size();
  }
  // one allocation, carved: first the sizes, then the pointers
  const size_t n = m->lv[0].d.padded();
  for (int pass = 0; pass < 2; pass++) {
    size_t off = 0;
    auto take = [&](auto *&p, size_t bytes) {
      if (pass) p = (std::remove_reference_t<decltype(p)>)((char *)m->slab + off);
      off += (bytes + 255) / 256 * 256;
    };
    for (size_t l = 0; l < m->lv.size(); l++) {
      pb_mg::Level &L = m->lv[l];
      const MgDims &q = L.d;
      take(L.ex64, q.nex() * 8); take(L.ey64, q.ney() * 8); take(L.ez64, q.nez() * 8);
      take(L.lam, q.nodes());
      if (l > 0 || !m->packed) {
        take(L.cx, q.padded() * 4); take(L.cy, q.padded() * 4); take(L.cz, q.padded() * 4);
        take(L.diag, q.padded() * 4); take(L.rd, q.padded() * 4);
      }
      take(L.z0, q.padded() * 4); take(L.z1, q.padded() * 4);
      take(L.r, q.padded() * 4); take(L.res, q.padded() * 4);
    }
    if (m->tail < m->lv.size()) take(m->block, (size_t)m->T.coef * 4);
    take(m->x, n * 8); take(m->r, n * 8); take(m->p, n * 8); take(m->ap, n * 8);
    take(m->part, MG_DOT_CTAS * 8);
    take(m->S, sizeof(MgScal));
    if (!pass) {
      const pb_status st = pb_dalloc(&m->slab, off);
      if (st) return fail(st);
    }
  }
  if (cudaMallocHost((void **)&m->hS, sizeof(MgScal)) != cudaSuccess) {
    cudaGetLastError();
    m->hS = nullptr;
    return fail(pb_fail(PB_ERR_OOM, "multigrid: pinned scalars"));
  }
  // level 0 from the grid, then coarsen
  const pb_mg::Level &L0 = m->lv[0];
  k_mg_level0<<<mg_blocks(L0.d.nex()), MG_NT, 0, s>>>(
      L0.d, g->g.px, g->code, (const double *)g->ex64, (const double *)g->ey64, (const double *)g->ez64,
      g->d.eps_in, g->d.eps_out, L0.ex64, L0.ey64, L0.ez64, L0.lam);
  unsigned long long launches = 1;
  for (size_t l = 0; l + 1 < m->lv.size(); l++) {
    const pb_mg::Level &F = m->lv[l], &C = m->lv[l + 1];
    k_mg_coarsen<<<mg_blocks(C.d.nex()), MG_NT, 0, s>>>(F.d, C.d, F.ex64, F.ey64, F.ez64, F.lam, C.ex64,
                                                        C.ey64, C.ez64, C.lam);
    launches++;
  }
  for (const pb_mg::Level &L : m->lv) {
    if (L.cx) {
      k_mg_finish<<<mg_blocks(L.d.padded()), MG_NT, 0, s>>>(L.d, L.kbh2, L.ex64, L.ey64, L.ez64, L.lam, L.cx, L.cy,
                                                            L.cz, L.diag, L.rd);
      launches++;
    }
    cudaMemsetAsync(L.z1, 0, L.d.padded() * 4, s);  // row pads that no kernel writes
  }
  for (size_t l = m->tail; l < m->lv.size(); l++) {
    const pb_mg::Level &L = m->lv[l];
    k_mg_tail_pack<<<8, MG_NT, 0, s>>>(m->T.lv[l - m->tail], L.cx, L.cy, L.cz, L.diag, L.rd, m->block);
    launches++;
  }
  cudaMemsetAsync(m->x, 0, n * 8, s);
  g->ctx->stats->launches += launches;
  if (cudaGetLastError() != cudaSuccess) return fail(pb_fail(PB_ERR_CUDA, "multigrid setup kernels"));
  // operators
  double dt[NDTAB];
  for (int nin = 0; nin <= 6; nin++)
    for (int lam = 0; lam <= 1; lam++) {
      double v = 0;
      for (int t = 0; t < 6; t++) v = v + (t < nin ? g->d.eps_in : g->d.eps_out);
      dt[2 * nin + lam] = v + g->kbh2 * lam;
    }
  for (size_t l = 0; l < m->lv.size(); l++) {
    pb_mg::Level &L = m->lv[l];
    MgOp &A = L.op;
    A = MgOp{};
    A.d = L.d;
    A.cx = L.cx; A.cy = L.cy; A.cz = L.cz; A.diag = L.diag; A.rd = L.rd;
    if (l == 0 && m->packed) {
      A.code = g->code;
      A.px = g->g.px;
      A.ein = (float)g->d.eps_in;
      A.eout = (float)g->d.eps_out;
      for (int t = 0; t < NDTAB; t++) {
        A.dt[t] = (float)dt[t];
        A.rt[t] = 1.0f / A.dt[t];
      }
    }
  }
  MgOp64 &D = m->op64;
  D = MgOp64{};
  D.d = L0.d;
  D.px = g->g.px;
  D.code = g->code;
  D.ex = (const double *)g->ex64; D.ey = (const double *)g->ey64; D.ez = (const double *)g->ez64;
  D.diag = (const double *)g->diag64;
  D.ein = g->d.eps_in;
  D.eout = g->d.eps_out;
  for (int t = 0; t < NDTAB; t++) D.dt[t] = dt[t];
  if (m->tail < m->lv.size()) {
    const pb_mg::Level &L = m->lv[m->tail];
    m->T.block = m->block;
    m->T.r = L.r;
    m->T.y = L.z0;
    m->T.z = L.z1;
  }
  *out = m;
  return PB_OK;
}

// Launch a column kernel over a level (its planes-a-column argument second).
template <typename A0, typename... Params, typename... Args>
static void mg_columns(const pb_mg *m, const MgDims &d, cudaStream_t s, unsigned long long &launches,
                       void (*k)(A0, int, Params...), const A0 &a0, Args... args) {
  const MgLaunch L = mg_plan(k, d, m->num_sms);
  mg_launch(k, dim3(L.ctas), MG_NT, 0, s, a0, L.zc, args...);
  launches++;
}
// ... of the two builds by operator storage
#define MG_BY_STORAGE(L, K, ...)                                                     \
  do {                                                                               \
    if ((L).op.code) mg_columns(m, (L).d, s, launches, K<true>, (L).op, __VA_ARGS__); \
    else mg_columns(m, (L).d, s, launches, K<false>, (L).op, __VA_ARGS__);           \
  } while (0)

// One sweep of a level.
static void mg_sweep(const pb_mg *m, const pb_mg::Level &L, const float *u, float *out, cudaStream_t s,
                     unsigned long long &launches) {
  MG_BY_STORAGE(L, k_mg_sweep, m->S, u, L.r, out);
}

// z_l = V(r_l) on level l, from L.r and its first sweep in L.z0; the result in L.z1.
static void vcycle(pb_mg *m, size_t l, cudaStream_t s, unsigned long long &launches) {
  pb_mg::Level &L = m->lv[l];
  if (l == m->tail) {  // the rest in one CTA
    mg_launch(k_mg_tail, dim3(1), MG_TAIL_NT, (size_t)m->T.all * 4, s, m->T, m->S);
    launches++;
    return;
  }
  const bool coarsest = l + 1 == m->lv.size();
  if (coarsest) {  // sweeps from zero: z0 is the first one; the last ends in z1
    for (int t = 1; t < MG_COARSE_SWEEPS; t++)
      mg_sweep(m, L, t & 1 ? L.z0 : L.z1, t & 1 ? L.z1 : L.z0, s, launches);
    return;
  }
  // pre-smoothing: z1 = S(S(0))
  mg_sweep(m, L, L.z0, L.z1, s, launches);
  pb_mg::Level &C = m->lv[l + 1];
  MG_BY_STORAGE(L, k_mg_residual, m->S, L.z1, L.r, L.res);
  mg_columns(m, C.d, s, launches, k_mg_restrict, C.d, L.d, m->S, L.res, C.diag, C.rd, C.r, C.z0);
  vcycle(m, l + 1, s, launches);
  mg_columns(m, L.d, s, launches, k_mg_prolong_add, L.d, C.d, m->S, C.z1, L.z1);
  // post-smoothing: z0 = S(z1), z1 = S(z0)
  mg_sweep(m, L, L.z1, L.z0, s, launches);
  mg_sweep(m, L, L.z0, L.z1, s, launches);
}

// The preconditioned CG of Sec. 2.2 with z = V(r), in FP64.  Its scalars
// stay on the device (MgScal), formed by the last CTA of the dot product they
// need: after the first direction, the host launches a CUDA graph of
// MG_GRAPH_ITERS iterations (the operator, the updates, a V-cycle and the
// direction each: 25 kernels at 129^3) and reads the scalars once per graph;
// kernels after convergence return at once.  Called by pb_pcg_solve for
// PB_PRECOND_GMG.
//
// Measured, an iteration at 33^3 / 129^3 / 257^3: 83 / 205 / 1,050 us.  With
// every sweep, transfer, dot product and scalar a kernel of its own, a node a
// thread (74 launches), and explicit coefficients on every level: 122 / 287 /
// 1,524 us.  What bounds it now: the FP64 work of the outer CG (13 operations a
// node, 44 us at 129^3), the passes over its FP64 vectors, and the launches of
// the levels of 65^3 and 33^3.
#ifndef MG_GRAPH_ITERS
#define MG_GRAPH_ITERS 4
#endif
pb_status pb_gmg_solve(pb_grid *g, const pb_solve_opts *o, double *phi, pb_solve_info *info) {
  cudaStream_t s = g->ctx->stream;
  if (!g->mg) {
    pb_status st = mg_build(g, &g->mg);
    if (st) return st;
  }
  pb_mg *m = g->mg;
  const pb_mg::Level &L0 = m->lv[0];
  const size_t n = L0.d.padded();
  const int nx = L0.d.nx, ny = L0.d.ny, nz = L0.d.nz, P = L0.d.pitch();
  unsigned long long launches = 0, n_reads = 0;
  pb_status st;
  MgScal *S = m->S, *hS = m->hS;
  float *r32 = L0.r, *y = L0.z0;
  auto read_scal = [&]() -> pb_status {  // *hS = *S
    CK(cudaMemcpyAsync(hS, S, sizeof(MgScal), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    n_reads++;
    return PB_OK;
  };
  // r = b - A x, S->rr = ||r||^2; r32: also the V-cycle's input
  auto true_residual = [&](double *r, float *r32) {
    if (m->packed)
      mg_columns(m, L0.d, s, launches, k_mg_true_residual<true>, m->op64, L0.op, m->x, g->b, r, r32, y);
    else
      mg_columns(m, L0.d, s, launches, k_mg_true_residual<false>, m->op64, L0.op, m->x, g->b, r, r32, y);
    mg_launch(k_mg_dot<DOT_RR, double>, dim3(MG_DOT_CTAS), MG_NT, 0, s, L0.d, S, r, r, m->part);
    launches++;
  };
  auto beta = [&]() {  // r.z and beta
    mg_launch(k_mg_dot<DOT_BETA, float>, dim3(MG_DOT_CTAS), MG_NT, 0, s, L0.d, S, m->r, L0.z1, m->part);
    launches++;
  };
  auto direction = [&](int first) {
    mg_launch(k_mg_direction, dim3(mg_blocks(n / 4)), MG_NT, 0, s, n / 4, S, first, L0.z1, m->p);
    launches++;
  };
  // One outer iteration, from p, r and rz: alpha, x and r, the stop test,
  // z = V(r), beta, p.
  auto iteration = [&]() {
    if (m->packed) mg_columns(m, L0.d, s, launches, k_mg_apply<true>, m->op64, S, m->p, m->ap);
    else mg_columns(m, L0.d, s, launches, k_mg_apply<false>, m->op64, S, m->p, m->ap);
    mg_launch(k_mg_dot<DOT_ALPHA, double>, dim3(MG_DOT_CTAS), MG_NT, 0, s, L0.d, S, m->p, m->ap, m->part);
    MG_BY_STORAGE(L0, k_mg_update, S, m->p, m->ap, m->x, m->r, r32, y);
    mg_launch(k_mg_dot<DOT_STOP, double>, dim3(MG_DOT_CTAS), MG_NT, 0, s, L0.d, S, m->r, m->r, m->part);
    launches += 2;
    vcycle(m, 0, s, launches);
    beta();
    direction(0);
  };
  // x0 = phi (warm start) or 0; r = b - A x0
  if (o->warm_start) {
    CK(launch_pack(phi, m->x, nx, ny, nz, P, s));  // (the row pads stay 0)
    launches++;
  } else {
    CK(cudaMemsetAsync(m->x, 0, n * 8, s));
  }
  const double bnorm = g->bnorm;
  MgScal h0;
  memset(&h0, 0, sizeof(h0));
  h0.stop2 = (o->rel_tol * bnorm) * (o->rel_tol * bnorm);
  h0.max_iter = o->max_iter;
  h0.status = PB_ERR_NOT_CONVERGED;
  h0.rz = 1.0;
  *hS = h0;
  CK(cudaMemcpyAsync(S, hS, sizeof(MgScal), cudaMemcpyHostToDevice, s));
  true_residual(m->r, r32);
  CK(cudaGetLastError());
  if ((st = read_scal())) return st;
  double rel = bnorm > 0 ? std::sqrt(hS->rr) / bnorm : 0.0;
  int it = 0, status = PB_OK;
  if (bnorm == 0.0) {
    CK(cudaMemsetAsync(m->x, 0, n * 8, s));
    rel = 0.0;
  } else if (!(rel < o->rel_tol) && o->max_iter > 0) {
    vcycle(m, 0, s, launches);
    beta();
    direction(1);
    CK(cudaGetLastError());
    if (!m->graph) {  // capture MG_GRAPH_ITERS iterations
      cudaGraph_t graph = nullptr;
      CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
      const unsigned long long before = launches;
      for (int k = 0; k < MG_GRAPH_ITERS; k++) iteration();
      const cudaError_t e = cudaGetLastError();
      m->graph_launches = launches - before;
      launches = before;  // counted when the graph runs
      const cudaError_t e2 = cudaStreamEndCapture(s, &graph);
      if (e != cudaSuccess || e2 != cudaSuccess) {
        if (graph) cudaGraphDestroy(graph);
        return pb_fail(PB_ERR_CUDA, std::string("multigrid graph capture: ") +
                                        cudaGetErrorString(e != cudaSuccess ? e : e2));
      }
      const cudaError_t e3 = cudaGraphInstantiate(&m->graph, graph, 0);
      cudaGraphDestroy(graph);
      if (e3 != cudaSuccess) {
        m->graph = nullptr;
        return pb_fail(PB_ERR_CUDA, std::string("multigrid graph: ") + cudaGetErrorString(e3));
      }
    }
    while (true) {
      CK(cudaGraphLaunch(m->graph, s));
      launches += m->graph_launches;
      if ((st = read_scal())) return st;
      if (hS->done) break;
    }
    it = hS->it;
    status = hS->status;
    rel = std::sqrt(hS->rr) / bnorm;
  } else if (!(rel < o->rel_tol)) {
    status = PB_ERR_NOT_CONVERGED;
  }
  // true residual of the result, then phi = x
  true_residual(m->ap, nullptr);
  CK(cudaGetLastError());
  CK(launch_unpack(m->x, phi, nx, ny, nz, P, s));
  launches++;
  if ((st = read_scal())) return st;
  const double rr_true = hS->rr;
  g->ctx->stats->launches += launches;
  g->ctx->stats->h2d += sizeof(MgScal);
  g->ctx->stats->d2h += sizeof(MgScal) * n_reads;
  if (info) {
    info->status = status;
    info->iterations = it;
    info->outer_steps = 1;
    info->relres = rel;
    info->relres_true = bnorm > 0 ? std::sqrt(rr_true) / bnorm : 0.0;
  }
  return status == PB_OK ? PB_OK : pb_fail(status, status == PB_ERR_BREAKDOWN ? "CG breakdown" : "not converged");
}
