// ops.cu -- helper kernels of libpb: dense <-> padded copies, the operator
// applied to a dense vector (Eq. 3-4), and the electrostatic energy.
#include <algorithm>

#include "coef.cuh"
#include "pb_internal.cuh"
#include "solve.cuh"

namespace pb {

static int blocks_for(size_t n, int nt) {
  size_t b = (n + nt - 1) / nt;
  return (int)(b < 152 * 32 ? (b ? b : 1) : 152 * 32);
}

// Node indices split in 32-bit arithmetic: a grid has at most 2e9 nodes
// (checked when it is created), and 32-bit division costs a fraction of
// 64-bit division per node.
__device__ __forceinline__ size_t padded_of(size_t t, int nx, int px) {
  const uint32_t tt = (uint32_t)t, row = tt / (uint32_t)nx;
  return (size_t)row * px + (tt - row * (uint32_t)nx);
}
__global__ void k_pack(const double *dense, double *padded, int nx, int ny, int nz, int px) {
  const size_t n = (size_t)nx * ny * nz;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n;
       t += (size_t)gridDim.x * blockDim.x)
    padded[padded_of(t, nx, px)] = dense[t];
}
__global__ void k_unpack(const double *padded, double *dense, int nx, int ny, int nz, int px) {
  const size_t n = (size_t)nx * ny * nz;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n;
       t += (size_t)gridDim.x * blockDim.x)
    dense[t] = padded[padded_of(t, nx, px)];
}

cudaError_t launch_pack(const double *dense, double *padded, int nx, int ny, int nz, int px,
                        cudaStream_t st) {
  k_pack<<<blocks_for((size_t)nx * ny * nz, 256), 256, 0, st>>>(dense, padded, nx, ny, nz, px);
  return cudaGetLastError();
}
cudaError_t launch_unpack(const double *padded, double *dense, int nx, int ny, int nz, int px,
                          cudaStream_t st) {
  k_unpack<<<blocks_for((size_t)nx * ny * nz, 256), 256, 0, st>>>(padded, dense, nx, ny, nz, px);
  return cudaGetLastError();
}

// (A u)_c = diag_c u_c - sum_nb eps_edge u_nb, ghosts zero; dense u and Au.
// Bound by the call on small grids (the descriptor travels as a kernel argument:
// uploading it first cost more than the kernel), by FP64 arithmetic or DRAM on
// large ones: a thread walks kz nodes of a z column, so that the index divisions
// are two a column and u is read five times a node instead of seven; CTAs run on
// into the next planes at a plane's end (3x3x20000 nodes, FP64, 34 -> 24 us).  Measured, a
// call, against the uploaded descriptor and one node a thread: 33^3 14.5 -> 12.7 us;
// 257^3 FP64 218 -> 216, FP32 packed 94 -> 77, BF16 112 -> 94, FP32 109 -> 97 (packed:
// kz = 16 and 1 94 and 133; explicit storage: two nodes in flight 110 .. 138).  Six
// CTAs an SM: left alone the compiler takes registers for fewer, 168.
template <typename T, int CM>
__global__ void __launch_bounds__(256, 6) k_apply(const __grid_constant__ Inst I,
                                                  const T *__restrict__ u,
                                                  T *__restrict__ au, int kz) {
  constexpr int UNROLL = CM == COEF_PACKED ? 2 : 1;
  const int nx = I.nx, ny = I.ny, nz = I.nz;
  const uint32_t plane = (uint32_t)nx * ny, t = blockIdx.x * 256u + threadIdx.x;
  const uint32_t run = t / plane, p = t - run * plane;  // run of kz planes, place in a plane
  const long k0 = (long)run * kz;
  if (k0 >= nz) return;
  const int j = (int)(p / (uint32_t)nx), i = (int)(p - (uint32_t)j * nx);
  const bool per = I.periodic != 0;
  // offsets of the in-plane neighbours (with wrap: modulo n)
  const long xm = i > 0 ? -1 : nx - 1, xp = i < nx - 1 ? 1 : 1 - nx;
  const long ym = j > 0 ? -nx : (long)plane - nx, yp = j < ny - 1 ? nx : nx - (long)plane;
  const bool has_xm = per || i > 0, has_xp = per || i < nx - 1, has_ym = per || j > 0, has_yp = per || j < ny - 1;
  const int k1 = (int)(k0 + kz < nz ? k0 + kz : nz);
  const T *uk = u + (size_t)k0 * plane + p;
  T *ak = au + (size_t)k0 * plane + p;
  size_t e = ((size_t)k0 * ny + j) * I.px + i;
  T below = 0, here = *uk;
  if (k0 > 0) below = uk[-(long)plane];
  else if (per) below = u[(size_t)(nz - 1) * plane + p];
#pragma unroll UNROLL
  for (int k = (int)k0; k < k1; k++) {
    T above = 0;
    if (k < nz - 1) above = uk[plane];
    else if (per) above = u[p];
    const NodeCoef<T> c = node_coef<T, CM>(I, e, k);
    T s = 0;
    if (has_xm) s += c.exm * uk[xm];
    if (has_xp) s += c.exp * uk[xp];
    if (has_ym) s += c.eym * uk[ym];
    if (has_yp) s += c.eyp * uk[yp];
    if (per || k > 0) s += c.ezm * below;
    if (per || k < nz - 1) s += c.ezp * above;
    *ak = c.diag * here - s;
    below = here;
    here = above;
    uk += plane;
    ak += plane;
    e += (size_t)I.px * ny;
  }
}

cudaError_t launch_apply(const Inst &I, const void *u, void *au, int dtype, int num_sms, cudaStream_t st) {
  // columns of up to 4 nodes while that leaves eight CTAs an SM and more
  const long plane = (long)I.nx * I.ny;
  const int kz = (int)std::max(1l, std::min(4l, plane * I.nz / (256l * 16l * num_sms)));
  const unsigned blocks = (unsigned)((plane * ((I.nz + kz - 1) / kz) + 255) / 256);
  if (dtype == 0) {  // FP64: exact coefficients
    if (I.coef == COEF_F64)
      k_apply<double, COEF_F64><<<blocks, 256, 0, st>>>(I, (const double *)u, (double *)au, kz);
    else
      k_apply<double, COEF_PACKED><<<blocks, 256, 0, st>>>(I, (const double *)u, (double *)au, kz);
  } else {
    if (I.coef == COEF_F32)
      k_apply<float, COEF_F32><<<blocks, 256, 0, st>>>(I, (const float *)u, (float *)au, kz);
    else if (I.coef == COEF_BF16)
      k_apply<float, COEF_BF16><<<blocks, 256, 0, st>>>(I, (const float *)u, (float *)au, kz);
    else
      k_apply<float, COEF_PACKED><<<blocks, 256, 0, st>>>(I, (const float *)u, (float *)au, kz);
  }
  return cudaGetLastError();
}

// Energy: 1/2 * 332.0637 * sum_a q_a * (trilinear interpolation of phi at x_a)
// with the weights of the charge spreading, so it equals 1/2 * 332.0637 *
// sum_nodes q_node phi_node up to rounding order.  Per-CTA partials, then one
// CTA sums them in order (deterministic).
constexpr int EN_NT = 256;
// px: row pitch of phi in elements (nx for a dense array).  An atom whose
// trilinear cell leaves the grid reads nothing and makes the energy NaN; on a
// periodic grid the cell's corners wrap modulo n.
__global__ void k_energy_partial(const dbl4 *xyzq, int n_atoms, int nx, int ny, int nz, int px,
                                 int periodic, double h, double ox, double oy, double oz,
                                 const double *phi, double *part) {
  __shared__ double red[EN_NT];
  double acc = 0.0;
  const int a = blockIdx.x * EN_NT + threadIdx.x;
  if (a < n_atoms) {
    const dbl4 A = xyzq[a];
    const double f[3] = {__ddiv_rn(__dsub_rn(A.x, ox), h), __ddiv_rn(__dsub_rn(A.y, oy), h),
                         __ddiv_rn(__dsub_rn(A.z, oz), h)};
    double w[3][2];
    long c0[3];
    const long n[3] = {nx, ny, nz};
    bool inside = true;
    for (int d = 0; d < 3; d++) {
      const double fl = floor(f[d]);
      c0[d] = (long)fl;
      w[d][1] = __dsub_rn(f[d], fl);
      w[d][0] = __dsub_rn(1.0, w[d][1]);
      // the cell's upper corner may be the last node only when its weight is 0
      if (periodic) inside = inside && isfinite(fl);
      else inside = inside && fl >= 0.0 && (c0[d] + 1 < n[d] || (c0[d] + 1 == n[d] && w[d][1] == 0.0));
    }
    if (!inside) {
      acc = __longlong_as_double(0x7ff8000000000000LL);  // NaN
    } else {
      for (int dk = 0; dk < 2; dk++)
        for (int dj = 0; dj < 2; dj++)
          for (int di = 0; di < 2; di++) {
            const double c = __dmul_rn(__dmul_rn(__dmul_rn(A.w, w[0][di]), w[1][dj]), w[2][dk]);
            long ci = c0[0] + di, cj = c0[1] + dj, ck = c0[2] + dk;
            if (periodic) {
              ci = ((ci % nx) + nx) % nx;
              cj = ((cj % ny) + ny) % ny;
              ck = ((ck % nz) + nz) % nz;
            } else if (ci >= nx || cj >= ny || ck >= nz) {
              continue;  // weight 0
            }
            const size_t t = ((size_t)ck * ny + cj) * px + ci;
            acc += c * phi[t];
          }
    }
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int s = EN_NT / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}
__global__ void k_energy_final(const double *part, int n, double *out) {
  __shared__ double red[EN_NT];
  double s = 0.0;
  for (int t = threadIdx.x; t < n; t += EN_NT) s += part[t];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = EN_NT / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = 0.5 * 332.0637 * red[0];
}

cudaError_t launch_energy(const dbl4 *xyzq, int n_atoms, int nx, int ny, int nz, int px,
                          int periodic, double h, double ox, double oy, double oz,
                          const double *phi, double *scratch, double *out, cudaStream_t st) {
  const int blocks = n_atoms > 0 ? (n_atoms + EN_NT - 1) / EN_NT : 0;
  if (blocks > 0)
    k_energy_partial<<<blocks, EN_NT, 0, st>>>(xyzq, n_atoms, nx, ny, nz, px, periodic, h, ox, oy,
                                               oz, phi, scratch);
  k_energy_final<<<1, EN_NT, 0, st>>>(scratch, blocks, out);
  return cudaGetLastError();
}

}  // namespace pb
