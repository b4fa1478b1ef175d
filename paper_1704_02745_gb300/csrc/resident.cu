// resident.cu -- one inner CG solve (Sec. 2.2 preconditioned CG, Sec. 2.4
// Jacobi, operator of Eq. 3-4) of a grid in one cooperative kernel that keeps
// the vectors on the chip; and of several grids of a batch side by side.
//
// What bounds the two-pass form (solve.cu) on one grid is not its bytes: a
// 129^3 iteration moves 82 MB, 12 us at the measured copy rate, and takes 40
// us; a 33^3 iteration moves 1.4 MB and takes 28 us.  Launches, pipeline fills
// and half-empty waves set the time.  A grid of a few million nodes fits the
// SMs' registers and shared memory, so here a CTA owns a brick of the grid
// for the whole inner solve (measured, us an iteration: 33^3 28 -> 6, 97^3
// 35 -> 8, 129^3 40 -> 13.3, 187x161x175 58 -> 38, FP64 129^3 147 -> 79):
//   - brick = all of x, by rows, kn planes; a thread owns one group of NV = 4
//     x nodes and its kn planes.  p sits in shared memory with a one-node halo
//     in y and z; z and the increment d in the thread's registers and Ap in
//     shared memory (G > 0), or all three in the grid's arrays, that is in L2
//     (G = 0: larger bricks, FP64).  A brick at 12 x 11 of a 129^3 grid: 93 KB
//     of p, 74 KB of Ap and codes, 96 of 168 registers.
//   - an iteration is p = z + beta p (halo cells included: a CTA reads its
//     neighbours' boundary z and keeps its own copy of their p), Ap and p.Ap;
//     a grid-wide sum; r = M z - alpha Ap, z = M^-1 r, r.z, r.r, the
//     boundary z written out; a grid-wide sum.  The same operations per node
//     as cg_tile, up to the order in which a surface node's six edges are
//     added; the partial sums are grouped by brick.
//   - the grid-wide sum is the barrier: each CTA stores its sum and an epoch as
//     one 16-byte word in a line of its own, and every CTA polls all CTAs'
//     words, one thread each, and adds them in CTA order, so every CTA holds
//     the same scalars after one trip through L2 and takes the same decisions.
//     Measured with 152 CTAs: 1,830 cycles (words side by side 4,060; pushed to
//     152 mailboxes 2,800; through a master CTA 2,600; clusters of 4 and their
//     leaders 3,900).  Polls are bounded: a CTA that gives up sets the error
//     word, the others leave on seeing it, and the host starts the solve over in
//     phase ticks, which need no CTA to run beside another.
//   - the scalars stay off the FP64 pipe in FP32 solves (a warp's FP64 add takes
//     19 cycles of an SM, a division 2,270 over 16 warps): sums and quotients
//     are unevaluated pairs of floats (48 bits and more).
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>
#include <iterator>
#include <type_traits>

#include "coef.cuh"
#include "pb_internal.cuh"
#include "resident.cuh"

namespace pb {

// ---------------------------------------------------------------------------
// Sums and scalars: FP64 for FP64 solves, pairs of floats (hi + lo, |lo| at
// most half an ulp of hi) for FP32 solves, whose terms are floats.

template <typename T> struct Sum;
template <> struct Sum<double> { double v; };
template <> struct Sum<float> { float h, l; };

__device__ __forceinline__ Sum<double> sum_of(double v) { return Sum<double>{v}; }
__device__ __forceinline__ Sum<float> sum_of(float v) { return Sum<float>{v, 0.f}; }
__device__ __forceinline__ Sum<double> add(Sum<double> a, Sum<double> b) { return Sum<double>{a.v + b.v}; }
// Knuth's error-free two-sum of the leading parts, then one renormalisation
__device__ __forceinline__ Sum<float> add(Sum<float> a, Sum<float> b) {
  const float s = __fadd_rn(a.h, b.h), t = __fsub_rn(s, a.h);
  float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
  e = __fadd_rn(e, __fadd_rn(a.l, b.l));
  const float h = __fadd_rn(s, e);
  return Sum<float>{h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ Sum<double> quotient(Sum<double> a, Sum<double> b) { return Sum<double>{a.v / b.v}; }
__device__ __forceinline__ Sum<float> quotient(Sum<float> a, Sum<float> b) {
  const float y = __frcp_rn(b.h), q = a.h * y;
  float r = fmaf(-q, b.h, a.h);  // exact: q is within two ulps of a.h / b.h
  r = __fadd_rn(r, fmaf(-q, b.l, a.l));
  const float q2 = r * y, h = __fadd_rn(q, q2);
  return Sum<float>{h, __fsub_rn(q2, __fsub_rn(h, q))};
}
__device__ __forceinline__ double value(Sum<double> a) { return a.v; }
__device__ __forceinline__ double value(Sum<float> a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ double lead(Sum<double> a) { return a.v; }
__device__ __forceinline__ float lead(Sum<float> a) { return a.h; }
__device__ __forceinline__ bool below(Sum<double> a, Sum<double> b) { return a.v < b.v; }
__device__ __forceinline__ bool below(Sum<float> a, Sum<float> b) { return a.h < b.h || (a.h == b.h && a.l < b.l); }
template <typename T> __device__ __forceinline__ Sum<T> from_double(double v);
template <> __device__ __forceinline__ Sum<double> from_double<double>(double v) { return Sum<double>{v}; }
template <> __device__ __forceinline__ Sum<float> from_double<float>(double v) {
  const float h = (float)v;
  return Sum<float>{h, (float)(v - (double)h)};
}
// Running sums: like add(), without the renormalisation (settle() does it
// once at the end), which leaves one addition and a shuffle in the chain.
__device__ __forceinline__ void gather(Sum<double> &a, Sum<double> b) { a.v += b.v; }
__device__ __forceinline__ void gather(Sum<float> &a, Sum<float> b) {
  const float s = __fadd_rn(a.h, b.h), t = __fsub_rn(s, a.h);
  const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
  a.l = __fadd_rn(__fadd_rn(a.l, b.l), e);
  a.h = s;
}
__device__ __forceinline__ void settle(Sum<double> &) {}
__device__ __forceinline__ void settle(Sum<float> &a) {
  const float h = __fadd_rn(a.h, a.l);
  a.l = __fsub_rn(a.l, __fsub_rn(h, a.h));
  a.h = h;
}
__device__ __forceinline__ Sum<double> shfl_xor(Sum<double> a, int o) {
  return Sum<double>{__shfl_xor_sync(0xffffffffu, a.v, o)};
}
__device__ __forceinline__ Sum<float> shfl_xor(Sum<float> a, int o) {
  return Sum<float>{__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o)};
}
// a[0] += a[1] + ... + a[C - 1], as a tree (C a power of two).
template <typename T, int C>
__device__ __forceinline__ void tree_sum(Sum<T> (&a)[C]) {
#pragma unroll
  for (int o = 1; o < C; o *= 2)
#pragma unroll
    for (int j = 0; j < C; j += 2 * o) gather(a[j], a[j + o]);
}
// Sum over the warp, the same bits in every lane (a two-sum's error is exact,
// so its operands' order does not matter).
template <typename T, int N>
__device__ __forceinline__ void warp_sum(Sum<T> (&a)[N]) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int n = 0; n < N; n++) gather(a[n], shfl_xor(a[n], o));
#pragma unroll
  for (int n = 0; n < N; n++) settle(a[n]);
}

// ---------------------------------------------------------------------------
// The words CTAs exchange: a sum and its epoch in one 16-byte access.

struct alignas(16) Packet { unsigned long long a, b; };
constexpr int PACKET_STRIDE = 16;  // packets (256 bytes) between CTAs' words

__device__ __forceinline__ void packet_store(Packet *p, unsigned long long a, unsigned long long b) {
  asm volatile("{\n .reg .b128 q;\n mov.b128 q, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], q;\n}\n" ::"l"(p),
               "l"(a), "l"(b)
               : "memory");
}
__device__ __forceinline__ Packet packet_load(const Packet *p) {
  Packet r;
  asm volatile("{\n .reg .b128 q;\n ld.relaxed.gpu.global.b128 q, [%2];\n mov.b128 {%0, %1}, q;\n}\n"
               : "=l"(r.a), "=l"(r.b)
               : "l"(p)
               : "memory");
  return r;
}
__device__ __forceinline__ unsigned long long bits(float lo, uint32_t hi) {
  return (unsigned long long)__float_as_uint(lo) | ((unsigned long long)hi << 32);
}
// Float sums travel in one word: one sum as {h, l, epoch}; two as {h0, l0, h1,
// the upper 24 bits of l1 (16 bits of it: the sum, r.r, to 2^-41) and 8 bits of the
// iteration's number (a word holds the previous epoch of its kind until it is
// rewritten, 0 before the first, which is 1).  The sums' FP32 terms are off by 1e-10
// to 4e-9 of the sum, as measured against FP64 over 2,000 to 78,000 threads of 1 to 48
// planes, the pairs by 4e-15, the word by 5e-13; with a word each, in full, an
// iteration of 33^3 takes 6.1 us for 5.7, of 129^3 12.3 for 11.8.
// Double sums take a word each, side by side.
template <int N>
__device__ __forceinline__ void wire_store(Packet *p, const Sum<float> (&s)[N], uint32_t epoch) {
  if constexpr (N == 1) {
    packet_store(p, bits(s[0].h, __float_as_uint(s[0].l)), epoch);
  } else {
    const uint32_t t = (__float_as_uint(s[1].l) & 0xFFFFFF00u) | (epoch >> 1 & 0xFFu);
    packet_store(p, bits(s[0].h, __float_as_uint(s[0].l)), bits(s[1].h, t));
  }
}
template <int N>
__device__ __forceinline__ bool wire_load(const Packet *p, Sum<float> (&s)[N], uint32_t epoch) {
  const Packet q = packet_load(p);
  s[0] = Sum<float>{__uint_as_float((uint32_t)q.a), __uint_as_float((uint32_t)(q.a >> 32))};
  if constexpr (N == 1) {
    return q.b == epoch;
  } else {
    const uint32_t t = (uint32_t)(q.b >> 32);
    s[1] = Sum<float>{__uint_as_float((uint32_t)q.b), __uint_as_float(t & 0xFFFFFF00u)};
    return (t & 0xFFu) == (epoch >> 1 & 0xFFu);
  }
}
template <int N>
__device__ __forceinline__ void wire_store(Packet *p, const Sum<double> (&s)[N], uint32_t epoch) {
#pragma unroll
  for (int n = 0; n < N; n++) packet_store(p + n, (unsigned long long)__double_as_longlong(s[n].v), epoch);
}
template <int N>
__device__ __forceinline__ bool wire_load(const Packet *p, Sum<double> (&s)[N], uint32_t epoch) {
  bool ok = true;
#pragma unroll
  for (int n = 0; n < N; n++) {
    const Packet q = packet_load(p + n);
    s[n].v = __longlong_as_double((long long)q.a);
    ok = ok && q.b == epoch;
  }
  return ok;
}
// (a fence of release and acquire; __threadfence() also orders sequentially
// consistent accesses and costs more)
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ int load_error(const int *p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// Polls before a wait gives up: about 4 s of L2 round trips, so that CTAs that got
// their SMs outlast long kernels of other streams that still hold the others'.
// Counted in polls, not in clock cycles, so that a preempted context does not
// time out.
constexpr int RES_MAX_POLLS = 8000000;

#ifdef PB_FAULT_TEST
// Test builds only: while positive, the first grid-wide wait of a CTA gives up.
__device__ int g_fault_abandon_sums;
__device__ __forceinline__ bool fault_abandon_sum() {
  return *(volatile int *)&g_fault_abandon_sums > 0 && atomicAdd(&g_fault_abandon_sums, -1) > 0;
}
#endif

constexpr int RES_MAX_CTAS = 160;  // CTAs of a launch at most (one per SM)
template <typename T, int NTH> struct SumScratch {  // shared memory of the sums
  T part[2][NTH];
  Sum<T> block[2], cta[2][RES_MAX_CTAS];
  Sum<T> grid[2];      // the sums
  Sum<T> rz, alpha, beta;  // r.z, r.z / p.Ap, r.z / (the last r.z)
  Sum<T> stop;         // r.r below which the solve ends
  int neighbour[4];    // CTAs whose boundary z this one reads (-1: none)
  int failed;          // a wait gave up; stays set
};

// Wait for CTA c's word of this epoch.
template <typename T, int N>
__device__ __forceinline__ bool await_word(const Packet *words, int c, Sum<T> (&x)[N], uint32_t epoch, const int *err) {
  int polls = 0;
#pragma unroll 1
  while (!wire_load(words + (size_t)PACKET_STRIDE * c, x, epoch)) {
    ++polls;
    if (polls >= RES_MAX_POLLS || ((polls & 255) == 0 && load_error(err) != 0)) return false;
  }
  return true;
}

// Sum of N values per thread over the whole grid, in a fixed order, and the
// scalar that follows from it (N = 1: p.Ap and alpha; N = 2: r.z, r.r and
// beta), left in S for every thread.  false: a wait gave up (here or in
// another CTA).
// words: this kind of sum's array; a kind is used again only after the other
// kind's sum, so a word is overwritten only when every CTA has read it.
// publish: what the CTA's threads stored before the call is visible to the
// neighbours' threads after it: a release fence before the CTA's word, and
// the last warp waits for the neighbours' words and fences, beside the sum.
// At least four warps a CTA.
template <typename T, int N, int NTH>
__device__ __forceinline__ bool grid_sum(T v0, T v1, Packet *words, int cta, int ncta, uint32_t epoch, bool publish,
                                         int *err, SumScratch<T, NTH> &S, bool first) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  S.part[0][threadIdx.x] = v0;
  if (N == 2) S.part[1][threadIdx.x] = v1;
  __syncthreads();
  if (warp <= N) {
    if (warp < N) {  // warp n: the block's sum n
      constexpr int C = 16;
      Sum<T> t[1] = {sum_of((T)0)};
#pragma unroll 1
      for (int w = 0; w < nw; w += C) {
        Sum<T> s[C];
#pragma unroll
        for (int j = 0; j < C; j++) s[j] = sum_of(w + j < nw ? S.part[warp][lane + 32 * (w + j)] : (T)0);
        tree_sum<T, C>(s);
        gather(t[0], s[0]);
      }
      warp_sum<T, 1>(t);
      if (lane == 0) S.block[warp] = t[0];
    } else if (publish && lane == 0) {
      fence_gpu();
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * (N + 1)) : "memory");
    if (warp == N && lane == 0) {
      Sum<T> s[N];
#pragma unroll
      for (int n = 0; n < N; n++) s[n] = S.block[n];
      wire_store(words + (size_t)PACKET_STRIDE * cta, s, epoch);
    }
  }
  const int pollers = min(nw - 1, (ncta + 31) >> 5);  // warps that poll
  bool ok = true;
  if (warp < pollers) {
#ifdef PB_FAULT_TEST
    if (first && threadIdx.x == 0) ok = !fault_abandon_sum();
#endif
#pragma unroll 1
    for (int c = threadIdx.x; c < ncta && ok; c += 32 * pollers) {
      Sum<T> x[N];
      ok = await_word<T, N>(words, c, x, epoch, err);
#pragma unroll
      for (int n = 0; n < N; n++) S.cta[n][c] = x[n];
    }
  } else if (publish && warp == nw - 1) {
    if (lane < 4 && S.neighbour[lane] >= 0) {
      Sum<T> x[N];
      ok = await_word<T, N>(words, S.neighbour[lane], x, epoch, err);
      fence_gpu();
    }
  }
  if (!ok) {
    atomicOr(err, 1);
    S.failed = 1;
  }
  __syncthreads();
  if (warp == 0) {  // every CTA's sums in CTA order
    Sum<T> s[N];
#pragma unroll
    for (int n = 0; n < N; n++) {
      constexpr int C = 8;  // RES_MAX_CTAS / 32 rounded up to a power of two
      Sum<T> x[C];
#pragma unroll
      for (int j = 0; j < C; j++) x[j] = lane + 32 * j < ncta ? S.cta[n][lane + 32 * j] : sum_of((T)0);
      tree_sum<T, C>(x);
      s[n] = x[0];
    }
    warp_sum<T, N>(s);
    if (lane == 0) {
      if (N == 1) {
        S.alpha = quotient(S.rz, s[0]);
      } else {
        S.beta = quotient(s[0], S.rz);
        S.rz = s[0];
      }
#pragma unroll
      for (int n = 0; n < N; n++) S.grid[n] = s[n];
    }
  }
  __syncthreads();
  return S.failed == 0;
}

// ---------------------------------------------------------------------------
// Groups of four values.  FP32 groups are two register pairs and use the
// packed FP32 instructions (two results an issue slot, each rounded as the
// scalar instruction rounds it).

template <typename T> struct Q4;
template <> struct Q4<float> { unsigned long long p[2]; };
template <> struct Q4<double> { double v[4]; };

__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ Q4<float> make4(float a, float b, float c, float d) {
  return Q4<float>{{pack2(a, b), pack2(c, d)}};
}
__device__ __forceinline__ Q4<double> make4(double a, double b, double c, double d) {
  return Q4<double>{{a, b, c, d}};
}
template <typename T> __device__ __forceinline__ Q4<T> dup4(T a) { return make4(a, a, a, a); }
__device__ __forceinline__ float elem(const Q4<float> &q, int u) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(q.p[u >> 1]));
  return u & 1 ? hi : lo;
}
__device__ __forceinline__ double elem(const Q4<double> &q, int u) { return q.v[u]; }
__device__ __forceinline__ Q4<float> fma4(const Q4<float> &a, const Q4<float> &b, const Q4<float> &c) {
  return Q4<float>{{fma2(a.p[0], b.p[0], c.p[0]), fma2(a.p[1], b.p[1], c.p[1])}};
}
__device__ __forceinline__ Q4<float> mul4(const Q4<float> &a, const Q4<float> &b) {
  return Q4<float>{{mul2(a.p[0], b.p[0]), mul2(a.p[1], b.p[1])}};
}
__device__ __forceinline__ Q4<float> add4(const Q4<float> &a, const Q4<float> &b) {
  return Q4<float>{{add2(a.p[0], b.p[0]), add2(a.p[1], b.p[1])}};
}
__device__ __forceinline__ Q4<double> fma4(const Q4<double> &a, const Q4<double> &b, const Q4<double> &c) {
  return Q4<double>{{fma(a.v[0], b.v[0], c.v[0]), fma(a.v[1], b.v[1], c.v[1]), fma(a.v[2], b.v[2], c.v[2]),
                     fma(a.v[3], b.v[3], c.v[3])}};
}
__device__ __forceinline__ Q4<double> mul4(const Q4<double> &a, const Q4<double> &b) {
  return Q4<double>{{a.v[0] * b.v[0], a.v[1] * b.v[1], a.v[2] * b.v[2], a.v[3] * b.v[3]}};
}
__device__ __forceinline__ Q4<double> add4(const Q4<double> &a, const Q4<double> &b) {
  return Q4<double>{{a.v[0] + b.v[0], a.v[1] + b.v[1], a.v[2] + b.v[2], a.v[3] + b.v[3]}};
}
// Dot products: FP32 keeps a pair of running sums, added at the end; FP64 one
// (its adds are what an FP64 solve waits for).
template <typename T> struct Dot;
template <> struct Dot<float> { unsigned long long s; };
template <> struct Dot<double> { double s; };
__device__ __forceinline__ void dot4(Dot<float> &d, const Q4<float> &a, const Q4<float> &b) {
  d.s = fma2(a.p[0], b.p[0], d.s);
  d.s = fma2(a.p[1], b.p[1], d.s);
}
__device__ __forceinline__ void dot4(Dot<double> &d, const Q4<double> &a, const Q4<double> &b) {
#pragma unroll
  for (int u = 0; u < 4; u++) d.s = fma(a.v[u], b.v[u], d.s);
}
__device__ __forceinline__ float total_of(const Dot<float> &d) {
  const Q4<float> q{{d.s, d.s}};
  return elem(q, 0) + elem(q, 1);
}
__device__ __forceinline__ double total_of(const Dot<double> &d) { return d.s; }

__device__ __forceinline__ Q4<float> q_load(const float *p) {
  const ulonglong2 a = *(const ulonglong2 *)p;
  return Q4<float>{{a.x, a.y}};
}
__device__ __forceinline__ Q4<double> q_load(const double *p) {
  const double2 a = ((const double2 *)p)[0], b = ((const double2 *)p)[1];
  return Q4<double>{{a.x, a.y, b.x, b.y}};
}
// another CTA's z: past L1
__device__ __forceinline__ Q4<float> q_load_l2(const float *p) {
  const ulonglong2 a = __ldcg((const ulonglong2 *)p);
  return Q4<float>{{a.x, a.y}};
}
__device__ __forceinline__ Q4<double> q_load_l2(const double *p) {
  const double2 a = __ldcg((const double2 *)p), b = __ldcg((const double2 *)p + 1);
  return Q4<double>{{a.x, a.y, b.x, b.y}};
}
__device__ __forceinline__ void q_store(float *p, const Q4<float> &r) {
  *(ulonglong2 *)p = make_ulonglong2(r.p[0], r.p[1]);
}
__device__ __forceinline__ void q_store(double *p, const Q4<double> &r) {
  ((double2 *)p)[0] = make_double2(r.v[0], r.v[1]);
  ((double2 *)p)[1] = make_double2(r.v[2], r.v[3]);
}
// zero in the lanes whose bit of the mask is not set
template <typename T>
__device__ __forceinline__ Q4<T> keep(const Q4<T> &q, uint32_t mask) {
  return make4(mask & 1u ? elem(q, 0) : (T)0, mask & 2u ? elem(q, 1) : (T)0, mask & 4u ? elem(q, 2) : (T)0,
               mask & 8u ? elem(q, 3) : (T)0);
}

// By code byte: {diag A, M^-1}, M (1 without preconditioner) and the negated
// coefficient of a node whose six edges lie on one side of the surface.
template <typename T> struct alignas(4 * sizeof(T)) CodeEntry { T d, m, i, ne; };

// A group is simple when its four code bytes are one byte whose six edges lie
// on one side of the surface: one table entry and one coefficient serve it.
__device__ __forceinline__ bool simple_group(uint32_t codes) {
  const uint32_t m6 = codes & 0x3F3F3F3Fu;
  return codes == (codes & 0xffu) * 0x01010101u && (m6 == 0u || m6 == 0x3F3F3F3Fu);
}
// A value the compiler cannot follow: addresses formed from it stay in the
// loop that uses them.  (Hoisted out of the iteration loop, the addresses of
// every plane took more registers than the planes, and each spilled one
// cost a trip to L2 after every fence.)
template <typename V> __device__ __forceinline__ V opaque(V v) {
  asm volatile("" : "+r"(v));
  return v;
}
// What the operator reads of a plane beside this column's p.
template <typename T> struct Fetch {
  Q4<T> pn, ym, yp;  // p of the plane above, of the rows below and above
  T xl, xr;          // x neighbours at the ends of a warp or of a row
  uint32_t codes;
  CodeEntry<T> t;
};
// Negated coefficients of one edge direction (bit of the code bytes).
template <typename T>
__device__ __forceinline__ Q4<T> edge_eps(uint32_t codes, int bit, T nei, T neo) {
  return make4(codes >> bit & 1u ? nei : neo, codes >> (bit + 8) & 1u ? nei : neo, codes >> (bit + 16) & 1u ? nei : neo,
               codes >> (bit + 24) & 1u ? nei : neo);
}
// Ap of one group from its code bytes (Eq. 3), the neighbour sums formed from
// negated coefficients: diag p + sum (-eps) p_nb.  An edge between two nodes
// of the group is decoded once, and so is one between two planes: lower holds
// the coefficients of the edges below the group on entry (carried: those the
// plane below left; else they are decoded here) and of those above on return.
template <typename T, bool PER>
__device__ __forceinline__ Q4<T> packed_ap(bool simple, bool carried, uint32_t codes, const CodeEntry<T> &t, const CodeEntry<T> *mtab,
                                           const Q4<T> &pm, const Q4<T> &pc, const Q4<T> &pn, const Q4<T> &ym,
                                           const Q4<T> &yp, T xl, T xr, T nei, T neo, Q4<T> &lower) {
  const Q4<T> pl = make4(xl, elem(pc, 0), elem(pc, 1), elem(pc, 2));
  const Q4<T> pr = make4(elem(pc, 1), elem(pc, 2), elem(pc, 3), xr);
  if (simple) {
    const Q4<T> s6 = add4(add4(add4(pl, pr), add4(ym, yp)), add4(pm, pn));
    return fma4(dup4(t.d), pc, mul4(dup4(t.ne), s6));
  }
  if (!carried) lower = edge_eps(codes, 4, nei, neo);
  Q4<T> s = mul4(lower, pm);
  lower = edge_eps(codes, 5, nei, neo);
  s = fma4(lower, pn, s);
  s = fma4(edge_eps(codes, 2, nei, neo), ym, s);
  s = fma4(edge_eps(codes, 3, nei, neo), yp, s);
  const Q4<T> ex = edge_eps(codes, 0, nei, neo);
  s = fma4(ex, pl, s);
  // (with wrap the last node of a row has an edge that the pad byte after it lacks)
  if (PER) s = fma4(edge_eps(codes, 1, nei, neo), pr, s);
  else s = fma4(make4(elem(ex, 1), elem(ex, 2), elem(ex, 3), codes >> 25 & 1u ? nei : neo), pr, s);
  const Q4<T> dg = make4(t.d, mtab[codes >> 8 & 127u].d, mtab[codes >> 16 & 127u].d,
                         mtab[codes >> 24 & 127u].d);
  return fma4(dg, pc, s);
}

// ---------------------------------------------------------------------------
// T: precision of the inner solve; CM: coefficient storage; G > 0: planes a
// thread can own, z and the increment d in registers, Ap in shared memory (so
// that the operator's loop, most of the code, is not unrolled); G = 0: z and d
// in the grid's arrays (L2), any number of planes; Ap is stored there by FP64
// solves (KEEP), whose arithmetic is what they wait for, and formed again from
// p by FP32 solves (8 B a node of L2 traffic less).  PER: periodic axes.
constexpr int RES_YH = 3;  // y-halo groups a thread can own
// CTAs on an SM: the small builds, of batches, come in pairs, one computing while
// the other waits for its sums
constexpr int ctas_per_sm(int threads) { return threads <= 256 ? 2 : 1; }

// The direction p (array gp) of a CTA's brick into ps: rows -1 .. rows of planes -1 .. kn,
// as an earlier launch left them.  Out of line: inlined, it took registers from the
// iterations (spills of the 8-plane build 64 -> 92 bytes; a burst of 129^3 167 -> 177 ms).
template <typename T, bool PER>
__device__ __noinline__ void load_direction(const ResArgs &R, const T *gp, int cta, T *ps) {
  const int gpr = R.gpr, by = R.by, ny = R.ny, nz = R.nz, rp = 4 * gpr + 4;
  const int cy = cta % R.nby, y0 = cy * by, z0 = cta / R.nby * R.bz;
  const int rows = min(by, ny - y0) + 2, planes = min(R.bz, nz - z0) + 2;
  for (int f = threadIdx.x; f < planes * rows * gpr; f += blockDim.x) {
    const int row = f / gpr, x = f - row * gpr, pl = row / rows, r = row - pl * rows;
    int j = y0 + r - 1, k = z0 + pl - 1;
    if (PER) {
      j = j < 0 ? ny - 1 : j == ny ? 0 : j;
      k = k < 0 ? nz - 1 : k == nz ? 0 : k;
    }
    if (j >= 0 && j < ny && k >= 0 && k < nz)
      q_store(ps + (pl * (by + 2) + r) * rp + 4 + 4 * x,
              q_load_l2(gp + ((uint32_t)k * ny + j) * R.px + 4 * x));
  }
}

template <typename T, int CM, int G, int NTH, bool PER, typename W>
__global__ void __launch_bounds__(NTH, ctas_per_sm(NTH)) k_cg_resident(const __grid_constant__ W wave) {
  int n_grid = 0, cta = blockIdx.x, ncta = gridDim.x;  // this CTA's grid, its number there
  if constexpr (std::is_same_v<W, ResWave>) {
    while (cta >= wave.first[n_grid + 1]) n_grid++;
    ncta = wave.first[n_grid + 1] - wave.first[n_grid];
    cta -= wave.first[n_grid];
  }
  const ResArgs &R = wave.grid[n_grid];
  constexpr bool SEP = sizeof(T) == 4;  // FP32 inner solves accumulate into d
  constexpr bool REG = G > 0, KEEP = REG || sizeof(T) == 8;
  // planes whose loads are issued together
  constexpr int BATCH = !REG ? 2 : G % 4 == 0 ? 4 : G % 3 == 0 ? 3 : G;
  static_assert(!REG || G % BATCH == 0, "whole batches");
  extern __shared__ __align__(128) uint8_t dyn[];
  __shared__ SumScratch<T, NTH> S;
  __shared__ CodeEntry<T> mtab[CM == COEF_PACKED ? 128 : 1];
  const Inst &I = *R.inst;
  Scal *Sp = I.s;
  const int was = *(volatile int *)&Sp->phase;
  constexpr bool ROUNDS = std::is_same_v<W, ResWave>;  // leaves a solve after `budget` iterations
  if (was != PH_START && !(ROUNDS && was == PH_INNER)) return;  // nothing to solve (the same for every CTA)
  const bool resume = ROUNDS && was == PH_INNER;  // goes on where an earlier launch left it
  if (threadIdx.x == 0) S.failed = 0;
  const int by = R.by, gpr = R.gpr, rp = 4 * gpr + 4, ps_plane = (by + 2) * rp;
  const int cy = cta % R.nby, cz = cta / R.nby;
  const int y0 = cy * by, z0 = cz * R.bz;
  const int ny = R.ny, nz = R.nz, nx = R.nx, px = R.px;
  const int rows = min(by, ny - y0), kn = min(R.bz, nz - z0);
  const int ty = threadIdx.x / gpr, xg = threadIdx.x - ty * gpr;
  const bool own = ty < rows;
  const uint32_t plane = (uint32_t)px * ny;
  // shared memory: p with its halo; REG: Ap and the code words
  T *ps = (T *)dyn;
  const int n_ps = (R.bz + 2) * ps_plane + 4;
#pragma unroll 1
  for (int t = threadIdx.x; t < n_ps; t += blockDim.x) ps[t] = (T)0;
  T *as = (T *)(dyn + R.off_ap) + 4 * threadIdx.x;  // REG: Ap, [plane][thread] groups
  const int group_stride = 4 * blockDim.x;
  uint32_t *cs = (uint32_t *)(dyn + R.off_codes) + threadIdx.x;  // REG: the code words, [plane][thread]
  if constexpr (CM == COEF_PACKED) {
    for (int t = threadIdx.x; t < 128; t += blockDim.x) {
      const int k = dtab_index(t);
      mtab[t] = CodeEntry<T>{tab_d<T>(I, k), I.precond ? tab_d<T>(I, k) : (T)1, I.precond ? tab_i<T>(I, k) : (T)1,
                             t & 1 ? -e_in<T>(I) : -e_out<T>(I)};
    }
  }
  const bool prec = I.precond != 0;
  const T nei = -e_in<T>(I), neo = -e_out<T>(I);
  uint32_t vmask = 0;
  if (own)
    for (int u = 0; u < 4; u++)
      if (4 * xg + u < nx) vmask |= 1u << u;
  const bool full = vmask == 0xFu;
  const uint32_t col = (uint32_t)(y0 + (own ? ty : 0)) * px + 4 * xg;  // this thread's column
  const uint32_t e0 = (uint32_t)z0 * plane + col;                      // ... its first plane's group
  T *const gz = (T *)R.z;
  T *const gd = SEP ? (T *)R.d : (T *)(Sp->xbuf ? R.x64b : R.x64);
  T *const ga = (T *)R.ap;
  // Boundary z alternates between the two direction buffers (p itself is in
  // shared memory): what an iteration writes is read in the next one and
  // overwritten in the one after, so only the second sum of an iteration has
  // to order it.
  T *const x0 = (T *)R.p1, *const x1 = (T *)R.p0;
  const int o0 = ps_plane + (ty + 1) * rp + 4 + 4 * xg;  // this thread's group in plane 0 of ps
  // z-halo planes of this thread's column (-1: outside the grid, p = 0)
  const int zb = z0 - 1 >= 0 ? z0 - 1 : PER ? nz - 1 : -1, zt = z0 + kn < nz ? z0 + kn : PER ? 0 : -1;
  // This thread's h-th group of the rows beside the brick: its place in ps and
  // in the grid's arrays; false: none, or outside the grid.
  auto y_halo = [&](int h, int &o, uint32_t &e) -> bool {
    const int f = threadIdx.x + h * blockDim.x;
    if (f >= 2 * kn * gpr) return false;
    const int side = f >= kn * gpr, g = f - side * kn * gpr;
    const int k = gpr == 1 ? g : (int)__umulhi(g, R.gpr_magic), x = g - k * gpr;
    int j = side ? y0 + rows : y0 - 1;
    if (PER) j = j < 0 ? ny - 1 : j == ny ? 0 : j;
    o = (k + 1) * ps_plane + (side ? rows + 1 : 0) * rp + 4 + 4 * x;
    e = (uint32_t)(z0 + k) * plane + (uint32_t)j * px + 4 * x;
    return j >= 0 && j < ny;
  };
  const bool y_edge = ty == 0 || ty == rows - 1;
  // x neighbours come from the lanes beside, or from shared memory at the ends
  // of a warp or of a row
  const uint32_t own_lanes = __ballot_sync(0xffffffffu, own);
  const bool left_edge = xg == 0 || (threadIdx.x & 31) == 0, right_edge = xg == gpr - 1 || (threadIdx.x & 31) == 31;
  if (threadIdx.x == 0) {
    const int b = cta, nby = R.nby, nbz = R.nbz;
    S.neighbour[0] = cy > 0 ? b - 1 : PER ? b + nby - 1 : -1;
    S.neighbour[1] = cy < nby - 1 ? b + 1 : PER ? b - nby + 1 : -1;
    S.neighbour[2] = cz > 0 ? b - nby : PER ? b + (nbz - 1) * nby : -1;
    S.neighbour[3] = cz < nbz - 1 ? b + nby : PER ? b - (nbz - 1) * nby : -1;
  }

  if (resume) {
    __syncthreads();  // ps is zero
    load_direction<T, PER>(R, (const T *)(Sp->pbuf ? R.p1 : R.p0), cta, ps);
  }
  const Q4<T> zero4 = dup4((T)0);
  Q4<T> z[REG ? G : 1], d[REG ? G : 1];
  if constexpr (REG) {
#pragma unroll
    for (int k = 0; k < G; k++) {
      z[k] = d[k] = zero4;
      if (own && k < kn) {
        z[k] = q_load_l2(gz + e0 + k * plane);
        if (!SEP || resume) d[k] = q_load(gd + e0 + k * plane);
      }
    }
  }
  if (own) {
#pragma unroll 1
    for (int k = 0; k < kn; k++) {
      const uint32_t e = e0 + k * plane;
      if (REG && CM == COEF_PACKED) cs[k * blockDim.x] = *(const uint32_t *)(R.code + e);
      if (!REG && SEP && !resume) q_store(gd + e, zero4);
    }
  }
  // Scalars of the recurrences.  Float sums are scaled by a power of two that
  // brings ||rhs||^2 near 1, so that neither they nor their low parts leave
  // the range of a float.
  T scale_t = (T)1;
  if (SEP) {
    int ex = 0;
    frexp(Sp->ref_norm, &ex);
    scale_t = (T)ldexp(1.0, max(-120, min(120, -2 * ex)));
  }
  if (threadIdx.x == 0) {
    const double tol = (I.mode == MODE_F32_REFINE ? Sp->itol : I.tol) * Sp->ref_norm;
    S.stop = from_double<T>(tol * tol * scale_t);  // ||r|| < tol as r.r < stop
    S.rz = from_double<T>(Sp->rz_old * scale_t);
    S.alpha = S.beta = sum_of((T)0);
    if constexpr (ROUNDS) {
      S.alpha = from_double<T>(resume ? Sp->alpha : 0.0);
      S.beta = from_double<T>(resume ? Sp->beta : 0.0);
    }
  }
  int iter = 0, total = Sp->total_iter, status = Sp->status, phase = PH_INNER;
  const int max_iter = I.max_iter;
  Packet *const words_a = (Packet *)R.packets;  // p.Ap
  Packet *const words_b = words_a + (size_t)PACKET_STRIDE * ncta;  // r.z, r.r
  auto code_of = [&](int k) -> uint32_t {
    if (CM != COEF_PACKED) return 0u;
    return REG ? cs[k * blockDim.x] : __ldg((const uint32_t *)(R.code + e0 + k * plane));
  };
  // Planes whose groups are not all simple, per warp: such a plane takes the
  // general form in every lane (both forms one after the other cost more).
  uint32_t general = 0;
  if constexpr (CM == COEF_PACKED) {
#pragma unroll 1
    for (int k = 0; k < kn; k++)
      if (__any_sync(0xffffffffu, own && !simple_group(code_of(k)))) general |= 1u << k;
  }
  // x += alpha p (the last iteration's, deferred; alpha = p = 0 in the first),
  // p = z + beta p of planes k0 .. k0 + BATCH - 1: their loads before their stores
  auto direction = [&](int k0, int o, const Q4<T> *zk, Q4<T> *dk, const Q4<T> &alpha_prev, const Q4<T> &beta) {
    Q4<T> po[BATCH];
#pragma unroll
    for (int j = 0; j < BATCH; j++) {
      if (k0 + j < kn) po[j] = q_load(ps + o + j * ps_plane);
      if (PER && !full) po[j] = keep(po[j], vmask);  // pad lanes hold wrapped values for the stencil
    }
#pragma unroll
    for (int j = 0; j < BATCH; j++)
      if (k0 + j < kn) {
        dk[j] = fma4(alpha_prev, po[j], dk[j]);
        q_store(ps + o + j * ps_plane, fma4(beta, po[j], zk[j]));
      }
  };
  auto halo = [&](int o, const Q4<T> &zh, const Q4<T> &beta) {
    q_store(ps + o, fma4(beta, q_load(ps + o), zh));
  };
  // The operator's inputs of plane k, whose group is at pp.
  auto fetch = [&](int k, const T *pp) -> Fetch<T> {
    Fetch<T> f;
    f.pn = q_load(pp + ps_plane);
    f.ym = q_load(pp - rp);
    f.yp = q_load(pp + rp);
    f.xl = f.xr = (T)0;
    if (left_edge) f.xl = pp[-1];
    if (right_edge) f.xr = pp[4];
    if constexpr (CM == COEF_PACKED) {
      f.codes = code_of(k);
      f.t = mtab[f.codes & 127u];
    }
    return f;
  };
  // Ap of plane k from the p of planes k-1, k and what was fetched
  auto operator_at = [&](int k, const Fetch<T> &f, const Q4<T> &pm, const Q4<T> &pc, Q4<T> &lower) -> Q4<T> {
    const Q4<T> &pn = f.pn, &ym = f.ym, &yp = f.yp;
    T xl = __shfl_up_sync(own_lanes, elem(pc, 3), 1), xr = __shfl_down_sync(own_lanes, elem(pc, 0), 1);
    if (left_edge) xl = f.xl;
    if (right_edge) xr = f.xr;
    Q4<T> a;
    if constexpr (CM == COEF_PACKED) {
      a = packed_ap<T, PER>(!(general >> k & 1u), k > 0 && (general >> (k - 1) & 1u), f.codes, f.t, mtab, pm, pc, pn,
                       ym, yp, xl, xr, nei, neo, lower);
    } else {
      const GroupCoef<T> c = group_coef<T, CM>(I, e0 + k * plane, z0 + k, (vmask >> 3) & 1u);
      const Q4<T> pl = make4(xl, elem(pc, 0), elem(pc, 1), elem(pc, 2));
      const Q4<T> pr = make4(elem(pc, 1), elem(pc, 2), elem(pc, 3), xr);
      Q4<T> s = mul4(make4(c.ex[0], c.ex[1], c.ex[2], c.ex[3]), pl);
      s = fma4(make4(c.ex[1], c.ex[2], c.ex[3], c.ex[4]), pr, s);
      s = fma4(make4(c.eym[0], c.eym[1], c.eym[2], c.eym[3]), ym, s);
      s = fma4(make4(c.eyp[0], c.eyp[1], c.eyp[2], c.eyp[3]), yp, s);
      s = fma4(make4(c.ezm[0], c.ezm[1], c.ezm[2], c.ezm[3]), pm, s);
      s = fma4(make4(c.ezp[0], c.ezp[1], c.ezp[2], c.ezp[3]), pn, s);
      a = fma4(make4(c.diag[0], c.diag[1], c.diag[2], c.diag[3]), pc, mul4(dup4((T)-1), s));
    }
    if (PER && !full) a = keep(a, vmask);  // (without wrap p = 0 there, and nalpha masks)
    return a;
  };
  // r = M z - alpha Ap, z = M^-1 r of plane k; adds r.z and r.r
  auto residual = [&](int k, uint32_t codes, const Q4<T> &zk, const Q4<T> &a, const Q4<T> &nalpha, Dot<T> &rz, Dot<T> &rr) -> Q4<T> {
    Q4<T> m, mi;
    if constexpr (CM == COEF_PACKED) {
      if (!(general >> k & 1u)) {
        const CodeEntry<T> t = mtab[codes & 127u];
        m = dup4(t.m);
        mi = dup4(t.i);
      } else {
        const CodeEntry<T> t0 = mtab[codes & 127u], t1 = mtab[codes >> 8 & 127u], t2 = mtab[codes >> 16 & 127u],
                           t3 = mtab[codes >> 24 & 127u];
        m = make4(t0.m, t1.m, t2.m, t3.m);
        mi = make4(t0.i, t1.i, t2.i, t3.i);
      }
    } else {
      m = prec ? q_load((const T *)R.diag + e0 + k * plane) : dup4((T)1);  // pads hold 1
      // FP32: the correctly rounded reciprocal, within an ulp of r / m
      if constexpr (sizeof(T) == 4)
        mi = make4(__frcp_rn(elem(m, 0)), __frcp_rn(elem(m, 1)), __frcp_rn(elem(m, 2)), __frcp_rn(elem(m, 3)));
    }
    const Q4<T> r = fma4(nalpha, a, mul4(m, zk));
    Q4<T> zn;
    if constexpr (CM == COEF_F64)
      zn = make4(elem(r, 0) / elem(m, 0), elem(r, 1) / elem(m, 1), elem(r, 2) / elem(m, 2), elem(r, 3) / elem(m, 3));
    else
      zn = mul4(r, mi);
    dot4(rz, r, zn);
    dot4(rr, r, r);
    return zn;
  };
  __syncthreads();

  for (;;) {
    const Q4<T> alpha_prev = dup4(lead(S.alpha)), beta = dup4(lead(S.beta));
    // neighbours' boundary z (in the first iteration the z that the residual
    // pass left, then the buffer the last iteration wrote), requested first,
    // used after the CTA's own groups
    const T *const gx = iter == 0 ? gz : (iter & 1) ? x0 : x1;
    T *const gw = (iter & 1) ? x1 : x0;  // this iteration's boundary z
    Q4<T> hb = zero4, ht = zero4, hy[RES_YH];
    if (own && zb >= 0) hb = q_load_l2(gx + (uint32_t)zb * plane + col);
    if (own && zt >= 0) ht = q_load_l2(gx + (uint32_t)zt * plane + col);
    int yo[RES_YH];
#pragma unroll
    for (int h = 0; h < RES_YH; h++) {
      uint32_t e;
      if (y_halo(h, yo[h], e)) hy[h] = q_load_l2(gx + e);
      else yo[h] = -1;
    }
    if (own) {
      if constexpr (REG) {
        int o = opaque(o0);
#pragma unroll
        for (int k = 0; k < G; k += BATCH) {
          if (k < kn) direction(k, o, z + k, d + k, alpha_prev, beta);
          o += BATCH * ps_plane;
        }
      } else {
#pragma unroll 1
        for (int k0 = 0; k0 < kn; k0 += BATCH) {  // a batch's loads before its stores
          Q4<T> zk[BATCH], dk[BATCH];
#pragma unroll
          for (int j = 0; j < BATCH; j++) {
            const uint32_t e = e0 + min(k0 + j, kn - 1) * plane;
            zk[j] = q_load(gz + e);
            dk[j] = q_load(gd + e);
          }
          direction(k0, o0 + k0 * ps_plane, zk, dk, alpha_prev, beta);
#pragma unroll
          for (int j = 0; j < BATCH; j++)
            if (k0 + j < kn) q_store(gd + e0 + (k0 + j) * plane, dk[j]);
        }
      }
      if (zb >= 0) halo(o0 - ps_plane, hb, beta);
      if (zt >= 0) halo(o0 + kn * ps_plane, ht, beta);
    }
#pragma unroll
    for (int h = 0; h < RES_YH; h++)
      if (yo[h] >= 0) halo(yo[h], hy[h], beta);
    __syncthreads();
    if (PER) {  // x images of the brick's rows: node -1 and node nx
      for (int f = threadIdx.x; f < rows * kn; f += blockDim.x) {
        const int k = f / rows, r = f - k * rows;
        T *row = ps + (k + 1) * ps_plane + (r + 1) * rp;
        row[3] = row[4 + nx - 1];
        row[4 + nx] = row[4];
      }
      __syncthreads();
    }
    // Ap, p.Ap
    Dot<T> acc = {};
    if (own) {
      const T *pp = ps + o0;
      Q4<T> pm = q_load(pp - ps_plane), pc = q_load(pp), lower = zero4;
#pragma unroll 1
      for (int k = 0; k < kn; k++) {
        const Fetch<T> fk = fetch(k, pp);
        pp += ps_plane;
        const Q4<T> a = operator_at(k, fk, pm, pc, lower);
        dot4(acc, pc, a);
        if (KEEP) q_store(REG ? as + k * group_stride : ga + e0 + k * plane, a);
        pm = pc;
        pc = fk.pn;
      }
    }
    // (the first sum also orders reading the residual pass's z before a
    // neighbour's G = 0 build overwrites it)
    if (!grid_sum<T, 1, NTH>(total_of(acc) * scale_t, (T)0, words_a, cta, ncta, 2u * iter + 1u, iter == 0, R.err, S,
                             iter == 0))
      return;
    if (!(lead(S.grid[0]) > (T)0) || !isfinite(lead(S.alpha))) {
      status = 6;  // PB_ERR_BREAKDOWN
      phase = PH_DONE;
      break;
    }
    const Q4<T> nalpha = keep(dup4(-lead(S.alpha)), opaque(vmask));  // r stays 0 at row pads
    Dot<T> rz = {}, rr = {};
    if (own) {
      if constexpr (REG) {
        int oa = opaque(0), oc = oa;
        uint32_t e = opaque(e0);
#pragma unroll
        for (int k = 0; k < G; k++) {
          if (k < kn) {
            z[k] = residual(k, CM == COEF_PACKED ? cs[oc] : 0u, z[k], q_load(as + oa), nalpha, rz, rr);
            if (y_edge || k == 0 || k == kn - 1) q_store(gw + e, z[k]);
          }
          oa += group_stride;
          oc += blockDim.x;
          e += plane;
        }
      } else {
        const T *pp = ps + o0;
        Q4<T> pm = q_load(pp - ps_plane), pc = q_load(pp), lower = zero4;
#pragma unroll 1
        for (int k0 = 0; k0 < kn; k0 += BATCH) {  // a batch's loads before its stores
          Q4<T> zk[BATCH], ak[BATCH];
#pragma unroll
          for (int j = 0; j < BATCH; j++) {
            const uint32_t e = e0 + min(k0 + j, kn - 1) * plane;
            zk[j] = q_load(gz + e);
            if (KEEP) ak[j] = q_load(ga + e);
          }
#pragma unroll
          for (int j = 0; j < BATCH; j++) {
            const int k = k0 + j;
            if (k < kn) {
              if (!KEEP) {
                const Fetch<T> fk = fetch(k, pp);
                pp += ps_plane;
                ak[j] = operator_at(k, fk, pm, pc, lower);
                pm = pc;
                pc = fk.pn;
              }
              const Q4<T> zn = residual(k, code_of(k), zk[j], ak[j], nalpha, rz, rr);
              q_store(gz + e0 + k * plane, zn);
              if (y_edge || k == 0 || k == kn - 1) q_store(gw + e0 + k * plane, zn);
            }
          }
        }
      }
    }
    if (!grid_sum<T, 2, NTH>(total_of(rz) * scale_t, total_of(rr) * scale_t, words_b, cta, ncta, 2u * iter + 2u, true,
                             R.err, S, false))
      return;
    if (!isfinite(lead(S.grid[0])) || !isfinite(lead(S.grid[1]))) {
      status = 6;
      phase = PH_DONE;
      break;
    }
    iter++;
    total++;
    const bool converged = below(S.grid[1], S.stop), end = converged || total >= max_iter;
    if (end && !converged) status = 5;  // PB_ERR_NOT_CONVERGED
    if (end) {
      phase = PH_RESID;
      break;
    }
    if (ROUNDS && iter >= R.budget) break;  // phase INNER
  }
  // hand over to the residual pass: d without the last step, p of the last
  // step in buffer 0, the scalars; and z, from which (as from the state after an
  // update pass) the next launch or phase ticks go on with the inner solve
  if (own) {
#pragma unroll 1
    for (int k = 0; k < kn; k++) {
      Q4<T> pv = q_load(ps + o0 + k * ps_plane);
      if (PER && !full) pv = keep(pv, vmask);
      q_store((T *)R.p0 + e0 + k * plane, pv);
    }
    if constexpr (REG) {
      uint32_t e = opaque(e0);
#pragma unroll
      for (int k = 0; k < G; k++) {
        if (k < kn) {
          q_store(gd + e, d[k]);
          if (ROUNDS && phase == PH_INNER) q_store(gz + e, z[k]);
        }
        e += plane;
      }
    }
  }
  if (cta == 0 && threadIdx.x == 0) {
    if (ROUNDS ? phase != PH_DONE : phase == PH_RESID) {
      Sp->alpha = value(S.alpha);
      Sp->beta = value(S.beta);
      Sp->rz_old = value(S.rz) / scale_t;
    }
    if (iter > 0 && isfinite(lead(S.grid[1]))) Sp->relres = sqrt(value(S.grid[1]) / scale_t) / Sp->ref_norm;
    Sp->pbuf = 0;
    Sp->iter = ROUNDS ? Sp->iter + iter : iter;  // (0 in the start phase)
    Sp->total_iter = total;
    Sp->status = status;
    Sp->phase = phase;
    if (phase == PH_RESID) R.resid_list[atomicAdd(R.resid_pending, 1)] = R.slot;
  }
}

// ---------------------------------------------------------------------------
// Host side: the builds, the plan, the launch.

namespace {

struct Build {
  int G, threads;
};
// Builds by planes a thread owns (0: any); threads: the most whose registers fit one SM.
constexpr Build F32_BUILDS[] = {{2, 512}, {4, 512}, {5, 512}, {6, 512}, {8, 512}, {12, 384}, {0, 1024}};
constexpr Build F64_BUILDS[] = {{0, 512}};
// Of a batch: an iteration of two grids of 97^3 takes 10.8 us in the pairs of {8, 256},
// 12.1 in {8, 512}, one of them alone 9.1 and 9.
constexpr Build BATCH_BUILDS[] = {{8, 512}, {12, 384}, {8, 256}, {12, 192}};  // FP32 grids of a batch, packed codes

size_t p_bytes(int by, int bz, int gpr, int es) {
  return ((size_t)((size_t)(bz + 2) * (by + 2) * (4 * gpr + 4) + 4) * es + 15) / 16 * 16;
}

struct Shape {  // of a launch
  int ctas, threads;
  size_t smem;
};
template <typename W, typename K>
cudaError_t launch_kernel(K *k, const Shape &P, const W &wave, cudaStream_t st) {
  const cudaError_t e = allow_all_smem(k);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(P.ctas);
  cfg.blockDim = dim3(P.threads);
  cfg.dynamicSmemBytes = P.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, wave);
}
// Shared memory: p, then (G > 0) Ap, then (packed codes) the code words, a
// thread's groups each.
size_t off_codes(const ResPlan &P, int es, int threads) {
  return (size_t)P.off_ap + (P.planes ? (size_t)4 * es * P.bz * threads : 0);
}
size_t smem_of(const ResPlan &P, int es, int coef, int threads) {
  return off_codes(P, es, threads) + (P.planes && coef == COEF_PACKED ? (size_t)4 * P.bz * threads : 0);
}
template <typename T, int CM, int G, int NTH, typename W = ResOne>
cudaError_t launch_build(const Shape &P, const W &wave, bool per, cudaStream_t st) {
  return per ? launch_kernel<W>(k_cg_resident<T, CM, G, NTH, true, W>, P, wave, st)
             : launch_kernel<W>(k_cg_resident<T, CM, G, NTH, false, W>, P, wave, st);
}

template <int CM>
cudaError_t launch_f32(int build, const Shape &P, const ResOne &R, bool per, cudaStream_t st) {
  switch (build) {
    case 0: return launch_build<float, CM, 2, 512>(P, R, per, st);
    case 1: return launch_build<float, CM, 4, 512>(P, R, per, st);
    case 2: return launch_build<float, CM, 5, 512>(P, R, per, st);
    case 3: return launch_build<float, CM, 6, 512>(P, R, per, st);
    case 4: return launch_build<float, CM, 8, 512>(P, R, per, st);
    case 5: return launch_build<float, CM, 12, 384>(P, R, per, st);
    default: return launch_build<float, CM, 0, 1024>(P, R, per, st);
  }
}
template <int CM>
cudaError_t launch_f64(const Shape &P, const ResOne &R, bool per, cudaStream_t st) {
  return launch_build<double, CM, 0, 512>(P, R, per, st);
}

cudaError_t launch_batch(int build, const Shape &P, const ResWave &R, bool per, cudaStream_t st) {
  switch (build) {
    case 0: return launch_build<float, COEF_PACKED, 8, 512>(P, R, per, st);
    case 1: return launch_build<float, COEF_PACKED, 12, 384>(P, R, per, st);
    case 2: return launch_build<float, COEF_PACKED, 8, 256>(P, R, per, st);
    default: return launch_build<float, COEF_PACKED, 12, 192>(P, R, per, st);
  }
}

// Kernel arguments of one grid; threads: of the launch.
ResArgs grid_args(const ResPlan &P, const Inst &I, const Inst *dI, const Batch &B, void *packets, int slot, int threads,
                  int budget) {
  ResArgs R;
  R.inst = dI;
  R.packets = packets;
  R.err = B.error + ERR_RESIDENT;
  R.resid_pending = B.resid_pending;
  R.resid_list = B.resid_list;
  R.z = I.z;
  R.d = I.d;
  R.ap = I.ap;
  R.p0 = I.p0;
  R.p1 = I.p1;
  R.x64 = I.x64;
  R.x64b = I.x64b;
  R.code = I.code;
  R.diag = I.diag;
  R.nx = I.nx;
  R.ny = I.ny;
  R.nz = I.nz;
  R.px = I.px;
  R.by = P.by;
  R.bz = P.bz;
  R.nby = P.nby;
  R.nbz = P.nbz;
  R.gpr = P.gpr;
  // g / gpr = umulhi(g, magic) for g * gpr < 2^32
  R.gpr_magic = P.gpr > 1 ? (uint32_t)(((1ull << 32) + P.gpr - 1) / P.gpr) : 0u;
  R.off_ap = P.off_ap;
  R.off_codes = off_codes(P, I.mode == MODE_F64 ? 8 : 4, threads);
  R.slot = slot;
  R.budget = budget;
  return R;
}

}  // namespace

// The plan of least cost: of an iteration (alone), or of an iteration of as many
// such grids as the device holds at once, a grid.
static bool best_plan(int nx, int ny, int nz, int mode, int coef, int num_sms, int max_smem, long l2_bytes, bool alone,
                      ResPlan *out) {
  const int es = mode == MODE_F64 ? 8 : 4, gpr = (nx + 3) / 4;
  const Build *builds = !alone ? BATCH_BUILDS : mode == MODE_F64 ? F64_BUILDS : F32_BUILDS;
  const int nb = !alone ? std::size(BATCH_BUILDS) : mode == MODE_F64 ? std::size(F64_BUILDS) : std::size(F32_BUILDS);
  // What an FP32 iteration of the G = 0 builds reads of L2: the coefficients, z, d.
  // More than 7/8 of L2 goes to memory in part, in the order of the bricks and
  // twice, and the two-pass form is faster (L2 of 135 MB, FP32 coefficients, us an
  // iteration in two passes -> here: 169^3, 116 MB, 72 -> 63; 173^3, 124 MB, 76 ->
  // 84; 177^3, 133 MB, 81 -> 96; BF16: 177^3, 89 MB, 76 -> 66).  (FP64 waits for its
  // arithmetic: 129^3 with explicit coefficients, 120 MB, 189 -> 148.)
  const int coef_bytes = coef == COEF_PACKED ? 1 : coef == COEF_BF16 ? 8 : 16;
  const bool in_l2 = mode == MODE_F64 || (long)nx * ny * nz * (coef_bytes + 8) <= l2_bytes / 8 * 7;
  // Explicit coefficients in the G = 0 builds: a plane waits for its loads, and a narrow,
  // deep brick has few warps to wait beside each other.  The two-pass form is faster
  // beyond these planes at these warps (us an iteration in two passes -> here: FP32
  // 17x17x1976, 13 planes, 34.6 -> 34.6, x2432, 16, 36.5 -> 44.3, 25x25x2432, 6 warps,
  // 45.9 -> 47.8, 9x65x2432, 7 warps, 58 -> 48; BF16 17x17x2432 37.0 -> 38.8, x2888, 19,
  // 40 -> 46; FP64 9x9x1976 82 -> 79, x2432 87 -> 97.  Packed codes: faster at any).
  const int few_warps = coef == COEF_F32 ? 6 : coef == COEF_BF16 ? 5 : coef == COEF_F64 ? 4 : 0;
  const int deep = coef == COEF_BF16 ? 16 : 13;
  bool found = false;
  double best = 0;
  for (int b = 0; b < nb; b++) {
    const Build &B = builds[b];
    if (B.G == 0 && !in_l2) continue;
    const int per_sm = ctas_per_sm(B.threads), room = per_sm * num_sms;
    // (an SM keeps 1 KB of each CTA's shared memory to itself)
    const int smem = (max_smem + 1024) / per_sm - 1024 - RES_STATIC_SMEM / per_sm;
    for (int bym = 1; bym * gpr <= B.threads && bym <= ny; bym++) {
      for (int bzm = 1; bzm <= (B.G ? B.G : nz) && bzm <= nz; bzm++) {
        const int nby = (ny + bym - 1) / bym, nbz = (nz + bzm - 1) / bzm;
        if ((long)nby * nbz > std::min(room, RES_MAX_CTAS)) continue;
        ResPlan P;
        P.build = b;
        P.planes = B.G;
        P.by = (ny + nby - 1) / nby;
        P.bz = (nz + nbz - 1) / nbz;
        P.gpr = gpr;
        P.threads = std::max(128, (P.by * gpr + 31) / 32 * 32);  // four warps: grid_sum
        if (P.threads > B.threads || P.bz > 32 || 2 * P.bz * gpr > RES_YH * P.threads) continue;
        if (B.G == 0 && P.threads <= 32 * few_warps && P.bz > deep) continue;
        P.off_ap = (int)p_bytes(P.by, P.bz, gpr, es);
        // (in a batch the launch has the threads of its largest plan)
        if ((long)smem_of(P, es, coef, alone ? P.threads : B.threads) > smem) continue;
        P.nby = (ny + P.by - 1) / P.by;
        P.nbz = (nz + P.bz - 1) / P.bz;
        P.ctas = P.nby * P.nbz;
        P.room = room;
        // Cycles of an iteration: a plane costs its groups' issue slots on four
        // schedulers and a latency, more in the builds whose registers spill;
        // the two grid-wide sums.  (Measured best and the model's choice differ
        // by 3% at most on cubes of 33 to 145 nodes a side.)
        const double group = es == 8 ? 900.0 : coef == COEF_PACKED ? 150.0 : 200.0;
        const double spill = B.G == 0 ? 2.5 : B.G >= 8 ? 1.2 : B.G >= 5 && coef != COEF_PACKED ? 1.15 : 1.0;
        const double issue = spill * P.bz * P.threads / 32.0 / 4.0 * group;
        double cost = issue + spill * P.bz * 400.0 + 6000.0 + 6.0 * nby * nbz;
        if (!alone) cost = std::max(cost, per_sm * issue + 2000.0) / (room / P.ctas);
        if (found && cost >= best) continue;
        found = true;
        best = cost;
        *out = P;
      }
    }
  }
  return found;
}
bool resident_plan(int nx, int ny, int nz, int mode, int coef, int num_sms, int max_smem, long l2_bytes, ResPlan *out) {
  return best_plan(nx, ny, nz, mode, coef, num_sms, max_smem, l2_bytes, true, out);
}
bool resident_batch_plan(int nx, int ny, int nz, int num_sms, int max_smem, ResPlan *out) {
  return best_plan(nx, ny, nz, MODE_F32_REFINE, COEF_PACKED, num_sms, max_smem, 0, false, out);
}

size_t resident_packet_bytes(int ctas) { return 2 * PACKET_STRIDE * sizeof(Packet) * (size_t)ctas; }

cudaError_t launch_resident(const ResPlan &P, const Inst &I, const Batch &B, void *packets, size_t packet_bytes,
                            cudaStream_t st) {
  const cudaError_t e = cudaMemsetAsync(packets, 0, packet_bytes, st);  // epochs count from 1 in every launch
  if (e != cudaSuccess) return e;
  const bool per = I.periodic != 0;
  ResOne R;
  R.grid[0] = grid_args(P, I, B.inst, B, packets, 0, P.threads, INT_MAX);
  const Shape L{P.ctas, P.threads, smem_of(P, I.mode == MODE_F64 ? 8 : 4, I.coef, P.threads)};
  if (I.mode == MODE_F64) {
    if (I.coef == COEF_F64) return launch_f64<COEF_F64>(L, R, per, st);
    return launch_f64<COEF_PACKED>(L, R, per, st);
  }
  if (I.coef == COEF_F32) return launch_f32<COEF_F32>(P.build, L, R, per, st);
  if (I.coef == COEF_BF16) return launch_f32<COEF_BF16>(P.build, L, R, per, st);
  return launch_f32<COEF_PACKED>(P.build, L, R, per, st);
}

cudaError_t launch_resident_batch(int n, const ResPlan *const *P, const Inst *const *I, const int *slot,
                                  const Batch &B, void *packets, size_t packet_bytes, int budget, cudaStream_t st) {
  const cudaError_t e = cudaMemsetAsync(packets, 0, packet_bytes, st);
  if (e != cudaSuccess) return e;
  Shape L{0, 0, 0};
  for (int k = 0; k < n; k++) L.threads = std::max(L.threads, P[k]->threads);
  ResWave W;
  W.n = n;
  for (int k = 0; k < n; k++) {
    W.first[k] = L.ctas;
    W.grid[k] = grid_args(*P[k], *I[k], B.inst + slot[k], B, (Packet *)packets + (size_t)2 * PACKET_STRIDE * L.ctas,
                          slot[k], L.threads, budget);
    L.ctas += P[k]->ctas;
    L.smem = std::max(L.smem, smem_of(*P[k], 4, COEF_PACKED, L.threads));
  }
  for (int k = n; k <= RES_MAX_GRIDS; k++) W.first[k] = L.ctas;
  const bool per = I[0]->periodic != 0;
  return launch_batch(P[0]->build, L, W, per, st);
}

}  // namespace pb

#ifdef PB_FAULT_TEST
// Test builds only: see g_fault_abandon_sums.
extern "C" int pb_test_abandon_sums(int count) {
  return cudaMemcpyToSymbol(pb::g_fault_abandon_sums, &count, sizeof(int)) == cudaSuccess ? 0 : 3;
}
#endif
