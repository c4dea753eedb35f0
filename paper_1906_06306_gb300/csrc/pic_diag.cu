// Diagnostics of the PIC state, held to at least double precision on the GPU:
// field and kinetic energies, the first-order charge on the nodes and the
// discrete Gauss residual div E - rho of Appendix B (arXiv:1906.06306).
#include "pic_kernels.h"

namespace pic {

static unsigned blocks_for(long long n) {
  long long b = (n + 255) / 256;
  if (b > 152LL * 16) b = 152LL * 16;
  return (unsigned)(b < 1 ? 1 : b);
}

// Blocks of a reduction: every thread ends in a block sum of FP64 exchanges
// (ten additions of the slow pipe), so a grid of 4 blocks per SM, each thread
// with several terms, measures faster than one that fills the SMs (field
// energy of a 1024^2 box 30.5 us with 16 blocks per SM).
static unsigned blocks_for_sum(long long n) {
  const unsigned b = blocks_for(n);
  return b < 152u * 4u ? b : 152u * 4u;
}

__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 32) {
    s = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  }
  return s;  // valid in thread 0
}

// The GPU's FP64 pipe issues one operation for some thirty FP32 ones, so the
// diagnostics form their terms and the sums of a thread's terms as sums of three
// floats, s0 + s1 + s2, each about 2^-24 of the one before: 64 bits and more,
// where FP64 holds 53.  The error-free sum is Knuth's, the error-free product
// the fused multiply-add's.  Two values go through each step as the halves of
// the packed FP32 instructions.
__device__ __forceinline__ float2 neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a + b = s + the return value
__device__ __forceinline__ float2 two_sum(float2 a, float2 b, float2& s) {
  s = add(a, b);
  const float2 t = add(s, neg(a));
  return add(add(a, neg(add(s, neg(t)))), add(b, neg(t)));
}
// a a = p + the return value
__device__ __forceinline__ float2 square(float2 a, float2& p) {
  p = mul(a, a);
  return fma(a, a, neg(p));
}
struct Sum3 {
  float2 s0, s1, s2;
  __device__ __forceinline__ void add_term(float2 h, float2 l) {
    const float2 e = two_sum(s0, h, s0);
    const float2 f = two_sum(s1, l, s1);
    const float2 g = two_sum(s1, e, s1);
    s2 = add(s2, add(f, g));
  }
  __device__ __forceinline__ double x() const { return (double)s0.x + ((double)s1.x + s2.x); }
  __device__ __forceinline__ double y() const { return (double)s0.y + ((double)s1.y + s2.y); }
};
// approximations with a relative error below 2^-21 for normal arguments
__device__ __forceinline__ float rsqrt_approx(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Whether the squares of three floats can be summed this way: the sum of their
// magnitudes is 0 or between 2^-40 and 2^60 (not for NaN and infinities).
// Others take FP64.
__device__ __forceinline__ bool sum3_range(float a, float b, float c) {
  const float m = fabsf(a) + fabsf(b) + fabsf(c);
  return (m >= 0x1p-40f && m <= 0x1p60f) || m == 0.f;
}

constexpr int kSumTerms = 16;  // points or pairs of a thread before its FP64 sum takes them

// Not inlined: a branch, not FP64 operations that every thread goes through.
__device__ __noinline__ double squares_fp64(float a, float b, float c) {
  return (double)a * a + (double)b * b + (double)c * c;
}

// Sums of E^2 and B^2, one in each half, four points of a thread at a time:
// 1024^2 box 15 us (FP64 products and sums 40; 38 with the rare FP64 form
// inlined, which the compiler then evaluates for every point).
__global__ void k_field_energy(const float* __restrict__ F, long long P, double* acc) {
  __shared__ double sh[32];
  double se = 0.0, sb = 0.0;
  Sum3 sum = {};
  int terms = 0;
  const long long stride = (long long)gridDim.x * blockDim.x;
  constexpr int U = 4;  // rounds whose loads are issued together
  for (long long base = blockIdx.x * (long long)blockDim.x + threadIdx.x; base < P;
       base += U * stride) {
    float2 v[U][3];
#pragma unroll
    for (int r = 0; r < U; ++r) {
      const long long i = base + r * stride;
#pragma unroll
      for (int a = 0; a < 3; ++a)
        v[r][a] = i < P ? make_float2(F[(EX + a) * P + i], F[(BX + a) * P + i]) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int r = 0; r < U; ++r) {
      if (!sum3_range(v[r][0].x, v[r][1].x, v[r][2].x)) {
        se += squares_fp64(v[r][0].x, v[r][1].x, v[r][2].x);
        v[r][0].x = v[r][1].x = v[r][2].x = 0.f;  // adds nothing below
      }
      if (!sum3_range(v[r][0].y, v[r][1].y, v[r][2].y)) {
        sb += squares_fp64(v[r][0].y, v[r][1].y, v[r][2].y);
        v[r][0].y = v[r][1].y = v[r][2].y = 0.f;
      }
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        float2 p;
        const float2 l = square(v[r][a], p);
        sum.add_term(p, l);
      }
    }
    terms += U;
    if (terms == kSumTerms) {
      terms = 0;
      se += sum.x();
      sb += sum.y();
      sum = {};
    }
  }
  se += sum.x();
  sb += sum.y();
  se = block_sum(se, sh);
  sb = block_sum(sb, sh);
  if (threadIdx.x == 0) {
    atomicAdd(acc, 0.5 * se);
    atomicAdd(acc + 1, 0.5 * sb);
  }
}

// t = gamma - 1 as t0 + t1 + t2, for components in sum3_range: the root of
// t (t + 2) = u^2.  u^2 is held to 2^-68 of its value, t0 is its FP32 value, and
// t1 and t2 are the corrections that the remainder u^2 - t (t + 2), formed from
// error-free products and sums, asks for (divided by 2 (t + 1), whose reciprocal
// is half of 1/gamma): the sum is good to 2^-62.
__device__ __forceinline__ void gamma_minus_1(float2 a, float2 b, float2 c, float2& t0, float2& t1,
                                              float2& t2) {
  float2 pa, pb, pc, s, u0, u1, m, q;
  const float2 la = square(a, pa), lb = square(b, pb), lc = square(c, pc);
  const float2 e1 = two_sum(pa, pb, s), e2 = two_sum(s, pc, u0);
  const float2 f1 = two_sum(e1, e2, m), f2 = two_sum(la, lb, q), f3 = two_sum(q, lc, q),
               f4 = two_sum(m, q, u1);
  const float2 u2 = add(add(f1, f2), add(f3, f4));
  const float2 x = add(u0, make_float2(1.f, 1.f));
  const float2 y = make_float2(rsqrt_approx(x.x), rsqrt_approx(x.y));
  const float2 g1 = fma(x, y, make_float2(1.f, 1.f));
  t0 = mul(u0, make_float2(rcp_approx(g1.x), rcp_approx(g1.y)));
  const float2 hy = mul(y, make_float2(0.5f, 0.5f)), tt = add(t0, t0);
  // u^2 - t0^2 - 2 t0: the leading parts agree to 2^-20, their difference is exact
  float2 p, d, r;
  const float2 lp = square(t0, p), ld = two_sum(p, tt, d);
  const float2 h1 = two_sum(add(u0, neg(d)), u1, r), h2 = two_sum(r, neg(ld), r),
               h3 = two_sum(r, neg(lp), r);
  const float2 rest = add(add(h1, h2), add(h3, u2));
  t1 = mul(r, hy);
  float2 w;  // 2 t0 + 2
  const float2 lw = two_sum(tt, make_float2(2.f, 2.f), w);
  const float2 r1 = add(fma(neg(t1), w, r), rest);
  t2 = mul(fma(neg(t1), add(lw, t1), r1), hy);
}

// Sum of m c^2 (gamma - 1).  With square root and quotient in FP64 the FP64
// pipe bounded it, 769 us for 16.8 M particles; with terms of three floats,
// two particles to an instruction, it takes 75 us, bound by FP32 arithmetic
// (some 115 packed operations a pair; the reads alone would take 30 us; terms of
// two floats, good to 2^-44 only, took 60).  16 blocks per SM, not the 4 of the
// other sums (81 us): with this much work in a thread, late blocks even out.
__global__ void __launch_bounds__(256) k_kinetic(const float* __restrict__ u, long long n,
                                                 long long ld, double mc2, double* acc) {
  __shared__ double sh[32];
  double s = 0.0;
  Sum3 sum = {};
  int terms = 0;
  const long long stride = (long long)gridDim.x * blockDim.x;
  constexpr int U = 4;  // rounds whose loads are issued together, two to a pair
  for (long long base = blockIdx.x * (long long)blockDim.x + threadIdx.x; base < n;
       base += U * stride) {
    float v[U][3];
#pragma unroll
    for (int r = 0; r < U; ++r) {
      const long long p = base + r * stride;
#pragma unroll
      for (int a = 0; a < 3; ++a) v[r][a] = p < n ? u[a * ld + p] : 0.f;
    }
#pragma unroll
    for (int r = 0; r < U; ++r) {
      if (!sum3_range(v[r][0], v[r][1], v[r][2])) {
        const double u2 = squares_fp64(v[r][0], v[r][1], v[r][2]);
        s += u2 / (sqrt(1.0 + u2) + 1.0);
        v[r][0] = v[r][1] = v[r][2] = 0.f;  // adds nothing below
      }
    }
#pragma unroll
    for (int r = 0; r < U; r += 2) {
      float2 t0, t1, t2;
      gamma_minus_1(make_float2(v[r][0], v[r + 1][0]), make_float2(v[r][1], v[r + 1][1]),
                    make_float2(v[r][2], v[r + 1][2]), t0, t1, t2);
      sum.add_term(t0, t1);
      sum.s2 = add(sum.s2, t2);
    }
    terms += U / 2;
    if (terms == kSumTerms) {
      terms = 0;
      s += sum.x() + sum.y();
      sum = {};
    }
  }
  s += sum.x() + sum.y();
  s = block_sum(s, sh);
  if (threadIdx.x == 0) atomicAdd(acc, mc2 * s);
}

// charge q with weights (1 - w, w) per gridded axis onto the 2^D nodes
template <int D>
__device__ __forceinline__ void rho_particle(const GridDev& g, int c, const float* o, double q,
                                             double* rho) {
  int ijk[3];
  ijk[0] = c % g.n[0];
  const int r = c / g.n[0];
  ijk[1] = r % g.n[1];
  ijk[2] = r / g.n[1];
  double w[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int d = 0; d < D; ++d) w[d] = o[d];
#pragma unroll
  for (int corner = 0; corner < (1 << D); ++corner) {
    double wt = q;
    int id[3] = {ijk[0], ijk[1], ijk[2]};
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const int up = (corner >> d) & 1;
      wt *= up ? w[d] : 1.0 - w[d];
      id[d] = up ? wrap1(id[d] + 1, g.n[d]) : id[d];
    }
    atomicAdd(&rho[id[0] + (long long)g.n[0] * (id[1] + (long long)g.n[1] * id[2])], wt);
  }
}

template <int D>
__global__ void k_rho(const GridDev g, const int* __restrict__ cell, const float* __restrict__ off,
                      long long first, long long n, long long ld, double q, double* rho) {
  for (long long p = first + blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n;
       p += (long long)gridDim.x * blockDim.x) {
    const int c = cell[p];
    if (c < 0 || (long long)c >= g.plane) continue;
    float o[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int d = 0; d < D; ++d) o[d] = off[d * ld + p];
    rho_particle<D>(g, c, o, q, rho);
  }
}

// The same charge for particles grouped by tile (1D and 2D), by fixed-point
// sums in shared memory.  A block takes its share of a tile's bucket and sums,
// for each cell of the tile's window, the particle count and the moments
// sum w_x, sum w_y, sum w_x w_y; the four corner weights of every particle are
// differences of these (w_x - w_x w_y, ...), so a node's charge is one integer
// sum over its four cells, rounded once to FP64.
// Nothing is cut off: an offset of 2^-8 or more (or 0) is whole in units of
// 2^-31, a product of two in units of 2^-62, and the node sums take 128-bit
// integers.  Each moment goes as 16-bit limbs into 32-bit words with native
// integer atomics (64-bit shared atomics are a compare-and-swap loop);
// kRhoBatch = 2^14 particles, a quarter of what a word holds, go between two
// folds.  Particles outside the window, or with other offsets (0.8 % of
// uniform ones on two axes), are queued and take the FP64 atomics of k_rho
// together, and so does the unsorted tail.  The global atomics bounded that
// kernel (one FP64 atomic per L2 slice and clock: 4 a particle, 338 us for
// 16.8 M in 2D); here a block issues one per window node, and the kernel takes
// 93 us, bound by instruction issue and 9 shared atomics a particle (87 us with
// moments cut at 2^-48, 8 atomics).  Four rounds of loads go out together.
constexpr int kRhoBatch = 1 << 14;
constexpr int kRhoQueue = 1024;

template <int D>
__host__ __device__ constexpr int rho_words() {
  return D == 1 ? 3 : 9;  // count; w_x, w_y in two limbs each; w_x w_y in four
}

__device__ __forceinline__ bool rho_whole(float w) { return (w >= 0x1p-8f && w < 1.0f) || w == 0.f; }

template <int D>
__global__ void __launch_bounds__(256, 6) k_rho_tiles(const GridDev g, const TileDev t, int splits,
                                                   FastDiv div0, const int* __restrict__ tstart,
                                                   const int* __restrict__ cell,
                                                   const float* __restrict__ off, long long ld,
                                                   double q, double* rho) {
  extern __shared__ unsigned sw[];
  __shared__ unsigned short queue[kRhoQueue];  // particles of the batch for the FP64 atomics
  __shared__ int queued;
  constexpr int NW = rho_words<D>();
  const int tile = blockIdx.x / splits, split = blockIdx.x - tile * splits;
  const int w0[2] = {(tile % t.nt[0]) * t.T[0] - t.H, D == 2 ? (tile / t.nt[0]) * t.T[1] - t.H : 0};
  const int W0 = t.W[0], W1 = D == 2 ? t.W[1] : 1, wc = W0 * W1;
  const bool near = W0 <= g.n[0] && (D < 2 || W1 <= g.n[1]);
  const long long lo = tstart[tile * t.nsub], len = tstart[(tile + 1) * t.nsub] - lo;
  const long long a = lo + len * split / splits, b = lo + len * (split + 1) / splits;
  for (long long first = a; first < b; first += kRhoBatch) {
    const long long last = first + kRhoBatch < b ? first + kRhoBatch : b;
    for (int w = threadIdx.x; w < NW * wc; w += blockDim.x) sw[w] = 0u;
    if (threadIdx.x == 0) queued = 0;
    __syncthreads();
    constexpr int U = 4;  // rounds whose loads are issued together
    const int here = (int)(last - first);
    for (int base = threadIdx.x; base < here; base += U * blockDim.x) {
      int cu[U];
      float ou[U][2];
#pragma unroll
      for (int r = 0; r < U; ++r) {
        const int p = base + r * blockDim.x;
        cu[r] = p < here ? cell[first + p] : -1;
        ou[r][0] = p < here ? off[first + p] : 0.f;
        ou[r][1] = D == 2 && p < here ? off[ld + first + p] : 0.f;
      }
#pragma unroll
      for (int r = 0; r < U; ++r) {
        const int c = cu[r];
        const float* o = ou[r];
        if (c < 0 || (long long)c >= g.plane) continue;
        const int j = D == 2 ? fdiv(c, div0) : 0, i = c - j * g.n[0];
        int l0 = i - w0[0], l1 = D == 2 ? j - w0[1] : 0;
        if (near) {  // at most one period away
          l0 = wrap1(l0, g.n[0]);
          if (D == 2) l1 = wrap1(l1, g.n[1]);
        } else {
          l0 = wrapi(l0, g.n[0]);
          if (D == 2) l1 = wrapi(l1, g.n[1]);
        }
        bool in = l0 < W0 - 1 && rho_whole(o[0]);
        if (D == 2) in &= l1 < W1 - 1 && rho_whole(o[1]);
        if (in) {
          unsigned* s = sw + l0 + W0 * l1;
          const unsigned x = __float2uint_rz(o[0] * 0x1p31f);
          atomicAdd(s, 1u);
          atomicAdd(s + wc, x & 0xffffu);
          atomicAdd(s + 2 * wc, x >> 16);
          if (D == 2) {
            const unsigned y = __float2uint_rz(o[1] * 0x1p31f);
            const unsigned long long xy = (unsigned long long)x * y;
            atomicAdd(s + 3 * wc, y & 0xffffu);
            atomicAdd(s + 4 * wc, y >> 16);
            atomicAdd(s + 5 * wc, (unsigned)xy & 0xffffu);
            atomicAdd(s + 6 * wc, (unsigned)xy >> 16);
            atomicAdd(s + 7 * wc, (unsigned)(xy >> 32) & 0xffffu);
            atomicAdd(s + 8 * wc, (unsigned)(xy >> 48));
          }
        } else {
          const int slot = atomicAdd(&queued, 1);
          if (slot < kRhoQueue)
            queue[slot] = (unsigned short)(base + r * blockDim.x);
          else
            rho_particle<D>(g, c, o, q, rho);
        }
      }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < min(queued, kRhoQueue); k += blockDim.x) {
      const long long p = first + queue[k];
      const float o[3] = {off[p], D == 2 ? off[ld + p] : 0.f, 0.f};
      rho_particle<D>(g, cell[p], o, q, rho);
    }
    for (int w = threadIdx.x; w < wc; w += blockDim.x) {
      const int lx = w % W0, ly = w / W0;
      // sums of cell v: {count, w_x, w_y} in units of 2^-31, w_x w_y in 2^-62
      const auto linear = [&](int v, long long* m) {
        m[0] = (long long)sw[v] << 31;
        m[1] = (long long)sw[v + wc] + ((long long)sw[v + 2 * wc] << 16);
        m[2] = D == 2 ? (long long)sw[v + 3 * wc] + ((long long)sw[v + 4 * wc] << 16) : 0;
      };
      const auto product = [&](int v) {
        const unsigned long long lo = sw[v + 5 * wc] + ((unsigned long long)sw[v + 6 * wc] << 16);
        const unsigned long long hi = sw[v + 7 * wc] + ((unsigned long long)sw[v + 8 * wc] << 16);
        return (__int128)lo + ((__int128)hi << 32);
      };
      long long sum = 0, m[3];  // units of 2^-31
      __int128 sum2 = 0;        // units of 2^-62
      linear(w, m);
      sum += m[0] - m[1] - m[2];
      if (D == 2) sum2 += product(w);
      if (lx > 0) {
        linear(w - 1, m);
        sum += m[1];
        if (D == 2) sum2 -= product(w - 1);
      }
      if (D == 2 && ly > 0) {
        linear(w - W0, m);
        sum += m[2];
        sum2 -= product(w - W0);
        if (lx > 0) sum2 += product(w - W0 - 1);
      }
      if (D == 2) sum2 += (__int128)sum << 31;
      if (D == 1 ? sum != 0 : sum2 != 0) {
        // at most 2^45 and 2^76: all but the last addition are exact
        const double charge = D == 1 ? (double)sum * 0x1p-31
                                     : (double)(long long)(sum2 >> 32) * 0x1p-30 +
                                           (double)(unsigned)sum2 * 0x1p-62;
        const int i = wrapi(w0[0] + lx, g.n[0]), j = D == 2 ? wrapi(w0[1] + ly, g.n[1]) : 0;
        atomicAdd(&rho[i + (long long)g.n[0] * j], q * charge);
      }
    }
    __syncthreads();
  }
}

// res = div- E - rho on the nodes with i_lo <= i < i_hi; max |res| (bit
// pattern of a non-negative double, which orders like the value) and sum res^2
template <int D>
__global__ void k_gauss(const GridDev g, const float* __restrict__ F, const double* __restrict__ rho,
                        int i_lo, int i_hi, unsigned long long* acc_max, double* acc_sq) {
  __shared__ double sh[32];
  __shared__ unsigned long long shm;
  if (threadIdx.x == 0) shm = 0ull;
  const long long P = g.plane;
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  double sq = 0.0, mx = 0.0;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < P;
       idx += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(idx % n0);
    const long long r = idx / n0;
    const int j = (int)(r % n1), k = (int)(r / n1);
    if (i < i_lo || i >= i_hi) continue;
    double div = (double)F[EX * P + idx] - (double)F[EX * P + idx - ((i > 0) ? 1 : 1 - n0)];
    if (D >= 2)
      div += (double)F[EY * P + idx] -
             (double)F[EY * P + idx - ((j > 0) ? n0 : (long long)n0 * (1 - n1))];
    if (D >= 3)
      div += (double)F[EZ * P + idx] -
             (double)F[EZ * P + idx - ((k > 0) ? (long long)n0 * n1 : (long long)n0 * n1 * (1 - n2))];
    const double res = div - rho[idx];
    sq += res * res;
    mx = fmax(mx, fabs(res));
  }
  sq = block_sum(sq, sh);
  __syncthreads();
  atomicMax(&shm, (unsigned long long)__double_as_longlong(mx));
  __syncthreads();
  if (threadIdx.x == 0) {
    atomicAdd(acc_sq, sq);
    atomicMax(acc_max, shm);
  }
}

cudaError_t launch_field_energy(const GridDev& g, const float* F, double* acc, cudaStream_t st) {
  k_field_energy<<<blocks_for_sum(g.plane), 256, 0, st>>>(F, g.plane, acc);
  return cudaGetLastError();
}

cudaError_t launch_kinetic(const float* u, long long n, long long ld, double mc2, double* acc,
                           cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_kinetic<<<blocks_for(n), 256, 0, st>>>(u, n, ld, mc2, acc);
  return cudaGetLastError();
}

static cudaError_t launch_rho_global(const GridDev& g, const int* cell, const float* off,
                                     long long first, long long n, long long ld, double q,
                                     double* rho, cudaStream_t st) {
  if (n <= first) return cudaSuccess;
  const unsigned nb = blocks_for(n - first);
  switch (g.dim) {
    case 1: k_rho<1><<<nb, 256, 0, st>>>(g, cell, off, first, n, ld, q, rho); break;
    case 2: k_rho<2><<<nb, 256, 0, st>>>(g, cell, off, first, n, ld, q, rho); break;
    case 3: k_rho<3><<<nb, 256, 0, st>>>(g, cell, off, first, n, ld, q, rho); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// The tile kernel for the grouped particles of 1D and 2D boxes (about 8192 of
// them to a block, so that zeroing and folding a window stay small), and the
// global one for what follows them.  3D takes the global kernel: eight moments
// of an 8x8x4 tile's window would take 134 KB of shared memory.
cudaError_t launch_rho(const GridDev& g, const TileDev& t, const int* tstart, const int* cell,
                       const float* off, long long sorted, long long n, long long ld, double q,
                       double* rho, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const size_t smem = sizeof(unsigned) * (g.dim == 1 ? rho_words<1>() : rho_words<2>()) * (size_t)t.wcells;
  if (g.dim == 3 || sorted == 0 || smem > 200 * 1024)
    return launch_rho_global(g, cell, off, 0, n, ld, q, rho, st);
  const void* k = g.dim == 1 ? (const void*)k_rho_tiles<1> : (const void*)k_rho_tiles<2>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  if (e != cudaSuccess) return e;
  long long splits = (sorted / t.ntiles + 8191) / 8192;
  splits = splits < 1 ? 1 : splits > 1024 ? 1024 : splits;
  const unsigned nb = (unsigned)(t.ntiles * splits);
  const FastDiv d0 = make_fastdiv(g.n[0]);
  if (g.dim == 1)
    k_rho_tiles<1><<<nb, 256, smem, st>>>(g, t, (int)splits, d0, tstart, cell, off, ld, q, rho);
  else
    k_rho_tiles<2><<<nb, 256, smem, st>>>(g, t, (int)splits, d0, tstart, cell, off, ld, q, rho);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_rho_global(g, cell, off, sorted, n, ld, q, rho, st);
}

cudaError_t launch_gauss(const GridDev& g, const float* F, const double* rho, int i_lo, int i_hi,
                         unsigned long long* acc_max, double* acc_sq, cudaStream_t st) {
  const unsigned nb = blocks_for_sum(g.plane);
  switch (g.dim) {
    case 1: k_gauss<1><<<nb, 256, 0, st>>>(g, F, rho, i_lo, i_hi, acc_max, acc_sq); break;
    case 2: k_gauss<2><<<nb, 256, 0, st>>>(g, F, rho, i_lo, i_hi, acc_max, acc_sq); break;
    case 3: k_gauss<3><<<nb, 256, 0, st>>>(g, F, rho, i_lo, i_hi, acc_max, acc_sq); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// One warp waits on a shared-memory barrier that nothing completes: its
// bounded wait gives up after about a second of SM clock and sets ST_TIMEOUT
// in the status word, as a particle block's wait on a tensor copy that never
// landed would.  No copy is in flight, so leaving is safe.
__global__ void k_wait_probe(int* status) {
  __shared__ unsigned long long bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_init_fence();
  }
  __syncthreads();
  mbar_wait(&bar, 0, status);
}

cudaError_t launch_wait_probe(int* status, cudaStream_t st) {
  k_wait_probe<<<1, 32, 0, st>>>(status);
  return cudaGetLastError();
}

}  // namespace pic
