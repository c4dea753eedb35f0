// FDTD2 and FDTD4 field updates (arXiv:1906.06306, Sect. 2.3.1, Eqs. (fdE),
// (fdB), Table 2) on periodic Yee planes, and the FP64 form of the Binomial2
// filter's sub-pass (the current's filter: pic_filter.cu).
// One thread per lattice point (or four), x fastest, so every plane is streamed
// with coalesced loads; neighbours one point away come from the same or adjacent
// rows and hit L1/L2.
#include "pic_kernels.h"

namespace pic {

// B -= (c/2) curl+ E (forward differences: B sits half a cell above E), and,
// when zero_j is set, clear J for the deposit that follows.
template <int D>
__device__ __forceinline__ void b_half_point(float* __restrict__ F, const GridDev& g, int i, int j,
                                             int k, float hc, int zero_j) {
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const long long P = g.plane;
  const long long idx = (long long)i + (long long)n0 * (j + (long long)n1 * k);
  const long long sx = (i + 1 < n0) ? 1 : 1 - n0;
  const long long sy = (D >= 2) ? ((j + 1 < n1) ? n0 : (long long)n0 * (1 - n1)) : 0;
  const long long sz = (D >= 3) ? ((k + 1 < n2) ? (long long)n0 * n1 : (long long)n0 * n1 * (1 - n2)) : 0;
  const float* Ex = F + EX * P;
  const float* Ey = F + EY * P;
  const float* Ez = F + EZ * P;
  const float ex = Ex[idx], ey = Ey[idx], ez = Ez[idx];
  float cx = 0.f, cy = 0.f, cz = 0.f;
  cy -= Ez[idx + sx] - ez;
  cz += Ey[idx + sx] - ey;
  if (D >= 2) {
    cx += Ez[idx + sy] - ez;
    cz -= Ex[idx + sy] - ex;
  }
  if (D >= 3) {
    cx -= Ey[idx + sz] - ey;
    cy += Ex[idx + sz] - ex;
  }
  F[BX * P + idx] = fmaf(-hc, cx, F[BX * P + idx]);
  F[BY * P + idx] = fmaf(-hc, cy, F[BY * P + idx]);
  F[BZ * P + idx] = fmaf(-hc, cz, F[BZ * P + idx]);
  if (zero_j) {
    F[JX * P + idx] = 0.f;
    F[JY * P + idx] = 0.f;
    F[JZ * P + idx] = 0.f;
  }
}

template <int D>
__global__ void k_b_half(float* __restrict__ F, const GridDev g, float hc, int zero_j,
                         int push_next) {
  grid_dependency(push_next);
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n0) return;
  FOR_ROWS(j, k) { b_half_point<D>(F, g, i, j, k, hc, zero_j); }
}

// E += c curl- B - J (backward differences: E sits half a cell below B).
template <int D>
__device__ __forceinline__ void e_update_point(float* __restrict__ F, const float* J,
                                               const GridDev& g, int i, int j, int k, float c) {
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const long long P = g.plane;
  const long long idx = (long long)i + (long long)n0 * (j + (long long)n1 * k);
  const long long sx = (i > 0) ? 1 : 1 - n0;
  const long long sy = (D >= 2) ? ((j > 0) ? n0 : (long long)n0 * (1 - n1)) : 0;
  const long long sz = (D >= 3) ? ((k > 0) ? (long long)n0 * n1 : (long long)n0 * n1 * (1 - n2)) : 0;
  const float* Bx = F + BX * P;
  const float* By = F + BY * P;
  const float* Bz = F + BZ * P;
  const float bx = Bx[idx], by = By[idx], bz = Bz[idx];
  float cx = 0.f, cy = 0.f, cz = 0.f;
  cy -= bz - Bz[idx - sx];
  cz += by - By[idx - sx];
  if (D >= 2) {
    cx += bz - Bz[idx - sy];
    cz -= bx - Bx[idx - sy];
  }
  if (D >= 3) {
    cx -= by - By[idx - sz];
    cy += bx - Bx[idx - sz];
  }
  const float jx = J[idx], jy = J[P + idx], jz = J[2 * P + idx];
  F[EX * P + idx] = fmaf(c, cx, F[EX * P + idx]) - jx;
  F[EY * P + idx] = fmaf(c, cy, F[EY * P + idx]) - jy;
  F[EZ * P + idx] = fmaf(c, cz, F[EZ * P + idx]) - jz;
  if (J != F + JX * P) {  // the filter left it in its buffer
    F[JX * P + idx] = jx;
    F[JY * P + idx] = jy;
    F[JZ * P + idx] = jz;
  }
}

template <int D>
__global__ void k_e_update(float* __restrict__ F, const float* J, const GridDev g, float c) {
  grid_dependency();
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n0) return;
  FOR_ROWS(j, k) { e_update_point<D>(F, J, g, i, j, k, c); }
}

// The second B half step and the E update of a small lattice by one block, in
// shared memory: the planes are read once, every point's B half step, a
// block barrier, every point's E update, and the planes are written once; the
// operations of k_b_half and k_e_update point by point, so the same bits.  One
// launch instead of two where launch and memory latency, not bandwidth, bound
// the step.  With `chain` set, after another barrier, the next step's first B
// half step (which clears J for its deposit) as well: one launch instead of
// three.  512 points: 7.0 us with the loads of a plane one after the other, 3.4
// with all nine in flight (5.6 us with every phase in global memory).
template <int D>
__global__ void __launch_bounds__(1024) k_fields_small(float* __restrict__ F, const float* J,
                                                       const GridDev g, float hc, float c,
                                                       int chain) {
  grid_dependency();
  extern __shared__ float sm[];  // the 9 planes
  const int n0 = g.n[0], n1 = g.n[1];
  const int cells = (int)g.plane;
  for (int t = threadIdx.x; t < cells; t += blockDim.x) {
    float v[9];  // all in flight together
#pragma unroll
    for (int q = 0; q < 9; ++q) v[q] = q < 6 ? F[q * cells + t] : J[(q - 6) * cells + t];
#pragma unroll
    for (int q = 0; q < 9; ++q) sm[q * cells + t] = v[q];
  }
  __syncthreads();
  const auto every_point = [&](auto fn) {
    for (int t = threadIdx.x; t < cells; t += blockDim.x) {
      const int r = D == 1 ? 0 : t / n0;
      fn(t - r * n0, D == 3 ? r % n1 : r, D == 3 ? r / n1 : 0);
    }
    __syncthreads();
  };
  every_point([&](int i, int j, int k) { b_half_point<D>(sm, g, i, j, k, hc, 0); });
  every_point([&](int i, int j, int k) { e_update_point<D>(sm, sm + 6 * cells, g, i, j, k, c); });
  if (chain) every_point([&](int i, int j, int k) { b_half_point<D>(sm, g, i, j, k, hc, 1); });
  const int planes = chain || J != F + JX * g.plane ? 9 : 6;
  for (int t = threadIdx.x; t < cells; t += blockDim.x) {
#pragma unroll
    for (int q = 0; q < 9; ++q)
      if (q < planes) F[q * cells + t] = sm[q * cells + t];
  }
}

// The same two updates with four consecutive x points per thread (rows whose
// length is a multiple of 4 and 16-byte aligned planes): 16-byte loads and
// stores of the thread's points, one scalar load for the x neighbour outside
// them.  Each point goes through the operations of k_b_half / k_e_update in
// the same order, so the results are the same bits.
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, const float v[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void arr4(const float4 a, float v[4]) {
  v[0] = a.x;
  v[1] = a.y;
  v[2] = a.z;
  v[3] = a.w;
}

template <int D>
__global__ void k_b_half_x4(float* __restrict__ F, const GridDev g, float hc, int zero_j,
                            int push_next) {
  grid_dependency(push_next);
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const long long P = g.plane;
  const int i = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n0) return;
  FOR_ROWS(j, k) {
    const long long idx = (long long)i + (long long)n0 * (j + (long long)n1 * k);
    const long long x4 = (i + 4 < n0) ? idx + 4 : idx + 4 - n0;  // x neighbour of the last point
    const long long sy = (D >= 2) ? ((j + 1 < n1) ? n0 : (long long)n0 * (1 - n1)) : 0;
    const long long sz = (D >= 3) ? ((k + 1 < n2) ? (long long)n0 * n1 : (long long)n0 * n1 * (1 - n2)) : 0;
    const float* Ex = F + EX * P;
    const float* Ey = F + EY * P;
    const float* Ez = F + EZ * P;
    float ex[4], ey[4], ez[4], eyx[4], ezx[4], ezy[4] = {}, exy[4] = {}, eyz[4] = {}, exz[4] = {};
    arr4(ld4(Ex + idx), ex);
    arr4(ld4(Ey + idx), ey);
    arr4(ld4(Ez + idx), ez);
    eyx[0] = ey[1], eyx[1] = ey[2], eyx[2] = ey[3], eyx[3] = Ey[x4];
    ezx[0] = ez[1], ezx[1] = ez[2], ezx[2] = ez[3], ezx[3] = Ez[x4];
    if (D >= 2) {
      arr4(ld4(Ez + idx + sy), ezy);
      arr4(ld4(Ex + idx + sy), exy);
    }
    if (D >= 3) {
      arr4(ld4(Ey + idx + sz), eyz);
      arr4(ld4(Ex + idx + sz), exz);
    }
    float bx[4], by[4], bz[4];
    arr4(ld4(F + BX * P + idx), bx);
    arr4(ld4(F + BY * P + idx), by);
    arr4(ld4(F + BZ * P + idx), bz);
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      float cx = 0.f, cy = 0.f, cz = 0.f;
      cy -= ezx[l] - ez[l];
      cz += eyx[l] - ey[l];
      if (D >= 2) {
        cx += ezy[l] - ez[l];
        cz -= exy[l] - ex[l];
      }
      if (D >= 3) {
        cx -= eyz[l] - ey[l];
        cy += exz[l] - ex[l];
      }
      bx[l] = fmaf(-hc, cx, bx[l]);
      by[l] = fmaf(-hc, cy, by[l]);
      bz[l] = fmaf(-hc, cz, bz[l]);
    }
    st4(F + BX * P + idx, bx);
    st4(F + BY * P + idx, by);
    st4(F + BZ * P + idx, bz);
    if (zero_j) {
      const float z[4] = {0.f, 0.f, 0.f, 0.f};
      st4(F + JX * P + idx, z);
      st4(F + JY * P + idx, z);
      st4(F + JZ * P + idx, z);
    }
  }
}

template <int D>
__global__ void k_e_update_x4(float* __restrict__ F, const float* J, const GridDev g, float c) {
  grid_dependency();
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const long long P = g.plane;
  const int i = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n0) return;
  FOR_ROWS(j, k) {
    const long long idx = (long long)i + (long long)n0 * (j + (long long)n1 * k);
    const long long xm = (i > 0) ? idx - 1 : idx + n0 - 1;  // x neighbour of the first point
    const long long sy = (D >= 2) ? ((j > 0) ? n0 : (long long)n0 * (1 - n1)) : 0;
    const long long sz = (D >= 3) ? ((k > 0) ? (long long)n0 * n1 : (long long)n0 * n1 * (1 - n2)) : 0;
    const float* Bx = F + BX * P;
    const float* By = F + BY * P;
    const float* Bz = F + BZ * P;
    float bx[4], by[4], bz[4], byx[4], bzx[4], bzy[4] = {}, bxy[4] = {}, byz[4] = {}, bxz[4] = {};
    arr4(ld4(Bx + idx), bx);
    arr4(ld4(By + idx), by);
    arr4(ld4(Bz + idx), bz);
    byx[0] = By[xm], byx[1] = by[0], byx[2] = by[1], byx[3] = by[2];
    bzx[0] = Bz[xm], bzx[1] = bz[0], bzx[2] = bz[1], bzx[3] = bz[2];
    if (D >= 2) {
      arr4(ld4(Bz + idx - sy), bzy);
      arr4(ld4(Bx + idx - sy), bxy);
    }
    if (D >= 3) {
      arr4(ld4(By + idx - sz), byz);
      arr4(ld4(Bx + idx - sz), bxz);
    }
    float ex[4], ey[4], ez[4], jx[4], jy[4], jz[4];
    arr4(ld4(F + EX * P + idx), ex);
    arr4(ld4(F + EY * P + idx), ey);
    arr4(ld4(F + EZ * P + idx), ez);
    arr4(ld4(J + idx), jx);
    arr4(ld4(J + P + idx), jy);
    arr4(ld4(J + 2 * P + idx), jz);
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      float cx = 0.f, cy = 0.f, cz = 0.f;
      cy -= bz[l] - bzx[l];
      cz += by[l] - byx[l];
      if (D >= 2) {
        cx += bz[l] - bzy[l];
        cz -= bx[l] - bxy[l];
      }
      if (D >= 3) {
        cx -= by[l] - byz[l];
        cy += bx[l] - bxz[l];
      }
      ex[l] = fmaf(c, cx, ex[l]) - jx[l];
      ey[l] = fmaf(c, cy, ey[l]) - jy[l];
      ez[l] = fmaf(c, cz, ez[l]) - jz[l];
    }
    st4(F + EX * P + idx, ex);
    st4(F + EY * P + idx, ey);
    st4(F + EZ * P + idx, ez);
    if (J != F + JX * P) {
      st4(F + JX * P + idx, jx);
      st4(F + JY * P + idx, jy);
      st4(F + JZ * P + idx, jz);
    }
  }
}

// One Binomial2 sub-pass along one axis: dst = (1/4, 1/2, 1/4) * src along
// `axis`, periodic.  Thread (x, y, z*ncomp) of a 3D launch grid owns one
// lattice value, so neighbours along every axis are coalesced loads.
template <typename T>
__global__ void k_filter_axis(const T* __restrict__ src, T* __restrict__ dst, const GridDev g,
                              int axis) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.n[0]) return;
  const int j = blockIdx.y;
  const int k = blockIdx.z % g.n[2];
  const long long comp = blockIdx.z / g.n[2];
  const long long P = g.plane;
  const long long idx = (long long)i + (long long)g.n[0] * (j + (long long)g.n[1] * k);
  const T* s = src + comp * P;
  const int a = axis == 0 ? i : axis == 1 ? j : k;
  const int na = g.n[axis];
  const long long stride = axis == 0 ? 1 : axis == 1 ? (long long)g.n[0] : (long long)g.n[0] * g.n[1];
  const long long lo = a > 0 ? idx - stride : idx + (long long)(na - 1) * stride;
  const long long hi = a + 1 < na ? idx + stride : idx - (long long)(na - 1) * stride;
  dst[comp * P + idx] = T(0.25) * s[lo] + T(0.5) * s[idx] + T(0.25) * s[hi];
}

// Offsets (elements) of the lattice points a-2, a-1, a+1, a+2 along an axis of
// n points with stride s, periodic.
struct Nb {
  long long m2, m1, p1, p2;
};
__device__ __forceinline__ Nb neighbours(int a, int n, long long s) {
  // From two points on one conditional wrap reaches every neighbour (eight
  // remainders a point before: a half step on 768 x 384 points 7.1 -> 5.7 us,
  // the E update 7.4 -> 6.4).
  if (n == 1) return Nb{0, 0, 0, 0};
  Nb r;
  r.m2 = (long long)(wrap1(a - 2, n) - a) * s;
  r.m1 = (long long)(wrap1(a - 1, n) - a) * s;
  r.p1 = (long long)(wrap1(a + 1, n) - a) * s;
  r.p2 = (long long)(wrap1(a + 2, n) - a) * s;
  return r;
}
// fourth-order staggered differences (FDTD4): at the point half a cell up
// (forward) or down (backward) the axis, coefficients 9/8 and -1/24
__device__ __forceinline__ float d4p(const float* A, long long i, const Nb& b) {
  return 1.125f * (A[i + b.p1] - A[i]) - (1.0f / 24.0f) * (A[i + b.p2] - A[i + b.m1]);
}
__device__ __forceinline__ float d4m(const float* A, long long i, const Nb& b) {
  return 1.125f * (A[i] - A[i + b.m1]) - (1.0f / 24.0f) * (A[i + b.p1] - A[i + b.m2]);
}

// FDTD4 versions of the two updates (same structure as above, wider stencil).
template <int D>
__global__ void k_b_half4(float* __restrict__ F, const GridDev g, float hc, int zero_j,
                          int push_next) {
  grid_dependency(push_next);
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const long long P = g.plane;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n0) return;
  FOR_ROWS(j, k) {
    const long long idx = (long long)i + (long long)n0 * (j + (long long)n1 * k);
    const Nb nx = neighbours(i, g.n[0], 1);
    const Nb ny = neighbours(j, g.n[1], g.n[0]);
    const Nb nz = neighbours(k, g.n[2], (long long)g.n[0] * g.n[1]);
    const float* Ex = F + EX * P;
    const float* Ey = F + EY * P;
    const float* Ez = F + EZ * P;
    float cx = 0.f, cy = 0.f, cz = 0.f;
    cy -= d4p(Ez, idx, nx);
    cz += d4p(Ey, idx, nx);
    if (D >= 2) {
      cx += d4p(Ez, idx, ny);
      cz -= d4p(Ex, idx, ny);
    }
    if (D >= 3) {
      cx -= d4p(Ey, idx, nz);
      cy += d4p(Ex, idx, nz);
    }
    F[BX * P + idx] = fmaf(-hc, cx, F[BX * P + idx]);
    F[BY * P + idx] = fmaf(-hc, cy, F[BY * P + idx]);
    F[BZ * P + idx] = fmaf(-hc, cz, F[BZ * P + idx]);
    if (zero_j) {
      F[JX * P + idx] = 0.f;
      F[JY * P + idx] = 0.f;
      F[JZ * P + idx] = 0.f;
    }
  }
}

template <int D>
__global__ void k_e_update4(float* __restrict__ F, const float* J, const GridDev g, float c) {
  grid_dependency();
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const long long P = g.plane;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n0) return;
  FOR_ROWS(j, k) {
    const long long idx = (long long)i + (long long)n0 * (j + (long long)n1 * k);
    const Nb nx = neighbours(i, g.n[0], 1);
    const Nb ny = neighbours(j, g.n[1], g.n[0]);
    const Nb nz = neighbours(k, g.n[2], (long long)g.n[0] * g.n[1]);
    const float* Bx = F + BX * P;
    const float* By = F + BY * P;
    const float* Bz = F + BZ * P;
    float cx = 0.f, cy = 0.f, cz = 0.f;
    cy -= d4m(Bz, idx, nx);
    cz += d4m(By, idx, nx);
    if (D >= 2) {
      cx += d4m(Bz, idx, ny);
      cz -= d4m(Bx, idx, ny);
    }
    if (D >= 3) {
      cx -= d4m(By, idx, nz);
      cy += d4m(Bx, idx, nz);
    }
    const float jx = J[idx], jy = J[P + idx], jz = J[2 * P + idx];
    F[EX * P + idx] = fmaf(c, cx, F[EX * P + idx]) - jx;
    F[EY * P + idx] = fmaf(c, cy, F[EY * P + idx]) - jy;
    F[EZ * P + idx] = fmaf(c, cz, F[EZ * P + idx]) - jz;
    if (J != F + JX * P) {
      F[JX * P + idx] = jx;
      F[JY * P + idx] = jy;
      F[JZ * P + idx] = jz;
    }
  }
}

// Launch of the four-points-per-thread kernels: rows of n0 / 4 threads.
static bool x4_ok(const GridDev& g, const float* F) {
  return g.n[0] % 4 == 0 && (reinterpret_cast<uintptr_t>(F) & 15) == 0;
}
static RowLaunch row_launch_x4(const GridDev& g) {
  GridDev q = g;
  q.n[0] = g.n[0] / 4;
  return row_launch(q);
}

cudaError_t launch_b_half(const GridDev& g, float* F, int zero_j, cudaStream_t st, int push_next) {
  const float hc = 0.5f * g.c;
  if (g.order == 2 && x4_ok(g, F)) {
    const RowLaunch L = row_launch_x4(g);
    switch (g.dim) {
      case 1: launch_kernel(g.pdl, k_b_half_x4<1>, L.grid, L.threads, 0, st, F, g, hc, zero_j, push_next); break;
      case 2: launch_kernel(g.pdl, k_b_half_x4<2>, L.grid, L.threads, 0, st, F, g, hc, zero_j, push_next); break;
      case 3: launch_kernel(g.pdl, k_b_half_x4<3>, L.grid, L.threads, 0, st, F, g, hc, zero_j, push_next); break;
      default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
  }
  const RowLaunch L = row_launch(g);
  switch (g.dim * 10 + g.order) {
    case 12: launch_kernel(g.pdl, k_b_half<1>, L.grid, L.threads, 0, st, F, g, hc, zero_j, push_next); break;
    case 22: launch_kernel(g.pdl, k_b_half<2>, L.grid, L.threads, 0, st, F, g, hc, zero_j, push_next); break;
    case 32: launch_kernel(g.pdl, k_b_half<3>, L.grid, L.threads, 0, st, F, g, hc, zero_j, push_next); break;
    case 14: launch_kernel(g.pdl, k_b_half4<1>, L.grid, L.threads, 0, st, F, g, hc, zero_j, push_next); break;
    case 24: launch_kernel(g.pdl, k_b_half4<2>, L.grid, L.threads, 0, st, F, g, hc, zero_j, push_next); break;
    case 34: launch_kernel(g.pdl, k_b_half4<3>, L.grid, L.threads, 0, st, F, g, hc, zero_j, push_next); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

bool fields_small_ok(const GridDev& g) {
  return PIC_SMALL_FIELDS && g.order == 2 && g.plane <= kSmallFieldCells;
}

cudaError_t launch_fields_small(const GridDev& g, float* F, const float* J, cudaStream_t st,
                                int chain) {
  const size_t smem = 9 * sizeof(float) * (size_t)g.plane;
  const int threads = g.plane < 1024 ? (int)((g.plane + 31) / 32 * 32) : 1024;
  const auto small = [&](auto kernel) {
    if (smem > 48 * 1024) {
      const cudaError_t e = cudaFuncSetAttribute(
          kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 9 * sizeof(float) * kSmallFieldCells);
      if (e != cudaSuccess) return e;
    }
    return launch_kernel(g.pdl, kernel, 1, threads, smem, st, F, J, g, 0.5f * g.c, g.c, chain);
  };
  switch (g.dim) {
    case 1: return small(k_fields_small<1>);
    case 2: return small(k_fields_small<2>);
    case 3: return small(k_fields_small<3>);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_e_update(const GridDev& g, float* F, const float* J, cudaStream_t st) {
  if (g.order == 2 && x4_ok(g, F) && (reinterpret_cast<uintptr_t>(J) & 15) == 0) {
    const RowLaunch L = row_launch_x4(g);
    switch (g.dim) {
      case 1: launch_kernel(g.pdl, k_e_update_x4<1>, L.grid, L.threads, 0, st, F, J, g, g.c); break;
      case 2: launch_kernel(g.pdl, k_e_update_x4<2>, L.grid, L.threads, 0, st, F, J, g, g.c); break;
      case 3: launch_kernel(g.pdl, k_e_update_x4<3>, L.grid, L.threads, 0, st, F, J, g, g.c); break;
      default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
  }
  const RowLaunch L = row_launch(g);
  switch (g.dim * 10 + g.order) {
    case 12: launch_kernel(g.pdl, k_e_update<1>, L.grid, L.threads, 0, st, F, J, g, g.c); break;
    case 22: launch_kernel(g.pdl, k_e_update<2>, L.grid, L.threads, 0, st, F, J, g, g.c); break;
    case 32: launch_kernel(g.pdl, k_e_update<3>, L.grid, L.threads, 0, st, F, J, g, g.c); break;
    case 14: launch_kernel(g.pdl, k_e_update4<1>, L.grid, L.threads, 0, st, F, J, g, g.c); break;
    case 24: launch_kernel(g.pdl, k_e_update4<2>, L.grid, L.threads, 0, st, F, J, g, g.c); break;
    case 34: launch_kernel(g.pdl, k_e_update4<3>, L.grid, L.threads, 0, st, F, J, g, g.c); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_filter(const GridDev& g, const T* src, T* dst, int ncomp, int axis,
                                 cudaStream_t st) {
  if (axis < 0 || axis >= g.dim || g.n[1] > 65535 || (long long)g.n[2] * ncomp > 65535)
    return cudaErrorInvalidValue;
  const dim3 grid((g.n[0] + 127) / 128, g.n[1], g.n[2] * ncomp);
  k_filter_axis<T><<<grid, 128, 0, st>>>(src, dst, g, axis);
  return cudaGetLastError();
}

cudaError_t launch_filter_f64(const GridDev& g, const double* src, double* dst, int ncomp,
                              int axis, cudaStream_t st) {
  return launch_filter<double>(g, src, dst, ncomp, axis, st);
}

}  // namespace pic
