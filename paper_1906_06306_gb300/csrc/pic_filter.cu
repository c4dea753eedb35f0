// Binomial2 current filter (arXiv:1906.06306, Table 2): passes of the
// (1/4, 1/2, 1/4) kernel along every gridded axis, x first, on periodic
// planes, up to four passes per launch.
//
// A pass alone streams the planes from and to memory (1024x128x128: 70 us a
// pass, 5.8 TB/s), so passes are fused: the threads march along the slowest
// axis (z in 3D, y in 2D) and keep each pass's partial sums of that axis in
// registers, one pass feeding the next one row or plane later.  A lane holds
// 4 consecutive x points, a warp 128 of them; x neighbours come by shuffle.
// The outermost 4 points on each side are halo (4 points, not K, so that
// copies and stores stay 16-byte aligned), which leaves 120 points of a warp.
// Every output goes through the sub-passes of one pass after the other, x
// first.  Measured (us, one launch of three planes): 4096^2, one pass 74, four
// passes 76; 768 x 384 (L2 resident), one pass 4, four passes 6.
#include "pic_kernels.h"

namespace pic {

__device__ __forceinline__ void cp_async4(void* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

constexpr int kOutX = 120;  // x points that a warp writes (of the 128 it holds)

// The x points of a lane: 4 from x on, wrapped; with vec (rows of a multiple
// of 4 points, 16-byte aligned) they stay together.
struct LaneX {
  int x[4];
  bool vec;
};
__device__ __forceinline__ LaneX lane_x(int x, int n0, int vec) {
  LaneX l;
  l.vec = vec != 0;
#pragma unroll
  for (int e = 0; e < 4; ++e) l.x[e] = wrapi(x + e, n0);
  return l;
}
__device__ __forceinline__ void copy_quad(float4* dst, const float* row, const LaneX& l) {
  if (l.vec) {
    cp_async16(dst, row + l.x[0]);
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) cp_async4(reinterpret_cast<float*>(dst) + e, row + l.x[e]);
  }
}
// wide: the quad is aligned and inside the row
__device__ __forceinline__ void store_quad(float* row, int gx, int n0, bool wide, float4 v) {
  if (wide) {
    *reinterpret_cast<float4*>(row + gx) = v;
  } else {
    if (gx < n0) row[gx] = v.x;
    if (gx + 1 < n0) row[gx + 1] = v.y;
    if (gx + 2 < n0) row[gx + 2] = v.z;
    if (gx + 3 < n0) row[gx + 3] = v.w;
  }
}

// Sub-passes are evaluated as l + 2 c + r, an addition and a fused multiply-add
// (two roundings, as for the weighted sum), and a pass's factor 4^-D, which
// is exact, is applied once, before it (no sum can overflow that the weighted
// sum would not): two operations a sub-pass instead of three.  A quad of x
// points is two pairs of the packed FP32 instructions.
struct Quad {
  float2 a, b;
};
__device__ __forceinline__ Quad to_quad(float4 v) {
  return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ float4 to_float4(const Quad& q) {
  return make_float4(q.a.x, q.a.y, q.b.x, q.b.y);
}
__device__ __forceinline__ Quad add(const Quad& u, const Quad& v) {
  return {__fadd2_rn(u.a, v.a), __fadd2_rn(u.b, v.b)};
}
__device__ __forceinline__ Quad twice_plus(const Quad& v, const Quad& s) {  // 2 v + s
  const float2 k = make_float2(2.0f, 2.0f);
  return {__ffma2_rn(k, v.a, s.a), __ffma2_rn(k, v.b, s.b)};
}
template <int D>
__device__ __forceinline__ Quad scaled(const Quad& v) {  // v 4^-D
  const float f = D == 1 ? 0.25f : D == 2 ? 0.0625f : 0.015625f;
  const float2 k = make_float2(f, f);
  return {__fmul2_rn(k, v.a), __fmul2_rn(k, v.b)};
}
// x sub-pass of a row held 4 points to a lane (the row's end points are not valid)
__device__ __forceinline__ Quad filter_x(const Quad& v) {
  const float l = __shfl_up_sync(0xffffffffu, v.b.y, 1);
  const float r = __shfl_down_sync(0xffffffffu, v.a.x, 1);
  return {make_float2(__fmaf_rn(2.0f, v.a.x, l + v.a.y), __fmaf_rn(2.0f, v.a.y, v.a.x + v.b.x)),
          make_float2(__fmaf_rn(2.0f, v.b.x, v.a.y + v.b.y), __fmaf_rn(2.0f, v.b.y, v.b.x + r))};
}

// The marching axis of one pass: `part` holds twice the last row's value plus
// the one before, `last` the last one.
struct March {
  Quad part, last;
  __device__ __forceinline__ Quad step(const Quad& v) {  // the row before v, filtered
    const Quad out = add(part, v);
    part = twice_plus(v, last);
    last = v;
    return out;
  }
};

// 1D: K passes of a plane, one warp per 120 outputs.
template <int K>
__global__ void __launch_bounds__(128) k_filter_x1(const float* __restrict__ src,
                                                   float* __restrict__ dst, const GridDev g,
                                                   int vec) {
  grid_dependency();
  const int lane = threadIdx.x & 31, n0 = g.n[0];
  const long long x0 = ((long long)blockIdx.x * 4 + (threadIdx.x >> 5)) * kOutX;
  if (x0 >= n0) return;
  const float* s = src + (long long)blockIdx.y * g.plane;
  float* d = dst + (long long)blockIdx.y * g.plane;
  const int gx = (int)x0 + 4 * (lane - 1);
  const LaneX l = lane_x(gx, n0, vec);
  Quad v;
  if (vec) {
    v = to_quad(*reinterpret_cast<const float4*>(s + l.x[0]));
  } else {
    v = {make_float2(s[l.x[0]], s[l.x[1]]), make_float2(s[l.x[2]], s[l.x[3]])};
  }
#pragma unroll
  for (int p = 0; p < K; ++p) v = filter_x(scaled<1>(v));
  if (lane >= 1 && lane <= 30) store_quad(d, gx, n0, vec && gx + 3 < n0, to_float4(v));
}

// 2D: K passes, one warp per strip of 120 outputs in x and run of `run` rows,
// marching over the run and K rows on either side of it.  Warps need nothing
// of each other.  A lane's rows come through a ring of kRows shared-memory
// slots of its own, copied kRows - 1 rows ahead.
constexpr int kRows = 8;
template <int K>
__global__ void __launch_bounds__(128) k_filter_y2(const float* __restrict__ src,
                                                   float* __restrict__ dst, const GridDev g,
                                                   int strips, int run, int vec) {
  grid_dependency();
  __shared__ float4 ring[kRows][128];
  const int lane = threadIdx.x & 31, n0 = g.n[0], n1 = g.n[1];
  const long long w = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
  const int strip = (int)(w % strips);
  const long long y0 = w / strips * run;
  if (y0 >= n1) return;
  const int yc = min((long long)run, n1 - y0);
  const float* s = src + (long long)blockIdx.y * g.plane;
  float* d = dst + (long long)blockIdx.y * g.plane;
  const int gx = strip * kOutX + 4 * (lane - 1);
  const LaneX l = lane_x(gx, n0, vec);
  const int steps = yc + 2 * K;
  const bool wide = vec && gx + 3 < n0, mine = lane >= 1 && lane <= 30;
  int yi = wrapi((int)y0 - K, n1);  // next row to copy
  const float* in = s + (long long)n0 * yi;
  auto issue = [&](int k) {  // row y0 - K + k
    if (k < steps) {
      copy_quad(&ring[k % kRows][threadIdx.x], in, l);
      in += n0;
      if (++yi == n1) {
        yi = 0;
        in = s;
      }
    }
    cp_async_commit();
  };
#pragma unroll
  for (int k = 0; k < kRows - 1; ++k) issue(k);
  March m[K];
#pragma unroll
  for (int p = 0; p < K; ++p) m[p] = March{};
  float* out = d + (long long)n0 * (y0 - 2 * K);
#pragma unroll 2
  for (int k = 0; k < steps; ++k, out += n0) {
    cp_async_wait<kRows - 2>();  // this lane's copy of row k has landed
    Quad v = to_quad(ring[k % kRows][threadIdx.x]);
    issue(k + kRows - 1);  // into the slot of row k - 1
#pragma unroll
    for (int p = 0; p < K; ++p) v = m[p].step(filter_x(scaled<2>(v)));
    if (k >= 2 * K && mine) store_quad(out, gx, n0, wide, to_float4(v));
  }
  cp_async_wait<0>();
}

// One full 3D Binomial2 pass (x, y, then z sub-pass) of one plane src -> dst,
// marching along z.  A block of 256 threads owns a ZX x ZY = 128 x 16 column
// of (x, y) points over a run of `zrun` z-planes; a thread owns a 4 (x) x 2
// (y) patch of it.  Each z-plane of the column plus its one-point periodic
// (x, y) halo is copied into a ring of ZS shared-memory stages, ZS - 1 planes
// ahead of the one being filtered.  BULK (rows of a multiple of 4 floats,
// 16-byte aligned planes, a status word): the ZY + 2 stage rows arrive by one
// bulk copy each (`cp.async.bulk`, issued by the lanes of warp 0, completing
// on the stage's mbarrier) and the two halo points of each row by 4-byte
// cp.async; otherwise every thread copies by cp.async (16-byte copies for the
// aligned interior, 4-byte ones for the halo and for ragged or wrapped rows).
// A thread reads its four rows (y - 1 .. y + 2) with one 16-byte and two
// 4-byte shared loads each, runs the x and y sub-passes in registers and keeps
// the last three y results for the z sub-pass.  Reads: the column, its (x, y)
// halo (rows of neighbouring columns, mostly from L2) and two extra planes per
// run; writes: the column, 16 bytes per store.  Every output goes through the
// x, y and z sub-passes in this order, with the arithmetic of the marched forms.
// Grid: x = column index + columns x run, y = plane.
constexpr int ZX = 128, ZY = 16, ZS = 4;
constexpr int ZROW = ZX + 8;  // stage row: [3] left halo, [4, 4 + ZX) interior, [4 + ZX] right
constexpr int ZPLANE = (ZY + 2) * ZROW;
constexpr int ZCH = ZX / 4 + 2;         // copy operations per stage row
constexpr int ZOPS = (ZY + 2) * ZCH;    // copy operations per stage (612)
constexpr int ZOPT = (ZOPS + 255) / 256;  // per thread (3)

// l + 2 c + r, and (l + 2 c + r) / 4, with the roundings of the fused passes
__device__ __forceinline__ float s3(float l, float c, float r) {
  return __fmaf_rn(2.0f, c, l + r);
}
__device__ __forceinline__ float b3(float l, float c, float r) {
  return __fmaf_rn(0.5f, c, __fmaf_rn(0.25f, l, 0.25f * r));
}
// the same along the marching axis, whose points come one after the other
__device__ __forceinline__ float b3_march(float l, float c, float r) {
  return __fmaf_rn(0.25f, r, __fmaf_rn(0.5f, c, 0.25f * l));
}

// A marching pass's wait, by every thread, for the bulk copies of step k
// (stage k % ZS, phase parity (k / ZS) & 1; steps k .. min(k + ZS - 2,
// nk - 1) are in flight); true when the whole block may go on.  When a wait
// ran out (the status word has the timeout bit), thread 0 waits once more,
// bounded, for each step still in flight, and the block leaves together.
__device__ __forceinline__ bool stage_landed(unsigned long long* full, int k, int nk, int* status) {
  const bool ok = mbar_wait(&full[k % ZS], (unsigned)(k / ZS) & 1u, status);
  if (!__syncthreads_or(!ok)) return true;
  if (threadIdx.x == 0)
    for (int j = k; j < k + ZS - 1 && j < nk; ++j)
      mbar_wait(&full[j % ZS], (unsigned)(j / ZS) & 1u, nullptr);
  cp_async_wait<0>();
  return false;
}

template <bool BULK>
__global__ void __launch_bounds__(256, 4) k_filter_z3(const float* __restrict__ src,
                                                     float* __restrict__ dst, const GridDev g,
                                                     int ncx, int ncy, int zrun, int vec,
                                                     int* status) {
  grid_dependency();
  __shared__ __align__(16) float stage[ZS][ZPLANE];
  __shared__ unsigned long long full[ZS];  // BULK: stage's rows have landed
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const long long nxy = (long long)n0 * n1;
  const int col = blockIdx.x % (ncx * ncy), run = blockIdx.x / (ncx * ncy);
  const int x0 = (col % ncx) * ZX, y0 = (col / ncx) * ZY, z0 = run * zrun;
  const int zc = min(zrun, n2 - z0);  // planes z0 .. z0 + zc - 1 are written
  const long long P = g.plane;
  const float* s = src + (long long)blockIdx.y * P;
  float* d = dst + (long long)blockIdx.y * P;
  const int len = min(ZX, n0 - x0);  // interior points of the column's rows

  // This thread's copy operations op = threadIdx.x + 256 j, the same for every
  // z-plane: stage row op / ZCH (y = y0 - 1 + row) and either a 4-point
  // interior chunk (c < ZX / 4), the left halo point (c = ZX / 4) or the right.
  // BULK: lane r < ZY + 2 of warp 0 copies the interior of stage row r, and
  // threads 64 .. 64 + 2 (ZY + 2) - 1 its halo points (the right one after
  // the last interior point, where a ragged column's x sub-pass reads it).
  long long yoff[ZOPT];
  int xs[ZOPT], dofs[ZOPT], kind[ZOPT];  // kind: 0 none, 1 16-byte, 2 four 4-byte, 3 one 4-byte
#pragma unroll
  for (int j = 0; j < ZOPT; ++j) {
    kind[j] = 0;
    yoff[j] = 0;
    xs[j] = 0;
    dofs[j] = 0;
  }
  if (BULK) {
    const int t = threadIdx.x;
    if (t < ZY + 2) {  // interior of row t
      yoff[0] = (long long)n0 * wrapi(y0 - 1 + t, n1);
      xs[0] = x0;
      dofs[0] = t * ZROW + 4;
      kind[0] = 1;
    } else if (t >= 64 && t < 64 + 2 * (ZY + 2)) {  // a halo point of row (t - 64) / 2
      const int row = (t - 64) >> 1, right = (t - 64) & 1;
      yoff[0] = (long long)n0 * wrapi(y0 - 1 + row, n1);
      xs[0] = wrapi(right ? x0 + len : x0 - 1, n0);
      dofs[0] = row * ZROW + (right ? 4 + len : 3);
      kind[0] = 3;
    }
    if (t == 0) {
      for (int i = 0; i < ZS; ++i) mbar_init(&full[i], 1);
      mbar_init_fence();
    }
    __syncthreads();  // the barriers are initialised before any copy or wait
  } else {
#pragma unroll
    for (int j = 0; j < ZOPT; ++j) {
      const int op = threadIdx.x + 256 * j;
      const int row = op / ZCH, c = op % ZCH;
      if (op < ZOPS) {
        yoff[j] = (long long)n0 * wrapi(y0 - 1 + row, n1);
        if (c < ZX / 4) {
          xs[j] = x0 + 4 * c;
          dofs[j] = row * ZROW + 4 + 4 * c;
          kind[j] = vec && xs[j] + 3 < n0 ? 1 : 2;
        } else {
          xs[j] = wrapi(c == ZX / 4 ? x0 - 1 : x0 + ZX, n0);
          dofs[j] = row * ZROW + (c == ZX / 4 ? 3 : 4 + ZX);
          kind[j] = 3;
        }
      }
    }
  }
  auto issue = [&](int k) {  // copy halo plane k (z = z0 - 1 + k) into stage k % ZS
    if (k < zc + 2) {
      int z = z0 - 1 + k;  // -1 <= z <= n2
      z = z < 0 ? z + n2 : (z >= n2 ? z - n2 : z);
      const float* base = s + nxy * z;
      float* st = stage[k % ZS];
      if (BULK) {
        if (threadIdx.x < 32) {
          if (threadIdx.x == 0)
            mbar_arrive_expect_tx(&full[k % ZS], (unsigned)((ZY + 2) * len * 4));
          __syncwarp();
          if (kind[0] == 1) {
            fence_proxy_async_smem();
            bulk_load(st + dofs[0], base + yoff[0] + xs[0], (unsigned)(len * 4), &full[k % ZS]);
          }
        } else if (kind[0] == 3) {
          cp_async4(st + dofs[0], base + yoff[0] + xs[0]);
        }
      } else {
#pragma unroll
        for (int j = 0; j < ZOPT; ++j) {
          const float* sr = base + yoff[j];
          if (kind[j] == 1) {
            cp_async16(st + dofs[j], sr + xs[j]);
          } else if (kind[j] == 3) {
            cp_async4(st + dofs[j], sr + xs[j]);
          } else if (kind[j] == 2) {
            for (int e = 0; e < 4; ++e) cp_async4(st + dofs[j] + e, sr + wrapi(xs[j] + e, n0));
          }
        }
      }
    }
    cp_async_commit();  // an empty group keeps the group count uniform
  };
#pragma unroll
  for (int k = 0; k < ZS - 1; ++k) issue(k);

  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int gx = x0 + 4 * tx, gy = y0 + 2 * ty;
  float pm[8], p0[8];  // y results of the two previous planes: [row * 4 + x]
#pragma unroll
  for (int i = 0; i < 8; ++i) pm[i] = p0[i] = 0.f;
  for (int k = 0; k < zc + 2; ++k) {
    cp_async_wait<ZS - 2>();  // this thread's copies of plane k have landed
    if (BULK) {
      // and the bulk copies of every thread's rows; then stage (k - 1) % ZS
      // is no longer read
      if (!stage_landed(full, k, zc + 2, status)) return;
    } else {
      __syncthreads();  // everyone's have; stage (k - 1) % ZS is no longer read
    }
    issue(k + ZS - 1);
    const float* a = stage[k % ZS] + 2 * ty * ZROW + 4 * tx + 3;  // row y - 1, column x - 1
    float xf[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {  // x sub-pass of rows y - 1 .. y + 2
      const float l = a[r * ZROW];
      const float4 m = *reinterpret_cast<const float4*>(a + r * ZROW + 1);
      const float rr = a[r * ZROW + 5];
      xf[r][0] = s3(l, m.x, m.y);
      xf[r][1] = s3(m.x, m.y, m.z);
      xf[r][2] = s3(m.y, m.z, m.w);
      xf[r][3] = s3(m.z, m.w, rr);
    }
    float p1[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // y sub-pass of rows y, y + 1, and both sub-passes' factor
      p1[i] = 0.0625f * s3(xf[0][i], xf[1][i], xf[2][i]);
      p1[4 + i] = 0.0625f * s3(xf[1][i], xf[2][i], xf[3][i]);
    }
    if (k >= 2) {  // z sub-pass of plane z0 + k - 2
      const int z = z0 + k - 2;
#pragma unroll
      for (int rw = 0; rw < 2; ++rw) {
        if (gy + rw >= n1) continue;
        float o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = b3_march(pm[4 * rw + i], p0[4 * rw + i], p1[4 * rw + i]);
        float* q = d + gx + (long long)n0 * (gy + rw) + nxy * z;
        if (vec && gx + 3 < n0) {
          *reinterpret_cast<float4*>(q) = make_float4(o[0], o[1], o[2], o[3]);
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (gx + i < n0) q[i] = o[i];
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      pm[i] = p0[i];
      p0[i] = p1[i];
    }
  }
  cp_async_wait<0>();
}

// 2D, a single pass of rows of a multiple of 4 points (16-byte aligned, with a
// status word for the bounded waits): marching along y, a block of 256 threads
// owns YX = 1024 x points (4 per thread) over a run of `yrun` rows.  Each row
// arrives by one bulk copy (`cp.async.bulk`, issued by thread 0, completing on
// the stage's mbarrier) and its two halo points by 4-byte cp.async, ZS - 1
// rows ahead in a ring of ZS stages.  Long rows written whole: 4096^2 in 70 us
// against 82 us for the 120-point strips of k_filter_y2<1>.
// Grid: x = x column + columns x run, y = plane.
constexpr int YX = 1024;
constexpr int YROW = YX + 8;  // stage row: [3] left halo, [4, 4 + YX) interior, [4 + YX] right

__global__ void __launch_bounds__(256) k_filter_y2_one(const float* __restrict__ src,
                                                      float* __restrict__ dst, const GridDev g,
                                                      int ncx, int yrun, int* status) {
  grid_dependency();
  __shared__ __align__(16) float stage[ZS][YROW];
  __shared__ unsigned long long full[ZS];  // the stage's row has landed
  const int n0 = g.n[0], n1 = g.n[1];
  const int col = blockIdx.x % ncx, run = blockIdx.x / ncx;
  const int x0 = col * YX, y0 = run * yrun;
  const int yc = min(yrun, n1 - y0);  // rows y0 .. y0 + yc - 1 are written
  const long long P = g.plane;
  const float* s = src + (long long)blockIdx.y * P;
  float* d = dst + (long long)blockIdx.y * P;
  const int t = threadIdx.x;
  const int len = min(YX, n0 - x0);  // interior points of the column's rows
  const int xs = x0 + 4 * t;
  const bool mine = xs < n0;
  // threads 0 and 1 copy the left and right halo point (the right one after the
  // last interior point, where a ragged column's x sub-pass reads it)
  const int hx = t == 0 ? wrapi(x0 - 1, n0) : wrapi(x0 + len, n0);
  const int hcol = t == 0 ? 3 : 4 + len;
  if (t == 0) {
    for (int i = 0; i < ZS; ++i) mbar_init(&full[i], 1);
    mbar_init_fence();
  }
  __syncthreads();  // the barriers are initialised before any copy or wait
  auto issue = [&](int k) {  // copy halo row k (y = y0 - 1 + k) into stage k % ZS
    if (k < yc + 2) {
      int y = y0 - 1 + k;  // -1 <= y <= n1
      y = y < 0 ? y + n1 : (y >= n1 ? y - n1 : y);
      const float* row = s + (long long)n0 * y;
      float* st = stage[k % ZS];
      if (t == 0) {
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(&full[k % ZS], (unsigned)(len * 4));
        bulk_load(st + 4, row + x0, (unsigned)(len * 4), &full[k % ZS]);
      }
      if (t < 2) cp_async4(st + hcol, row + hx);
    }
    cp_async_commit();  // an empty group keeps the group count uniform
  };
#pragma unroll
  for (int k = 0; k < ZS - 1; ++k) issue(k);

  float pm[4] = {0.f, 0.f, 0.f, 0.f}, p0[4] = {0.f, 0.f, 0.f, 0.f};
  for (int k = 0; k < yc + 2; ++k) {
    cp_async_wait<ZS - 2>();  // this thread's copy of row k has landed
    // and the row's bulk copy; then stage (k - 1) % ZS is no longer read
    if (!stage_landed(full, k, yc + 2, status)) return;
    issue(k + ZS - 1);
    const float* a = stage[k % ZS] + 4 * t + 3;  // column x - 1
    const float l = a[0];
    const float4 m = *reinterpret_cast<const float4*>(a + 1);
    const float r = a[5];
    const float p1[4] = {b3(l, m.x, m.y), b3(m.x, m.y, m.z), b3(m.y, m.z, m.w), b3(m.z, m.w, r)};
    if (k >= 2) {  // y sub-pass of row y0 + k - 2
      float o[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) o[i] = b3_march(pm[i], p0[i], p1[i]);
      float* q = d + (long long)n0 * (y0 + k - 2) + xs;
      if (mine) *reinterpret_cast<float4*>(q) = make_float4(o[0], o[1], o[2], o[3]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      pm[i] = p0[i];
      p0[i] = p1[i];
    }
  }
  cp_async_wait<0>();
}

// 3D: two passes, one block of 8 warps per column of 120 x 28 outputs and run
// of `run` planes, marching over the run and K = 2 planes on either side.
// A warp holds R = 4 rows of the column's 32 (K of halo on either side); the
// rows next to its own come from the neighbouring warps through shared memory,
// one exchange and block barrier per pass and plane (two exchange buffers in
// turn: a buffer is written again only after the barrier that follows its
// reads).  A lane's rows come through a ring of kPlanes slots of its own,
// copied kPlanes - 1 planes ahead.  1024x128x128: 104 us for the two passes,
// bound by latency at 16 warps per SM (the passes' state is 64 registers a
// thread), against 141 us for two launches of the one-pass kernel above; the
// one-pass form of this kernel takes 81 us against 70.  Two rows a lane (32
// warps per SM) 132 us; rows by bulk copies 127 us; four passes 343 us.
constexpr int kPlanes = 4;
constexpr int kColY = 32;
constexpr int kRowsZ = 4;                // rows of a lane
constexpr int kWarpsZ = kColY / kRowsZ;  // warps of a block
struct Z3Smem {
  float4 ring[kPlanes][kRowsZ][32 * kWarpsZ];
  float4 edge[2][kWarpsZ][2][32];  // [buffer][warp][first, last row][lane]
};
__global__ void __launch_bounds__(32 * kWarpsZ, 2)
    k_filter_z3_two(const float* __restrict__ src, float* __restrict__ dst, const GridDev g, int ncx,
                int ncy, int run, int vec) {
  grid_dependency();
  extern __shared__ __align__(16) unsigned char smem[];
  Z3Smem& S = *reinterpret_cast<Z3Smem*>(smem);
  constexpr int K = 2, R = kRowsZ, kOutY = kColY - 2 * K;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const long long nxy = (long long)n0 * n1;
  const int col = blockIdx.x % (ncx * ncy), z0 = blockIdx.x / (ncx * ncy) * run;
  const int zc = min(run, n2 - z0);
  const float* s = src + (long long)blockIdx.y * g.plane;
  float* d = dst + (long long)blockIdx.y * g.plane;
  const int gx = col % ncx * kOutX + 4 * (lane - 1);
  const int gy = col / ncx * kOutY - K + R * w;  // this warp's first row
  const LaneX l = lane_x(gx, n0, vec);
  int row[R];        // of the plane: its points number fewer than 2^31
  unsigned out = 0;  // bit r: row r is an output of the column and on the lattice
#pragma unroll
  for (int r = 0; r < R; ++r) {
    row[r] = n0 * wrapi(gy + r, n1);
    const int i = R * w + r - K;
    if (lane >= 1 && lane <= 30 && i >= 0 && i < kOutY && gy + r < n1) out |= 1u << r;
  }
  const bool wide = vec && gx + 3 < n0;
  const int steps = zc + 2 * K;
  int zi = wrapi(z0 - K, n2);  // next plane to copy
  const float* in = s + nxy * zi;
  auto issue = [&](int k) {  // plane z0 - K + k
    if (k < steps) {
#pragma unroll
      for (int r = 0; r < R; ++r) copy_quad(&S.ring[k % kPlanes][r][threadIdx.x], in + row[r], l);
      in += nxy;
      if (++zi == n2) {
        zi = 0;
        in = s;
      }
    }
    cp_async_commit();
  };
#pragma unroll
  for (int k = 0; k < kPlanes - 1; ++k) issue(k);
  March m[K][R];
#pragma unroll
  for (int p = 0; p < K; ++p)
#pragma unroll
    for (int r = 0; r < R; ++r) m[p][r] = March{};
  const int wu = w > 0 ? w - 1 : 0, wd = w < kWarpsZ - 1 ? w + 1 : kWarpsZ - 1;
  float* o = d + nxy * (z0 - 2 * K) + (long long)n0 * gy;  // used from plane z0 on
#pragma unroll 2
  for (int k = 0; k < steps; ++k, o += nxy) {
    cp_async_wait<kPlanes - 2>();  // this lane's copies of plane k have landed
    Quad v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = to_quad(S.ring[k % kPlanes][r][threadIdx.x]);
    issue(k + kPlanes - 1);  // into the slots of plane k - 1
#pragma unroll
    for (int p = 0; p < K; ++p) {
      const int buf = (k * K + p) & 1;
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = filter_x(scaled<3>(v[r]));
      S.edge[buf][w][0][lane] = to_float4(v[0]);
      S.edge[buf][w][1][lane] = to_float4(v[R - 1]);
      __syncthreads();
      // the column's outermost rows have no neighbour: halo, not valid
      Quad below = to_quad(S.edge[buf][wu][1][lane]);
      const Quad above = to_quad(S.edge[buf][wd][0][lane]);
#pragma unroll
      for (int r = 0; r < R; ++r) {  // y sub-pass, then z
        const Quad t = twice_plus(v[r], add(below, r + 1 < R ? v[r + 1 < R ? r + 1 : r] : above));
        below = v[r];
        v[r] = m[p][r].step(t);
      }
    }
    if (k >= 2 * K) {
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (out >> r & 1) store_quad(o + (long long)n0 * r, gx, n0, wide, to_float4(v[r]));
    }
  }
  cp_async_wait<0>();
}

// 16-byte copies and stores need 16-byte aligned rows: plane bases and n0
// multiples of 4 floats
static int aligned_rows(const GridDev& g, const float* src, const float* dst) {
  return ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15) == 0 &&
         g.n[0] % 4 == 0 && g.plane % 4 == 0;
}

static int device_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    sms = 152;
  return sms;
}

// The z-marching 3D pass.  The z-runs are as long as they can be with every
// block resident at once (one wave: no block re-reads a run's two halo planes
// from DRAM after its neighbour has evicted them, no tail wave); a grid with
// more columns than resident blocks gets one run per column.
static cudaError_t launch_pass_z3(const GridDev& g, const float* src, float* dst, int ncomp,
                                  cudaStream_t st, int* status) {
  static int resident = 0;
  if (resident == 0) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_filter_z3<true>, 256, 0);
    resident = sms * per_sm > 0 ? sms * per_sm : 1;
  }
  const int ncx = (g.n[0] + ZX - 1) / ZX, ncy = (g.n[1] + ZY - 1) / ZY;
  const long long streams = (long long)ncx * ncy * ncomp;
  long long runs = resident / streams;
  if (runs < 1) runs = 1;
  if (runs > g.n[2]) runs = g.n[2];
  const int zrun = (int)((g.n[2] + runs - 1) / runs);
  const long long blocks = (long long)ncx * ncy * ((g.n[2] + zrun - 1) / zrun);
  if (blocks > 0x7fffffffLL || ncomp > 65535) return cudaErrorInvalidValue;
  const int vec = aligned_rows(g, src, dst);
  // bulk row copies where a status word can report a wait that ran out
  const dim3 grid((unsigned)blocks, (unsigned)ncomp);
  if (vec && status)
    launch_kernel(g.pdl, k_filter_z3<true>, grid, 256, 0, st, src, dst, g, ncx, ncy, zrun, vec, status);
  else
    launch_kernel(g.pdl, k_filter_z3<false>, grid, 256, 0, st, src, dst, g, ncx, ncy, zrun, vec, status);
  return cudaGetLastError();
}


// The y-marching 2D pass; runs as long as one wave of resident blocks allows.
static cudaError_t launch_one_y2(const GridDev& g, const float* src, float* dst, int ncomp,
                                  cudaStream_t st, int* status) {
  static int resident = 0;
  if (resident == 0) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_filter_y2_one, 256, 0);
    resident = sms * per_sm > 0 ? sms * per_sm : 1;
  }
  const int ncx = (g.n[0] + YX - 1) / YX;
  const long long streams = (long long)ncx * ncomp;
  long long runs = resident / streams;
  if (runs < 1) runs = 1;
  if (runs > g.n[1]) runs = g.n[1];
  const int yrun = (int)((g.n[1] + runs - 1) / runs);
  const long long blocks = (long long)ncx * ((g.n[1] + yrun - 1) / yrun);
  if (blocks > 0x7fffffffLL || ncomp > 65535) return cudaErrorInvalidValue;
  launch_kernel(g.pdl, k_filter_y2_one, dim3((unsigned)blocks, (unsigned)ncomp), 256, 0, st, src, dst, g, ncx, yrun, status);
  return cudaGetLastError();
}

// Two 3D passes: one wave of resident blocks.
static cudaError_t launch_two_z3(const GridDev& g, const float* src, float* dst, int ncomp,
                                 cudaStream_t st) {
  const int vec = aligned_rows(g, src, dst);
  const int outy = kColY - 4;
  const int ncx = (g.n[0] + kOutX - 1) / kOutX, ncy = (g.n[1] + outy - 1) / outy;
  const long long columns = (long long)ncx * ncy;
  long long runs = 2LL * device_sms() / (columns * ncomp);
  runs = runs < 1 ? 1 : runs > g.n[2] ? g.n[2] : runs;
  const int run = (int)((g.n[2] + runs - 1) / runs);
  const long long blocks = columns * ((g.n[2] + run - 1) / run);
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  const cudaError_t e = cudaFuncSetAttribute(
      k_filter_z3_two, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Z3Smem));
  if (e != cudaSuccess) return e;
  launch_kernel(g.pdl, k_filter_z3_two, dim3((unsigned)blocks, ncomp), 32 * kWarpsZ, sizeof(Z3Smem), st, src, dst, g, ncx, ncy, run, vec);
  return cudaGetLastError();
}

template <int K>
static cudaError_t launch_k(const GridDev& g, const float* src, float* dst, int ncomp,
                            cudaStream_t st) {
  const int vec = aligned_rows(g, src, dst);
  const int sms = device_sms();
  const long long strips = ((long long)g.n[0] + kOutX - 1) / kOutX;
  if (g.dim == 1) {
    launch_kernel(g.pdl, k_filter_x1<K>, dim3((unsigned)((strips + 3) / 4), ncomp), 128, 0, st, src, dst, g, vec);
  } else if (g.dim == 2) {
    // runs short enough for 16 warps per SM, but no shorter than the K rows
    // of halo on either side
    const long long warps = 16LL * sms;
    long long run = (g.n[1] * strips * ncomp + warps - 1) / warps;
    run = run < 2 * K ? 2 * K : run;
    const long long runs = (g.n[1] + run - 1) / run;
    launch_kernel(g.pdl, k_filter_y2<K>, dim3((unsigned)((strips * runs + 3) / 4), ncomp), 128, 0, st, src, dst, g, (int)strips, (int)run, vec);
  }
  return cudaGetLastError();
}

int filter_launches(int dim, int passes) {
  // an even number, so that the result is back in the planes it started
  // from; a single pass is one launch and a copy.  Up to four passes to a
  // launch in 1D and 2D, two in 3D.
  const int most = dim == 3 ? 2 : 4;
  return passes <= 0 ? 0 : passes == 1 ? 1 : 2 * ((passes + 2 * most - 1) / (2 * most));
}

cudaError_t launch_filter(const GridDev& g, const float* src, float* dst, int ncomp, int passes,
                          cudaStream_t st, int* status) {
  switch (g.dim == 3 ? 30 + passes : passes) {
    case 1:
      if (g.dim == 2 && status && aligned_rows(g, src, dst))
        return launch_one_y2(g, src, dst, ncomp, st, status);
      return launch_k<1>(g, src, dst, ncomp, st);
    case 2: return launch_k<2>(g, src, dst, ncomp, st);
    case 3: return launch_k<3>(g, src, dst, ncomp, st);
    case 4: return launch_k<4>(g, src, dst, ncomp, st);
    case 31: return launch_pass_z3(g, src, dst, ncomp, st, status);
    case 32: return launch_two_z3(g, src, dst, ncomp, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pic
