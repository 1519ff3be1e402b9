// Device kernels of the tdmps library beside the block GEMMs: sparse MPO-tensor
// application, block gather/scatter, one-sided Jacobi SVD, Gram-Schmidt QR, the
// truncation rule, and the small Krylov algebra.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <mutex>
#include <set>
#include <tuple>

#include "kernels.hpp"

namespace tdmps {

// Raise a kernel's dynamic shared-memory limit once per (device, kernel, size).
// Thread-safe; a failure is left for the launch to report.
void set_smem_limit(const void* func, int bytes) {
  static std::mutex mu;
  static std::set<std::tuple<int, const void*, int>> done;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return;
  std::lock_guard<std::mutex> lk(mu);
  auto key = std::make_tuple(dev, func, bytes);
  if (done.count(key)) return;
  if (cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess)
    done.insert(key);
}


// ------------------------------------------------------------------ complex helpers

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 cscale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
__device__ __forceinline__ double cabs2(double2 a) { return a.x * a.x + a.y * a.y; }
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 c) {   // a*b + c
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}
__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
  double d = b.x * b.x + b.y * b.y;
  return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ------------------------------------------------------------------ W stage

template <class T>
__device__ __forceinline__ double2 ld2(const T* p, size_t i);
template <>
__device__ __forceinline__ double2 ld2<double2>(const double2* p, size_t i) { return p[i]; }
template <>
__device__ __forceinline__ double2 ld2<float2>(const float2* p, size_t i) {
  float2 v = p[i];
  return make_double2(v.x, v.y);
}
template <class T>
__device__ __forceinline__ void st2(T* p, size_t i, double2 v);
template <>
__device__ __forceinline__ void st2<double2>(double2* p, size_t i, double2 v) { p[i] = v; }
template <>
__device__ __forceinline__ void st2<float2>(float2* p, size_t i, double2 v) {
  p[i] = make_float2((float)v.x, (float)v.y);
}

// One thread per (output channel w, column b) and group of up to WS_ROWS
// rows a of a block: the CSR row of w (entries w_in, value) is walked once
// and applied to all of those rows, so the entry loads, the loop control and
// the index arithmetic are shared by WS_ROWS outputs; consecutive threads
// take consecutive columns, so every X read and Y write is coalesced along b.
// Complex FP64 data: bound by the FP64 pipe (74% of it at L = 16, D = 256).
constexpr int WS_ROWS = 2;

// the task of work item idx, searched once, then stepped forward
__device__ __forceinline__ int ws_find(const WTask* __restrict__ tasks, int ntasks, int64_t idx) {
  int lo = 0, hi = ntasks - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tasks[mid].work_base <= idx) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__global__ void __launch_bounds__(256) k_wstage(const WTask* __restrict__ tasks, int ntasks,
                                                int64_t total, const int* __restrict__ rowptr,
                                                const int* __restrict__ ent_w,
                                                const double* __restrict__ ent_v) {
  // each CTA owns one contiguous range of the flat work index
  const int64_t per = (total + gridDim.x - 1) / gridDim.x;
  const int64_t beg = (int64_t)blockIdx.x * per;
  const int64_t end = beg + per < total ? beg + per : total;
  int lo = beg + threadIdx.x < end ? ws_find(tasks, ntasks, beg + threadIdx.x) : 0;
  for (int64_t idx = beg + threadIdx.x; idx < end; idx += blockDim.x) {
    while (lo + 1 < ntasks && tasks[lo + 1].work_base <= idx) ++lo;
    const WTask& t = tasks[lo];
    // 32-bit index split (a task holds fewer than 2^31 work items)
    const int loc = (int)(idx - t.work_base);
    const int cols = t.cols, wout = t.wout;
    const int rw = loc / cols;
    const int b = loc - rw * cols;
    const int q = rw / wout;            // row group
    const int w = rw - q * wout;
    const int a0 = q * WS_ROWS;
    const int nr = t.rows - a0 < WS_ROWS ? t.rows - a0 : WS_ROWS;
    double ax[WS_ROWS], ay[WS_ROWS];
#pragma unroll
    for (int r = 0; r < WS_ROWS; ++r) ax[r] = ay[r] = 0.0;
    for (int s = 0; s < 4; ++s) {
      if (t.csr[s] < 0) continue;
      const int* rp = rowptr + t.csr[s];
      const size_t rstride = (size_t)t.win[s] * cols;
      const double2* X = (const double2*)t.X[s] + (size_t)a0 * rstride + b;
      const int e1 = rp[w + 1];
      for (int e = rp[w]; e < e1; ++e) {
        const double v = ent_v[e];
        const double2* xp = X + (size_t)ent_w[e] * cols;
#pragma unroll
        for (int r = 0; r < WS_ROWS; ++r) {
          if (r < nr) {   // constant indices: the accumulators stay in registers
            const double2 x = xp[r * rstride];
            ax[r] = fma(v, x.x, ax[r]);
            ay[r] = fma(v, x.y, ay[r]);
          }
        }
      }
    }
    const size_t ystride = (size_t)wout * cols;
    double2* y = (double2*)t.Y + (size_t)a0 * ystride + (size_t)w * cols + b;
#pragma unroll
    for (int r = 0; r < WS_ROWS; ++r) {
      if (r < nr) {
        double2* yr = y + r * ystride;
        if (t.beta) { ax[r] += yr->x; ay[r] += yr->y; }
        *yr = make_double2(ax[r], ay[r]);
      }
    }
  }
}

// The same stage on complex FP32 data, where the loads bound it and not the
// arithmetic: one thread takes WS_GROUP consecutive output channels and
// WS_ROWS rows of one column.  The table lists, per group of channels, every
// input channel that one of them uses, with its WS_GROUP values (zero where a
// channel does not use it): four loads feed 16 multiply-adds, where the rows
// of the single channels took four loads for four.  Every output sums its
// inputs in the same order as the CSR row; the zeros are skipped, so that an
// infinity in one channel stays out of the others' sums (2.98 ms instead of
// 2.96 at L = 24, D = 128).
// Measured against the CSR kernel: the centre-site local operator at L = 16,
// D = 256 (8 launches) 2.38 -> 1.26 ms, a fitted H|psi> there (47 launches)
// 3.0 -> 2.0 ms, at L = 24, D = 128 (71) 3.7 -> 3.1 ms.
constexpr int WS_GROUP = 4;

__global__ void __launch_bounds__(256) k_wstage_f32(const WTask* __restrict__ tasks, int ntasks,
                                                    int64_t total, const int* __restrict__ grp_ptr,
                                                    const int* __restrict__ grp_w,
                                                    const float4* __restrict__ grp_v) {
  const int64_t per = (total + gridDim.x - 1) / gridDim.x;
  const int64_t beg = (int64_t)blockIdx.x * per;
  const int64_t end = beg + per < total ? beg + per : total;
  int lo = beg + threadIdx.x < end ? ws_find(tasks, ntasks, beg + threadIdx.x) : 0;
  for (int64_t idx = beg + threadIdx.x; idx < end; idx += blockDim.x) {
    while (lo + 1 < ntasks && tasks[lo + 1].work_base <= idx) ++lo;
    const WTask& t = tasks[lo];
    const int loc = (int)(idx - t.work_base);
    const int cols = t.cols, wout = t.wout;
    const int ngrp = (wout + WS_GROUP - 1) / WS_GROUP;
    const int rw = loc / cols;
    const int b = loc - rw * cols;
    const int q = rw / ngrp;
    const int g = rw - q * ngrp;
    const int a0 = q * WS_ROWS;
    const int nr = t.rows - a0 < WS_ROWS ? t.rows - a0 : WS_ROWS;
    float2 acc[WS_ROWS][WS_GROUP];
#pragma unroll
    for (int r = 0; r < WS_ROWS; ++r)
#pragma unroll
      for (int j = 0; j < WS_GROUP; ++j) acc[r][j] = make_float2(0.f, 0.f);
    for (int s = 0; s < 4; ++s) {
      if (t.csr[s] < 0) continue;
      const int* gp = grp_ptr + t.csr[s] + g;
      const size_t rstride = nr > 1 ? (size_t)t.win[s] * cols : 0;   // a missing row repeats the first
      const float2* X = (const float2*)t.X[s] + (size_t)a0 * t.win[s] * cols + b;
      const int e1 = gp[1];
#pragma unroll 2
      for (int e = gp[0]; e < e1; ++e) {
        const float4 v = grp_v[e];
        const float2* xp = X + (size_t)grp_w[e] * cols;
#pragma unroll
        for (int r = 0; r < WS_ROWS; ++r) {
          const float2 x = xp[r * rstride];
          if (v.x != 0.f) {
            acc[r][0].x = fmaf(v.x, x.x, acc[r][0].x);
            acc[r][0].y = fmaf(v.x, x.y, acc[r][0].y);
          }
          if (v.y != 0.f) {
            acc[r][1].x = fmaf(v.y, x.x, acc[r][1].x);
            acc[r][1].y = fmaf(v.y, x.y, acc[r][1].y);
          }
          if (v.z != 0.f) {
            acc[r][2].x = fmaf(v.z, x.x, acc[r][2].x);
            acc[r][2].y = fmaf(v.z, x.y, acc[r][2].y);
          }
          if (v.w != 0.f) {
            acc[r][3].x = fmaf(v.w, x.x, acc[r][3].x);
            acc[r][3].y = fmaf(v.w, x.y, acc[r][3].y);
          }
        }
      }
    }
    const size_t ystride = (size_t)wout * cols;
    float2* y = (float2*)t.Y + (size_t)a0 * ystride + (size_t)g * WS_GROUP * cols + b;
#pragma unroll
    for (int r = 0; r < WS_ROWS; ++r) {
#pragma unroll
      for (int j = 0; j < WS_GROUP; ++j) {
        if (r < nr && g * WS_GROUP + j < wout) {
          float2* yr = y + r * ystride + (size_t)j * cols;
          float2 o = acc[r][j];
          if (t.beta) { o.x += yr->x; o.y += yr->y; }
          *yr = o;
        }
      }
    }
  }
}

int64_t wstage_items(int rows, int wout, int cols, int et) {
  const int64_t w = et == 0 ? wout : (wout + WS_GROUP - 1) / WS_GROUP;
  return (int64_t)((rows + WS_ROWS - 1) / WS_ROWS) * w * cols;
}
int wstage_group() { return WS_GROUP; }

void launch_wstage(const WTask* d_tasks, int ntasks, int64_t total_work, const WTables& tb, int et,
                   cudaStream_t st) {
  if (total_work <= 0) return;
  int64_t blocks = (total_work + 255) / 256;
  if (blocks > 152 * 64) blocks = 152 * 64;
  if (et == 0)
    k_wstage<<<(int)blocks, 256, 0, st>>>(d_tasks, ntasks, total_work, tb.rowptr, tb.ent_w, tb.ent_v);
  else
    k_wstage_f32<<<(int)blocks, 256, 0, st>>>(d_tasks, ntasks, total_work, tb.grp_ptr, tb.grp_w,
                                              (const float4*)tb.grp_v);
}

template <class T>
__global__ void k_to_double(const T* in, double2* out, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    out[i] = ld2(in, i);
}

void launch_to_double(const void* in, int et, double2* out, size_t n, cudaStream_t st) {
  if (n == 0) return;
  size_t blocks = (n + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  if (et == 0) k_to_double<double2><<<(unsigned)blocks, 256, 0, st>>>((const double2*)in, out, n);
  else k_to_double<float2><<<(unsigned)blocks, 256, 0, st>>>((const float2*)in, out, n);
}

__global__ void k_to_float(const double2* in, float2* out, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const double2 v = in[i];
    out[i] = make_float2((float)v.x, (float)v.y);
  }
}

void launch_to_float(const double2* in, float2* out, size_t n, cudaStream_t st) {
  if (n == 0) return;
  size_t blocks = (n + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  k_to_float<<<(unsigned)blocks, 256, 0, st>>>(in, out, n);
}

__global__ void k_fill_one(void* p, int et) {
  if (et == 0) *(double2*)p = make_double2(1.0, 0.0);
  else *(float2*)p = make_float2(1.f, 0.f);
}

void launch_fill_one(void* p, int et, cudaStream_t st) { k_fill_one<<<1, 1, 0, st>>>(p, et); }

// ------------------------------------------------------------------ gather / scatter

__global__ void k_copy(const CopyTask* __restrict__ tasks, int to_work) {
  const CopyTask t = tasks[blockIdx.x];
  int n = t.rows * t.cols;
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    int i = e / t.cols, j = e % t.cols;
    size_t w = t.conj_t ? (size_t)(t.row0 + i) * t.ldw + (t.col0 + j)
                        : (size_t)(t.col0 + j) * t.ldw + (t.row0 + i);
    double2* b = t.blk + (size_t)i * t.ld + j;
    if (to_work) {
      double2 v = cmul(t.scale, *b);
      t.work[w] = t.conj_t ? cconj(v) : v;
    } else {
      double2 v = t.work[w];
      if (t.conj_t) v = cconj(v);
      *b = cmul(t.scale, v);
    }
  }
}

void launch_copy(const CopyTask* d_tasks, int ntasks, int to_work, cudaStream_t st) {
  if (ntasks <= 0) return;
  k_copy<<<ntasks, 256, 0, st>>>(d_tasks, to_work);
}

__global__ void k_scatter(const ScatterTask* __restrict__ tasks) {
  const ScatterTask t = tasks[blockIdx.x];
  int n = t.rows * t.cols;
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    int i = e / t.cols, j = e % t.cols;
    double2 v = t.conj_t ? cconj(t.src[(size_t)(t.c0 + i) * t.lds + t.r0 + j])
                         : t.src[(size_t)(t.c0 + j) * t.lds + t.r0 + i];
    if (t.scale_dim == 1) v = cscale(v, t.s[j]);
    else if (t.scale_dim == 2) v = cscale(v, t.s[i]);
    t.blk[(size_t)i * t.ld + j] = v;
  }
}

void launch_scatter(const ScatterTask* d_tasks, int ntasks, cudaStream_t st) {
  if (ntasks <= 0) return;
  k_scatter<<<ntasks, 256, 0, st>>>(d_tasks);
}

// dst = src^H for square column-major n x n matrices (one CTA per task)
__global__ void k_adjoint(const FactTask* __restrict__ src, const FactTask* __restrict__ dst) {
  const FactTask a = src[blockIdx.x], b = dst[blockIdx.x];
  const int n = b.n;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int i = e % n, j = e / n;
    b.A[(size_t)j * n + i] = cconj(a.V[(size_t)i * n + j]);
  }
}

void launch_adjoint(const FactTask* d_src, const FactTask* d_dst, int n, cudaStream_t st) {
  if (n <= 0) return;
  k_adjoint<<<n, 256, 0, st>>>(d_src, d_dst);
}

__global__ void k_zero(double2* p, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    p[i] = make_double2(0.0, 0.0);
}

void launch_zero(double2* p, size_t n, cudaStream_t st) {
  if (n == 0) return;
  size_t blocks = (n + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  k_zero<<<(unsigned)blocks, 256, 0, st>>>(p, n);
}

__global__ void k_scale(double2* x, size_t n, double2 a) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    x[i] = cmul(a, x[i]);
}

void launch_scale(double2* x, size_t n, double2 a, cudaStream_t st) {
  if (n == 0) return;
  size_t blocks = (n + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  k_scale<<<(unsigned)blocks, 256, 0, st>>>(x, n, a);
}

__global__ void k_axpby(double2* y, const double2* x, size_t n, double2 a, double2 b) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    y[i] = cadd(cmul(a, y[i]), cmul(b, x[i]));
}

void launch_axpby(double2* y, const double2* x, size_t n, double2 a, double2 b, cudaStream_t st) {
  if (n == 0) return;
  size_t blocks = (n + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  k_axpby<<<(unsigned)blocks, 256, 0, st>>>(y, x, n, a, b);
}

// ------------------------------------------------------------------ Jacobi SVD

// One-sided (Hestenes) Jacobi on the columns of a column-major m x n matrix
// (n <= m): pairs of columns are rotated until mutually orthogonal to m*eps
// relative; round-robin pairing lets every warp rotate a disjoint pair.
// Columns below 1e-13 of the Frobenius norm are numerically zero and are not
// rotated (their singular values fall under the truncation floor).
// Afterwards sigma_j = |a_j|, u_j = a_j / sigma_j, columns sorted descending.
// The matrix and V live in shared memory when both fit (smem_budget bytes).
constexpr int SVD_THREADS = 1024;
constexpr int SVD_MAX_SWEEPS = 60;

// Rotation of the column pair with squared norms al, be and inner product
// gr + i gi (conj(a_p) a_q): c and s e^{i phi}, or false when the pair is
// already orthogonal to tol or a column is numerically zero.  Taken by one
// thread per pair: these square roots and divisions run on the FP64 pipe,
// which is the scarce unit on this part, and a warp that computed them on
// every lane would spend 32 times the pipe time.
__device__ __forceinline__ bool jacobi_rotation(double al, double be, double gr, double gi,
                                                double negl, double tol, double* c,
                                                double2* sph) {
  const double g = sqrt(gr * gr + gi * gi);
  if (g == 0.0 || al <= negl || be <= negl || g <= tol * sqrt(al * be)) return false;
  const double zeta = (be - al) / (2.0 * g);
  const double tt = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
  const double cc = 1.0 / sqrt(1.0 + tt * tt), sn = cc * tt;
  *c = cc;
  *sph = cscale(make_double2(gr / g, gi / g), sn);   // s e^{i phi}
  return true;
}

__global__ void __launch_bounds__(SVD_THREADS) k_svd(const FactTask* __restrict__ tasks,
                                                     int* status, int smem_budget) {
  extern __shared__ double2 svd_sh[];
  const FactTask t = tasks[blockIdx.x];
  const int m = t.m, n = t.n;
  const bool a_sh = (size_t)m * n * sizeof(double2) <= (size_t)smem_budget && n <= 1024;
  const bool v_sh = a_sh && (size_t)(m * n + n * n) * sizeof(double2) <= (size_t)smem_budget;
  double2* A = a_sh ? svd_sh : t.A;
  double2* V = v_sh ? svd_sh + (size_t)m * n : t.V;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  __shared__ int rotated;
  __shared__ double fro2;
  __shared__ int perm[1024];
  __shared__ double2 pr[1024];   // per pair: sums, then rotation parameters
  if (threadIdx.x == 0) fro2 = 0.0;
  if (a_sh)
    for (size_t e = threadIdx.x; e < (size_t)m * n; e += blockDim.x) A[e] = t.A[e];
  for (int e = threadIdx.x; e < n * n; e += blockDim.x)
    V[e] = make_double2((e % n) == (e / n) ? 1.0 : 0.0, 0.0);
  __syncthreads();
  {
    // Frobenius norm: warp partial sums added in warp order (the same
    // rounding on every run, so the negligibility threshold is reproducible)
    __shared__ double part[32];
    double s2 = 0.0;
    for (size_t e = threadIdx.x; e < (size_t)m * n; e += blockDim.x) s2 += cabs2(A[e]);
    s2 = warp_sum(s2);
    if (lane == 0) part[warp] = s2;
    __syncthreads();
    if (threadIdx.x == 0) {
      double f = 0.0;
      for (int w = 0; w < nwarp; ++w) f += part[w];
      fro2 = f;
    }
  }
  __syncthreads();
  const double negl = 1e-26 * fro2;
  // the computed inner product carries ~m eps relative rounding error
  const double tol = 2.2e-16 * fmax(16.0, (double)m);
  const int np = (n + 1) & ~1;   // even number of players
  int sweep = 0;
  for (; sweep < SVD_MAX_SWEEPS; ++sweep) {
    if (threadIdx.x == 0) rotated = 0;
    __syncthreads();
    for (int r = 0; r < np - 1; ++r) {
      // the pair sums and the rotation parameters (one thread per pair),
      // then the rotations (one thread per (pair, row)): no warp
      // reductions and no FP64 work repeated across lanes; pr holds each
      // pair's c and s e^{i phi}
      for (int k = threadIdx.x; k < np / 2; k += blockDim.x) {
        int pa = k, pb = np - 1 - k;
        int p = pa == 0 ? 0 : ((pa - 1 + r) % (np - 1)) + 1;
        int q = ((pb - 1 + r) % (np - 1)) + 1;
        double al = 0.0, be = 0.0, gr = 0.0, gi = 0.0;
        if (p < n && q < n) {
          if (p > q) { int tmp = p; p = q; q = tmp; }
          const double2* ap = A + (size_t)p * m;
          const double2* aq = A + (size_t)q * m;
          for (int i = 0; i < m; ++i) {
            double2 x = ap[i], y = aq[i];
            al += cabs2(x);
            be += cabs2(y);
            gr += x.x * y.x + x.y * y.y;     // conj(x) * y
            gi += x.x * y.y - x.y * y.x;
          }
        }
        double c = 1.0;
        double2 sph = make_double2(0.0, 0.0);
        const bool go = p < n && q < n && jacobi_rotation(al, be, gr, gi, negl, tol, &c, &sph);
        pr[2 * k] = make_double2(c, go ? 1.0 : 0.0);
        pr[2 * k + 1] = sph;
        if (go) rotated = 1;
      }
      __syncthreads();
      const int per = m + n;
      for (int idx = threadIdx.x; idx < (np / 2) * per; idx += blockDim.x) {
        const int k = idx / per, i = idx - k * per;
        if (pr[2 * k].y == 0.0) continue;
        int pa = k, pb = np - 1 - k;
        int p = pa == 0 ? 0 : ((pa - 1 + r) % (np - 1)) + 1;
        int q = ((pb - 1 + r) % (np - 1)) + 1;
        if (p > q) { int tmp = p; p = q; q = tmp; }
        const double c = pr[2 * k].x;
        const double2 sph = pr[2 * k + 1];                   // s e^{i phi}
        const double2 sphc = cconj(sph);                     // s e^{-i phi}
        double2* xp = i < m ? A + (size_t)p * m + i : V + (size_t)p * n + (i - m);
        double2* yp = i < m ? A + (size_t)q * m + i : V + (size_t)q * n + (i - m);
        const double2 x = *xp, y = *yp;
        *xp = csub(cscale(x, c), cmul(sphc, y));
        *yp = cadd(cmul(sph, x), cscale(y, c));
      }
      __syncthreads();
    }
    int any = rotated;
    __syncthreads();
    if (!any) break;
  }
  if (threadIdx.x == 0 && sweep == SVD_MAX_SWEEPS) atomicExch(status, 1);
  // singular values
  for (int j = warp; j < n; j += nwarp) {
    const double2* aj = A + (size_t)j * m;
    double s2 = 0.0;
    for (int i = lane; i < m; i += 32) s2 += cabs2(aj[i]);
    s2 = warp_sum(s2);
    if (lane == 0) t.s[j] = sqrt(s2);
  }
  __syncthreads();
  if (a_sh) {
    // descending order (ties: lower index first) written straight out
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
      double sj = t.s[j];
      int rank = 0;
      for (int k = 0; k < n; ++k) {
        double sk = t.s[k];
        rank += (sk > sj) || (sk == sj && k < j);
      }
      perm[rank] = j;
      pr[j].x = sj > 0.0 ? 1.0 / sj : 0.0;   // 1/sigma once per column (pairs are done)
    }
    __syncthreads();
    for (size_t e = threadIdx.x; e < (size_t)m * n; e += blockDim.x) {
      int j = (int)(e / m), i = (int)(e % m);
      t.A[e] = cscale(A[(size_t)perm[j] * m + i], pr[perm[j]].x);
    }
    __syncthreads();
    if (!v_sh) {   // A's shared buffer is free: stage V there (n*n <= m*n)
      for (size_t e = threadIdx.x; e < (size_t)n * n; e += blockDim.x) svd_sh[e] = t.V[e];
      __syncthreads();
      V = svd_sh;
    }
    for (size_t e = threadIdx.x; e < (size_t)n * n; e += blockDim.x) {
      int j = (int)(e / n), i = (int)(e % n);
      t.V[e] = V[(size_t)perm[j] * n + i];
    }
    // permute the singular values: one thread per value (n <= 1024 = blockDim)
    double mine = threadIdx.x < n ? t.s[perm[threadIdx.x]] : 0.0;
    __syncthreads();
    if (threadIdx.x < n) t.s[threadIdx.x] = mine;
    return;
  }
  for (int j = warp; j < n; j += nwarp) {
    double2* aj = A + (size_t)j * m;
    double sv = t.s[j];
    double inv = sv > 0.0 ? 1.0 / sv : 0.0;
    for (int i = lane; i < m; i += 32) aj[i] = cscale(aj[i], inv);
  }
  __syncthreads();
  // selection sort in global memory, descending (ties: lower index first)
  __shared__ int sel;
  for (int j = 0; j < n - 1; ++j) {
    if (threadIdx.x == 0) {
      int b = j;
      for (int k = j + 1; k < n; ++k)
        if (t.s[k] > t.s[b]) b = k;
      sel = b;
    }
    __syncthreads();
    int b = sel;
    if (b != j) {
      for (int i = threadIdx.x; i < m; i += blockDim.x) {
        double2 x = A[(size_t)j * m + i];
        A[(size_t)j * m + i] = A[(size_t)b * m + i];
        A[(size_t)b * m + i] = x;
      }
      for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double2 x = V[(size_t)j * n + i];
        V[(size_t)j * n + i] = V[(size_t)b * n + i];
        V[(size_t)b * n + i] = x;
      }
      if (threadIdx.x == 0) {
        double x = t.s[j];
        t.s[j] = t.s[b];
        t.s[b] = x;
      }
    }
    __syncthreads();
  }
}

// One-CTA Jacobi SVD of a small matrix (m x n, n <= m), in three stages:
//   1. one-sided Jacobi in FP32 on a copy scaled by a power of two: this part's
//      FP32 pipe is 64 times as wide as its FP64 pipe, so the sweeps that bring
//      the columns from arbitrary to orthogonal within 1e-6 cost little;
//   2. the accumulated rotations V, unitary to FP32 rounding, made unitary to
//      FP64 rounding by two Newton steps V <- V - V (V^H V - 1) / 2 (the
//      defect in FP64; the correction, a product of the small defect, in
//      FP32), and A V in FP64;
//   3. one-sided Jacobi in FP64 from there, to the same criterion as the
//      kernels below.  Two or three sweeps remain of seven to nine.  A
//      rotation's tangent is taken in FP32 (any tangent is a rotation; a
//      relative error of 1e-7 in it leaves 1e-7 of the inner product), its
//      cosine and sine in FP64, so V stays unitary to FP64 rounding.
// What bounds it is the FP64 pipe in the rotations of stage 3 (12 operations
// per row and pair of A and V).  Measured against FP64 Jacobi from the start
// (one CTA below n = 24, a cluster from there): compression 256 -> 128 at L = 16
// (15 launches, n <= 25) 17.3 -> 6.3 ms; a two-site Runge-Kutta step at L = 8,
// D = 64 (224 launches, n <= 36) 76.4 -> 29.1 ms; at L = 12, D = 128 (n up to
// 56) 342 -> 160 ms, of which 262 with the line at n = 32.  256 threads: 7.5 ms.
constexpr int SVDS_THREADS = 512;
constexpr int SVDS_MAX_N = 64;   // 164 KB of shared memory

__host__ __device__ inline size_t svds_bytes(int m, int n) {
  return 16 * ((size_t)m * n + (size_t)n * n) + 8 * (size_t)n * n;
}

__global__ void __launch_bounds__(SVDS_THREADS) k_svd_small(const FactTask* __restrict__ tasks,
                                                            int* status) {
  extern __shared__ double2 svd_sh[];
  const FactTask t = tasks[blockIdx.x];
  const int m = t.m, n = t.n;
  double2* A = svd_sh;                        // [n][m], stage 3
  double2* V = A + (size_t)m * n;             // [n][n]
  float2* E = (float2*)(V + (size_t)n * n);   // [n][n], stage 2
  float2* Af = (float2*)svd_sh;               // [n][m], stage 1, where A will be
  float2* Vf = Af + (size_t)m * n;            // [n][n], stages 1 and 2, the same
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = SVDS_THREADS / 32;
  __shared__ int rotated, expo;
  __shared__ double nrm[SVDS_MAX_N];          // squared column norms, tracked
  __shared__ double2 pr[SVDS_MAX_N];          // per pair: c, whether it rotates
  __shared__ double2 sc_sh[SVDS_MAX_N];       // per pair: s e^{i phi}
  __shared__ int perm[SVDS_MAX_N];
  if (tid == 0) expo = 0;
  __syncthreads();
  // power of two at the largest element, so that FP32 neither over- nor underflows
  {
    int e = 0;
    for (int i = tid; i < m * n; i += SVDS_THREADS) {
      const double2 x = t.A[i];
      e = max(e, max((__double2hiint(x.x) >> 20) & 0x7ff, (__double2hiint(x.y) >> 20) & 0x7ff));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) atomicMax(&expo, e);
  }
  __syncthreads();
  const int ex = max(expo, 1) - 1022;         // |x| < 2^ex
  const double down = scalbn(1.0, -max(-1000, min(1000, ex)));
  for (int i = tid; i < m * n; i += SVDS_THREADS) {
    const double2 x = t.A[i];
    Af[i] = make_float2((float)(x.x * down), (float)(x.y * down));
  }
  for (int i = tid; i < n * n; i += SVDS_THREADS) Vf[i] = make_float2(i % n == i / n ? 1.f : 0.f, 0.f);
  const int np = (n + 1) & ~1;   // even number of players
  // the round's k-th pair, p < q; q == n: a bye
  auto pair_of = [&](int k, int r, int& p, int& q) {
    const int pb = np - 1 - k;
    p = k == 0 ? 0 : ((k - 1 + r) % (np - 1)) + 1;
    q = ((pb - 1 + r) % (np - 1)) + 1;
    if (p > q) { const int x = p; p = q; q = x; }
  };

  // ---- stage 1: FP32, a warp per pair
  for (int sweep = 0; sweep < 12 && expo < 0x7ff; ++sweep) {
    __syncthreads();
    if (tid == 0) rotated = 0;
    __syncthreads();
    for (int r = 0; r < np - 1; ++r) {
      for (int k = warp; k < np / 2; k += NW) {
        int p, q;
        pair_of(k, r, p, q);
        if (q >= n) continue;
        float2 *ap = Af + (size_t)p * m, *aq = Af + (size_t)q * m;
        float al = 0.f, be = 0.f, gr = 0.f, gi = 0.f;
        for (int i = lane; i < m; i += 32) {
          const float2 x = ap[i], y = aq[i];
          al += x.x * x.x + x.y * x.y;
          be += y.x * y.x + y.y * y.y;
          gr += x.x * y.x + x.y * y.y;
          gi += x.x * y.y - x.y * y.x;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          al += __shfl_xor_sync(0xffffffffu, al, o);
          be += __shfl_xor_sync(0xffffffffu, be, o);
          gr += __shfl_xor_sync(0xffffffffu, gr, o);
          gi += __shfl_xor_sync(0xffffffffu, gi, o);
        }
        const float g2 = gr * gr + gi * gi;
        if (!(al > 1e-30f && be > 1e-30f && g2 > 1e-12f * al * be && g2 > 1e-36f)) continue;
        const float g = sqrtf(g2), z = (be - al) / (2.f * g);
        const float tt = (z >= 0.f ? 1.f : -1.f) / (fabsf(z) + sqrtf(1.f + z * z));
        const float c = 1.f / sqrtf(1.f + tt * tt);
        const float sx = c * tt * gr / g, sy = c * tt * gi / g;
        auto rot = [&](float2& x, float2& y) {
          const float2 a = x, b = y;
          x = make_float2(c * a.x - (sx * b.x + sy * b.y), c * a.y - (sx * b.y - sy * b.x));
          y = make_float2(c * b.x + (sx * a.x - sy * a.y), c * b.y + (sx * a.y + sy * a.x));
        };
        for (int i = lane; i < m; i += 32) rot(ap[i], aq[i]);
        for (int i = lane; i < n; i += 32) rot(Vf[(size_t)p * n + i], Vf[(size_t)q * n + i]);
        if (lane == 0) rotated = 1;
      }
      __syncthreads();
    }
    if (!rotated) break;
  }
  __syncthreads();

  // ---- stage 2: V unitary in FP64, then A V
  for (int i = tid; i < n * n; i += SVDS_THREADS) V[i] = make_double2(Vf[i].x, Vf[i].y);
  for (int it = 0; it < 2; ++it) {
    __syncthreads();
    for (int e = tid; e < n * n; e += SVDS_THREADS) {
      const int p = e % n, q = e / n;
      if (p > q) continue;
      const double2 *x = V + (size_t)p * n, *y = V + (size_t)q * n;
      double re = p == q ? -1.0 : 0.0, im = 0.0;
      for (int i = 0; i < n; ++i) {
        re = fma(x[i].x, y[i].x, fma(x[i].y, y[i].y, re));
        im = fma(x[i].x, y[i].y, fma(-x[i].y, y[i].x, im));
      }
      const float2 d = make_float2((float)re, (float)im);
      E[(size_t)q * n + p] = d;                     // (V^H V - 1)(p, q)
      E[(size_t)p * n + q] = make_float2(d.x, p == q ? d.y : -d.y);
    }
    __syncthreads();
    for (int e = tid; e < n * n; e += SVDS_THREADS) {
      const int i = e % n, q = e / n;
      float re = 0.f, im = 0.f;
      for (int p = 0; p < n; ++p) {
        const float2 v = Vf[(size_t)p * n + i], d = E[(size_t)q * n + p];
        re += v.x * d.x - v.y * d.y;
        im += v.x * d.y + v.y * d.x;
      }
      V[e] = make_double2(V[e].x - 0.5 * (double)re, V[e].y - 0.5 * (double)im);
    }
  }
  __syncthreads();   // Vf is done with: A takes its place
  for (int e = tid; e < m * n; e += SVDS_THREADS) {
    const int i = e % m, q = e / m;
    double2 acc = make_double2(0.0, 0.0);
    for (int p = 0; p < n; ++p) acc = cfma(t.A[(size_t)p * m + i], V[(size_t)q * n + p], acc);
    A[e] = cscale(acc, down);
  }
  __syncthreads();

  // ---- stage 3: FP64
  __shared__ double fro2;
  // the computed inner product carries ~m eps relative rounding error
  const double tol = 2.2e-16 * fmax(16.0, (double)m), tol2 = tol * tol;
  int sweep = 0;
  for (; sweep < SVD_MAX_SWEEPS; ++sweep) {
    // column norms, four lanes each (tracked within the sweep)
    for (int c = tid >> 2; c < ((n + 7) & ~7); c += SVDS_THREADS / 4) {
      double s = 0.0;
      if (c < n)
        for (int i = tid & 3; i < m; i += 4) s += cabs2(A[(size_t)c * m + i]);
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      if (c < n && (tid & 3) == 0) nrm[c] = s;
    }
    if (tid == 0) rotated = 0;
    __syncthreads();
    if (sweep == 0 && tid == 0) {
      double f = 0.0;
      for (int c = 0; c < n; ++c) f += nrm[c];
      fro2 = f;
    }
    __syncthreads();
    const double negl = 1e-26 * fro2;
    for (int r = 0; r < np - 1; ++r) {
      // inner products, four lanes per pair (whole warps enter: np / 2 * 4
      // rounded up to 32)
      for (int k0 = tid >> 2; k0 < ((np / 2 + 7) & ~7); k0 += SVDS_THREADS / 4) {
        int p = 0, q = n;
        if (k0 < np / 2) pair_of(k0, r, p, q);
        double gr = 0.0, gi = 0.0;
        if (q < n) {
          const double2 *ap = A + (size_t)p * m, *aq = A + (size_t)q * m;
          for (int i = tid & 3; i < m; i += 4) {
            const double2 x = ap[i], y = aq[i];
            gr = fma(x.x, y.x, fma(x.y, y.y, gr));
            gi = fma(x.x, y.y, fma(-x.y, y.x, gi));
          }
        }
        gr += __shfl_xor_sync(0xffffffffu, gr, 1);
        gi += __shfl_xor_sync(0xffffffffu, gi, 1);
        gr += __shfl_xor_sync(0xffffffffu, gr, 2);
        gi += __shfl_xor_sync(0xffffffffu, gi, 2);
        if ((tid & 3) == 0 && k0 < np / 2) {
          double c = 1.0;
          double2 s = make_double2(0.0, 0.0);
          bool go = false;
          if (q < n) {
            const double al = nrm[p], be = nrm[q], g2 = gr * gr + gi * gi;
            go = al > negl && be > negl && g2 > tol2 * al * be;
            if (go) {
              double tr, ti;   // tan e^{i phi}
              if (g2 > 1e-32) {
                const float gf = sqrtf((float)g2), z = (float)(be - al) / (2.f * gf);
                const float tt = fabsf(z) > 1e9f ? 0.5f / z
                                                 : copysignf(1.f, z) / (fabsf(z) + sqrtf(1.f + z * z));
                tr = (double)(tt * ((float)gr / gf));
                ti = (double)(tt * ((float)gi / gf));
              } else {
                const double g = sqrt(g2), z = (be - al) / (2.0 * g);
                const double tt = (z >= 0.0 ? 1.0 : -1.0) / (fabs(z) + sqrt(1.0 + z * z));
                tr = tt * gr / g;
                ti = tt * gi / g;
              }
              const double h = tr * tr + ti * ti;
              if (h < 1e-5)   // 1 / sqrt(1 + h), next term 63/256 h^5
                c = 1.0 + h * (-0.5 + h * (0.375 + h * (-0.3125 + h * 0.2734375)));
              else
                c = 1.0 / sqrt(1.0 + h);
              s = make_double2(c * tr, c * ti);
              const double d = tr * gr + ti * gi;   // tan |g|
              nrm[p] = al - d;
              nrm[q] = be + d;
              rotated = 1;
            }
          }
          pr[k0] = make_double2(c, go ? 1.0 : 0.0);
          sc_sh[k0] = s;
        }
      }
      __syncthreads();
      const int per = m + n;
      for (int idx = tid; idx < (np / 2) * per; idx += SVDS_THREADS) {
        const int k = idx / per, i = idx - k * per;
        if (__double2hiint(pr[k].y) == 0) continue;
        int p, q;
        pair_of(k, r, p, q);
        const double c = pr[k].x;
        const double2 s = sc_sh[k];
        double2* xp = i < m ? A + (size_t)p * m + i : V + (size_t)p * n + (i - m);
        double2* yp = i < m ? A + (size_t)q * m + i : V + (size_t)q * n + (i - m);
        const double2 x = *xp, y = *yp;
        *xp = make_double2(fma(c, x.x, fma(-s.x, y.x, -s.y * y.y)), fma(c, x.y, fma(-s.x, y.y, s.y * y.x)));
        *yp = make_double2(fma(c, y.x, fma(s.x, x.x, -s.y * x.y)), fma(c, y.y, fma(s.x, x.y, s.y * x.x)));
      }
      __syncthreads();
    }
    const int any = rotated;
    __syncthreads();
    if (!any) break;
  }
  if (tid == 0 && sweep == SVD_MAX_SWEEPS) atomicExch(status, 1);

  // singular values, descending (ties: lower index first)
  for (int c = warp; c < n; c += NW) {
    double s = 0.0;
    for (int i = lane; i < m; i += 32) s += cabs2(A[(size_t)c * m + i]);
    s = warp_sum(s);
    if (lane == 0) nrm[c] = sqrt(s);
  }
  if (tid < n) perm[tid] = tid;   // with NaN the ranks below do not cover every place
  __syncthreads();
  int rk = 0;
  if (tid < n) {
    const double sj = nrm[tid];
    for (int k = 0; k < n; ++k) rk += (nrm[k] > sj) || (nrm[k] == sj && k < tid);
    perm[rk] = tid;
    pr[tid].x = sj > 0.0 ? 1.0 / sj : 0.0;
  }
  __syncthreads();
  if (tid < n) t.s[tid] = nrm[perm[tid]] * scalbn(1.0, max(-1000, min(1000, ex)));
  __syncthreads();
  for (int e = tid; e < m * n; e += SVDS_THREADS) {
    const int j = e / m, i = e % m, pj = perm[j];
    t.A[e] = cscale(A[(size_t)pj * m + i], pr[pj].x);
  }
  for (int e = tid; e < n * n; e += SVDS_THREADS) {
    const int j = e / n, i = e % n;
    t.V[e] = V[(size_t)perm[j] * n + i];
  }
}

// The same one-sided Jacobi SVD with one matrix spread over a cluster of
// SVDC_CS CTAs: CTA `rank` holds rows [rank*mc, rank*mc + mc) of A in shared
// memory and rows [rank*nc, rank*nc + nc) of V in global memory.  Each round
// of the round-robin ordering computes the partial inner products (|a_p|^2,
// |a_q|^2, a_p^H a_q) of all its n/2 disjoint column pairs over the local
// rows, sums them across the cluster in one reduction (slots in every CTA's
// shared memory, rank-ordered sums, so every CTA takes the same rotation
// decisions), and rotates its own rows.  One cluster barrier per round
// instead of one SM doing all of the FP64 work.
constexpr int SVDC_CS = 8;
constexpr int SVDC_THREADS = 512;

__host__ __device__ inline size_t svdc_elems(int m, int n) {
  const size_t mc = (m + SVDC_CS - 1) / SVDC_CS;
  const size_t np = (size_t)((n + 1) & ~1);
  const size_t SL = np > (size_t)n ? np : (size_t)n;
  return mc * n + SL + 2 * (size_t)SVDC_CS * SL + (size_t)n + 16;
}

__global__ void __launch_bounds__(SVDC_THREADS) k_svd_cl(const FactTask* __restrict__ tasks,
                                                         int* status) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ double2 shv[];
  const int rank = (int)cl.block_rank();
  const FactTask t = tasks[blockIdx.x / SVDC_CS];
  const int m = t.m, n = t.n;
  const int mc = (m + SVDC_CS - 1) / SVDC_CS, nc = (n + SVDC_CS - 1) / SVDC_CS;
  const int row0 = rank * mc, ml = max(0, min(mc, m - row0));
  const int vr0 = rank * nc, nl = max(0, min(nc, n - vr0));
  const int np = (n + 1) & ~1;
  const int SL = np > n ? np : n;
  double2* A = shv;                          // [n][mc]
  double2* part = A + (size_t)mc * n;        // [SL]: pair k -> (al, be), (gr, gi) at 2k, 2k+1
  double2* slots = part + SL;                // [2][CS][SL]
  double* sv = (double*)(slots + 2 * (size_t)SVDC_CS * SL);   // [n]
  int* perm = (int*)(sv + n);                // [n]
  __shared__ int rotated;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  int red = 0;
  auto allreduce = [&](double2* buf, int len) {
    const int b = red & 1;
    ++red;
    for (int r = 0; r < SVDC_CS; ++r) {
      double2* dst = cl.map_shared_rank(slots, r) + ((size_t)b * SVDC_CS + rank) * SL;
      for (int i = threadIdx.x; i < len; i += blockDim.x) dst[i] = buf[i];
    }
    cl.sync();
    for (int i = threadIdx.x; i < len; i += blockDim.x) {
      double2 acc = make_double2(0.0, 0.0);
      for (int r = 0; r < SVDC_CS; ++r) acc = cadd(acc, slots[((size_t)b * SVDC_CS + r) * SL + i]);
      buf[i] = acc;
    }
    __syncthreads();
  };
  for (int c = 0; c < n; ++c)
    for (int i = threadIdx.x; i < ml; i += blockDim.x) A[(size_t)c * mc + i] = t.A[(size_t)c * m + row0 + i];
  for (int c = 0; c < n; ++c)
    for (int i = threadIdx.x; i < nl; i += blockDim.x)
      t.V[(size_t)c * n + vr0 + i] = make_double2(vr0 + i == c ? 1.0 : 0.0, 0.0);
  // the rows were staged by every thread; warp 0 reads all of them
  __syncthreads();
  // Frobenius norm
  {
    if (warp == 0) {
      double s2 = 0.0;
      for (size_t e = lane; e < (size_t)ml * n; e += 32) {
        const size_t c = e / ml, i = e % ml;
        s2 += cabs2(A[c * mc + i]);
      }
      s2 = warp_sum(s2);
      if (lane == 0) part[0] = make_double2(s2, 0.0);
    }
    __syncthreads();
    allreduce(part, 1);
  }
  const double negl = 1e-26 * part[0].x;
  const double tol = 2.2e-16 * fmax(16.0, (double)m);
  __syncthreads();
  int sweep = 0;
  for (; sweep < SVD_MAX_SWEEPS; ++sweep) {
    if (threadIdx.x == 0) rotated = 0;
    __syncthreads();
    for (int r = 0; r < np - 1; ++r) {
      // the partial sums of every pair over the local rows, one thread per
      // pair (the local rows are few: no warp reduction, whose shuffles and
      // adds would cost the FP64 pipe on every lane)
      for (int k = threadIdx.x; k < np / 2; k += blockDim.x) {
        int pa = k, pb = np - 1 - k;
        int p = pa == 0 ? 0 : ((pa - 1 + r) % (np - 1)) + 1;
        int q = ((pb - 1 + r) % (np - 1)) + 1;
        double al = 0.0, be = 0.0, gr = 0.0, gi = 0.0;
        if (p < n && q < n) {
          if (p > q) { int tmp = p; p = q; q = tmp; }
          const double2* ap = A + (size_t)p * mc;
          const double2* aq = A + (size_t)q * mc;
          for (int i = 0; i < ml; ++i) {
            const double2 x = ap[i], y = aq[i];
            al += cabs2(x);
            be += cabs2(y);
            gr += x.x * y.x + x.y * y.y;     // conj(x) * y
            gi += x.x * y.y - x.y * y.x;
          }
        }
        part[2 * k] = make_double2(al, be);
        part[2 * k + 1] = make_double2(gr, gi);
      }
      __syncthreads();
      allreduce(part, np);
      // rotation parameters, one thread per pair, in place of the sums
      for (int k = threadIdx.x; k < np / 2; k += blockDim.x) {
        int pa = k, pb = np - 1 - k;
        int p = pa == 0 ? 0 : ((pa - 1 + r) % (np - 1)) + 1;
        int q = ((pb - 1 + r) % (np - 1)) + 1;
        double c = 1.0;
        double2 sph = make_double2(0.0, 0.0);
        const bool go = p < n && q < n &&
                        jacobi_rotation(part[2 * k].x, part[2 * k].y, part[2 * k + 1].x,
                                        part[2 * k + 1].y, negl, tol, &c, &sph);
        part[2 * k] = make_double2(c, go ? 1.0 : 0.0);
        part[2 * k + 1] = sph;
        if (go) rotated = 1;
      }
      __syncthreads();
      // the rotations, one thread per (pair, local row of A or V)
      const int per = ml + nl;
      for (int idx = threadIdx.x; idx < (np / 2) * per; idx += blockDim.x) {
        const int k = idx / per, i = idx - k * per;
        if (part[2 * k].y == 0.0) continue;
        int pa = k, pb = np - 1 - k;
        int p = pa == 0 ? 0 : ((pa - 1 + r) % (np - 1)) + 1;
        int q = ((pb - 1 + r) % (np - 1)) + 1;
        if (p > q) { int tmp = p; p = q; q = tmp; }
        const double c = part[2 * k].x;
        const double2 sph = part[2 * k + 1];                // s e^{i phi}
        const double2 sphc = cconj(sph);                    // s e^{-i phi}
        double2* xp;
        double2* yp;
        if (i < ml) {
          xp = A + (size_t)p * mc + i;
          yp = A + (size_t)q * mc + i;
        } else {
          xp = t.V + (size_t)p * n + vr0 + (i - ml);
          yp = t.V + (size_t)q * n + vr0 + (i - ml);
        }
        const double2 x = *xp, y = *yp;
        *xp = csub(cscale(x, c), cmul(sphc, y));
        *yp = cadd(cmul(sph, x), cscale(y, c));
      }
      __syncthreads();
    }
    const int any = rotated;   // identical in every CTA of the cluster
    __syncthreads();
    if (!any) break;
  }
  if (rank == 0 && threadIdx.x == 0 && sweep == SVD_MAX_SWEEPS) atomicExch(status, 1);
  // singular values: column norms over all rows
  for (int j = warp; j < n; j += nwarp) {
    const double2* aj = A + (size_t)j * mc;
    double s2 = 0.0;
    for (int i = lane; i < ml; i += 32) s2 += cabs2(aj[i]);
    s2 = warp_sum(s2);
    if (lane == 0) part[j] = make_double2(s2, 0.0);
  }
  __syncthreads();
  allreduce(part, n);
  for (int j = threadIdx.x; j < n; j += blockDim.x) sv[j] = sqrt(part[j].x);
  __syncthreads();
  // descending order, ties: lower index first
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const double sj = sv[j];
    int rk = 0;
    for (int k = 0; k < n; ++k) rk += (sv[k] > sj) || (sv[k] == sj && k < j);
    perm[rk] = j;
    part[j].x = sj > 0.0 ? 1.0 / sj : 0.0;   // 1/sigma once per column
  }
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    const int pj = perm[j];
    const double inv = part[pj].x;
    for (int i = threadIdx.x; i < ml; i += blockDim.x)
      t.A[(size_t)j * m + row0 + i] = cscale(A[(size_t)pj * mc + i], inv);
  }
  if (rank == 0)
    for (int j = threadIdx.x; j < n; j += blockDim.x) t.s[j] = sv[perm[j]];
  // V columns permuted; each CTA owns its rows of V, staged through the A
  // buffer (free now; the launcher requires m >= n, so nc <= mc)
  __syncthreads();
  for (int c = 0; c < n; ++c)
    for (int i = threadIdx.x; i < nl; i += blockDim.x) A[(size_t)c * nc + i] = t.V[(size_t)c * n + vr0 + i];
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    const int pj = perm[j];
    for (int i = threadIdx.x; i < nl; i += blockDim.x)
      t.V[(size_t)j * n + vr0 + i] = A[(size_t)pj * nc + i];
  }
  // no CTA may leave while others can still write into its slots
  cl.sync();
}

void launch_svd(const FactTask* d_tasks, int ntasks, int* d_status, cudaStream_t st,
                size_t max_bytes, const FactTask* h_tasks) {
  if (ntasks <= 0) return;
  // One kernel per launch: k_svd_small when every matrix of the bond fits it
  // (SVDS_MAX_N; its comment has both sides), else the cluster kernel if all
  // fit that one, else one CTA per matrix in global memory.
  {
    size_t need = 0;
    bool all_small = h_tasks != nullptr;
    for (int i = 0; h_tasks && i < ntasks; ++i) {
      if (h_tasks[i].n > SVDS_MAX_N || h_tasks[i].m < h_tasks[i].n) all_small = false;
      need = std::max(need, svds_bytes(h_tasks[i].m, h_tasks[i].n));
    }
    const size_t cap_small = 200 * 1024;
    if (all_small && need <= cap_small) {
      set_smem_limit((const void*)k_svd_small, (int)cap_small);
      k_svd_small<<<ntasks, SVDS_THREADS, need, st>>>(d_tasks, d_status);
      return;
    }
  }
  {
    const size_t cap_cl = 200 * 1024;
    size_t need = 0;
    bool shape_ok = h_tasks != nullptr;
    for (int i = 0; h_tasks && i < ntasks; ++i) {
      need = std::max(need, svdc_elems(h_tasks[i].m, h_tasks[i].n) * sizeof(double2));
      if (h_tasks[i].m < h_tasks[i].n || h_tasks[i].n > 2048) shape_ok = false;
    }
    if (shape_ok && need <= cap_cl) {
      set_smem_limit((const void*)k_svd_cl, (int)cap_cl);
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)(ntasks * SVDC_CS));
      cfg.blockDim = dim3(SVDC_THREADS);
      cfg.dynamicSmemBytes = need;
      cfg.stream = st;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = SVDC_CS;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      cudaLaunchKernelEx(&cfg, k_svd_cl, d_tasks, d_status);
      return;
    }
  }
  // static shared: perm (4 KB), the pair array (16 KB) and scalars
  const size_t cap = 227 * 1024 - 21 * 1024;
  size_t dyn = max_bytes < cap ? max_bytes : cap;
  set_smem_limit((const void*)k_svd, (int)cap);
  k_svd<<<ntasks, SVD_THREADS, dyn, st>>>(d_tasks, d_status, (int)dyn);
}

// ------------------------------------------------------------------ Gram-Schmidt QR

// Modified Gram-Schmidt with conditional re-orthogonalisation on column-major
// m x n matrices: A = Q R, one matrix per cluster of CS CTAs (CS = 1: one CTA).
// CTA `rank` holds rows [rank*mc, rank*mc + mc), in shared memory when they
// fit, else in place in global memory.
//
// Right-looking: at step j the pivot v = a_j (already orthogonal to the
// accepted columns) is multiplied with every remaining column at once,
//   p_c = v^H a_c (c >= j; p_j = |v|^2),   a_c -= v p_c / p_j,
// so a step is one set of independent inner products, one cluster reduction
// and one rank-one update; nothing is summed serially over the earlier
// columns, and roots and the normalisation wait until the end (the FP64 pipe
// does two multiply-adds per clock and SM, so serial chains and work repeated
// on every lane are what costs here).  Each CTA writes its partial products
// into a slot of every CTA, the cluster barrier publishes them, and every CTA
// adds the slots in rank order: all hold the same bits and take the same
// branches.  Slots are double buffered: the barrier of reduction r also tells
// a CTA that every CTA has read the buffer of reduction r - 1.
//
// A column that lost more than half of its squared norm to the earlier ones
// (the Daniel-Gragg-Kaufman-Stewart criterion, on norms down-dated by
// |p_c|^2 / p_j) is projected once more against all accepted columns before
// it becomes the pivot.  A column whose residual norm is <= 1e-12 times the
// largest input column norm adds no direction.  Accepted directions are
// stored compactly in the first columns (at most k = min(m, n)), the others
// of the first k columns are zero.  R (n x n, column-major) holds the
// coefficients.
//
// Measured (one fitted H|psi>, L = 16, D = 256: 45 launches of ~38 sectors, n up
// to 25): 3.5 ms, where a left-looking form with five to seven block barriers
// and serial sums per column took 8.75 ms.  256 threads: 3.6 ms, 512: 4.2 ms;
// clusters of 4 CTAs: 3.5 ms.
constexpr int QR_THREADS = 128;
constexpr int QR_CS = 8;
// m n^2 from which a matrix gets a cluster.  With the line at 0 / 4000 / 12000 /
// 30000 / never: QR of a two-site Runge-Kutta step at L = 8, D = 64 17.5 / 15.4 / 15.4 /
// 14.9 / 14.9 ms, of the fitted H|psi> above 3.38 / 3.31 / 3.38 / 3.57 / 5.39 ms.
constexpr double QR_CLUSTER_WORK = 12000;
constexpr int QR_SMEM = 200 * 1024;
constexpr double QR_SQ_MIN = 0x1p-800, QR_SQ_MAX = 0x1p800;   // largest squared norm used as it is
constexpr double QR_SHIFT = 0x1p700;
constexpr int QR_BATCH = 512;         // columns of one reduction
constexpr int QR_BATCH_GLOBAL = 256;  // the same when the matrix stays in global memory

__host__ __device__ inline int qr_mc(int m, int cs) { return (m + cs - 1) / cs; }
// complex elements of dynamic shared memory: slots, factors, squared pivots
// and column norms, projection partials; then the rows
__host__ __device__ inline size_t qr_fixed(int n, int cs, int batch) {
  const size_t nb = n < batch ? n : batch;
  return 2 * (size_t)cs * nb + nb + (3 * (size_t)n + 1) / 2 + ((size_t)n + 3) / 4 + 1 + QR_THREADS;
}

template <int CS>
__global__ void __launch_bounds__(QR_THREADS) k_qr(const FactTask* __restrict__ tasks, int batch,
                                                   int smem_elems) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ double2 qr_sh[];
  const int rank = CS > 1 ? (int)cl.block_rank() : 0;
  const FactTask t = tasks[blockIdx.x / CS];
  const int m = t.m, n = t.n, kmax = m < n ? m : n;
  const int mc = qr_mc(m, CS), row0 = rank * mc;
  const int ml = max(0, min(mc, m - row0));   // rows held here
  const int NB = n < batch ? n : batch;
  double2* slots = qr_sh;                        // [2][CS][NB]
  double2* fac = slots + 2 * (size_t)CS * NB;    // [NB]
  double2* pp = fac + NB;                        // [QR_THREADS]
  double* piv = (double*)(pp + QR_THREADS);      // [n] squared norms of the accepted columns
  double* orig = piv + n;                        // [n] squared column norms
  double* est = orig + n;                        // [n] the same, down-dated
  int* again = (int*)(est + n);                  // [n] the column needs the second projection
  __shared__ int keep_sh;
  const size_t fixed = qr_fixed(n, CS, batch);
  const bool a_sh = fixed + (size_t)mc * n <= (size_t)smem_elems;
  double2* A = a_sh ? qr_sh + fixed : t.A + row0;   // column c at A + c * lda
  const size_t lda = a_sh ? mc : m;
  const int tid = threadIdx.x;
  int red = 0;

  // partial products conj(x) . y of the local rows for the columns [c0, c0 + cnt),
  // 1 to 8 lanes per column, into this CTA's slot of every CTA; then the barrier.
  // self: |a_c|^2 of each column, else column x times column c
  auto products = [&](const double2* x, int c0, int cnt, bool self) {
    const int lpc = cnt * 8 <= QR_THREADS ? 8 : cnt * 4 <= QR_THREADS ? 4 : cnt * 2 <= QR_THREADS ? 2 : 1;
    const int sub = tid & (lpc - 1), step = QR_THREADS / lpc;
    const int b = red & 1;
    // every lane of a warp takes part in the shuffles
    for (int k0 = 0; k0 < cnt; k0 += step) {
      const int k = k0 + tid / lpc;
      double re = 0.0, im = 0.0;
      if (k < cnt) {
        const double2* y = A + (size_t)(c0 + k) * lda;
        const double2* p = self ? y : x;
        for (int i = sub; i < ml; i += lpc) {
          const double2 u = p[i], w = y[i];
          re = fma(u.x, w.x, fma(u.y, w.y, re));
          im = fma(u.x, w.y, fma(-u.y, w.x, im));
        }
      }
      for (int o = lpc >> 1; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
      }
      if (k < cnt)
        for (int r = sub; r < CS; r += lpc) {
          double2* dst = CS > 1 ? cl.map_shared_rank(slots, r) : slots;
          dst[((size_t)b * CS + rank) * NB + k] = make_double2(re, im);
        }
    }
    if (CS > 1) cl.sync(); else __syncthreads();
    ++red;
  };
  // entry k of the last reduction
  auto total = [&](int k) {
    const double2* s = slots + (size_t)((red - 1) & 1) * CS * NB + k;
    double2 v = s[0];
#pragma unroll
    for (int r = 1; r < CS; ++r) v = cadd(v, s[(size_t)r * NB]);
    return v;
  };

  if (a_sh)
    for (int c = tid >> 5; c < n; c += QR_THREADS / 32)
      for (int i = tid & 31; i < ml; i += 32) A[c * lda + i] = t.A[(size_t)c * m + row0 + i];
  if (rank == 0)
    for (int e = tid; e < n * n; e += QR_THREADS) t.V[e] = make_double2(0.0, 0.0);
  __syncthreads();
  long long big = 0;
  double back = 1.0;   // what R is multiplied with in the end
  for (int pass = 0;; ++pass) {
    for (int c0 = 0; c0 < n; c0 += NB) {
      const int cnt = min(NB, n - c0);
      products(nullptr, c0, cnt, true);
      for (int k = tid; k < cnt; k += QR_THREADS) {
        orig[c0 + k] = est[c0 + k] = total(k).x;
        again[c0 + k] = 0;
      }
    }
    __syncthreads();
    // non-negative FP64 numbers order like their bit patterns
    big = 0;
    for (int c = 0; c < n; ++c) big = max(big, __double_as_longlong(orig[c]));
    // Squared norms far out are brought in by a power of two, once (the same
    // decision in every CTA): an accepted pivot is down to 1e-24 of the largest
    // square, and its reciprocal has to be a number.
    const bool tiny = big < __double_as_longlong(QR_SQ_MIN);
    if (pass || (!tiny && big <= __double_as_longlong(QR_SQ_MAX))) break;
    const double f = tiny ? QR_SHIFT : 1.0 / QR_SHIFT;
    back = 1.0 / f;
    for (int c = tid >> 5; c < n; c += QR_THREADS / 32)
      for (int i = tid & 31; i < ml; i += 32) A[c * lda + i] = cscale(A[c * lda + i], f);
    __syncthreads();
  }

  int nq = 0;
  for (int j = 0; j < n && nq < kmax; ++j) {
    double2* v = A + (size_t)j * lda;
    if (again[j]) {
      // once more against the accepted columns
      for (int c0 = 0; c0 < nq; c0 += NB) {
        const int cnt = min(NB, nq - c0);
        // conj(v) . q is the conjugate of q^H v
        products(v, c0, cnt, false);
        for (int k = tid; k < cnt; k += QR_THREADS) {
          const double2 d = cconj(total(k));
          fac[k] = cscale(d, 1.0 / piv[c0 + k]);
          if (rank == 0) {
            double2* rr = t.V + (size_t)j * n + c0 + k;
            *rr = cadd(*rr, d);
          }
        }
        __syncthreads();
        // v -= sum_k q_k fac_k: `seg` threads per row, then their partial sums
        const int seg = ml > 0 ? max(1, min(32, QR_THREADS / ml)) : 1;
        const int rows = QR_THREADS / seg;
        for (int i0 = 0; i0 < ml; i0 += rows) {
          const int i = i0 + tid % rows, sg = tid / rows;
          double2 acc = make_double2(0.0, 0.0);
          if (i < ml && sg < seg)
            for (int k = sg; k < cnt; k += seg) acc = cfma(fac[k], A[(size_t)(c0 + k) * lda + i], acc);
          pp[tid] = acc;
          __syncthreads();
          if (tid < rows && i < ml) {
            for (int s = 1; s < seg; ++s) acc = cadd(acc, pp[s * rows + tid]);
            v[i] = csub(v[i], acc);
          }
          __syncthreads();
        }
      }
    }
    double inv = 0.0;
    bool keep = false;
    for (int c0 = j; c0 < n; c0 += NB) {
      const int cnt = min(NB, n - c0);
      products(v, c0, cnt, false);
      // only the threads that form the factors of this batch touch the FP64 pipe
      if (tid < cnt) {
        bool ok = true;
        if (c0 == j) {
          const double pj = total(0).x;
          ok = pj > 1e-24 * __longlong_as_double(big);
          if (ok) inv = 1.0 / pj;
          if (tid == 0) {
            keep_sh = ok;
            piv[nq] = pj;
          }
        }
        for (int k = tid; ok && k < cnt; k += QR_THREADS) {
          const double2 p = total(k);
          const double2 f = cscale(p, inv);
          fac[k] = f;
          const double left = est[c0 + k] - (p.x * f.x + p.y * f.y);
          est[c0 + k] = left;
          again[c0 + k] = left < 0.5 * orig[c0 + k];
          if (rank == 0) t.V[(size_t)(c0 + k) * n + nq] = p;   // scaled by 1 / |v| at the end
        }
      }
      __syncthreads();
      keep = keep_sh != 0;
      if (!keep) break;
      // a_c -= v f_c
      const int k1 = c0 == j ? 1 : 0;
      const int w = cnt - k1;
      const int lpc = w * 8 <= QR_THREADS ? 8 : w * 4 <= QR_THREADS ? 4 : w * 2 <= QR_THREADS ? 2 : 1;
      const int sub = tid & (lpc - 1);
      for (int k = k1 + tid / lpc; k < cnt; k += QR_THREADS / lpc) {
        const double2 f = make_double2(-fac[k].x, -fac[k].y);
        double2* y = A + (size_t)(c0 + k) * lda;
        for (int i = sub; i < ml; i += lpc) y[i] = cfma(f, v[i], y[i]);
      }
      __syncthreads();
    }
    if (keep) {
      if (nq != j) {
        for (int i = tid; i < ml; i += QR_THREADS) A[(size_t)nq * lda + i] = v[i];
        __syncthreads();
      }
      ++nq;
    }
  }
  __syncthreads();
  // 1 / |v| of the accepted columns, once
  for (int q = tid; q < nq; q += QR_THREADS) est[q] = 1.0 / sqrt(piv[q]);
  __syncthreads();
  for (int c = tid >> 5; c < kmax; c += QR_THREADS / 32)
    for (int i = tid & 31; i < ml; i += 32)
      t.A[(size_t)c * m + row0 + i] = c < nq ? cscale(A[c * lda + i], est[c]) : make_double2(0.0, 0.0);
  if (rank == 0)
    for (int e = tid; e < n * n; e += QR_THREADS) {
      const int q = e % n;
      if (q < nq) t.V[e] = cscale(cscale(t.V[e], est[q]), back);
    }
  // no CTA may leave while others can still write into its slots
  if (CS > 1) cl.sync();
}

void launch_qr(const FactTask* d_tasks, int ntasks, cudaStream_t st, const FactTask* h_tasks) {
  if (ntasks <= 0) return;
  // A cluster per matrix when one of them is too much for one SM's FP64 pipe
  // (4 m n^2 multiply-adds at 1.7 per clock), else a CTA per matrix, which
  // saves the cluster barrier of every column.  The shared memory asked for
  // is what the largest matrix needs; one that does not fit stays in global
  // memory.
  bool large = false;
  for (int i = 0; i < ntasks; ++i)
    if ((double)h_tasks[i].m * h_tasks[i].n * h_tasks[i].n >= QR_CLUSTER_WORK) large = true;
  const int cs = large ? QR_CS : 1;
  const size_t cap = QR_SMEM / sizeof(double2);
  size_t need = 0;
  bool fits = true;
  for (int i = 0; i < ntasks; ++i) {
    const int m = h_tasks[i].m, n = h_tasks[i].n;
    const size_t e = qr_fixed(n, cs, QR_BATCH) + (size_t)qr_mc(m, cs) * n;
    if (e > cap) fits = false;
    need = std::max(need, std::min(e, cap));
  }
  const int batch = fits ? QR_BATCH : QR_BATCH_GLOBAL;
  if (!fits) need = cap;
  if (!large) {
    set_smem_limit((const void*)k_qr<1>, QR_SMEM);
    k_qr<1><<<ntasks, QR_THREADS, need * sizeof(double2), st>>>(d_tasks, batch, (int)need);
    return;
  }
  set_smem_limit((const void*)k_qr<QR_CS>, QR_SMEM);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(ntasks * QR_CS));
  cfg.blockDim = dim3(QR_THREADS);
  cfg.dynamicSmemBytes = need * sizeof(double2);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = QR_CS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_qr<QR_CS>, d_tasks, batch, (int)need);
}


// ------------------------------------------------------------------ truncation rule

// Singular values of all sectors of one bond (each sector descending, sector
// ids ascending): sort descending with ties by position; drop values <=
// 1e-12 * max; keep at most D and the fewest whose discarded weight is <= eps
// of the total; move a cut inside a cluster (gaps <= 1e-10 * max) down to the
// cluster edge (up if the cluster starts at the top).
__global__ void k_trunc(const double* __restrict__ s, const int* __restrict__ sec, int nv,
                        int nsec, int D, double eps, int* kept, double* w, double* sorted,
                        int* sorted_sec) {
  for (int i = threadIdx.x; i < nv; i += blockDim.x) {
    double si = s[i];
    int rank = 0;
    for (int j = 0; j < nv; ++j) {
      double sj = s[j];
      rank += (sj > si) || (sj == si && j < i);
    }
    sorted[rank] = si;
    sorted_sec[rank] = sec[i];
  }
  for (int i = threadIdx.x; i < nsec; i += blockDim.x) kept[i] = 0;
  __syncthreads();
  if (threadIdx.x == 0) {
    double total = 0.0;
    for (int i = nv - 1; i >= 0; --i) total += sorted[i] * sorted[i];
    int k = 0;
    double disc = total;
    if (nv > 0 && sorted[0] > 0.0) {
      const double smax = sorted[0];
      int nz = 0;
      while (nz < nv && sorted[nz] > 1e-12 * smax) ++nz;
      // tail[j] = sum_{i >= j} sorted[i]^2
      k = nz;
      double tail = 0.0;
      for (int i = nv - 1; i >= nz; --i) tail += sorted[i] * sorted[i];
      // try dropping index k-1 while allowed
      while (k > 1) {
        double t2 = tail + sorted[k - 1] * sorted[k - 1];
        if (t2 <= eps * total) { tail = t2; --k; } else break;
      }
      if (k > D) k = D;
      if (k < nz) {
        int j = k;
        while (j > 0 && sorted[j - 1] - sorted[j] <= 1e-10 * smax) --j;
        if (j > 0) k = j;
        else
          while (k < nz && sorted[k - 1] - sorted[k] <= 1e-10 * smax) ++k;
      }
      disc = 0.0;
      for (int i = nv - 1; i >= k; --i) disc += sorted[i] * sorted[i];
      for (int i = 0; i < k; ++i) kept[sorted_sec[i]] += 1;
    }
    w[0] = disc;
    w[1] = total;
  }
}

void launch_trunc(const double* d_s, const int* d_sec, int nv, int nsec, int D, double eps,
                  int* d_kept, double* d_w, double* d_sorted, int* d_sorted_sec, cudaStream_t st) {
  k_trunc<<<1, 1024, 0, st>>>(d_s, d_sec, nv, nsec, D, eps, d_kept, d_w, d_sorted, d_sorted_sec);
}

// ------------------------------------------------------------------ Krylov algebra

constexpr int KMAX = 16;

// Cyclic Jacobi eigen-decomposition of a Hermitian n x n matrix (row-major,
// in place); eigenvectors in columns of V.
__device__ void herm_eig(double2* A, double2* V, double* w, int n) {
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j) V[i * n + j] = make_double2(i == j ? 1.0 : 0.0, 0.0);
  for (int sweep = 0; sweep < 60; ++sweep) {
    double off = 0.0, tot = 0.0;
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j) {
        tot += cabs2(A[i * n + j]);
        if (i != j) off += cabs2(A[i * n + j]);
      }
    if (off <= 1e-30 * tot || off == 0.0) break;
    for (int p = 0; p < n - 1; ++p)
      for (int q = p + 1; q < n; ++q) {
        double2 apq = A[p * n + q];
        double g = sqrt(cabs2(apq));
        if (g == 0.0) continue;
        double a = A[p * n + p].x, b = A[q * n + q].x;
        double2 ph = make_double2(apq.x / g, apq.y / g);   // e^{i phi}
        double zeta = (b - a) / (2.0 * g);
        double tt = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
        double c = 1.0 / sqrt(1.0 + tt * tt), s = c * tt;
        // J = [[c, s],[ -s e^{-i phi}, c e^{-i phi}]] on (p, q); A <- J^H A J, V <- V J
        double2 phc = cconj(ph);
        for (int k = 0; k < n; ++k) {   // columns: A J
          double2 x = A[k * n + p], y = A[k * n + q];
          A[k * n + p] = csub(cscale(x, c), cmul(cscale(phc, s), y));
          A[k * n + q] = cadd(cscale(x, s), cmul(cscale(phc, c), y));
          double2 vx = V[k * n + p], vy = V[k * n + q];
          V[k * n + p] = csub(cscale(vx, c), cmul(cscale(phc, s), vy));
          V[k * n + q] = cadd(cscale(vx, s), cmul(cscale(phc, c), vy));
        }
        for (int k = 0; k < n; ++k) {   // rows: J^H (A J)
          double2 x = A[p * n + k], y = A[q * n + k];
          A[p * n + k] = csub(cscale(x, c), cmul(cscale(ph, s), y));
          A[q * n + k] = cadd(cscale(x, s), cmul(cscale(ph, c), y));
        }
        A[p * n + q] = make_double2(0.0, 0.0);
        A[q * n + p] = make_double2(0.0, 0.0);
      }
  }
  for (int i = 0; i < n; ++i) w[i] = A[i * n + i].x;
}

__global__ void k_krylov_small(const double2* Nm, const double2* Hm, int m, double dt,
                               double2* c, int* status) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double2 A[KMAX * KMAX], V[KMAX * KMAX], X[KMAX * KMAX], M[KMAX * KMAX], U[KMAX * KMAX];
  double w[KMAX], lam[KMAX];
  int bad = 0;
  for (int i = 0; i < m * m; ++i) {
    if (!isfinite(Nm[i].x) || !isfinite(Nm[i].y) || !isfinite(Hm[i].x) || !isfinite(Hm[i].y)) bad = 1;
  }
  // N and H arrive with their upper triangles (i <= j) filled; complete them
  // as Hermitian matrices
  double2 Nf[KMAX * KMAX], Hf[KMAX * KMAX];
  for (int i = 0; i < m; ++i)
    for (int j = 0; j < m; ++j) {
      double2 n = i <= j ? Nm[i * m + j] : cconj(Nm[j * m + i]);
      double2 h = i <= j ? Hm[i * m + j] : cconj(Hm[j * m + i]);
      if (i == j) { n.y = 0.0; h.y = 0.0; }
      Nf[i * m + j] = n;
      Hf[i * m + j] = h;
      A[i * m + j] = n;
    }
  herm_eig(A, V, w, m);
  double wmax = 0.0;
  for (int i = 0; i < m; ++i) wmax = fmax(wmax, w[i]);
  int r = 0;
  for (int k = 0; k < m; ++k)
    if (w[k] > 1e-12 * wmax) {
      double inv = 1.0 / sqrt(w[k]);
      for (int i = 0; i < m; ++i) X[i * KMAX + r] = cscale(V[i * m + k], inv);
      ++r;
    }
  // M = X^H H X  (r x r)
  for (int a = 0; a < r; ++a)
    for (int b = 0; b < r; ++b) {
      double2 acc = make_double2(0.0, 0.0);
      for (int i = 0; i < m; ++i)
        for (int j = 0; j < m; ++j) {
          acc = cadd(acc, cmul(cmul(cconj(X[i * KMAX + a]), Hf[i * m + j]), X[j * KMAX + b]));
        }
      M[a * r + b] = acc;
    }
  if (r > 0) herm_eig(M, U, lam, r);
  // b = X^H N e0
  double2 bvec[KMAX], tmp[KMAX];
  for (int a = 0; a < r; ++a) {
    double2 acc = make_double2(0.0, 0.0);
    for (int i = 0; i < m; ++i) acc = cadd(acc, cmul(cconj(X[i * KMAX + a]), Nf[i * m + 0]));
    bvec[a] = acc;
  }
  for (int a = 0; a < r; ++a) {   // tmp = exp(-i dt lam) U^H b
    double2 acc = make_double2(0.0, 0.0);
    for (int b2 = 0; b2 < r; ++b2) acc = cadd(acc, cmul(cconj(U[b2 * r + a]), bvec[b2]));
    double ph = -dt * lam[a];
    tmp[a] = cmul(make_double2(cos(ph), sin(ph)), acc);
  }
  for (int i = 0; i < m; ++i) {
    double2 acc = make_double2(0.0, 0.0);
    for (int a = 0; a < r; ++a) {
      double2 ua = make_double2(0.0, 0.0);
      for (int b2 = 0; b2 < r; ++b2) ua = cadd(ua, cmul(U[a * r + b2], tmp[b2]));
      acc = cadd(acc, cmul(X[i * KMAX + a], ua));
    }
    c[i] = acc;
    if (!isfinite(acc.x) || !isfinite(acc.y)) bad = 1;
  }
  status[0] = m - r;
  status[1] = bad;
}

void launch_krylov_small(const double2* d_N, const double2* d_H, int m, double dt, double2* d_c,
                         int* d_status, cudaStream_t st) {
  k_krylov_small<<<1, 32, 0, st>>>(d_N, d_H, m, dt, d_c, d_status);
}

// ------------------------------------------------------------------ scalar helpers

__global__ void k_scalar_div_neg(const double2* num, const double2* den, double2* out) {
  double2 q = cdiv(*num, *den);
  *out = make_double2(-q.x, -q.y);
}

void launch_scalar_div_neg(const double2* num, const double2* den, double2* out, cudaStream_t st) {
  k_scalar_div_neg<<<1, 1, 0, st>>>(num, den, out);
}

__global__ void k_normalize(double2* x, size_t n, double2* norm_out) {
  __shared__ double part[32];
  double s2 = 0.0;
  for (size_t i = threadIdx.x; i < n; i += blockDim.x) s2 += cabs2(x[i]);
  s2 = warp_sum(s2);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s2;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.0;
    v = warp_sum(v);
    if (threadIdx.x == 0) part[0] = v;
  }
  __syncthreads();
  double nrm = sqrt(part[0]);
  double inv = nrm > 0.0 ? 1.0 / nrm : 0.0;
  for (size_t i = threadIdx.x; i < n; i += blockDim.x) x[i] = cscale(x[i], inv);
  if (threadIdx.x == 0 && norm_out) *norm_out = make_double2(nrm, 0.0);
}

void launch_normalize(double2* x, size_t n, double2* d_norm_out, cudaStream_t st) {
  k_normalize<<<1, 1024, 0, st>>>(x, n, d_norm_out);
}

// out[w] += sum_{a, b} E[a][w][b] * R[a][b]   (rows x nch x cols and rows x cols)
template <class T>
__global__ void k_trace_channels(const T* E, int rows, int nch, int cols, const T* R,
                                 double2* out) {
  const int w = blockIdx.x;
  double re = 0.0, im = 0.0;
  for (int e = threadIdx.x; e < rows * cols; e += blockDim.x) {
    int a = e / cols, b = e % cols;
    double2 v = cmul(ld2(E, ((size_t)a * nch + w) * cols + b), ld2(R, (size_t)a * cols + b));
    re += v.x;
    im += v.y;
  }
  __shared__ double pr[32], pi[32];
  re = warp_sum(re);
  im = warp_sum(im);
  if ((threadIdx.x & 31) == 0) { pr[threadIdx.x >> 5] = re; pi[threadIdx.x >> 5] = im; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double sr = 0.0, si = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) { sr += pr[k]; si += pi[k]; }
    out[w] = cadd(out[w], make_double2(sr, si));
  }
}

void launch_trace_channels(const void* E, int rows, int nch, int cols, const void* R, int et,
                           double2* out, cudaStream_t st) {
  if (nch <= 0 || rows * cols == 0) return;
  if (et == 0)
    k_trace_channels<double2><<<nch, 256, 0, st>>>((const double2*)E, rows, nch, cols, (const double2*)R, out);
  else
    k_trace_channels<float2><<<nch, 256, 0, st>>>((const float2*)E, rows, nch, cols, (const float2*)R, out);
}

}  // namespace tdmps
