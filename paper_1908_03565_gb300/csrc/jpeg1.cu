// JPEG1 direct rasterisation (M.6): dequantisation and IDCT per 8x8 block,
// block-conditional Gaborish, 2x linear chroma upsampling and YCbCr -> RGB.
//
//  k_jpeg_cond_rows / k_jpeg_cond_cols  M.6.1.1 plateau scans, one thread
//               per block row / column.
//  k_jpeg_idct  sample planes of the components that need one (subsampled, or
//               with the M.6.3 side channel), all in one launch: 128 threads =
//               16 blocks x 8 rows.  A thread loads one coefficient row (8 x
//               int16, one 128-bit load), dequantises it with the prescaled
//               table and transforms it; the block's transpose goes through
//               shared memory within the warp (a block's 8 rows are 8 lanes of
//               one warp), then the column transform and the row store.
//  k_jpeg_gab   one 8x8 block per 64-thread CTA: J.4 on the plane (mirrored
//               at its bounds), the M.6.3 count by __syncthreads_count, and
//               the block's smoothed or original samples.
//  k_jpeg_out   one row of an 8x8 block of the image per thread: the samples of
//               full-resolution components straight from their coefficients
//               (the transform of k_jpeg_idct, without a plane in between), of
//               the others from their planes with M.6.4 (separable linear,
//               weights 3/4 and 1/4), then M.6.5 and the output encoding, 8
//               pixels stored as 8- or 16-byte words where rows allow it.
//
//               k_jpeg_out_420 is the same for the usual 4:2:0 stream.
//
// Bound by the latency of the loads and by instruction issue (50% busy), not
// by bandwidth: a 4:2:0 stream reads 2 bytes per sample, keeps its chroma
// planes (8 bytes per 4 pixels) in L2 and writes 3 bytes per pixel.  Measured
// at 4096^2, 4:2:0, u8 (whole request): 0.196 ms with a plane for every
// component and one thread per output pixel, 0.108 with luma straight from
// its coefficients and 8 pixels per thread (k_jpeg_out), 0.100 with the loads
// of k_jpeg_out_420 a block row ahead.  The dequantisation table is read from
// shared memory: indexed by the lane's row in constant memory, each of its
// reads was replayed for 8 rows.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstring>

#include "jpeg1.h"

namespace jxlr {

namespace {

// cos((2n+1) (2j+1) pi / 16), n, j < 4, and cos((2n+1) (2j+1) pi / 8), n, j < 2:
// the odd parts of the unscaled 8- and 4-point inverse DCT.
__constant__ float c_jodd8[16];
__constant__ float c_jodd4[4];
__constant__ float c_jodd2;   // cos(pi / 4)

// Unscaled 8-point inverse DCT: x_n = sum_k c_k cos((2n+1) k pi / 16).
__device__ __forceinline__ void idct8(float (&x)[8]) {
  // even part: 4-point on c0, c2, c4, c6
  const float e0 = x[0] + x[4] * c_jodd2, e1 = x[0] - x[4] * c_jodd2;
  const float o0 = x[2] * c_jodd4[0] + x[6] * c_jodd4[1];
  const float o1 = x[2] * c_jodd4[2] + x[6] * c_jodd4[3];
  const float ev[4] = {e0 + o0, e1 + o1, e1 - o1, e0 - o0};
  float od[4];
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) s = fmaf(x[2 * j + 1], c_jodd8[n * 4 + j], s);
    od[n] = s;
  }
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    x[n] = ev[n] + od[n];
    x[7 - n] = ev[n] - od[n];
  }
}

// M.6.1.1 along one line of n blocks (rows: step 1 block; columns: step bw
// blocks), in binary32, operation by operation (the comparisons decide which
// coefficients are replaced).  acx: index of the AC coefficient of the scan
// direction (1 horizontal, 8 vertical).
__device__ void cond_line(const int16_t* coef, int first, int stride, int n, int acx, float q,
                          float max_gap, float min_step, float* approx, float* slope,
                          uint8_t* has) {
  auto dc = [&](int i) { return static_cast<int>(coef[static_cast<size_t>(first + i * stride) * 64]); };
  auto ac = [&](int i) { return static_cast<int>(coef[static_cast<size_t>(first + i * stride) * 64 + acx]); };
  int x = 0;
  while (x < n) {
    const int d = dc(x);
    int end = x;
    bool zero = ac(x) == 0;
    while (end + 1 < n && dc(end + 1) == d) {
      ++end;
      zero = zero && ac(end) == 0;
    }
    const int start = x;
    x = end + 1;
    bool sane = false;
    float frm = 0.f, to = 0.f;
    if (zero && !(start == 0 && end == n - 1)) {
      const float cur = static_cast<float>(d);
      frm = start == 0 ? cur
                       : 0.5f * __fadd_rn(__fadd_rn(cur, static_cast<float>(dc(start - 1))),
                                          __fmul_rn(q, static_cast<float>(ac(start - 1))));
      to = end == n - 1 ? cur
                        : 0.5f * __fadd_rn(__fadd_rn(cur, static_cast<float>(dc(end + 1))),
                                           __fmul_rn(q, static_cast<float>(ac(end + 1))));
      sane = fabsf(__fsub_rn(to, cur)) <= max_gap && fabsf(__fsub_rn(cur, frm)) <= max_gap &&
             fabsf(__fsub_rn(to, frm)) > min_step;
    }
    const float ratio = sane ? __fdiv_rn(__fsub_rn(to, frm), static_cast<float>(end - start + 1)) : 0.f;
    for (int i = start; i <= end; ++i) {
      const size_t o = static_cast<size_t>(first + i * stride);
      has[o] = sane ? 1 : 0;
      approx[o] = sane ? __fadd_rn(frm, __fmul_rn(__fadd_rn(0.5f, static_cast<float>(i - start)), ratio)) : 0.f;
      slope[o] = sane ? -0.5f * ratio : 0.f;
    }
  }
}

__global__ void __launch_bounds__(128) k_jpeg_cond_rows(const __grid_constant__ JpegCondArgs a) {
  const int y = blockIdx.x * blockDim.x + threadIdx.x;
  if (y >= a.bh) return;
  cond_line(a.coef, y * a.bw, 1, a.bw, 1, a.q_h, a.max_gap, a.min_step, a.out.h_approx,
            a.out.h_slope, a.out.has_h);
}

__global__ void __launch_bounds__(128) k_jpeg_cond_cols(const __grid_constant__ JpegCondArgs a) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= a.bw) return;
  cond_line(a.coef, x, a.bw, a.bh, 8, a.q_v, a.max_gap, a.min_step, a.out.v_approx,
            a.out.v_slope, a.out.has_v);
}

// Row r (0..7) of the samples of block blk, in x, by the 8 threads of one warp
// that hold the block's rows; on: the block exists (else zeros take part).  dq:
// the component's prescaled table in shared memory; T: the block's scratch
// (kBlockScratch floats, rows of 12: 16-byte row accesses and the column
// accesses of a warp's 4 blocks without bank conflicts); raw: the coefficients
// of row r.
constexpr int kBlockScratch = 8 * 12 + 8;
__device__ __forceinline__ int4 load_row(const JpegIdctArgs& a, int blk, int r, bool on) {
  return on ? __ldg(reinterpret_cast<const int4*>(a.coef + static_cast<size_t>(blk) * 64 + 8 * r))
            : make_int4(0, 0, 0, 0);
}
__device__ __forceinline__ void block_row(const JpegIdctArgs& a, const float* dq, float* T,
                                          const int4& raw, int blk, int r, bool on, float (&x)[8]) {
  if (on) {
    const int16_t* h = reinterpret_cast<const int16_t*>(&raw);
    const float4 d0 = *reinterpret_cast<const float4*>(dq + 8 * r);
    const float4 d1 = *reinterpret_cast<const float4*>(dq + 8 * r + 4);
    const float d[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = static_cast<float>(h[j]) * d[j];
    if (a.cond && r < 2) {   // M.6.1.1: coefficients 0 and 1 (row 0), 8 (row 1)
      const bool hh = a.c.has_h[blk] != 0, vh = a.c.has_v[blk] != 0;
      if (r == 0) {
        float dcv = static_cast<float>(h[0]);
        if (hh && vh) dcv = 0.5f * __fadd_rn(a.c.h_approx[blk], a.c.v_approx[blk]);
        else if (hh) dcv = a.c.h_approx[blk];
        else if (vh) dcv = a.c.v_approx[blk];
        x[0] = dcv * a.m0;
        if (hh) x[1] = a.c.h_slope[blk] * a.m1;
      } else if (vh) {
        x[0] = a.c.v_slope[blk] * a.m1;
      }
    }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = 0.f;
  }
  // row r holds the coefficients of vertical frequency r: transform along
  // the horizontal frequencies first
  idct8(x);
  float4* row = reinterpret_cast<float4*>(T + 12 * r);
  row[0] = make_float4(x[0], x[1], x[2], x[3]);
  row[1] = make_float4(x[4], x[5], x[6], x[7]);
  __syncwarp();
  // column r: the vertical transform of horizontal position r
#pragma unroll
  for (int j = 0; j < 8; ++j) x[j] = T[12 * j + r];
  idct8(x);
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 8; ++j) T[12 * j + r] = x[j];
  __syncwarp();
  const float4 lo = row[0], hi = row[1];
  x[0] = lo.x; x[1] = lo.y; x[2] = lo.z; x[3] = lo.w;
  x[4] = hi.x; x[5] = hi.y; x[6] = hi.z; x[7] = hi.w;
  __syncwarp();   // the caller may transform another component's block
}

struct JpegIdctSet {
  JpegIdctArgs c[3];
};

__global__ void __launch_bounds__(128) k_jpeg_idct(const __grid_constant__ JpegIdctSet set) {
  const JpegIdctArgs& a = set.c[blockIdx.y];
  __shared__ __align__(16) float sT[16][kBlockScratch];
  __shared__ __align__(16) float s_dq[64];
  const int tid = threadIdx.x;
  const int lb = tid >> 3, r = tid & 7;
  const int blk = blockIdx.x * 16 + lb;
  const int nblk = a.bw * a.bh;
  if (blockIdx.x * 16 >= nblk) return;
  if (tid < 64) s_dq[tid] = a.dq[tid];
  __syncthreads();
  float x[8];
  block_row(a, s_dq, sT[lb], load_row(a, blk, r, blk < nblk), blk, r, blk < nblk, x);
  if (blk < nblk) {
    const int by = blk / a.bw, bx = blk - by * a.bw;
    float* dst = a.plane + static_cast<size_t>(8 * by + r) * (8 * a.bw) + 8 * bx;
    reinterpret_cast<float4*>(dst)[0] = make_float4(x[0], x[1], x[2], x[3]);
    reinterpret_cast<float4*>(dst)[1] = make_float4(x[4], x[5], x[6], x[7]);
  }
}

__device__ __forceinline__ int mirror_plane(int c, int n) {
  // 6.5, for coordinates at most one step outside [0, n)
  return c < 0 ? -c - 1 : c >= n ? 2 * n - 1 - c : c;
}

__global__ void __launch_bounds__(64) k_jpeg_gab(const __grid_constant__ JpegGabArgs a) {
  const int bx = blockIdx.x, by = blockIdx.y;
  const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
  const int w = 8 * a.bw, h = 8 * a.bh;
  const int x = 8 * bx + tx, y = 8 * by + ty;
  float acc_c = 0.f, acc_e = 0.f, acc_d = 0.f;
#pragma unroll
  for (int dy = -1; dy <= 1; ++dy) {
    const float* row = a.src + static_cast<size_t>(mirror_plane(y + dy, h)) * w;
#pragma unroll
    for (int dx = -1; dx <= 1; ++dx) {
      const float v = __ldg(row + mirror_plane(x + dx, w));
      if (dx == 0 && dy == 0) acc_c += v;
      else if (dx == 0 || dy == 0) acc_e += v;
      else acc_d += v;
    }
  }
  const float s = fmaf(a.w2n, acc_d, fmaf(a.w1n, acc_e, a.w0n * acc_c));
  const float p = a.src[static_cast<size_t>(y) * w + x];
  const bool inner = tx >= 1 && tx < 7 && ty >= 1 && ty < 7;
  const int count = __syncthreads_count(inner && fabsf(p - s) > a.threshold);
  a.dst[static_cast<size_t>(y) * w + x] = count < a.limit ? s : p;
}

// M.6.4 source index and weight of the second tap for output index o of a
// 2x upsampled axis of n samples: o = 2i -> (i, i-1), o = 2i+1 -> (i, i+1),
// index -1 reading 1 and index n reading n-2.
__device__ __forceinline__ void up_taps(int o, int n, int& i0, int& i1) {
  i0 = o >> 1;
  int j = (o & 1) ? i0 + 1 : i0 - 1;
  if (j < 0) j = -j;
  if (j >= n) j = 2 * n - 2 - j;
  i1 = min(max(j, 0), n - 1);
}

__device__ __forceinline__ float sample_up(const JpegPlane& p, int x, int y) {
  const float* s = p.data;
  if (!p.up_x && !p.up_y) return s[static_cast<size_t>(y) * p.w + x];
  int x0 = x, x1 = x, y0 = y, y1 = y;
  if (p.up_x) up_taps(x, p.w, x0, x1);
  if (p.up_y) up_taps(y, p.h, y0, y1);
  const float* r0 = s + static_cast<size_t>(y0) * p.w;
  const float* r1 = s + static_cast<size_t>(y1) * p.w;
  // horizontal first (M.6.4), then vertical
  const float h0 = p.up_x ? fmaf(0.75f, r0[x0], 0.25f * r0[x1]) : r0[x0];
  if (!p.up_y) return h0;
  const float h1 = p.up_x ? fmaf(0.75f, r1[x0], 0.25f * r1[x1]) : r1[x0];
  return fmaf(0.75f, h0, 0.25f * h1);
}

// The 8 samples of pixels x .. x + 7 (x a multiple of 8) of image row y from
// p's plane; columns at xs and beyond are not used (n of them are inside).
__device__ __forceinline__ void plane_row(const JpegPlane& p, int x, int y, int n, float (&v)[8]) {
  if (!p.up_x && !p.up_y) {
    const float4* s = reinterpret_cast<const float4*>(p.data + static_cast<size_t>(y) * p.w + x);
    const float4 a = __ldg(s), b = __ldg(s + 1);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    return;
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = j < n ? sample_up(p, x + j, y) : 0.f;
}

// M.6.5, M.6.6 and the output encoding of pixels x .. x + n - 1 (n <= 8) of row y.
__device__ __forceinline__ void color_row(const JpegOutArgs& a, int x, int y, int n,
                                          const float (&v)[3][8]) {
  float o[24];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float yv = v[0][j] + 128.f;
    if (a.ncomp == 1) {
      o[3 * j] = o[3 * j + 1] = o[3 * j + 2] = yv;
    } else {
      const float cb = v[1][j], cr = v[2][j];
      o[3 * j] = fmaf(1.402f, cr, yv);
      o[3 * j + 1] = fmaf(-0.71414f, cr, fmaf(-0.34414f, cb, yv));
      o[3 * j + 2] = fmaf(1.772f, cb, yv);
    }
  }
  char* row = static_cast<char*>(a.out) + static_cast<size_t>(y) * a.stride;
  if (a.dtype == 2) {   // u8: clamp, round half up (truncated by adding 2^23 toward zero)
    uint32_t w[24];
#pragma unroll
    for (int k = 0; k < 24; ++k)
      w[k] = __float_as_uint(__fadd_rz(fminf(fmaxf(o[k], 0.f), 255.f) + 0.5f, 8388608.f));
    uint8_t* p = reinterpret_cast<uint8_t*>(row) + 3 * x;
    if (n == 8 && (reinterpret_cast<uintptr_t>(p) & 7) == 0) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        uint32_t d[2];
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          const uint32_t* q = w + 8 * k + 4 * m;
          d[m] = __byte_perm(__byte_perm(q[0], q[1], 0x0040), __byte_perm(q[2], q[3], 0x0040), 0x5410);
        }
        reinterpret_cast<uint2*>(p)[k] = make_uint2(d[0], d[1]);
      }
    } else {
#pragma unroll
      for (int k = 0; k < 24; ++k)
        if (k < 3 * n) p[k] = static_cast<uint8_t>(w[k]);
    }
    return;
  }
#pragma unroll
  for (int k = 0; k < 24; ++k) o[k] *= 1.f / 255.f;
  if (a.dtype == 1) {
    __half* p = reinterpret_cast<__half*>(row) + 3 * x;
    if (n == 8 && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        uint32_t d[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const __half2 h = __floats2half2_rn(o[8 * k + 2 * m], o[8 * k + 2 * m + 1]);
          d[m] = *reinterpret_cast<const uint32_t*>(&h);
        }
        reinterpret_cast<uint4*>(p)[k] = make_uint4(d[0], d[1], d[2], d[3]);
      }
    } else {
#pragma unroll
      for (int k = 0; k < 24; ++k)
        if (k < 3 * n) p[k] = __float2half_rn(o[k]);
    }
  } else {
    float* p = reinterpret_cast<float*>(row) + 3 * x;
    if (n == 8 && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
#pragma unroll
      for (int k = 0; k < 24; k += 4)
        *reinterpret_cast<float4*>(p + k) = make_float4(o[k], o[k + 1], o[k + 2], o[k + 3]);
    } else {
#pragma unroll
      for (int k = 0; k < 24; ++k)
        if (k < 3 * n) p[k] = o[k];
    }
  }
}

__global__ void __launch_bounds__(128) k_jpeg_out(const __grid_constant__ JpegOutArgs a) {
  __shared__ __align__(16) float sT[16][kBlockScratch];
  __shared__ __align__(16) float s_dq[3][64];
  const int tid = threadIdx.x;
  const int lb = tid >> 3, r = tid & 7;
  for (int k = tid; k < 64 * a.ncomp; k += 128)
    if (a.direct[k >> 6]) s_dq[k >> 6][k & 63] = a.i[k >> 6].dq[k & 63];
  __syncthreads();
  const int bx = blockIdx.x * 16 + lb, x = 8 * bx, y = 8 * blockIdx.y + r;
  const bool in = x < a.xs;                    // the block has pixels (the same for its 8 rows)
  const int n = in && y < a.ys ? min(8, a.xs - x) : 0;
  float v[3][8];
  // all loads before the first transform
  int4 raw[3];
#pragma unroll
  for (int c = 0; c < 3; ++c)
    if (c < a.ncomp && a.direct[c]) raw[c] = load_row(a.i[c], blockIdx.y * a.i[c].bw + bx, r, in);
#pragma unroll
  for (int c = 0; c < 3; ++c)
    if (c < a.ncomp && !a.direct[c] && n > 0) plane_row(a.p[c], x, y, n, v[c]);
#pragma unroll
  for (int c = 0; c < 3; ++c)
    if (c < a.ncomp && a.direct[c])
      block_row(a.i[c], s_dq[c], sT[lb], raw[c], blockIdx.y * a.i[c].bw + bx, r, in, v[c]);
  if (n == 0) return;
  color_row(a, x, y, n, v);
}

// The usual form, 4:2:0 without the side channels of M.6.3: luma direct, both
// chroma components upsampled along both axes.  A CTA takes kRows420 block
// rows of 16 blocks, the next row's coefficients loaded before the current
// one's transform and the chroma samples before the luma transform.
constexpr int kRows420 = 4;
__global__ void __launch_bounds__(128) k_jpeg_out_420(const __grid_constant__ JpegOutArgs a) {
  __shared__ __align__(16) float sT[16][kBlockScratch];
  __shared__ __align__(16) float s_dq[64];
  const int tid = threadIdx.x;
  const int lb = tid >> 3, r = tid & 7;
  const int bx = blockIdx.x * 16 + lb, x = 8 * bx;
  const bool in = x < a.xs;
  int by = blockIdx.y * kRows420;
  const int by1 = min(by + kRows420, (a.ys + 7) >> 3);
  int4 next = load_row(a.i[0], by * a.i[0].bw + bx, r, in);
  if (tid < 64) s_dq[tid] = a.i[0].dq[tid];
  __syncthreads();
  // columns i0 - 1 .. i0 + 4 of the chroma planes, the outer ones mirrored (M.6.4)
  const int w = a.p[1].w, i0 = in ? x >> 1 : 0;
  const int left = i0 > 0 ? i0 - 1 : 1, right = i0 + 4 < w ? i0 + 4 : w - 2;
  for (; by < by1; ++by) {
    const int4 raw = next;
    const int y = 8 * by + r;
    const int n = in && y < a.ys ? min(8, a.xs - x) : 0;
    if (by + 1 < by1) next = load_row(a.i[0], (by + 1) * a.i[0].bw + bx, r, in);
    int y0 = 0, y1 = 0;
    if (n) up_taps(y, a.p[1].h, y0, y1);
    float ch[2][2][6];
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float* row = a.p[1 + c].data + static_cast<size_t>(k ? y1 : y0) * w;
        const float4 m = __ldg(reinterpret_cast<const float4*>(row + i0));
        ch[c][k][0] = __ldg(row + left);
        ch[c][k][1] = m.x; ch[c][k][2] = m.y; ch[c][k][3] = m.z; ch[c][k][4] = m.w;
        ch[c][k][5] = __ldg(row + right);
      }
    float v[3][8];
    block_row(a.i[0], s_dq, sT[lb], raw, by * a.i[0].bw + bx, r, in, v[0]);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      float h[2][8];
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          h[k][2 * j] = fmaf(0.75f, ch[c][k][j + 1], 0.25f * ch[c][k][j]);
          h[k][2 * j + 1] = fmaf(0.75f, ch[c][k][j + 1], 0.25f * ch[c][k][j + 2]);
        }
#pragma unroll
      for (int j = 0; j < 8; ++j) v[1 + c][j] = fmaf(0.75f, h[0][j], 0.25f * h[1][j]);
    }
    if (n) color_row(a, x, y, n, v);
  }
}

}  // namespace

bool upload_jpeg_constants(const float* odd8, const float* odd4, float odd2) {
  return cudaMemcpyToSymbol(c_jodd8, odd8, sizeof(float) * 16) == cudaSuccess &&
         cudaMemcpyToSymbol(c_jodd4, odd4, sizeof(float) * 4) == cudaSuccess &&
         cudaMemcpyToSymbol(c_jodd2, &odd2, sizeof(float)) == cudaSuccess;
}

void launch_jpeg_idct(const JpegIdctArgs* a, int n, cudaStream_t s) {
  JpegIdctSet set;
  std::memset(&set, 0, sizeof(set));
  int most = 1;
  for (int c = 0; c < n; ++c) {
    set.c[c] = a[c];
    const int nblk = a[c].bw * a[c].bh;
    most = nblk > most ? nblk : most;
  }
  k_jpeg_idct<<<dim3((most + 15) / 16, n), 128, 0, s>>>(set);
}

int launch_jpeg_cond(const JpegCondArgs& a, cudaStream_t s) {
  k_jpeg_cond_rows<<<(a.bh + 127) / 128, 128, 0, s>>>(a);
  k_jpeg_cond_cols<<<(a.bw + 127) / 128, 128, 0, s>>>(a);
  return 2;
}

void launch_jpeg_gab(const JpegGabArgs& a, cudaStream_t s) {
  k_jpeg_gab<<<dim3(a.bw, a.bh), 64, 0, s>>>(a);
}

void launch_jpeg_out(const JpegOutArgs& a, cudaStream_t s) {
  const auto both = [&](int c) { return !a.direct[c] && a.p[c].up_x && a.p[c].up_y; };
  const int rows = (a.ys + 7) / 8;
  if (a.ncomp == 3 && a.direct[0] && both(1) && both(2) && a.p[1].w == a.p[2].w &&
      a.p[1].h == a.p[2].h)
    k_jpeg_out_420<<<dim3((a.xs + 127) / 128, (rows + kRows420 - 1) / kRows420), 128, 0, s>>>(a);
  else
    k_jpeg_out<<<dim3((a.xs + 127) / 128, rows), 128, 0, s>>>(a);
}

}  // namespace jxlr
