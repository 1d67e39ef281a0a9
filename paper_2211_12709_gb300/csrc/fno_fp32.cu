// fno_fp32.cu -- the FP32 CUDA-core form of every stage of the spectral FNO
// block (the "plain form"), plus the table, reduction and fill kernels that
// every precision shares.
//
// Stage map (Alg. 2, Sec. IV-C of the paper; the forward truncated DFT runs
// over the non-partitioned axes y, z, t first and over x last, the inverse is
// the same chain in reverse order):
//   k_fwd_tz_f32   pruned DFT over t then z of each (b, c, x, y) column, a warp each
//   k_fwd_tz_cta_f32  the same with a CTA a column
//   k_line_f32     one complex DFT axis (forward y, x; inverse x, y)
//   k_mix_f32      per-mode complex channel mixing (the einsum of Alg. 2)
//   k_mix_adj_f32  its adjoint: weight gradient and input-spectrum gradient
//   k_epi_f32      inverse z then t, fused with the 1x1 linear, bias and GELU
//                  (or their gradients)
#include <cuda_bf16.h>

#include <algorithm>

#include "fno_internal.h"

namespace fno {


static int persistent_grid(const void* kern, int threads, size_t smem, int64_t work) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  int64_t g = (int64_t)per_sm * sm_count();
  if (g > work) g = work;
  if (g < 1) g = 1;
  return (int)g;
}

// ---------------------------------------------------------------------------
// Basis tables: exp(sign * 2 pi i * (k n mod N) / N), evaluated in FP64 with
// sincospi on the exactly reduced residue, optionally scaled by c(kt)/Ng.
// ---------------------------------------------------------------------------
struct TabSeg {
  float2* dst;
  int rows, cols, N, m, k_on_row, sign, scale;
};
struct TabParams {
  TabSeg seg[10];
  long long start[11];
  int nseg;
  int Nt;
  double invNg;
  int* err;
  EpiTables et;
  int Nz, mz, Jt;
  long long ncz, nct;  // threads of the epilogue's z and t fragments (0: none)
};

// FP32 value of sc exp(+2 pi i k n / N)
__device__ float2 root_of_unity(long long k, long long n, long long N, double sc) {
  long long rr = (k * n) % N;
  if (rr < 0) rr += N;
  double sn, cs;
  sincospi(2.0 * (double)rr / (double)N, &sn, &cs);
  return make_float2((float)(cs * sc), (float)(sn * sc));
}

// three exact BF16 parts of two floats
__device__ void three_parts(float a, float b, uint32_t (&p)[3]) {
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    const float2 f = __bfloat1622float2(h);
    p[q] = *reinterpret_cast<const uint32_t*>(&h);
    a -= f.x;
    b -= f.y;
  }
}

// Fragments of the epilogue's bases (see EpiTables): thread e < ncz one lane of
// one (16-plane tile, k-step) of the z basis, the others one lane of one
// 8-point t sub-tile (rows (kt, cos), then (kt, -sin)).
__device__ void epi_fragments(const TabParams& p, long long e) {
  const EpiTables& c = p.et;
  const int lane = (int)(e % 32), g = lane / 4, q = lane % 4;
  e /= 32;
  uint32_t w[4][3];
  if (e < p.ncz / 32) {
    const int ks = (int)(e % c.KS), zt = (int)(e / c.KS);
#pragma unroll 1
    for (int r = 0; r < 4; ++r) {
      const int z = 16 * zt + g + 8 * (r & 1), jz = 8 * ks + q + 4 * (r >> 1);
      float2 f = make_float2(0.f, 0.f);
      if (z < p.Nz && jz < 2 * p.mz) f = root_of_unity(jz < p.mz ? jz : jz - 2 * p.mz, z, p.Nz, 1.0);
      three_parts(f.x, -f.y, w[r]);
    }
    for (int k = 0; k < 3; ++k) c.zf[(e * 3 + k) * 32 + lane] = make_uint4(w[0][k], w[1][k], w[2][k], w[3][k]);
    return;
  }
  e -= p.ncz / 32;
  const bool scaled = e < 2 * c.NTT;
  if (!scaled) e -= 2 * c.NTT;
  const int h = (int)(e % 2), T = (int)(e / 2);
  const int t = 16 * T + (c.perm ? 4 * (g / 2) + 2 * h + g % 2 : 8 * h + g);
  float cv[2], sv[2];
#pragma unroll 1
  for (int u = 0; u < 2; ++u) {
    const int kt = 2 * q + u;
    const bool single = kt == 0 || (p.Nt % 2 == 0 && 2 * kt == p.Nt);
    const double sc = scaled ? (single ? 1.0 : 2.0) * p.invNg : 1.0;
    float2 f = make_float2(0.f, 0.f);
    if (t < p.Nt && kt < p.Jt) f = root_of_unity(kt, t, p.Nt, sc);
    cv[u] = f.x;
    sv[u] = -f.y;
  }
  three_parts(cv[0], cv[1], w[0]);
  three_parts(sv[0], sv[1], w[1]);
  uint2* dst = scaled ? c.tfs : c.tfu;
  for (int k = 0; k < 3; ++k) dst[(e * 3 + k) * 32 + lane] = make_uint2(w[0][k], w[1][k]);
}

EpiTables epi_tables(const Dims& d, void* base) {
  EpiTables c{};
  c.NZ = (int)((d.Nz + 15) / 16);
  c.KS = (int)((d.Jz + 7) / 8);
  c.NTT = (int)((d.Nt + 15) / 16);
  c.H = d.Nt > 16 ? 2 : 1;
  c.perm = (c.H == 2 && d.Nt % 4 == 0) ? 1 : 0;
  c.zf = static_cast<uint4*>(base);
  c.tfs = reinterpret_cast<uint2*>(c.zf + (size_t)c.NZ * c.KS * 3 * 32);
  c.tfu = c.tfs + (size_t)c.NTT * 2 * 3 * 32;
  return c;
}
size_t epi_tables_bytes(const Dims& d) {
  const EpiTables c = epi_tables(d, nullptr);
  return sizeof(uint4) * (size_t)c.NZ * c.KS * 3 * 32 + 2 * sizeof(uint2) * (size_t)c.NTT * 2 * 3 * 32;
}

__global__ void k_tables(TabParams p) {
  long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx == 0 && p.err) *p.err = 0;
  // the fragments first: their threads have the longest chains
  if (idx < p.ncz + p.nct) {
    epi_fragments(p, idx);
    return;
  }
  idx -= p.ncz + p.nct;
  if (idx >= p.start[p.nseg]) return;
  int s = 0;
  while (s + 1 < p.nseg && idx >= p.start[s + 1]) ++s;
  const TabSeg g = p.seg[s];
  long long e = idx - p.start[s];
  int r = (int)(e / g.cols), c = (int)(e % g.cols);
  int j = g.k_on_row ? r : c;
  int n = g.k_on_row ? c : r;
  long long k = (g.m > 0) ? (j < g.m ? j : j - 2 * g.m) : j;
  long long rr = (k * n) % g.N;
  if (rr < 0) rr += g.N;
  double sn, cs;
  sincospi(2.0 * (double)rr / (double)g.N, &sn, &cs);
  double sc = 1.0;
  if (g.scale) {
    bool single = (k == 0) || ((p.Nt % 2 == 0) && (2 * k == p.Nt));
    sc = (single ? 1.0 : 2.0) * p.invNg;
  }
  g.dst[e] = make_float2((float)(cs * sc), (float)((double)g.sign * sn * sc));
}

cudaError_t launch_tables(const Dims& d, const Tables& T, const EpiTables* et, int* err, cudaStream_t s) {
  TabParams p{};
  p.err = err;
  if (et) {
    p.et = *et;
    p.Nz = (int)d.Nz;
    p.mz = (int)d.mz;
    p.Jt = (int)d.Jt;
    p.ncz = 32LL * et->NZ * et->KS;
    p.nct = 32LL * 4 * et->NTT;
  }
  auto add = [&](float2* dst, int64_t rows, int64_t cols, int64_t N, int64_t m, int kr, int sign,
                 int scale) {
    p.seg[p.nseg] = TabSeg{dst, (int)rows, (int)cols, (int)N, (int)m, kr, sign, scale};
    p.start[p.nseg + 1] = p.start[p.nseg] + rows * cols;
    ++p.nseg;
  };
  p.start[0] = 0;
  add(T.Fx, d.Jx, d.Nx, d.Nx, d.mx, 1, -1, 0);
  add(T.Fy, d.Jy, d.Ny, d.Ny, d.my, 1, -1, 0);
  add(T.Fz, d.Jz, d.Nz, d.Nz, d.mz, 1, -1, 0);
  add(T.Ft, d.Jt, d.Nt, d.Nt, 0, 1, -1, 0);
  add(T.Fta, d.Jt, d.Nt, d.Nt, 0, 1, -1, 1);
  add(T.Ix, d.Nx, d.Jx, d.Nx, d.mx, 0, +1, 0);
  add(T.Iy, d.Ny, d.Jy, d.Ny, d.my, 0, +1, 0);
  add(T.Iz, d.Nz, d.Jz, d.Nz, d.mz, 0, +1, 0);
  add(T.Its, d.Jt, d.Nt, d.Nt, 0, 1, +1, 1);
  add(T.Itu, d.Jt, d.Nt, d.Nt, 0, 1, +1, 0);
  p.Nt = (int)d.Nt;
  p.invNg = 1.0 / (double)d.Ng;
  long long total = p.start[p.nseg] + p.ncz + p.nct;
  // one warp a block: an SM does about two FP64 operations a clock, so the
  // entries (some fifty operations each) are spread over all of them
  int threads = 32;
  int blocks = (int)((total + threads - 1) / threads);
  FNO_LAUNCH("fno_tables", k_tables, blocks, threads, 0, s, p);
  return cudaSuccess;
}

// ---------------------------------------------------------------------------
// Forward pruned DFT over t, then z, of each column [Nz][Nt] (real input):
//   P[z][jt]  = sum_t x[z][t] ft[jt][t]
//   T1[jz][jt] = sum_z fz[jz][z] P[z][jt]
// One warp per column.  t stage: a lane owns one or two z rows and folds t and
// Nt - t (the sum meets the cosines, the difference the sines), so a basis value
// read once (16-byte broadcasts) serves two points of each row.  z stage: a lane
// owns one jt and up to three |kz| and folds z and Nz - z likewise; the sums over
// cosines and sines give +kz and -kz together.  Together a quarter of the
// multiply-adds of the plain sums.
// Rows of a multiple of four floats are read straight from global memory, 16
// bytes per lane; other rows are copied to shared memory as they lie, 32 or 64 at
// a time (an odd row stride has no bank conflicts, Nt % 4 = 2 two-way ones; whole
// columns of 22 KB left eight warps on an SM and took 4.27 ms at 20 x 64^3 x 86), or
// read 4 bytes at a time where the copies would leave few warps (tz_f32_form).
// Issue bounds it.  One thread per row and per output with one basis read per two
// multiply-adds took 641 us at 2 x 20 x 64^3 x 16 and 132 us at 2 x 12 x 45 x 37
// x 27 x 21; this form 314 and 66 (three CTAs of 80 registers on an SM; two: 314
// and 82).
// ---------------------------------------------------------------------------
// shared memory of the CTA form, which bounds the sizes that are accepted
size_t fwd_tz_smem_bytes(const Dims& d) {
  return sizeof(float2) * (size_t)(d.Jt * d.Nt + d.Jz * (d.Nz + 1) + d.Nz * d.Jt);
}

constexpr int kTzfP = 10;  // float2 stride of a row of P (8 used): 16-byte stores without conflicts

// How a lane reads its rows: 16 bytes at a time (rows of a multiple of four
// floats), from copied rows, or 4 bytes at a time where copies of 32 rows a warp
// would leave few warps on an SM.
enum TzfRows { TZF_VEC4, TZF_COPIED, TZF_DIRECT };

// rows copied at a time (TZF_COPIED)
__host__ __device__ inline int tzf_rows_at_once(int Nz, int Nt) { return Nz > 32 && Nt <= 32 ? 64 : 32; }

// shared memory of W warps: tables, then per warp P and the copied rows
static size_t tzf_smem(const Dims& d, TzfRows rows, int W) {
  const size_t tab = sizeof(float2) * ((size_t)((d.Jt + 7) / 8) * (d.Nt / 2 + 1) * 8 +
                                       (((size_t)(d.Nz / 2 + 1) * (d.mz + 1) + 1) & ~(size_t)1));
  const size_t col =
      rows != TZF_COPIED ? 0 : sizeof(float) * (((size_t)std::min<int64_t>(d.Nz, tzf_rows_at_once((int)d.Nz, (int)d.Nt)) * d.Nt + 3) & ~(size_t)3);
  return tab + (size_t)W * (sizeof(float2) * kTzfP * (size_t)d.Nz + col);
}

// t stage of rows z0 + lane + 32 r (r < R): P[z][0..7] of one group of eight jt.
// F: [Nt / 2 + 1][8] (cos, -sin).
template <bool V4, int R>
__device__ __forceinline__ void tzf_rows(const float* __restrict__ src, float2* sP, const float2* F, int z0, int Nz,
                                         int Nt, int lane) {
  float ar[R][8], ai[R][8];
  const float* row[R];
#pragma unroll
  for (int r = 0; r < R; ++r) row[r] = src + (long long)min(z0 + lane + 32 * r, Nz - 1) * Nt;
  auto basis = [&](int t, float (&c)[8], float (&n)[8]) {
    const float4* f = reinterpret_cast<const float4*>(F + t * 8);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 v = f[q];
      c[2 * q] = v.x;
      n[2 * q] = v.y;
      c[2 * q + 1] = v.z;
      n[2 * q + 1] = v.w;
    }
  };
  // t and Nt - t
  auto pair = [&](int t, const float (&u)[R], const float (&v)[R]) {
    float c[8], n[8];
    basis(t, c, n);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float s = u[r] + v[r], d = u[r] - v[r];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        ar[r][q] = fmaf(s, c[q], ar[r][q]);
        ai[r][q] = fmaf(d, n[q], ai[r][q]);
      }
    }
  };
  // t = 0 and t = Nt / 2 stand alone; their sines are zero
  auto single = [&](int t, const float (&u)[R]) {
    float c[8], n[8];
    basis(t, c, n);
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int q = 0; q < 8; ++q) ar[r][q] = fmaf(u[r], c[q], ar[r][q]);
  };
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int q = 0; q < 8; ++q) ar[r][q] = ai[r][q] = 0.f;
  if (V4) {
    // 16 bytes from the head and 16 from the tail of the rows at a time
    float carry[R], u[R], v[R];
    const int C = Nt / 8;
#pragma unroll 1
    for (int c = 0; c < C; ++c) {
      float4 h[R], w[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        h[r] = __ldg(reinterpret_cast<const float4*>(row[r] + 4 * c));
        w[r] = __ldg(reinterpret_cast<const float4*>(row[r] + Nt - 4 - 4 * c));
      }
#pragma unroll
      for (int r = 0; r < R; ++r) u[r] = h[r].x;
      if (c == 0)
        single(0, u);
      else
        pair(4 * c, u, carry);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        u[r] = h[r].y;
        v[r] = w[r].w;
      }
      pair(4 * c + 1, u, v);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        u[r] = h[r].z;
        v[r] = w[r].z;
      }
      pair(4 * c + 2, u, v);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        u[r] = h[r].w;
        v[r] = w[r].y;
        carry[r] = w[r].x;
      }
      pair(4 * c + 3, u, v);
    }
    if (Nt % 8 == 0) {
      single(Nt / 2, carry);
    } else {  // four values are left in the middle
      float4 h[R];
#pragma unroll
      for (int r = 0; r < R; ++r) h[r] = __ldg(reinterpret_cast<const float4*>(row[r] + 4 * C));
#pragma unroll
      for (int r = 0; r < R; ++r) u[r] = h[r].x;
      if (C == 0)
        single(0, u);
      else
        pair(4 * C, u, carry);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        u[r] = h[r].y;
        v[r] = h[r].w;
      }
      pair(4 * C + 1, u, v);
#pragma unroll
      for (int r = 0; r < R; ++r) u[r] = h[r].z;
      single(Nt / 2, u);
    }
  } else {
    float u[R], v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) u[r] = row[r][0];
    single(0, u);
#pragma unroll 2
    for (int t = 1; 2 * t < Nt; ++t) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        u[r] = row[r][t];
        v[r] = row[r][Nt - t];
      }
      pair(t, u, v);
    }
    if (Nt % 2 == 0) {
#pragma unroll
      for (int r = 0; r < R; ++r) u[r] = row[r][Nt / 2];
      single(Nt / 2, u);
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int z = z0 + lane + 32 * r;
    if (z < Nz) {
      float4* dst = reinterpret_cast<float4*>(sP + z * kTzfP);
#pragma unroll
      for (int q = 0; q < 4; ++q) dst[q] = make_float4(ar[r][2 * q], ai[r][2 * q], ar[r][2 * q + 1], ai[r][2 * q + 1]);
    }
  }
}

template <TzfRows ROWS>
__global__ void __launch_bounds__(256, 3)
    k_fwd_tz_f32(const float* __restrict__ in, float2* __restrict__ out, long long ncol, int Nz,
                 int Nt, int mz, int Jt, const float2* __restrict__ ft, const float2* __restrict__ fz) {
  extern __shared__ float4 smem4[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
  const int J8 = (Jt + 7) / 8, TH = Nt / 2 + 1, ZH = Nz / 2 + 1, KP = mz + 1, Jz = 2 * mz;
  constexpr bool V4 = ROWS == TZF_VEC4, COPY = ROWS == TZF_COPIED;
  const int CR = COPY ? tzf_rows_at_once(Nz, Nt) : 64;
  const size_t colf = !COPY ? 0 : (((size_t)min(Nz, CR) * Nt + 3) & ~(size_t)3);
  float2* sF = reinterpret_cast<float2*>(smem4);  // [J8][TH][8] (cos, -sin) * scale
  float2* sZ = sF + J8 * TH * 8;                  // [ZH][KP] (cos, sin) of k z
  float2* sP = sZ + ((ZH * KP + 1) & ~1) + (size_t)warp * (kTzfP * Nz + colf / 2);  // [Nz][kTzfP]
  float* sX = reinterpret_cast<float*>(sP + kTzfP * Nz);                            // [CR][Nt] (COPY)
  for (int e = threadIdx.x; e < J8 * TH * 8; e += blockDim.x) {
    const int q = e % 8, t = (e / 8) % TH, j = 8 * (e / (8 * TH)) + q;
    sF[e] = j < Jt ? ft[(long long)j * Nt + t] : make_float2(0.f, 0.f);
  }
  for (int e = threadIdx.x; e < ZH * KP; e += blockDim.x) {
    const int k = e % KP, z = e / KP;
    const float2 f = fz[(long long)k * Nz + z];  // k < mz: exp(-i k z); k = mz: stored as -mz
    sZ[e] = make_float2(f.x, k < mz ? -f.y : f.y);
  }
  __syncthreads();
  const int jt = lane & 7, kg = lane >> 3;
  for (long long col = (long long)blockIdx.x * W + warp; col < ncol; col += (long long)gridDim.x * W) {
    const float* src = in + col * (long long)Nz * Nt;
    for (int j8 = 0; j8 < J8; ++j8) {
      const float2* F = sF + j8 * TH * 8;
      for (int z0 = 0; z0 < Nz; z0 += CR) {
        const float* rows = src;
        if (COPY) {
          const int n = min(CR, Nz - z0) * Nt;
          const float* from = src + (long long)z0 * Nt;
          __syncwarp();
          for (int e0 = lane; e0 < n; e0 += 32 * 8) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = e0 + 32 * u < n ? __ldg(from + e0 + 32 * u) : 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u)
              if (e0 + 32 * u < n) sX[e0 + 32 * u] = v[u];
          }
          __syncwarp();
          rows = sX - (long long)z0 * Nt;
        }
        if (CR == 64 && Nz - z0 > 32)
          tzf_rows<V4, 2>(rows, sP, F, z0, Nz, Nt, lane);
        else
          tzf_rows<V4, 1>(rows, sP, F, z0, Nz, Nt, lane);
      }
      __syncwarp();
      const float2* P = sP + jt;
      const int j = 8 * j8 + jt;
      float2* dst = out + col * (long long)(Jz * Jt) + j;
      for (int kc = 0; kc < KP; kc += 12) {
        float2 A[3], Bs[3];  // sums over cosines and sines, (re, im)
        const float2* f0[3];
        const float2 p0 = P[0];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          f0[r] = sZ + min(kc + kg + 4 * r, KP - 1);
          A[r] = p0;
          Bs[r] = make_float2(0.f, 0.f);
        }
#pragma unroll 4
        for (int z = 1; 2 * z < Nz; ++z) {
          const float2 a = P[z * kTzfP], b = P[(Nz - z) * kTzfP];
          const float sr = a.x + b.x, si = a.y + b.y, dr = a.x - b.x, di = a.y - b.y;
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            const float2 f = f0[r][z * KP];
            A[r].x = fmaf(f.x, sr, A[r].x);
            A[r].y = fmaf(f.x, si, A[r].y);
            Bs[r].x = fmaf(f.y, dr, Bs[r].x);
            Bs[r].y = fmaf(f.y, di, Bs[r].y);
          }
        }
        if (Nz % 2 == 0) {
          const float2 a = P[(Nz / 2) * kTzfP];
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            const float c = f0[r][(Nz / 2) * KP].x;
            A[r].x = fmaf(c, a.x, A[r].x);
            A[r].y = fmaf(c, a.y, A[r].y);
          }
        }
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          const int k = kc + kg + 4 * r;
          if (j < Jt && k < KP) {
            if (k < mz) dst[(long long)k * Jt] = make_float2(A[r].x + Bs[r].y, A[r].y - Bs[r].x);
            if (k > 0) dst[(long long)(Jz - k) * Jt] = make_float2(A[r].x - Bs[r].y, A[r].y + Bs[r].x);
          }
        }
      }
      __syncwarp();  // P (and the column) may be overwritten
    }
  }
}

// The same by a CTA of 128 threads per column, a thread per z row in the t stage and
// per (jz, jt) output in the z stage, plain sums: a third of the shared memory on
// long axes, and a column's rows in parallel.
template <bool VEC4>
__global__ void __launch_bounds__(128)
    k_fwd_tz_cta_f32(const float* __restrict__ in, float2* __restrict__ out, long long ncol, int Nz,
                     int Nt, int Jz, int Jt, const float2* __restrict__ ft,
                     const float2* __restrict__ fz) {
  extern __shared__ float4 smem4[];
  float2* sFt = reinterpret_cast<float2*>(smem4);  // [Jt][Nt]
  float2* sFz = sFt + Jt * Nt;                      // [Jz][Nz + 1]
  float2* sP = sFz + Jz * (Nz + 1);                 // [Nz][Jt]
  for (int e = threadIdx.x; e < Jt * Nt; e += blockDim.x) sFt[e] = ft[e];
  for (int e = threadIdx.x; e < Jz * Nz; e += blockDim.x) {
    int r = e / Nz, c = e - r * Nz;
    sFz[r * (Nz + 1) + c] = fz[e];
  }
  __syncthreads();
  const int JZT = Jz * Jt;
  for (long long col = blockIdx.x; col < ncol; col += gridDim.x) {
    const float* src = in + col * (long long)Nz * Nt;
    for (int z = threadIdx.x; z < Nz; z += blockDim.x) {
      const float* row = src + (long long)z * Nt;
      for (int j0 = 0; j0 < Jt; j0 += 8) {
        float ar[8], ai[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) { ar[q] = 0.f; ai[q] = 0.f; }
        if (VEC4) {
          for (int t = 0; t < Nt; t += 4) {
            float4 v4 = __ldg(reinterpret_cast<const float4*>(row + t));
            float vv[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                if (j0 + q < Jt) {
                  float2 f = sFt[(j0 + q) * Nt + t + u];
                  ar[q] = fmaf(vv[u], f.x, ar[q]);
                  ai[q] = fmaf(vv[u], f.y, ai[q]);
                }
              }
            }
          }
        } else {
          for (int t = 0; t < Nt; ++t) {
            float v = __ldg(row + t);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              if (j0 + q < Jt) {
                float2 f = sFt[(j0 + q) * Nt + t];
                ar[q] = fmaf(v, f.x, ar[q]);
                ai[q] = fmaf(v, f.y, ai[q]);
              }
            }
          }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (j0 + q < Jt) sP[z * Jt + j0 + q] = make_float2(ar[q], ai[q]);
      }
    }
    __syncthreads();
    float2* dst = out + col * (long long)JZT;
    for (int o = threadIdx.x; o < JZT; o += blockDim.x) {
      int jz = o / Jt, jt = o - jz * Jt;
      const float2* f = sFz + jz * (Nz + 1);
      float re = 0.f, im = 0.f;
      for (int z = 0; z < Nz; ++z) {
        float2 a = f[z], b = sP[z * Jt + jt];
        re = fmaf(a.x, b.x, re);
        re = fmaf(-a.y, b.y, re);
        im = fmaf(a.x, b.y, im);
        im = fmaf(a.y, b.x, im);
      }
      dst[o] = make_float2(re, im);
    }
    __syncthreads();
  }
}

// warps of a CTA of the warp-per-column form: fewer than eight where their rows of
// P and their copied rows do not fit two CTAs on an SM
static int tzf_warps(const Dims& d, TzfRows rows) {
  int W = 8;
  while (W > 1 && tzf_smem(d, rows, W) > 110 * 1024) W /= 2;
  return W;
}
// warps of that form that an SM holds (0: not even one)
static int tzf_warps_per_sm(const Dims& d, TzfRows rows) {
  const int W = tzf_warps(d, rows);
  const size_t smem = tzf_smem(d, rows, W);
  if (smem > kMaxSmem) return 0;
  return W * (int)std::min<size_t>(3, 228 * 1024 / (smem + 1024));
}

// Which form runs.  The plan of the warp-per-column form grows with Nz (80 bytes a
// z row and warp) and, with copied rows, with Nt (32 rows a warp): the CTA form takes
// every size whose warps do not fit, and what check_support admits is its plan.
// Times in us at 1024 columns (256 where given), mt up to 8, warp / CTA form:
//   16-byte rows: 1.1 to 2 times faster while an SM holds two warps (768 x 32: 172 /
//     187; 512 x 1024, 256 columns: 543 / 704), slower with one (1024 x 16: 248 / 185;
//     2500 x 8: 455 / 285).
//   Copied rows: with 12 warps or more 10 / 12 (45 x 22) to 21 / 24 (64 x 86).  With
//     fewer, short rows are faster read 4 bytes at a time, which keeps the copies out
//     of shared memory (copied / direct / CTA: 262 x 22 43 / 23 / 49, 512 x 18 66 / 49 /
//     86), unless one warp is left (1024 x 18 687 / 311 / 244).  Long rows thrash L1 that
//     way (100 x 86: 31 / 58 / 56, 200 x 86: 168 / 217 / 144) and keep the copies down to
//     six warps; with fewer, few planes leave L1 the room (32 x 510: 296 / 88 / 209), more
//     do not (100 x 1022: 3032 / 1506 / 813).
//   Long columns that are too few to give each scheduler a warp: 208 / 107 at 256
//     columns of 64 x 1024, 227 / 103 at 130 x 512.
enum TzForm { TZ_VEC4, TZ_COPIED, TZ_DIRECT, TZ_CTA };
static TzForm tz_f32_form(const Dims& d, int64_t ncol) {
  if (d.Nz > 48 && d.Nz * d.Nt >= 16384 && ncol < 4 * (int64_t)sm_count()) return TZ_CTA;
  if (d.Nt % 4 == 0) return tzf_warps_per_sm(d, TZF_VEC4) >= 2 ? TZ_VEC4 : TZ_CTA;
  if (tzf_warps_per_sm(d, TZF_COPIED) >= (d.Nt < 32 ? 12 : 6)) return TZ_COPIED;
  if (d.Nt >= 32 && d.Nz > 48) return TZ_CTA;
  return tzf_warps_per_sm(d, TZF_DIRECT) >= 2 ? TZ_DIRECT : TZ_CTA;
}

template <TzfRows ROWS>
static cudaError_t launch_tzf(const float* in, float2* out, int64_t ncol, const Dims& d, const float2* ft,
                              const float2* fz, cudaStream_t s) {
  const int W = tzf_warps(d, ROWS);
  const size_t smem = tzf_smem(d, ROWS, W);
  const void* k = (const void*)k_fwd_tz_f32<ROWS>;
  cudaError_t e = allow_smem(k, smem);
  if (e != cudaSuccess) return e;
  const int grid = persistent_grid(k, 32 * W, smem, (ncol + W - 1) / W);
  FNO_LAUNCH("fno_fwd_tz_f32", k_fwd_tz_f32<ROWS>, grid, 32 * W, smem, s, in, out, (long long)ncol, (int)d.Nz,
             (int)d.Nt, (int)d.mz, (int)d.Jt, ft, fz);
  return cudaSuccess;
}

template <bool VEC4>
static cudaError_t launch_tz_cta(const float* in, float2* out, int64_t ncol, const Dims& d, const float2* ft,
                                 const float2* fz, cudaStream_t s) {
  const size_t smem = fwd_tz_smem_bytes(d);
  const void* k = (const void*)k_fwd_tz_cta_f32<VEC4>;
  cudaError_t e = allow_smem(k, smem);
  if (e != cudaSuccess) return e;
  const int grid = persistent_grid(k, 128, smem, ncol);
  FNO_LAUNCH("fno_fwd_tz_cta_f32", k_fwd_tz_cta_f32<VEC4>, grid, 128, smem, s, in, out, (long long)ncol, (int)d.Nz,
             (int)d.Nt, (int)d.Jz, (int)d.Jt, ft, fz);
  return cudaSuccess;
}

cudaError_t launch_fwd_tz_f32(const float* in, float2* out, int64_t ncol, const Dims& d,
                              const float2* ft, const float2* fz, cudaStream_t s) {
  if (ncol <= 0) return cudaSuccess;
  switch (tz_f32_form(d, ncol)) {
    case TZ_VEC4: return launch_tzf<TZF_VEC4>(in, out, ncol, d, ft, fz, s);
    case TZ_COPIED: return launch_tzf<TZF_COPIED>(in, out, ncol, d, ft, fz, s);
    case TZ_DIRECT: return launch_tzf<TZF_DIRECT>(in, out, ncol, d, ft, fz, s);
    default: break;
  }
  if (d.Nt % 4 == 0) return launch_tz_cta<true>(in, out, ncol, d, ft, fz, s);
  return launch_tz_cta<false>(in, out, ncol, d, ft, fz, s);
}

// ---------------------------------------------------------------------------
// One complex DFT axis: out[o][q][i] = sum_n tab[q][n] in[o][n][i].
// A CTA stages an [nin][32] slab of the input in shared memory; a warp owns a
// group of QB output rows for 32 consecutive i.
// ---------------------------------------------------------------------------
size_t line_smem_bytes(int nin, int nout) {
  return sizeof(float2) * (size_t)(nout * nin + nin * 32);
}

template <int QB>
__global__ void __launch_bounds__(256)
    k_line_f32(const float2* __restrict__ in, float2* __restrict__ out, long long outer, int nin,
               int nout, long long inner, const float2* __restrict__ tab) {
  extern __shared__ float4 smem4[];
  float2* sTab = reinterpret_cast<float2*>(smem4);  // [nout][nin]
  float2* sIn = sTab + nout * nin;                   // [nin][32]
  const int lane = threadIdx.x, ty = threadIdx.y;
  const int tid = ty * 32 + lane;
  for (int e = tid; e < nout * nin; e += 256) sTab[e] = tab[e];
  const long long ntile = (inner + 31) / 32;
  const long long nwork = outer * ntile;
  for (long long w = blockIdx.x; w < nwork; w += gridDim.x) {
    const long long o = w / ntile;
    const long long i = (w - o * ntile) * 32 + lane;
    const bool ok = i < inner;
    __syncthreads();
    for (int n = ty; n < nin; n += 8)
      sIn[n * 32 + lane] = ok ? in[(o * nin + n) * inner + i] : make_float2(0.f, 0.f);
    __syncthreads();
    for (int q0 = ty * QB; q0 < nout; q0 += 8 * QB) {
      float2 acc[QB];
#pragma unroll
      for (int qq = 0; qq < QB; ++qq) acc[qq] = make_float2(0.f, 0.f);
      for (int n = 0; n < nin; ++n) {
        float2 v = sIn[n * 32 + lane];
#pragma unroll
        for (int qq = 0; qq < QB; ++qq) {
          if (q0 + qq < nout) {
            float2 f = sTab[(q0 + qq) * nin + n];
            acc[qq].x = fmaf(f.x, v.x, acc[qq].x);
            acc[qq].x = fmaf(-f.y, v.y, acc[qq].x);
            acc[qq].y = fmaf(f.x, v.y, acc[qq].y);
            acc[qq].y = fmaf(f.y, v.x, acc[qq].y);
          }
        }
      }
      if (ok) {
#pragma unroll
        for (int qq = 0; qq < QB; ++qq)
          if (q0 + qq < nout) out[(o * nout + q0 + qq) * inner + i] = acc[qq];
      }
    }
  }
}

// The same with two i a lane, 32 apart.  Shared-memory reads bound both forms (one
// of the slab for each i and one of the table for each row, per 4 multiply-adds
// and row), so a table value serves two i here.  Rows past nout repeat the last
// one and are not stored.  Eight launches of a step: 20 x 64^3 x 32, modes
// 12/12/8/8 455 us with one i, 354 with two; 2 x 20 x 64^3 x 16 422 and 404.
static size_t line_pair_smem(int nin, int nout) {
  return sizeof(float2) * (size_t)(nout * nin + nin * 64);
}

template <int QB>
__global__ void __launch_bounds__(256)
    k_line_pair_f32(const float2* __restrict__ in, float2* __restrict__ out, long long outer,
                    int nin, int nout, long long inner, const float2* __restrict__ tab) {
  extern __shared__ float4 smem4[];
  float2* sTab = reinterpret_cast<float2*>(smem4);  // [nout][nin]
  float2* sIn = sTab + nout * nin;                   // [nin][64]
  const int lane = threadIdx.x, ty = threadIdx.y;
  const int tid = ty * 32 + lane;
  for (int e = tid; e < nout * nin; e += 256) sTab[e] = tab[e];
  const long long ntile = (inner + 63) / 64;
  const long long nwork = outer * ntile;
  for (long long w = blockIdx.x; w < nwork; w += gridDim.x) {
    const long long o = w / ntile;
    const long long i = (w - o * ntile) * 64 + lane;
    __syncthreads();
    for (int n = ty; n < nin; n += 8)
#pragma unroll
      for (int v = 0; v < 2; ++v)
        sIn[n * 64 + 32 * v + lane] =
            i + 32 * v < inner ? in[(o * nin + n) * inner + i + 32 * v] : make_float2(0.f, 0.f);
    __syncthreads();
    for (int q0 = ty * QB; q0 < nout; q0 += 8 * QB) {
      float2 acc[QB][2];
      const float2* f[QB];
#pragma unroll
      for (int qq = 0; qq < QB; ++qq) {
        f[qq] = sTab + min(q0 + qq, nout - 1) * nin;
        acc[qq][0] = acc[qq][1] = make_float2(0.f, 0.f);
      }
#pragma unroll 4
      for (int n = 0; n < nin; ++n) {
        const float2 x[2] = {sIn[n * 64 + lane], sIn[n * 64 + 32 + lane]};
#pragma unroll
        for (int qq = 0; qq < QB; ++qq) {
          const float2 t = f[qq][n];
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            acc[qq][v].x = fmaf(t.x, x[v].x, acc[qq][v].x);
            acc[qq][v].x = fmaf(-t.y, x[v].y, acc[qq][v].x);
            acc[qq][v].y = fmaf(t.x, x[v].y, acc[qq][v].y);
            acc[qq][v].y = fmaf(t.y, x[v].x, acc[qq][v].y);
          }
        }
      }
#pragma unroll
      for (int qq = 0; qq < QB; ++qq)
#pragma unroll
        for (int v = 0; v < 2; ++v)
          if (q0 + qq < nout && i + 32 * v < inner)
            out[(o * nout + q0 + qq) * inner + i + 32 * v] = acc[qq][v];
    }
  }
}

cudaError_t launch_line_f32(const float2* in, float2* out, int64_t outer, int nin, int nout,
                            int64_t inner, const float2* tab, cudaStream_t s) {
  if (outer <= 0 || inner <= 0) return cudaSuccess;
  // Two i a lane where the tiles of 64 are hardly emptier than those of 32 (inner
  // 96: a quarter of them idle), there are two for each SM, and four CTAs fit on
  // one (64 -> 16 rows: 41 KB).  Axes that do not fit so keep one i a lane.
  const int64_t t2 = (inner + 63) / 64, t1 = (inner + 31) / 32;
  if (20 * t2 <= 11 * t1 && outer * t2 >= 2 * sm_count() &&
      line_pair_smem(nin, nout) <= 56 * 1024) {
    const size_t smem = line_pair_smem(nin, nout);
    const void* k = (const void*)k_line_pair_f32<4>;
    cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    const int grid = persistent_grid(k, 256, smem, outer * t2);
    FNO_LAUNCH("fno_line_pair_f32", k_line_pair_f32<4>, grid, dim3(32, 8), smem, s, in, out,
               (long long)outer, nin, nout, (long long)inner, tab);
    return cudaSuccess;
  }
  size_t smem = line_smem_bytes(nin, nout);
  const void* k = (const void*)k_line_f32<4>;
  cudaError_t e = allow_smem(k, smem);
  if (e != cudaSuccess) return e;
  int64_t work = outer * ((inner + 31) / 32);
  int grid = persistent_grid(k, 256, smem, work);
  FNO_LAUNCH("fno_line_f32", k_line_f32<4>, grid, dim3(32, 8), smem, s, in, out,
             (long long)outer, nin, nout, (long long)inner, tab);
  return cudaSuccess;
}

// ---------------------------------------------------------------------------
// Spectral convolution and its adjoint (FP32 complex multiply-adds).
//   forward  yh[b][o][j]  = sum_i xh[b][i][j] w[i][o][j]
//   adjoint  gxh[b][i][j] = sum_o conj(w[i][o][j]) g[b][o][j]
//            dw[i][o][j]  = sum_b conj(xh[b][i][j]) g[b][o][j]
// A CTA owns a tile of kMixJ consecutive modes and has one group of kMixJ
// threads per channel (output channels forward, input channels in the adjoint;
// at most kMixG groups, which then take several in turn; kMixMin for fewer channels
// with many rows to stage, the others helping there and, in the adjoint, sharing the
// output channels of dW).  It stages the tile's
// spectra for a chunk of BC batch entries in shared memory (rows of kMixJ
// complex values: 128-byte coalesced loads), then each thread walks the summed
// channel with kMixU weights in flight at a time, read straight from HBM in
// coalesced 128-byte rows; the first ones are under way before the staging.  W,
// dW and the outputs cross HBM once per batch chunk (once when B <= BC), and
// every sum runs in a fixed order.
// HBM bounds it (W, and dW in the adjoint).  With 16 fixed groups (20 channels:
// two rounds, the second a quarter full) and 4 or 8 weights in flight the
// forward and its adjoint took 59 and 57 us at 24576 modes, B = 2, width 20 (W 79
// MB), here 27 and 42; 72 and 107, here 51 and 87 at 73728 modes, B = 1; 263 and
// 361, here 207 and 354 at 110592 modes, B = 2, width 32.  20 weights in flight
// measured slower (registers), 5 about as fast.  One group and no more for a single
// channel (20 -> 1 forward, 1 -> 20 adjoint, 24576 modes, B = 16) took 304 and 360 us,
// 66 and 68 in 16 fixed groups, 60 and 75 here (mix_widen).
// ---------------------------------------------------------------------------
constexpr int kMixJ = 16;  // modes per tile
constexpr int kMixG = 32;    // most channel groups of a CTA
constexpr int kMixMin = 16;  // groups where many rows are staged for few channels
constexpr int kMixU = 10;  // weights in flight per thread

__device__ __forceinline__ void cmac(float2& acc, const float2 a, const float2 b) {
  acc.x = fmaf(a.x, b.x, acc.x);
  acc.x = fmaf(-a.y, b.y, acc.x);
  acc.y = fmaf(a.x, b.y, acc.y);
  acc.y = fmaf(a.y, b.x, acc.y);
}
// acc += conj(a) b
__device__ __forceinline__ void cmac_conj(float2& acc, const float2 a, const float2 b) {
  acc.x = fmaf(a.x, b.x, acc.x);
  acc.x = fmaf(a.y, b.y, acc.x);
  acc.y = fmaf(a.x, b.y, acc.y);
  acc.y = fmaf(-a.y, b.x, acc.y);
}

// stage src[b0 + q][c][j0 .. j0 + kMixJ) for q < nb, c < C into dst[q][c][kMixJ]
__device__ __forceinline__ void mix_stage(float2* dst, const float2* __restrict__ src, int b0,
                                          int nb, int BC, int C, long long Mk, long long j0) {
  for (int e = threadIdx.x; e < BC * C * kMixJ; e += blockDim.x) {
    const int jl = e % kMixJ, c = (e / kMixJ) % C, q = e / (kMixJ * C);
    const long long j = j0 + jl;
    dst[e] = (q < nb && j < Mk) ? src[((long long)(b0 + q) * C + c) * Mk + j]
                                : make_float2(0.f, 0.f);
  }
}
// weights u0 .. u0 + kMixU of a row of n, `step` apart
__device__ __forceinline__ void mix_load(float2 (&wv)[kMixU], const float2* __restrict__ wp, long long step,
                                         int u0, int n, bool in) {
#pragma unroll
  for (int u = 0; u < kMixU; ++u)
    wv[u] = (in && u0 + u < n) ? __ldg(wp + (u0 + u) * step) : make_float2(0.f, 0.f);
}

template <int BC>
__global__ void __launch_bounds__(kMixJ * kMixG, 2)
    k_mix_f32(const float2* __restrict__ xh, const float2* __restrict__ w, float2* __restrict__ yh,
              int B, int Ci, int Co, long long Mk) {
  extern __shared__ float2 mix_sm[];
  float2* xs = mix_sm;  // [BC][Ci][kMixJ]
  const int jl = threadIdx.x % kMixJ, grp = threadIdx.x / kMixJ, ngrp = blockDim.x / kMixJ;
  const long long j0 = (long long)blockIdx.x * kMixJ, j = j0 + jl;
  const bool inj = j < Mk;
  const long long step = (long long)Co * Mk;
  for (int b0 = 0; b0 < B; b0 += BC) {
    const int nb = min(BC, B - b0);
    float2 wv[kMixU];
    mix_load(wv, w + (long long)grp * Mk + j, step, 0, Ci, inj && grp < Co);
    __syncthreads();
    mix_stage(xs, xh, b0, nb, BC, Ci, Mk, j0);
    __syncthreads();
    if (!inj) continue;
    for (int o = grp; o < Co; o += ngrp) {
      float2 acc[BC];
#pragma unroll
      for (int q = 0; q < BC; ++q) acc[q] = make_float2(0.f, 0.f);
      const float2* wp = w + (long long)o * Mk + j;
      for (int i0 = 0; i0 < Ci; i0 += kMixU) {
        if (i0 > 0 || o != grp) mix_load(wv, wp, step, i0, Ci, true);
#pragma unroll
        for (int u = 0; u < kMixU; ++u) {
          if (i0 + u < Ci) {
#pragma unroll
            for (int q = 0; q < BC; ++q) cmac(acc[q], xs[(q * Ci + i0 + u) * kMixJ + jl], wv[u]);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < BC; ++q)
        if (q < nb) yh[((long long)(b0 + q) * Co + o) * Mk + j] = acc[q];
    }
  }
}

// SPLIT: several groups of threads per input channel, which share dW's outputs
template <int BC, bool SPLIT>
__global__ void __launch_bounds__(kMixJ * kMixG, 2)
    k_mix_adj_f32(const float2* __restrict__ xh, const float2* __restrict__ w,
                  const float2* __restrict__ g, float2* __restrict__ dw, float2* __restrict__ gxh,
                  int B, int Ci, int Co, long long Mk, int GI) {
  extern __shared__ float2 mix_sm[];
  float2* xs = mix_sm;                   // [BC][Ci][kMixJ]
  float2* gs = mix_sm + BC * Ci * kMixJ; // [BC][Co][kMixJ]
  // group (gi, go): input channels gi, gi + GI, ..; dW's outputs go, go + GO, ..
  const int jl = threadIdx.x % kMixJ, grp = threadIdx.x / kMixJ;
  const int GO = SPLIT ? blockDim.x / (kMixJ * GI) : 1;
  const int gi = SPLIT ? grp % GI : grp, go = SPLIT ? grp / GI : 0;
  const long long j0 = (long long)blockIdx.x * kMixJ, j = j0 + jl;
  const bool inj = j < Mk;
  for (int b0 = 0; b0 < B; b0 += BC) {
    const int nb = min(BC, B - b0);
    float2 wv[kMixU];
    mix_load(wv, w + (long long)gi * Co * Mk + j, Mk, 0, Co, inj && gxh && go == 0);
    __syncthreads();
    if (dw) mix_stage(xs, xh, b0, nb, BC, Ci, Mk, j0);
    mix_stage(gs, g, b0, nb, BC, Co, Mk, j0);
    __syncthreads();
    if (!inj) continue;
    if (gxh && go == 0) {
      for (int i = gi; i < Ci; i += GI) {
        float2 ga[BC];
#pragma unroll
        for (int q = 0; q < BC; ++q) ga[q] = make_float2(0.f, 0.f);
        const float2* wp = w + (long long)i * Co * Mk + j;
        for (int o0 = 0; o0 < Co; o0 += kMixU) {
          if (o0 > 0 || i != gi) mix_load(wv, wp, Mk, o0, Co, true);
#pragma unroll
          for (int u = 0; u < kMixU; ++u) {
            if (o0 + u < Co) {
#pragma unroll
              for (int q = 0; q < BC; ++q) cmac_conj(ga[q], wv[u], gs[(q * Co + o0 + u) * kMixJ + jl]);
            }
          }
        }
#pragma unroll
        for (int q = 0; q < BC; ++q)
          if (q < nb) gxh[((long long)(b0 + q) * Ci + i) * Mk + j] = ga[q];
      }
    }
    // dW after it: reads of W and writes of dW in one loop measured slower
    if (dw) {
      for (int i = gi; i < Ci; i += GI) {
        float2 xv[BC];
#pragma unroll
        for (int q = 0; q < BC; ++q) xv[q] = xs[(q * Ci + i) * kMixJ + jl];
        float2* dp = dw + ((long long)i * Co + go) * Mk + j;
#pragma unroll 4
        for (int o = go; o < Co; o += GO, dp += GO * Mk) {
          float2 da = make_float2(0.f, 0.f);
#pragma unroll
          for (int q = 0; q < BC; ++q) cmac_conj(da, xv[q], gs[(q * Co + o) * kMixJ + jl]);
          if (b0 == 0) {
            *dp = da;
          } else {
            const float2 p = *dp;
            *dp = make_float2(p.x + da.x, p.y + da.y);
          }
        }
      }
    }
  }
}

// Channel groups of a CTA: one per channel up to 24 and, in the forward, 32; otherwise
// two channels in turn.  21 to 24 groups put two CTAs of 64-register threads on an SM where
// half as many put five: taken where the tiles fill the chip (24 channels, 73728
// modes, B = 2: forward 104 us in 24 groups, 90 in 12; adjoint 177 and 154), not on
// few tiles (2048 modes: 8.1 and 10.4, 10.9 and 14.3) and not in the adjoint with
// eight batch entries at a time (B = 16: 810 and 893).  Other widths, adjoint: 32 at B
// = 2 330 us in 16 groups, 371 in 32; 20 46 in 16, 38 in 20.
static bool mix_halve(int64_t C, unsigned tiles) { return C >= 21 && C <= 24 && tiles >= 4u * (unsigned)sm_count(); }
static int mix_groups(int64_t Co, unsigned tiles) {
  return mix_halve(Co, tiles) ? (int)(Co + 1) / 2 : (int)std::min<int64_t>(kMixG, Co);
}
static int mix_adj_groups(int64_t Ci, int BC, unsigned tiles) {
  if (Ci > 32 || (BC <= 4 && mix_halve(Ci, tiles))) return (int)(Ci + 1) / 2;
  return Ci <= 24 ? (int)Ci : 16;
}

// Whether a CTA of `groups` groups takes kMixMin of them instead: so many rows to
// stage that its few threads would take longer over them than over the sums.  Many
// tiles hide the staging of one CTA behind others, so the line lies higher there
// (rows a group, us without and with: 20, 128 tiles 12.3 / 6.7; 40, 1536 tiles 22.7 / 14.6,
// 4608 tiles 30.4 / 33.3; 80, 4608 tiles 137 / 69).
static bool mix_widen(int64_t rows, int groups, unsigned tiles) {
  if (groups >= kMixMin) return false;
  const unsigned sms = (unsigned)sm_count();
  return rows > groups * (int64_t)(tiles < 4 * sms ? 8 : tiles < 16 * sms ? 32 : 44);
}

static int mix_bc(int64_t B) { return B <= 1 ? 1 : B <= 2 ? 2 : B <= 4 ? 4 : 8; }

template <int BC>
static cudaError_t launch_mix_bc(const Dims& d, const float2* xh, const float2* w, float2* yh,
                                 cudaStream_t s) {
  const size_t smem = sizeof(float2) * (size_t)BC * (size_t)d.Ci * kMixJ;
  cudaError_t e = allow_smem((const void*)k_mix_f32<BC>, smem);
  if (e != cudaSuccess) return e;
  const unsigned grid = (unsigned)((d.Mk + kMixJ - 1) / kMixJ);
  int groups = mix_groups(d.Co, grid);
  if (mix_widen(BC * d.Ci, groups, grid)) groups = kMixMin;
  FNO_LAUNCH("fno_mix_f32", k_mix_f32<BC>, grid, kMixJ * groups, smem, s, xh, w, yh, (int)d.B, (int)d.Ci,
             (int)d.Co, (long long)d.Mk);
  return cudaSuccess;
}

template <int BC>
static cudaError_t launch_mix_adj_bc(const Dims& d, const float2* xh, const float2* w,
                                     const float2* g, float2* dw, float2* gxh, cudaStream_t s) {
  const size_t smem = sizeof(float2) * (size_t)BC * (size_t)(d.Ci + d.Co) * kMixJ;
  const unsigned grid = (unsigned)((d.Mk + kMixJ - 1) / kMixJ);
  const int GI = mix_adj_groups(d.Ci, BC, grid);
  const bool split = mix_widen(BC * (d.Co + (dw ? d.Ci : 0)), GI, grid);
  const int threads = kMixJ * GI * (split ? kMixMin / GI : 1);
  const void* k = split ? (const void*)k_mix_adj_f32<BC, true> : (const void*)k_mix_adj_f32<BC, false>;
  cudaError_t e = allow_smem(k, smem);
  if (e != cudaSuccess) return e;
  if (split)
    FNO_LAUNCH("fno_mix_adjoint_f32", (k_mix_adj_f32<BC, true>), grid, threads, smem, s, xh, w, g, dw, gxh, (int)d.B,
               (int)d.Ci, (int)d.Co, (long long)d.Mk, GI);
  else
    FNO_LAUNCH("fno_mix_adjoint_f32", (k_mix_adj_f32<BC, false>), grid, threads, smem, s, xh, w, g, dw, gxh, (int)d.B,
               (int)d.Ci, (int)d.Co, (long long)d.Mk, GI);
  return cudaSuccess;
}

cudaError_t launch_mix_f32(const Dims& d, const float2* xh, const float2* w, float2* yh,
                           cudaStream_t s) {
  if (d.B <= 0) return cudaSuccess;
  switch (mix_bc(d.B)) {
    case 1: return launch_mix_bc<1>(d, xh, w, yh, s);
    case 2: return launch_mix_bc<2>(d, xh, w, yh, s);
    case 4: return launch_mix_bc<4>(d, xh, w, yh, s);
    default: return launch_mix_bc<8>(d, xh, w, yh, s);
  }
}

cudaError_t launch_mix_adjoint_f32(const Dims& d, const float2* xh, const float2* w,
                                   const float2* g, float2* dw, float2* gxh, cudaStream_t s) {
  if (d.B <= 0) return cudaSuccess;
  switch (mix_bc(d.B)) {
    case 1: return launch_mix_adj_bc<1>(d, xh, w, g, dw, gxh, s);
    case 2: return launch_mix_adj_bc<2>(d, xh, w, g, dw, gxh, s);
    case 4: return launch_mix_adj_bc<4>(d, xh, w, g, dw, gxh, s);
    default: return launch_mix_adj_bc<8>(d, xh, w, g, dw, gxh, s);
  }
}

// ---------------------------------------------------------------------------
// Inverse z, t stages fused with the pointwise epilogue (FP32 CUDA cores).
// A 128-thread CTA walks a contiguous range of tiles; a tile is P = 128
// consecutive points (z, t) of one (b, x, y) column (fewer at the column's
// end) and all its channels, one thread per point.  When Nt divides 128 a
// tile is 128 / Nt whole z-planes; otherwise it starts and ends inside planes
// and touches at most ZM = 1 + ceil(127 / Nt) of them.
//   Q[zz][jt][o] = inverse z stage of the column spectrum, with +-k pairing:
//       Q(z) = sum_{k=0..mz} E_k cos(k th) + i sum_{k=1..mz} O_k sin(k th)
//       E_0 = U_0, E_k = U_k + U_-k, O_k = U_k - U_-k, E_mz = U_-mz, O_mz = -U_-mz
//   per point and 4 outputs at a time (shared-memory vector broadcasts):
//       A_o = bias_o + sum_jt (Qr[jt][o] c_jt(t) - Qi[jt][o] s_jt(t)) + sum_i W(i, o) L_i
// Even Nt (EO, up to 8 kt and 32 inputs): with the even and the odd kt summed apart,
// S(t) = E + O and S(t + Nt / 2) = E - O, so a thread owns the points t and t + Nt /
// 2 of a plane: half of the inverse-t multiply-adds, and each weight and Q value
// read once for two points (tiles are then 128 such pairs).  The dA mode keeps one
// point per thread and forms the same two sums, so that it finds the forward's A
// bit for bit.  Forward and dX at 2 x 20 x 64^3 x 16: 1252 and 994 us with one point
// a thread (a shared-memory read per four multiply-adds), 1078 and 818 here; at 20
// x 64^3 x 86 2874 and 2178, here 2265 and 1546.  Sizes whose pair tiles need more
// than 56 KB of shared memory keep one point a thread.
//   SPECTRAL: out = A (no bias, no linear term)   FWD: out = GELU(A)
//   DA: out = dA = dz GELU'(A), and dW_lin / db partial sums   DX: out = A
// ---------------------------------------------------------------------------
struct EpiK {
  EpiArgs a;
  long long NxNy, ntiles;
  long long nzc;        // tiles per column: ceil(Nz * Nt / 128)
  int Nz, Nt, Jz, Jt, mz;
  int ZM;               // z-planes a tile touches at most
  int P;                // points per tile, min(128, Nz * Nt)
  int CS4;
  int IB, OB, KG;       // EPI_DA: 4x4 (i, o) blocks of dW_lin, point groups
  int CLW;              // weight rows held in shared memory (the template's channel bound)
  uint32_t off[8];      // shared-memory region offsets (16-byte aligned)
};

constexpr int kEpiP = 128;  // points per tile (one per thread)

// points per tile and the most z-planes a tile touches
static int epi_points(const Dims& d) { return (int)std::min<int64_t>(kEpiP, d.Nz * d.Nt); }
static int epi_planes(const Dims& d) {
  int64_t zm = (kEpiP % d.Nt == 0) ? kEpiP / d.Nt : 1 + (kEpiP - 1 + d.Nt - 1) / d.Nt;
  return (int)std::min<int64_t>(zm, d.Nz);
}

// channel bound of the lin-input register array (template CLM) for Cl channels
static int epi_clm(int Cl) {
  if (Cl <= 0) return 0;
  static const int b[] = {4, 8, 12, 16, 20, 24, 32, 48, 64};
  for (int v : b)
    if (Cl <= v) return v;
  return 64;
}

static void epi_layout(const Dims& d, int mode, int Cs, int Cl, size_t off[8], size_t& total) {
  const int ZM = epi_planes(d);
  const int P = epi_points(d);
  const int CS4 = (Cs + 3) / 4 * 4;
  auto al = [](size_t x) { return (x + 15) / 16 * 16; };
  size_t o = 0;
  off[0] = o;  // eo: [Cs][Jt][mz+1] float4
  o = al(o + sizeof(float4) * (size_t)(Cs * d.Jt * (d.mz + 1)));
  off[1] = o;  // cs: [Nz][mz+1] float2
  o = al(o + sizeof(float2) * (size_t)(d.Nz * (d.mz + 1)));
  off[2] = o;  // qs: [ZM][Jt][2][CS4] float
  o = al(o + sizeof(float) * (size_t)(ZM * d.Jt * 2 * CS4));
  off[3] = o;  // w: [CLW][CS4], CLW = Cl rounded up to the kernel's channel bound
  o = al(o + sizeof(float) * (size_t)(epi_clm(Cl) * CS4));
  off[4] = o;  // bias: [CS4]
  o = al(o + sizeof(float) * (size_t)CS4);
  off[5] = o;  // DA: x tile [Cl][P+1]
  if (mode == EPI_DA) o = al(o + sizeof(float) * (size_t)(Cl * (P + 1)));
  off[6] = o;  // DA: dA tile [CS4][P+1]
  if (mode == EPI_DA) o = al(o + sizeof(float) * (size_t)(CS4 * (P + 1)));
  // DA: Kahan (sum, compensation) pairs [IB*OB - 128][2][16] of the 4x4 (i, o)
  // blocks beyond the first 128 (each thread keeps its first block in
  // registers).  Placed past the first 8 KB, which the final reduction reuses
  // for the register-held sums.
  if (mode == EPI_DA) o = std::max(o, (size_t)(128 * 16 * sizeof(float)));
  off[7] = o;
  if (mode == EPI_DA) {
    const int nblk = ((Cl + 1 + 3) / 4) * (CS4 / 4);
    if (nblk > 128) o = al(o + sizeof(float) * 32 * (size_t)(nblk - 128));
  }
  total = o;
}

size_t epilogue_smem_bytes(const Dims& d, int mode, int Cs, int Cl) {
  size_t off[8], total;
  epi_layout(d, mode, Cs, Cl, off, total);
  // in DA mode the final reduction reuses the first 8 KB (128 items x 16
  // sums), which epi_layout already keeps below the spill region
  return total;
}

int epilogue_max_grid() { return 1024; }

template <int MODE, int CLM, int JTM, bool EO>
__global__ void __launch_bounds__(128, 4) k_epi_f32(const EpiK k) {
  extern __shared__ float4 smem4[];
  const EpiArgs& a = k.a;
  const int Cs = a.Cs, Cl = (MODE == EPI_SPECTRAL) ? 0 : a.Cl;
  constexpr bool TWO = EO && MODE != EPI_DA;  // two points (t, t + Nt / 2) per thread
  const int Jz = k.Jz, Jt = k.Jt, Nz = k.Nz, mz = k.mz, P = k.P, CS4 = k.CS4;
  const int Nt = TWO ? k.Nt / 2 : k.Nt;  // t positions of a tile's points
  const int PP = P + 1;
  unsigned char* base = reinterpret_cast<unsigned char*>(smem4);
  float4* eo = reinterpret_cast<float4*>(base + k.off[0]);
  float2* cs = reinterpret_cast<float2*>(base + k.off[1]);
  float* qs = reinterpret_cast<float*>(base + k.off[2]);
  float* sw = reinterpret_cast<float*>(base + k.off[3]);
  float* sbias = reinterpret_cast<float*>(base + k.off[4]);
  float* sx = reinterpret_cast<float*>(base + k.off[5]);
  float* sda = reinterpret_cast<float*>(base + k.off[6]);
  const int tid = threadIdx.x;

  for (int e = tid; e < Nz * (mz + 1); e += 128) {
    const int z = e / (mz + 1), kk = e - z * (mz + 1);
    const float2 f = a.Iz[z * Jz + kk];  // jz = kk: kz = kk (kk < mz), kz = -mz (kk = mz)
    cs[e] = (kk < mz) ? f : make_float2(f.x, -f.y);
  }
  if (MODE != EPI_SPECTRAL) {
    for (int e = tid; e < k.CLW * CS4; e += 128) {
      const int i = e / CS4, c = e - i * CS4;
      sw[e] = (c < Cs && i < Cl) ? a.wlin[(long long)i * a.w_si + (long long)c * a.w_sc] : 0.f;
    }
  }
  for (int c = tid; c < CS4; c += 128)
    sbias[c] = ((MODE == EPI_FWD || MODE == EPI_DA) && c < Cs) ? a.bias[c] : 0.f;

  // this thread's point is p of each tile; its t (and so the inverse-t
  // factors) changes between tiles only when Nt does not divide 128
  const int p = tid;
  int cur_t = -1;
  float itr[JTM], iti[JTM];
  float osign = 1.f;  // EO, dA mode: the sign of the odd kt at this thread's t

  // EPI_DA: work items are (4x4 block of (i, o), point group) pairs, item
  // it = g * nblk + block.  KG point groups split the points when there are
  // fewer than 128 blocks; with more (KG = 1), a thread owns blocks tid,
  // tid + 128, ...  Its first item's Kahan running sums live in registers, the
  // others' in shared memory (racc).
  const int nblk = k.IB * k.OB;
  const int nitem = nblk * k.KG;
  const bool wthread = (MODE == EPI_DA) && tid < nitem;
  float* racc = reinterpret_cast<float*>(base + k.off[7]);
  if (MODE == EPI_DA)
    for (int e = tid; e < (nitem - 128) * 32; e += 128) racc[e] = 0.f;
  float wsum[16], wcmp[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    wsum[q] = 0.f;
    wcmp[q] = 0.f;
  }

  const long long plane = (long long)Nz * Nt;
  const long long chan = k.NxNy * (TWO ? 2 * plane : plane);
  const long long t_begin = k.ntiles * blockIdx.x / gridDim.x;
  const long long t_end = k.ntiles * (blockIdx.x + 1) / gridDim.x;
  long long cur_col = -1;
  for (long long tau = t_begin; tau < t_end; ++tau) {
    const long long col = tau / k.nzc;
    const long long s0 = (tau - col * k.nzc) * kEpiP;  // first point of the tile in the column
    const int valid = (int)min((long long)kEpiP, plane - s0);
    const int z0 = (int)(s0 / Nt);                      // first plane the tile touches
    const int tf = (int)(s0 - (long long)z0 * Nt);      // its first point's t
    const int zn = (tf + valid - 1) / Nt + 1;           // planes touched, <= ZM
    const long long b = col / k.NxNy, xy = col - b * k.NxNy;
    const int zz_p = (tf + p) / Nt, t = (tf + p) - zz_p * Nt;
    if (t != cur_t) {
      const int tb = (EO && !TWO && t >= k.Nt / 2) ? t - k.Nt / 2 : t;
      if (EO && !TWO) osign = tb == t ? 1.f : -1.f;
#pragma unroll
      for (int jt = 0; jt < JTM; ++jt) {
        if (jt < Jt) {
          const float2 f = __ldg(a.It + jt * k.Nt + tb);
          itr[jt] = f.x;
          iti[jt] = -f.y;
        } else {
          itr[jt] = 0.f;
          iti[jt] = 0.f;
        }
      }
      cur_t = t;
    }
    __syncthreads();  // previous tile's shared-memory reads are done
    if (col != cur_col) {
      const int JZT = Jz * Jt;
      const int neo = Cs * Jt * (mz + 1);
      for (int e0 = tid; e0 < neo; e0 += 4 * 128) {
        float2 av[4], mv[4];
#pragma unroll
        for (int u4 = 0; u4 < 4; ++u4) {
          const int e = e0 + u4 * 128;
          av[u4] = make_float2(0.f, 0.f);
          mv[u4] = make_float2(0.f, 0.f);
          if (e < neo) {
            const int kk = e % (mz + 1), jt = (e / (mz + 1)) % Jt, c = e / ((mz + 1) * Jt);
            const float2* u = a.U + ((b * Cs + c) * k.NxNy + xy) * JZT + jt;
            if (kk < mz) av[u4] = __ldg(u + kk * Jt);
            if (kk > 0) mv[u4] = __ldg(u + (2 * mz - kk) * Jt);
          }
        }
#pragma unroll
        for (int u4 = 0; u4 < 4; ++u4) {
          const int e = e0 + u4 * 128;
          if (e < neo) {
            const float2 av_ = av[u4], mv_ = mv[u4];
            eo[e] = make_float4(av_.x + mv_.x, av_.y + mv_.y, av_.x - mv_.x, av_.y - mv_.y);
          }
        }
      }
      cur_col = col;
      __syncthreads();
    }
    // lin inputs of this point (issued early; consumed after Q is ready)
    float x[CLM > 0 ? CLM : 1], x2[TWO && CLM > 0 ? CLM : 1];
    const long long pofs =
        TWO ? xy * 2 * plane + (long long)(z0 + zz_p) * k.Nt + t : xy * plane + s0 + p;
    const bool pv = p < valid;
    if (MODE != EPI_SPECTRAL) {
      const float* xp = a.lin_in + (b * Cl) * chan + pofs;
#pragma unroll
      for (int i = 0; i < CLM; ++i) {
        x[i] = (i < Cl && pv) ? __ldg(xp + (long long)i * chan) : 0.f;
        if (TWO) x2[TWO ? i : 0] = (i < Cl && pv) ? __ldg(xp + (long long)i * chan + Nt) : 0.f;
      }
    }
    // Q of this tile's planes: one (o, jt, zz) unit per step
    {
      const int units = Cs * Jt * zn;
      for (int e = tid; e < units; e += 128) {
        const int zz = e % zn, cj = e / zn;
        const int jt = cj % Jt, c = cj / Jt;
        const float4* src = eo + (size_t)(c * Jt + jt) * (mz + 1);
        const float2* cz = cs + (size_t)(z0 + zz) * (mz + 1);
        float qr = 0.f, qi = 0.f, qr2 = 0.f, qi2 = 0.f;
        int kk = 0;
        for (; kk + 1 <= mz; kk += 2) {
          const float4 r0 = src[kk], r1 = src[kk + 1];
          const float2 t0 = cz[kk], t1 = cz[kk + 1];
          qr = fmaf(r0.x, t0.x, qr);
          qr = fmaf(-r0.w, t0.y, qr);
          qi = fmaf(r0.y, t0.x, qi);
          qi = fmaf(r0.z, t0.y, qi);
          qr2 = fmaf(r1.x, t1.x, qr2);
          qr2 = fmaf(-r1.w, t1.y, qr2);
          qi2 = fmaf(r1.y, t1.x, qi2);
          qi2 = fmaf(r1.z, t1.y, qi2);
        }
        if (kk <= mz) {
          const float4 r0 = src[kk];
          const float2 t0 = cz[kk];
          qr = fmaf(r0.x, t0.x, qr);
          qr = fmaf(-r0.w, t0.y, qr);
          qi = fmaf(r0.y, t0.x, qi);
          qi = fmaf(r0.z, t0.y, qi);
        }
        float* qd = qs + ((size_t)(zz * Jt + jt) * 2) * CS4 + c;
        qd[0] = qr + qr2;
        qd[CS4] = qi + qi2;
      }
      // zero the padded output columns once per tile (read by the vector loads)
      for (int e = tid; e < zn * Jt * 2 * (CS4 - Cs); e += 128) {
        const int c = Cs + e % (CS4 - Cs), r = e / (CS4 - Cs);
        qs[(size_t)r * CS4 + c] = 0.f;
      }
    }
    __syncthreads();
    // per point: 4 outputs at a time (only threads that own a point of this tile)
    if (pv) {
      const float* qp = qs + (size_t)(zz_p * Jt) * 2 * CS4;
      float* optr = a.out + (b * Cs) * chan + pofs;
      const float* dzp = (MODE == EPI_DA) ? a.dz + (b * Cs) * chan + pofs : nullptr;
      for (int c0 = 0; c0 < Cs; c0 += 4) {
        float dzq[4];
        if (MODE == EPI_DA) {
#pragma unroll
          for (int q = 0; q < 4; ++q) dzq[q] = (c0 + q < Cs) ? __ldg(dzp + (long long)(c0 + q) * chan) : 0.f;
        }
        float4 acc = *reinterpret_cast<const float4*>(sbias + c0);
        float4 odd = make_float4(0.f, 0.f, 0.f, 0.f);  // EO: the odd kt
#pragma unroll
        for (int jt = 0; jt < JTM; ++jt) {
          if (jt < Jt) {
            const float4 qr = *reinterpret_cast<const float4*>(qp + (size_t)(jt * 2) * CS4 + c0);
            const float4 qi = *reinterpret_cast<const float4*>(qp + (size_t)(jt * 2 + 1) * CS4 + c0);
            float4& s = (EO && (jt & 1)) ? odd : acc;
            s.x = fmaf(qr.x, itr[jt], fmaf(qi.x, iti[jt], s.x));
            s.y = fmaf(qr.y, itr[jt], fmaf(qi.y, iti[jt], s.y));
            s.z = fmaf(qr.z, itr[jt], fmaf(qi.z, iti[jt], s.z));
            s.w = fmaf(qr.w, itr[jt], fmaf(qi.w, iti[jt], s.w));
          }
        }
        float4 acc2 = acc;  // TWO: the point at t + Nt / 2
        if (TWO) {
          acc2 = make_float4(acc.x - odd.x, acc.y - odd.y, acc.z - odd.z, acc.w - odd.w);
          acc = make_float4(acc.x + odd.x, acc.y + odd.y, acc.z + odd.z, acc.w + odd.w);
        } else if (EO) {
          acc = make_float4(acc.x + osign * odd.x, acc.y + osign * odd.y, acc.z + osign * odd.z, acc.w + osign * odd.w);
        }
        if (MODE != EPI_SPECTRAL) {
          const float* wp = sw + c0;
#pragma unroll
          for (int i = 0; i < CLM; ++i) {
            const float4 w4 = *reinterpret_cast<const float4*>(wp + (size_t)i * CS4);
            acc.x = fmaf(w4.x, x[i], acc.x);
            acc.y = fmaf(w4.y, x[i], acc.y);
            acc.z = fmaf(w4.z, x[i], acc.z);
            acc.w = fmaf(w4.w, x[i], acc.w);
            if (TWO) {
              const float v = x2[TWO ? i : 0];
              acc2.x = fmaf(w4.x, v, acc2.x);
              acc2.y = fmaf(w4.y, v, acc2.y);
              acc2.z = fmaf(w4.z, v, acc2.z);
              acc2.w = fmaf(w4.w, v, acc2.w);
            }
          }
        }
        const float av[4] = {acc.x, acc.y, acc.z, acc.w};
        const float av2[4] = {acc2.x, acc2.y, acc2.z, acc2.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int c = c0 + q;
          if (c < Cs) {
            float* o = optr + (long long)c * chan;
            if (MODE == EPI_FWD) {
              *o = gelu_f(av[q]);
              if (TWO) o[Nt] = gelu_f(av2[q]);
              if (a.gp) {  // training forward
                a.gp[o - a.out] = gelu_grad_f(av[q]);
                if (TWO) a.gp[o - a.out + Nt] = gelu_grad_f(av2[q]);
              }
            } else if (MODE == EPI_DA) {
              const float da = dzq[q] * gelu_grad_f(av[q]);
              *o = da;
              sda[c * PP + p] = da;
            } else {
              *o = av[q];
              if (TWO) o[Nt] = av2[q];
            }
          } else if (MODE == EPI_DA && c < CS4) {
            sda[c * PP + p] = 0.f;
          }
        }
      }
    }
    if (MODE == EPI_DA) {
      if (p < P) {
        if (!pv)
          for (int c = 0; c < CS4; ++c) sda[c * PP + p] = 0.f;
#pragma unroll
        for (int i = 0; i < CLM; ++i)
          if (i < Cl) sx[i * PP + p] = x[i];
      }
      __syncthreads();
      if (wthread) {
        for (int it = tid; it < nitem; it += 128) {
          const int bl = it % nblk, kg = it / nblk;
          const int i0 = (bl / k.OB) * 4, o0w = (bl % k.OB) * 4;
          const int pa = kg * P / k.KG, pb = min((kg + 1) * P / k.KG, valid);
          float part[16];
#pragma unroll
          for (int q = 0; q < 16; ++q) part[q] = 0.f;
          for (int pt = pa; pt < pb; ++pt) {
            float xv[4], dv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int i = i0 + u;
              xv[u] = i < Cl ? sx[i * PP + pt] : (i == Cl ? 1.f : 0.f);
              dv[u] = sda[(o0w + u) * PP + pt];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
              for (int v = 0; v < 4; ++v) part[u * 4 + v] = fmaf(xv[u], dv[v], part[u * 4 + v]);
          }
          if (it < 128) {
#pragma unroll
            for (int q = 0; q < 16; ++q) {
              const float y = part[q] - wcmp[q];
              const float s = wsum[q] + y;
              wcmp[q] = (s - wsum[q]) - y;
              wsum[q] = s;
            }
          } else {
            float* r = racc + (it - 128) * 32;
#pragma unroll
            for (int q = 0; q < 16; ++q) {
              const float y = part[q] - r[16 + q];
              const float s = r[q] + y;
              r[16 + q] = (s - r[q]) - y;
              r[q] = s;
            }
          }
        }
      }
    }
  }
  if (MODE == EPI_DA) {
    __syncthreads();
    float* red = reinterpret_cast<float*>(base);
    if (wthread) {
#pragma unroll
      for (int q = 0; q < 16; ++q) red[tid * 16 + q] = wsum[q] - wcmp[q];
    }
    __syncthreads();
    const int npair = Cl * Cs + Cs;
    for (int e = tid; e < nblk * 16; e += 128) {
      const int bl = e / 16, q = e % 16;
      const int i = (bl / k.OB) * 4 + q / 4, c = (bl % k.OB) * 4 + q % 4;
      float s = 0.f, comp = 0.f;
      for (int g = 0; g < k.KG; ++g) {
        const int it = g * nblk + bl;
        const float v = it < 128 ? red[it * 16 + q]
                                 : racc[(it - 128) * 32 + q] - racc[(it - 128) * 32 + 16 + q];
        const float y = v - comp;
        const float tt = s + y;
        comp = (tt - s) - y;
        s = tt;
      }
      if (c < Cs && i <= Cl) {
        const int idx = (i < Cl) ? i * Cs + c : Cl * Cs + c;
        a.part[(long long)blockIdx.x * npair + idx] = s;
      }
    }
  }
}

// Even Nt with two points per thread (see the top): by the sizes of the block
// alone, so that the forward and the dA mode agree.  Not where a column is one tile
// either way, whose threads then are half idle (forward at 20 channels, 64 x 64 x 8 x
// 4: 53 us with one point, 70 with two), and not where rows of an odd, small number of
// pairs, which tiles cut, meet tiles that are not half as many and more than 12
// channels (20 channels, 32 x 32 x 64 x 14: 176 and 195, spectral form 129 and 157; 24
// at 64 x 32 x 64 x 10: 304 and 342; 4 at 64 x 64 x 64 x 10: 123 and 109).
static Dims half_t(Dims d) {
  d.Nt /= 2;
  return d;
}
static bool epi_even_odd(const Dims& d, int Cs, int Cl) {
  if (d.Nt % 2 != 0 || d.Jt > 8 || Cl > 32) return false;
  const int64_t points = (d.Nz * d.Nt + kEpiP - 1) / kEpiP, pairs = (d.Nz * d.Nt / 2 + kEpiP - 1) / kEpiP;
  if (pairs == points) return false;
  if (2 * pairs > points && d.Nt < 16 && d.Nt % 4 != 0 && std::max(Cs, Cl) > 12) return false;
  return epilogue_smem_bytes(half_t(d), EPI_FWD, Cs, Cl) <= 56 * 1024;
}

template <int MODE, int CLM, int JTM, bool EO>
static cudaError_t launch_epi_t(const Dims& d0, const EpiArgs& a, int* grid_used, cudaStream_t s) {
  const Dims d = (EO && MODE != EPI_DA) ? half_t(d0) : d0;  // tiles of points or of pairs
  EpiK k{};
  k.a = a;
  k.NxNy = d.Nx * d.Ny;
  k.Nz = (int)d.Nz;
  k.Nt = (int)d0.Nt;
  k.Jz = (int)d.Jz;
  k.Jt = (int)d.Jt;
  k.mz = (int)d.mz;
  k.ZM = epi_planes(d);
  k.P = epi_points(d);
  k.nzc = (d.Nz * d.Nt + kEpiP - 1) / kEpiP;
  k.CS4 = (a.Cs + 3) / 4 * 4;
  const int Cl = MODE == EPI_SPECTRAL ? 0 : a.Cl;
  k.IB = (Cl + 1 + 3) / 4;
  k.OB = k.CS4 / 4;
  k.KG = std::max(1, 128 / (k.IB * k.OB));
  k.CLW = epi_clm(Cl);
  k.ntiles = d.B * d.Nx * d.Ny * (long long)k.nzc;
  {
    size_t off[8], total;
    epi_layout(d, MODE, a.Cs, Cl, off, total);
    for (int q = 0; q < 8; ++q) k.off[q] = (uint32_t)off[q];
  }
  const size_t smem = epilogue_smem_bytes(d, MODE, a.Cs, Cl);
  const void* kern = (const void*)k_epi_f32<MODE, CLM, JTM, EO>;
  cudaError_t e = allow_smem(kern, smem);
  if (e != cudaSuccess) return e;
  int grid = persistent_grid(kern, 128, smem, k.ntiles);
  if (grid > epilogue_max_grid()) grid = epilogue_max_grid();
  if (grid_used) *grid_used = grid;
  static const char* names[4] = {"fno_epi_spectral_f32", "fno_epi_fwd_f32", "fno_epi_da_f32",
                                 "fno_epi_dx_f32"};
  // the forward of a training step also stores GELU'(A)
  const char* name = (MODE == EPI_FWD && a.gp) ? "fno_epi_fwd_train_f32" : names[MODE];
  FNO_LAUNCH(name, (k_epi_f32<MODE, CLM, JTM, EO>), grid, 128, smem, s, k);
  return cudaSuccess;
}

template <int MODE, int JTM, bool EO>
static cudaError_t launch_epi_j(const Dims& d, const EpiArgs& a, int* g, cudaStream_t s) {
  if constexpr (MODE == EPI_SPECTRAL) {
    return launch_epi_t<MODE, 0, JTM, EO>(d, a, g, s);
  } else {
    switch (epi_clm(a.Cl)) {
      case 4: return launch_epi_t<MODE, 4, JTM, EO>(d, a, g, s);
      case 8: return launch_epi_t<MODE, 8, JTM, EO>(d, a, g, s);
      case 12: return launch_epi_t<MODE, 12, JTM, EO>(d, a, g, s);
      case 16: return launch_epi_t<MODE, 16, JTM, EO>(d, a, g, s);
      case 20: return launch_epi_t<MODE, 20, JTM, EO>(d, a, g, s);
      case 24: return launch_epi_t<MODE, 24, JTM, EO>(d, a, g, s);
      case 32: return launch_epi_t<MODE, 32, JTM, EO>(d, a, g, s);
      default: break;
    }
    if constexpr (!EO) {
      if (epi_clm(a.Cl) == 48) return launch_epi_t<MODE, 48, JTM, EO>(d, a, g, s);
      return launch_epi_t<MODE, 64, JTM, EO>(d, a, g, s);
    } else {
      return cudaErrorInvalidValue;  // not reached: EO has at most 32 inputs
    }
  }
}

template <int MODE>
static cudaError_t launch_epi_m(const Dims& d, const EpiArgs& a, int* g, cudaStream_t s) {
  const int Cl = MODE == EPI_SPECTRAL ? 0 : a.Cl;
  if (epi_even_odd(d, a.Cs, Cl)) return launch_epi_j<MODE, 8, true>(d, a, g, s);
  if (d.Jt <= 8) return launch_epi_j<MODE, 8, false>(d, a, g, s);
  return launch_epi_j<MODE, 16, false>(d, a, g, s);
}

cudaError_t launch_epilogue_f32(const Dims& d, const EpiArgs& a, int* grid_used, cudaStream_t s) {
  if (d.B <= 0) {
    if (grid_used) *grid_used = 0;
    return cudaSuccess;
  }
  switch (a.mode) {
    case EPI_SPECTRAL: return launch_epi_m<EPI_SPECTRAL>(d, a, grid_used, s);
    case EPI_FWD: return launch_epi_m<EPI_FWD>(d, a, grid_used, s);
    case EPI_DA: return launch_epi_m<EPI_DA>(d, a, grid_used, s);
    default: return launch_epi_m<EPI_DX>(d, a, grid_used, s);
  }
}

// ---------------------------------------------------------------------------
// Final reduction of the per-CTA partial sums (Kahan-compensated, fixed order)
// and a zero fill.
// ---------------------------------------------------------------------------
__global__ void k_reduce_parts(const float* __restrict__ part, int rows, int npair, int CiCo,
                               float* __restrict__ dwl, float* __restrict__ db) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= npair) return;
  float sum = 0.f, comp = 0.f;
  for (int r = 0; r < rows; ++r) {
    float y = part[(long long)r * npair + e] - comp;
    float t = sum + y;
    comp = (t - sum) - y;
    sum = t;
  }
  if (e < CiCo)
    dwl[e] = sum;
  else
    db[e - CiCo] = sum;
}

cudaError_t launch_reduce_partials(const float* part, int rows, int Ci, int Co, float* dwl,
                                   float* db, cudaStream_t s) {
  const int npair = Ci * Co + Co;
  FNO_LAUNCH("fno_reduce_partials", k_reduce_parts, (npair + 127) / 128, 128, 0, s, part, rows,
             npair, Ci * Co, dwl, db);
  return cudaSuccess;
}

__global__ void k_fill_zero(float* __restrict__ p, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    p[i] = 0.f;
}

cudaError_t launch_fill_zero(float* p, int64_t n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  int blocks = (int)std::min<int64_t>((n + 255) / 256, 4096);
  FNO_LAUNCH("fno_fill_zero", k_fill_zero, blocks, 256, 0, s, p, (long long)n);
  return cudaSuccess;
}

}  // namespace fno
