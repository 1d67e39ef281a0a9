// fno_epi_col.cu -- the last stage of the inverse transform of Alg. 2 (inverse
// z, then inverse t; Sec. IV-C runs the inverse as the adjoint of the forward
// DFT) fused with the block's pointwise 1x1 channel linear, bias and GELU, for
// split BF16 and any even Nt up to 128 (modes EPI_FWD, EPI_DX and EPI_SPECTRAL), and
// for plain BF16 in the last two.
//
// Work unit: 16 z-planes of one (b, x, y) column, every channel, by a CTA of
// four to eight warps.
//   z phase: the warps share the output channel pairs.  For each channel o
//       V[z][kt] = sum_kz U[o][kz][kt] Iz[z][kz]   (complex)
//     as mma.sync m16n8k16 with A = the z basis (rows z, k = (kz, re/im)) and
//     B = the column's spectrum, staged by cp.async (the pair (re, im) of one
//     kz is one 32-bit B register, so U enters as it lies in memory).  The
//     fragments of V, split into BF16 parts, are exactly the A fragments of the
//     t phase: rows g of one fragment are 8 planes of the pair's first channel,
//     rows g + 8 the same planes of its second channel.  They pass through
//     shared memory to the warps that need them.
//   t phase: a warp takes 8 planes x 8 H points (H = 2, or 1 where Nt <= 16).
//     Its lane holds 2 H points of every input channel in registers (all loads
//     in flight at once; with H = 2 the first item's are issued before the z
//     phase) and walks the channel pairs:
//       S[o][z][t] = sum_kt V[o][z][kt] It[kt][t]   (mma.sync)
//       A = bias + sum_i W[i][o] x[i][z][t] + S     (FP32, packed FMAs)
//     then GELU (and GELU'), two values per instruction, and the stores.
//
// What bounds it.  HBM asks for 2.46 ms (forward with GELU') and 1.66 ms (dX) at
// 128^3 x 32, width 20; measured 3.48 and 2.61 ms (the tcgen05 form: 4.58 and
// 4.04).  Neither the tensor pipe nor the FMA pipe is full (a t phase without
// memory or z phase takes 2.8 and 1.9 ms): warps wait on one another's phases,
// with 12 warps on an SM.  Measured on the way, forward + dX at that size:
//   TF32 in place of BF16 parts in the DFT stages       6.90 ms
//   x staged by cp.async a unit ahead, 8 warps on an SM 9.62 ms
//   three CTAs of 168 registers or four of 128          6.20 / 6.26 ms
//   x loads before the z phase instead of after         6.08 ms
//   every warp alone with the 1x1 on mma.sync (3xTF32)  9.25 ms
// A packed FMA takes 2.3 cycles a scheduler, an mma.sync of this shape 8 (tf32
// m16n8k8 as well, for half the products).  At Nt = 84 and 86 a unit has twelve
// items, and what decides is L1: rows of 336 or 344 bytes share sectors and lines
// between items.  Training forward + dX at 262 x 118 x 64 x 86 and training forward
// (with GELU'(A)) at 130^3 x 84:
// two CTAs of six warps 18.4 and 12.4 ms, two of four 20.7 and 13.8, three of
// four 22.1 and 17.8, one of eight 24.6 and 16.5 (synthesis path 34.0 and 20.7;
// HBM asks for 10.4 and 6.6).  A form that took 14 ms for the forward there took 9
// with its two stores left out and no less without the loads of x: the partly
// written sectors of 8-byte-aligned rows are the likely reason, not a measured one.
//
// Precision (accumulation FP32; the 1x1 is FP32, its operands rounded to BF16
// before it where lin_round says so).  U, V and the bases enter as NP BF16
// parts: 3 with six products, 2 with three, 1 with one.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "fno_internal.h"
#include "packed_math.h"
#include "warp_mma.h"

namespace fno {

namespace {

// the products of NP-part operands that are kept, small terms first
template <int NP>
struct Prods;
template <>
struct Prods<3> {
  static constexpr int n = 6;
  static __device__ constexpr int a(int q) { return q == 0 ? 2 : q == 2 || q == 3 ? 1 : 0; }
  static __device__ constexpr int b(int q) { return q == 1 ? 2 : q == 2 || q == 4 ? 1 : 0; }
};
template <>
struct Prods<2> {
  static constexpr int n = 3;
  static __device__ constexpr int a(int q) { return q == 0 ? 1 : 0; }
  static __device__ constexpr int b(int q) { return q == 1 ? 1 : 0; }
};
template <>
struct Prods<1> {
  static constexpr int n = 1;
  static __device__ constexpr int a(int) { return 0; }
  static __device__ constexpr int b(int) { return 0; }
};

// BF16 parts of two floats, packed in pairs
template <int NP>
__device__ __forceinline__ void bf16_parts(float a, float b, uint32_t (&p)[NP]) {
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    p[q] = *reinterpret_cast<const uint32_t*>(&h);
    if (q + 1 < NP) {
      const float2 f = __bfloat1622float2(h);
      a -= f.x;
      b -= f.y;
    }
  }
}

}  // namespace

struct EpiCol {
  EpiArgs a;
  const uint4* zf;  // z basis A fragments [NZ16][KS][3 parts][32 lanes]
  const uint2* tf;  // t basis B fragments [NTT][2][3 parts][32 lanes]
  long long NxNy, plane, chan;
  unsigned nunits;
  int Nz, Nt, Jz, Jt, KS, NZ16, NPAIR;
  int NTI;        // t items of 8 H points
  int perm;       // t mapping: a lane's four points are consecutive
  int lin_round;  // 1x1 operands rounded to BF16
};

__device__ __forceinline__ float lin_round(float v, int on) {
  return on ? __bfloat162float(__float2bfloat16_rn(v)) : v;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One t-phase item: the NPAIR channel pairs at this lane's points, H
// sub-tiles of 8 points.
template <int MODE, int CM, int NP, int H, int CH>
__device__ __forceinline__ void col_item(const EpiCol& k, const uint4* sV, const uint4* sT, const ulonglong2* sW,
                                         const float2* sB, const u64 (&x)[CM > 0 ? CM : 1][H], char* out, char* gp,
                                         uint32_t pos, bool ok0, bool ok1) {
  typedef Prods<NP> P;
  const long long chan = 4 * k.chan;
  const int Cs = k.a.Cs;
#pragma unroll 1
  for (int p = 0; p < k.NPAIR; ++p) {
    float s[H][4];
#pragma unroll
    for (int h = 0; h < H; ++h)
#pragma unroll
      for (int q = 0; q < 4; ++q) s[h][q] = 0.f;
    uint4 A[NP], tb[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      A[q] = sV[(p * 2 * NP + q) * 32];
      tb[q] = sT[q * 32];
    }
#pragma unroll
    for (int q = 0; q < P::n; ++q)
#pragma unroll
      for (int h = 0; h < H; ++h) {
        const uint4 f = A[P::a(q)], t = tb[P::b(q)];
        wm::mma16(s[h], f.x, f.y, f.z, f.w, h == 0 ? t.x : t.z, h == 0 ? t.y : t.w);
      }
    // the 1x1 in CH chains of FP32 sums, the first from the bias; S starts the second
    // chain of several and is added to a single one
    constexpr int K = CH > 2 ? CH : 2;
    auto chain = [](int i) { return CH == 1 ? 0 : CH * i / CM; };
    u64 a1[K][H], a2[K][H];
    const float2 bias = (MODE == EPI_FWD) ? sB[p] : make_float2(0.f, 0.f);
#pragma unroll
    for (int h = 0; h < H; ++h) {
      a1[0][h] = pack2(bias.x, bias.x);
      a2[0][h] = pack2(bias.y, bias.y);
      a1[1][h] = pack2(s[h][0], s[h][1]);
      a2[1][h] = pack2(s[h][2], s[h][3]);
#pragma unroll
      for (int q = 2; q < K; ++q) a1[q][h] = a2[q][h] = 0;
    }
    if (MODE != EPI_SPECTRAL) {
      const ulonglong2* w = sW + p * CM;
#pragma unroll
      for (int i = 0; i < CM; ++i) {
        const ulonglong2 wv = w[i];
#pragma unroll
        for (int h = 0; h < H; ++h) {
          fma2(a1[chain(i)][h], wv.x, x[i][h]);
          fma2(a2[chain(i)][h], wv.y, x[i][h]);
        }
      }
    }
#pragma unroll
    for (int h = 0; h < H; ++h) {
#pragma unroll
      for (int q = 2; q < K; ++q) {
        a1[q - 2][h] = add2(a1[q - 2][h], a1[q][h]);
        a2[q - 2][h] = add2(a2[q - 2][h], a2[q][h]);
      }
      a1[0][h] = add2(a1[0][h], a1[1][h]);
      a2[0][h] = add2(a2[0][h], a2[1][h]);
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      u64 z[H], d[H];
#pragma unroll
      for (int h = 0; h < H; ++h) {
        z[h] = c == 0 ? a1[0][h] : a2[0][h];
        if (MODE == EPI_FWD) gelu2(z[h], z[h], d[h]);
      }
      if (2 * p + c < Cs) {
        char* op = out + c * chan + pos;
        char* dp = gp + c * chan + pos;
        if (H == 2 && k.perm) {
          if (ok0) {
            *reinterpret_cast<ulonglong2*>(op) = make_ulonglong2(z[0], z[H - 1]);
            if (MODE == EPI_FWD && k.a.gp) *reinterpret_cast<ulonglong2*>(dp) = make_ulonglong2(d[0], d[H - 1]);
          }
        } else {
          if (ok0) *reinterpret_cast<u64*>(op) = z[0];
          if (H == 2 && ok1) *reinterpret_cast<u64*>(op + 32) = z[H - 1];
          if (MODE == EPI_FWD && k.a.gp) {
            if (ok0) *reinterpret_cast<u64*>(dp) = d[0];
            if (H == 2 && ok1) *reinterpret_cast<u64*>(dp + 32) = d[H - 1];
          }
        }
      }
    }
    out += 2 * chan;
    gp += 2 * chan;
  }
}

// CM: bound of the 1x1 input channels (register array), 0 for EPI_SPECTRAL.
// H: sub-tiles of 8 t points of an item.  CH: chains of the 1x1's sums (1, 2, 4).
template <int MODE, int CM, int NP, int H, int CH, int NW, int MINB>
__global__ void __launch_bounds__(32 * NW, MINB) k_epi_col(const __grid_constant__ EpiCol k) {
  typedef Prods<NP> P;
  extern __shared__ __align__(16) unsigned char smem_col[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // uniform
  const int g = lane >> 2, q4 = lane & 3;
  const EpiArgs& a = k.a;
  const int NPAIR = k.NPAIR, Nt = k.Nt, Nz = k.Nz, Jt = k.Jt, Jz = k.Jz, KS = k.KS, JZT = Jz * Jt;
  uint4* sV = reinterpret_cast<uint4*>(smem_col);                          // [NPAIR][2 halves][NP][32]: A fragments
  uint4* sT = sV + NPAIR * 2 * NP * 32;                                    // [NTI][NP][32]: B fragments of sub-tiles 0, 1
  ulonglong2* sW = reinterpret_cast<ulonglong2*>(sT + k.NTI * NP * 32);    // [NPAIR][CM]: (w1, w1), (w2, w2)
  float2* sB = reinterpret_cast<float2*>(sW + NPAIR * CM);       // [NPAIR]
  float2* sU = sB + ((NPAIR + 1) & ~1);                          // [Cs][Jz][Jt]

  if (MODE != EPI_SPECTRAL)
    for (int e = tid; e < NPAIR * CM; e += 32 * NW) {
      const int p = e / (CM > 0 ? CM : 1), i = e - p * CM;
      float w[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int o = 2 * p + c;
        w[c] = (o < a.Cs && i < a.Cl)
                   ? lin_round(a.wlin[(long long)i * a.w_si + (long long)o * a.w_sc], k.lin_round)
                   : 0.f;
      }
      sW[e] = make_ulonglong2(pack2(w[0], w[0]), pack2(w[1], w[1]));
    }
  if (MODE == EPI_FWD)
    for (int p = tid; p < NPAIR; p += 32 * NW)
      sB[p] = make_float2(a.bias[2 * p], 2 * p + 1 < a.Cs ? a.bias[2 * p + 1] : 0.f);
  for (int e = tid; e < k.NTI * NP * 32; e += 32 * NW) {
    const int ln = e % 32, q = e / 32 % NP, t8 = H * (e / (32 * NP));
    const uint2 lo = k.tf[(t8 * 3 + q) * 32 + ln];
    const uint2 hi = (H == 2) ? k.tf[((t8 + 1) * 3 + q) * 32 + ln] : make_uint2(0u, 0u);
    sT[e] = make_uint4(lo.x, lo.y, hi.x, hi.y);
  }

  // the spectrum of a column, channel by channel
  const uint32_t dU = static_cast<uint32_t>(__cvta_generic_to_shared(sU));
  const int uchunks = JZT / 2;  // 16-byte chunks of a channel (Jz is even)
  auto fetch_u = [&](unsigned col) {
    const unsigned b = col / (unsigned)k.NxNy, xy = col - b * (unsigned)k.NxNy;
    const char* src = reinterpret_cast<const char*>(a.U) + 8 * ((long long)b * a.Cs * k.NxNy + xy) * JZT;
    const long long us = 8 * k.NxNy * (long long)JZT;
    for (int e = tid; e < a.Cs * uchunks; e += 32 * NW) {
      const int o = e / uchunks, r = e - o * uchunks;
      cp_async16(dU + 16 * e, src + o * us + 16 * r);
    }
  };

  // a contiguous range of units: U is fetched once a column
  const unsigned u0 = (unsigned)((unsigned long long)k.nunits * blockIdx.x / gridDim.x);
  const unsigned u1 = (unsigned)((unsigned long long)k.nunits * (blockIdx.x + 1) / gridDim.x);
  if (u0 >= u1) return;
  unsigned col = u0 / (unsigned)k.NZ16;
  int z16 = (int)(u0 - col * (unsigned)k.NZ16);
  fetch_u(col);
  const int ukt = min(g, Jt - 1);
  for (unsigned u = u0; u < u1; ++u) {
    const unsigned b = col / (unsigned)k.NxNy, xy = col - b * (unsigned)k.NxNy;
    cp_async_wait();
    __syncthreads();  // U of this column has arrived; V is free
    // t-phase items: (8-plane half, t tile); a half past Nz does not exist
    const int nit = (16 * z16 + 8 < Nz ? 2 : 1) * k.NTI;
    const char* xbase = reinterpret_cast<const char*>(a.lin_in + (long long)b * a.Cl * k.chan);
    char* obase = reinterpret_cast<char*>(a.out + (long long)b * a.Cs * k.chan);
    char* gbase = (MODE == EPI_FWD && a.gp) ? reinterpret_cast<char*>(a.gp + (long long)b * a.Cs * k.chan) : obase;
    const long long pt = (long long)xy * k.plane;
    const int z0 = 16 * z16;
    u64 x[CM > 0 ? CM : 1][H];
    uint32_t pos = 0;
    bool ok0 = false, ok1 = false;
    auto load_x = [&](int it) {
      const int sub = it / k.NTI, T = it - sub * k.NTI;
      const int z = z0 + 8 * sub + g, t = 8 * H * T + (H == 2 && k.perm ? 4 : 2) * q4;
      ok0 = z < Nz && t < Nt;
      ok1 = H == 2 && z < Nz && t + (k.perm ? 2 : 8) < Nt;
      pos = 4 * (uint32_t)(pt + (long long)z * Nt + t);
      if (MODE == EPI_SPECTRAL) return;
      // points past the column read its first one: their results are not stored
      const uint32_t p0 = ok0 ? pos : 4 * (uint32_t)pt;
      const char* xp = xbase;
      if (H == 2 && k.perm) {
#pragma unroll
        for (int i = 0; i < CM; ++i, xp += 4 * k.chan) {
          ulonglong2 v = make_ulonglong2(0, 0);
          if (i < a.Cl) v = *reinterpret_cast<const ulonglong2*>(xp + p0);
          x[i][0] = v.x;
          x[i][H - 1] = v.y;
        }
      } else {
        const uint32_t p1 = ok1 ? pos + 32 : p0;
#pragma unroll
        for (int i = 0; i < CM; ++i, xp += 4 * k.chan) {
          x[i][0] = x[i][H - 1] = 0;
          if (i < a.Cl) {
            x[i][0] = *reinterpret_cast<const u64*>(xp + p0);
            if (H == 2) x[i][H - 1] = *reinterpret_cast<const u64*>(xp + p1);
          }
        }
      }
    };
    // two sub-tiles: the first item's points are on their way during the z phase
    // (one sub-tile: the registers are better spent on more warps)
    if (H == 2 && warp < nit) load_x(warp);
    // ---- z phase: V of the warp's channel pairs.  Rows kz >= Jz and columns
    // kt >= Jt repeat the last one: their basis is zero.
    const uint4* zfb = k.zf + (size_t)z16 * KS * 3 * 32 + lane;
#pragma unroll 1
    for (int p = warp; p < NPAIR; p += NW) {
      float cr[2][4], ci[2][4];
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          cr[c][q] = 0.f;
          ci[c][q] = 0.f;
        }
      const float2* up0 = sU + 2 * p * JZT + ukt;
      const float2* up1 = sU + min(2 * p + 1, a.Cs - 1) * JZT + ukt;
#pragma unroll 2
      for (int ks = 0; ks < KS; ++ks) {
        const int k0 = min(8 * ks + q4, Jz - 1) * Jt, k1 = min(8 * ks + q4 + 4, Jz - 1) * Jt;
        uint4 A[NP], I[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q) {
          A[q] = __ldg(zfb + (ks * 3 + q) * 32);
          // rows (Ir, -Ii) of the real part -> (Ii, Ir) of the imaginary part
          I[q].x = __byte_perm(A[q].x, 0, 0x1032) ^ 0x00008000u;
          I[q].y = __byte_perm(A[q].y, 0, 0x1032) ^ 0x00008000u;
          I[q].z = __byte_perm(A[q].z, 0, 0x1032) ^ 0x00008000u;
          I[q].w = __byte_perm(A[q].w, 0, 0x1032) ^ 0x00008000u;
        }
        uint32_t B[2][2][NP];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const float2 v0 = (c == 0 ? up0 : up1)[k0], v1 = (c == 0 ? up0 : up1)[k1];
          bf16_parts<NP>(v0.x, v0.y, B[c][0]);
          bf16_parts<NP>(v1.x, v1.y, B[c][1]);
        }
#pragma unroll
        for (int q = 0; q < P::n; ++q)
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const uint4 z = A[P::a(q)], y = I[P::a(q)];
            wm::mma16(cr[c], z.x, z.y, z.z, z.w, B[c][0][P::b(q)], B[c][1][P::b(q)]);
            wm::mma16(ci[c], y.x, y.y, y.z, y.w, B[c][0][P::b(q)], B[c][1][P::b(q)]);
          }
      }
#pragma unroll
      for (int sub = 0; sub < 2; ++sub) {
        uint32_t f[4][NP];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          bf16_parts<NP>(cr[c][2 * sub], cr[c][2 * sub + 1], f[c]);
          bf16_parts<NP>(ci[c][2 * sub], ci[c][2 * sub + 1], f[2 + c]);
        }
#pragma unroll
        for (int q = 0; q < NP; ++q)
          sV[((p * 2 + sub) * NP + q) * 32 + lane] = make_uint4(f[0][q], f[1][q], f[2][q], f[3][q]);
      }
    }
    __syncthreads();  // V is complete; U is free
    if (++z16 == k.NZ16) {
      z16 = 0;
      ++col;
      if (u + 1 < u1) fetch_u(col);
    }
    // ---- t phase ----
    if (H == 1 && warp < nit) load_x(warp);
#pragma unroll 1
    for (int it = warp; it < nit;) {
      const int sub = it / k.NTI, T = it - sub * k.NTI;
      if (MODE != EPI_SPECTRAL && k.lin_round) {
#pragma unroll
        for (int i = 0; i < CM; ++i)
#pragma unroll
          for (int h = 0; h < H; ++h) {
            const float2 v = unpack2(x[i][h]);
            x[i][h] = pack2(lin_round(v.x, k.lin_round), lin_round(v.y, k.lin_round));
          }
      }
      col_item<MODE, CM, NP, H, CH>(k, sV + sub * NP * 32 + lane, sT + T * NP * 32 + lane, sW, sB, x, obase, gbase, pos,
                                ok0, ok1);
      it += NW;
      if (it < nit) load_x(it);
    }
  }
}

// ---------------------------------------------------------------------------
bool epilogue_col_supported(const Dims& d, int mode, int Cs, int Cl) {
  if (mode == EPI_DA) return false;
  if (d.Nt % 2 != 0 || d.Nt > 128 || d.Jt > 8 || d.Jz > 64) return false;
  if (Cs < 1 || Cs > 32) return false;
  // 32-bit byte offsets within a channel, 32-bit unit numbers
  if (4 * d.Ng >= (1LL << 32) || d.B * d.Nx * d.Ny * ((d.Nz + 15) / 16) >= (1LL << 31)) return false;
  return mode == EPI_SPECTRAL || (Cl >= 1 && Cl <= 32);
}

template <int MODE, int CM, int NP, int H, int CH, int NW, int MINB>
static cudaError_t launch_col_t(EpiCol k, const char* name, cudaStream_t s) {
  const int threads = 32 * NW;
  const size_t smem = sizeof(uint4) * (size_t)k.NPAIR * 2 * NP * 32 + sizeof(uint4) * (size_t)k.NTI * NP * 32 +
                      sizeof(ulonglong2) * (size_t)k.NPAIR * CM + sizeof(float2) * (size_t)((k.NPAIR + 1) & ~1) +
                      sizeof(float2) * (size_t)k.a.Cs * k.Jz * k.Jt;
  const void* kern = (const void*)k_epi_col<MODE, CM, NP, H, CH, NW, MINB>;
  cudaError_t e = allow_smem(kern, smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess || per_sm < 1)
    per_sm = 1;
  const long long g = std::max<long long>(1, std::min<long long>((long long)per_sm * sm_count(), k.nunits));
  FNO_LAUNCH(name, (k_epi_col<MODE, CM, NP, H, CH, NW, MINB>), (int)g, threads, smem, s, k);
  return cudaSuccess;
}

// Chains of the 1x1's FP32 sums: one for plain BF16, two with three-part operands (z
// error at Nt = 84 1.29e-7 against 1.47e-7 in one, in the same time).  With two parts
// one chain of up to 24 channels is more exact than the tcgen05 form's 3xTF32 was
// (z 1.6e-7 against 2.4e-7 at 20 channels); four chains are for what replaces the
// six-product 1x1 of k_epi_mma (fine): z 1.62e-7 with one and 1.16e-7 with four
// chains, 1.18e-7 in k_epi_mma, at 32 channels and Nt = 16, in the same time (32
// channels: 488 us a dX either way at 64^3 x 16).  At 20 channels and Nt = 32 they
// cost 4 to 7 %.
template <int MODE, int NP>
static cudaError_t launch_col_c(const EpiCol& k, bool narrow, bool fine, const char* name, cudaStream_t s) {
  constexpr int C1 = NP == 3 ? 2 : 1, C4 = NP == 2 ? 4 : C1;
  if constexpr (MODE == EPI_SPECTRAL) {
    if (narrow) return launch_col_t<EPI_SPECTRAL, 0, NP, 2, 1, 4, 4>(k, name, s);
    return launch_col_t<EPI_SPECTRAL, 0, NP, 1, 1, 4, 4>(k, name, s);
  } else if (narrow) {
    if (k.a.Cl <= 8) return launch_col_t<MODE, 8, NP, 2, C1, 4, 4>(k, name, s);
    if (k.a.Cl <= 12) return launch_col_t<MODE, 12, NP, 2, C1, 4, 4>(k, name, s);
    constexpr int NW = NP == 3 ? 6 : 4, MINB = NP == 3 ? 2 : 3;
    if (k.a.Cl <= 20) {
      if (fine) return launch_col_t<MODE, 20, NP, 2, C4, NW, MINB>(k, name, s);
      return launch_col_t<MODE, 20, NP, 2, C1, NW, MINB>(k, name, s);
    }
    if (k.a.Cl <= 24) {
      if (fine) return launch_col_t<MODE, 24, NP, 2, C4, NW, MINB>(k, name, s);
      return launch_col_t<MODE, 24, NP, 2, C1, NW, MINB>(k, name, s);
    }
    if constexpr (NP > 1) return launch_col_t<MODE, 32, NP, 2, C4, 4, 2>(k, name, s);
  } else {
    if (k.a.Cl <= 8) return launch_col_t<MODE, 8, NP, 1, C1, 4, 5>(k, name, s);
    if (k.a.Cl <= 20) {
      if (fine) return launch_col_t<MODE, 20, NP, 1, C4, 4, 5>(k, name, s);
      return launch_col_t<MODE, 20, NP, 1, C1, 4, 5>(k, name, s);
    }
    if (k.a.Cl <= 24) {
      if (fine) return launch_col_t<MODE, 24, NP, 1, C4, 4, 4>(k, name, s);
      return launch_col_t<MODE, 24, NP, 1, C1, 4, 4>(k, name, s);
    }
    if constexpr (NP > 1) return launch_col_t<MODE, 32, NP, 1, C4, 8, 2>(k, name, s);
  }
  return cudaErrorInvalidValue;  // not reached: plain BF16 has at most 24 inputs here
}

template <int NP>
static cudaError_t launch_col_m(const EpiCol& k, bool narrow, bool fine, const char* name, cudaStream_t s) {
  if (k.a.mode == EPI_SPECTRAL) return launch_col_c<EPI_SPECTRAL, NP>(k, narrow, fine, name, s);
  if (k.a.mode == EPI_DX) return launch_col_c<EPI_DX, NP>(k, narrow, fine, name, s);
  if constexpr (NP > 1) return launch_col_c<EPI_FWD, NP>(k, narrow, fine, name, s);
  return cudaErrorInvalidValue;  // not reached: plain BF16 runs its forward on k_epi_mma
}

cudaError_t launch_epilogue_col(const Dims& d, const EpiArgs& a, bool split, bool exact, bool lin_round,
                                bool fine, const EpiTables& ct, bool scaled, cudaStream_t s) {
  EpiCol k{};
  k.a = a;
  if (a.mode == EPI_SPECTRAL) k.a.Cl = 0;
  k.zf = ct.zf;
  k.tf = scaled ? ct.tfs : ct.tfu;
  k.NxNy = d.Nx * d.Ny;
  k.plane = d.Nz * d.Nt;
  k.chan = d.Ng;
  k.Nz = (int)d.Nz;
  k.Nt = (int)d.Nt;
  k.Jz = (int)d.Jz;
  k.Jt = (int)d.Jt;
  k.KS = ct.KS;
  k.NZ16 = ct.NZ;
  k.NTI = (int)((d.Nt + 8 * ct.H - 1) / (8 * ct.H));
  k.NPAIR = (a.Cs + 1) / 2;
  k.perm = ct.perm;
  k.lin_round = lin_round ? 1 : 0;
  k.nunits = (unsigned)(d.B * k.NxNy * ct.NZ);
  static const char* const names[4][2] = {{"fno_epi_spectral_cmma_bf16", "fno_epi_spectral_cmma_bf16x3"},
                                          {"fno_epi_dx_cmma_bf16", "fno_epi_dx_cmma_bf16x3"},
                                          {"", "fno_epi_fwd_cmma_bf16x3"},
                                          {"", "fno_epi_fwd_train_cmma_bf16x3"}};
  const char* name = names[a.mode == EPI_SPECTRAL ? 0 : a.mode == EPI_DX ? 1 : a.gp ? 3 : 2][split ? 1 : 0];
  const bool narrow = ct.H == 2;
  if (!split) return launch_col_m<1>(k, narrow, fine, name, s);
  if (exact) return launch_col_m<3>(k, narrow, fine, name, s);
  return launch_col_m<2>(k, narrow, fine, name, s);
}

}  // namespace fno
