// fno_tz_reg.cu -- the pruned DFT over t then z of every (b, c, x, y) column (the
// first half of F_yzt, S_yzt in Alg. 2) on mma.sync, columns loaded straight
// into registers.
//
// The arithmetic is that of k_fwd_tz_mma (fno_mma.cu), product by product: the t
// stage with the basis as A operand (rows re/im x kt) and the column as B (k = t,
// n = z), whose C fragments of two n-tiles are the B fragment of one z k-step.
// Here a warp loads the rows of its next D z-steps (16 z each) itself: lane (z
// row, t quarter) reads 16 bytes (8 where rows are not 16-byte aligned), and a
// step's registers are refilled as soon as it is done, also across columns.  No
// staging, no producer, no barrier after the prologue: a warp never waits for
// another one's column.
//
// What bounds it: HBM (4 bytes a point in, the spectrum out).  With staging in a
// ring of 16 KB bulk copies a column of more than one stage is consumed by one
// warp while it fills the ring for all.  One launch in split BF16, width 20, in
// the ring and here: 130^3 x 84 (43.7 KB columns, a ring of four stages) 8.40 and
// 2.57 ms (15.5 GB: 0.89 of 6.8 TB/s), 262 x 118 x 64 x 86 3.49 and 2.31 ms,
// 128^3 x 32 1.28 and 1.07 ms, 64^3 x 16 135 and 116 us, 64^3 x 8 286 and 216
// us.  Plain BF16 at Nt <= 16, one product a step, stays in the ring (64^3 x 16:
// 93 and 106 us; at Nt = 32 149 and 146).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "fno_internal.h"
#include "warp_mma.h"

namespace fno {

namespace {
constexpr int kTzrWarps = 8;
}

struct TzR {
  const float* in;   // [ncol][Nz][Nt]
  float2* out;       // [ncol][Jz][Jt]
  const float2* Ft;  // [Jt][Nt]  (cos, -sin) * scale
  const float2* Fz;  // [Jz][Nz]  (cos, -sin)
  long long ncol;
  int Nz, Nt, Jz, Jt, KT, KZ;
};

// MZ: z m-tiles (16 kz each).  KT: bound of the t k-steps (16 t each).
template <int MZ, int KT, bool SPLIT, bool TF>
__global__ void __launch_bounds__(32 * kTzrWarps, MZ <= 2 ? 2 : 1) k_fwd_tz_reg(const __grid_constant__ TzR p) {
  constexpr int D = KT == 1 ? 4 : KT == 2 ? 2 : 1;  // z-steps in flight: 32 to 64 registers
  constexpr bool TREG = KT <= 2;                    // t basis in registers (else shared memory)
  extern __shared__ __align__(16) unsigned char sm_tzr[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int g8 = lane >> 2, t4 = lane & 3;
  const int Nt = p.Nt, Nz = p.Nz, KZ = p.KZ;
  uint4* fzf = reinterpret_cast<uint4*>(sm_tzr);  // [MZ][KZ][re hi, re lo, im hi, im lo][32]
  uint4* ftf = fzf + (size_t)MZ * KZ * 4 * 32;    // [KT][hi, lo][32]

  // z basis in A-fragment order: rows kz, cols z
  for (int e = tid; e < MZ * KZ * 32; e += 32 * kTzrWarps) {
    const int ln = e & 31, ks = (e >> 5) % KZ, mt = (e >> 5) / KZ;
    const int r0 = 16 * mt + (ln >> 2), c0 = 16 * ks + 2 * (ln & 3);
    auto F = [&](int kz, int z, int im) -> float {
      if (kz >= p.Jz || z >= Nz) return 0.f;
      const float2 f = p.Fz[(long long)kz * Nz + z];
      return wm::rnd<TF>(im ? f.y : f.x);
    };
#pragma unroll
    for (int im = 0; im < 2; ++im) {
      uint32_t h[4], l[4];
      wm::split2(F(r0, c0, im), F(r0, c0 + 1, im), h[0], l[0]);
      wm::split2(F(r0 + 8, c0, im), F(r0 + 8, c0 + 1, im), h[1], l[1]);
      wm::split2(F(r0, c0 + 8, im), F(r0, c0 + 9, im), h[2], l[2]);
      wm::split2(F(r0 + 8, c0 + 8, im), F(r0 + 8, c0 + 9, im), h[3], l[3]);
      uint4* dst = fzf + ((mt * KZ + ks) * 4 + 2 * im) * 32 + ln;
      dst[0] = make_uint4(h[0], h[1], h[2], h[3]);
      dst[32] = make_uint4(l[0], l[1], l[2], l[3]);
    }
  }
  // t basis in A-fragment order: rows ri * 8 + jt, k slots 2 t4 + {0,1} <-> t = 16
  // ks + 4 t4 + {0,1} and 2 t4 + 8 + {0,1} <-> + {2,3}
  auto t_frag = [&](int ks, int ln, uint4& hi, uint4& lo) {
    const int jt = ln >> 2, t0 = 16 * ks + 4 * (ln & 3);
    auto F = [&](int ri, int t) -> float {
      if (jt >= p.Jt || t >= Nt) return 0.f;
      const float2 f = p.Ft[(long long)jt * Nt + t];
      return wm::rnd<TF>(ri ? f.y : f.x);
    };
    wm::split2(F(0, t0), F(0, t0 + 1), hi.x, lo.x);
    wm::split2(F(1, t0), F(1, t0 + 1), hi.y, lo.y);
    wm::split2(F(0, t0 + 2), F(0, t0 + 3), hi.z, lo.z);
    wm::split2(F(1, t0 + 2), F(1, t0 + 3), hi.w, lo.w);
  };
  uint4 frh[TREG ? KT : 1], frl[TREG ? KT : 1];
  if (TREG) {
#pragma unroll
    for (int ks = 0; ks < (TREG ? KT : 1); ++ks) t_frag(ks, lane, frh[ks], frl[ks]);
  } else {
    for (int e = tid; e < KT * 32; e += 32 * kTzrWarps)
      t_frag(e >> 5, e & 31, ftf[(e >> 5) * 64 + (e & 31)], ftf[(e >> 5) * 64 + 32 + (e & 31)]);
  }
  __syncthreads();

  const long long nw = (long long)gridDim.x * kTzrWarps;
  long long col = (long long)blockIdx.x * kTzrWarps + (tid >> 5);
  if (col >= p.ncol) return;
  const bool vec4 = (Nt & 3) == 0;  // 16-byte rows; otherwise 8-byte (Nt even)
  const long long plane = (long long)Nz * Nt;
  float4 v[D][2][KT];
  // the rows of a z-step into one slot: rows past Nz and times past Nt enter as zeros
  auto load = [&](float4 (&s)[2][KT], long long c, int kz) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int z = 16 * kz + 8 * h + g8;
      const float* row = p.in + c * plane + (long long)z * Nt + 4 * t4;
      const bool zin = c < p.ncol && z < Nz;
#pragma unroll
      for (int ks = 0; ks < KT; ++ks) {
        const int tt = 16 * ks + 4 * t4;
        float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
        if (vec4) {
          if (zin && tt < Nt) w = __ldg(reinterpret_cast<const float4*>(row + 16 * ks));
        } else {
          if (zin && tt < Nt) {
            const float2 a = __ldg(reinterpret_cast<const float2*>(row + 16 * ks));
            w.x = a.x;
            w.y = a.y;
          }
          if (zin && tt + 2 < Nt) {
            const float2 a = __ldg(reinterpret_cast<const float2*>(row + 16 * ks + 2));
            w.z = a.x;
            w.w = a.y;
          }
        }
        s[h][ks] = w;
      }
    }
  };
  // the z-step to load next
  long long lc = col;
  int lk = 0;
  auto advance = [&]() {
    if (++lk == KZ) {
      lk = 0;
      lc += nw;
    }
  };
#pragma unroll
  for (int i = 0; i < D; ++i) {
    load(v[i], lc, lk);
    advance();
  }
  float tre[MZ][4], tim[MZ][4];
#pragma unroll
  for (int mt = 0; mt < MZ; ++mt)
#pragma unroll
    for (int q = 0; q < 4; ++q) tre[mt][q] = tim[mt][q] = 0.f;
  int kz = 0;
  while (col < p.ncol) {
#pragma unroll
    for (int i = 0; i < D; ++i) {
      if (col < p.ncol) {
        // t stage of z = 16 kz .. 16 kz + 15 (two n-tiles)
        float pc[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int q = 0; q < 4; ++q) pc[h][q] = 0.f;
#pragma unroll
        for (int ks = 0; ks < KT; ++ks) {
          if (KT <= 2 || ks < p.KT) {
            const uint4 fh = TREG ? frh[TREG ? ks : 0] : ftf[ks * 64 + lane];
            uint4 fl = make_uint4(0u, 0u, 0u, 0u);
            if (SPLIT) fl = TREG ? frl[TREG ? ks : 0] : ftf[ks * 64 + 32 + lane];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const float4 x = v[i][h][ks];
              uint32_t bh0, bl0, bh1, bl1;
              wm::split2(wm::rnd<TF>(x.x), wm::rnd<TF>(x.y), bh0, bl0);
              wm::split2(wm::rnd<TF>(x.z), wm::rnd<TF>(x.w), bh1, bl1);
              if (SPLIT) {
                wm::mma16(pc[h], fl.x, fl.y, fl.z, fl.w, bh0, bh1);
                wm::mma16(pc[h], fh.x, fh.y, fh.z, fh.w, bl0, bl1);
              }
              wm::mma16(pc[h], fh.x, fh.y, fh.z, fh.w, bh0, bh1);
            }
          }
        }
        load(v[i], lc, lk);
        advance();
        // z stage k-step kz: B fragments straight from the t-stage accumulators
        uint32_t rh0, rl0, rh1, rl1, ih0, il0, ih1, il1;
        wm::split2(wm::rnd<TF>(pc[0][0]), wm::rnd<TF>(pc[0][1]), rh0, rl0);  // P_re, z + 0..7
        wm::split2(wm::rnd<TF>(pc[1][0]), wm::rnd<TF>(pc[1][1]), rh1, rl1);  // P_re, z + 8..15
        wm::split2(wm::rnd<TF>(pc[0][2]), wm::rnd<TF>(pc[0][3]), ih0, il0);  // P_im
        wm::split2(wm::rnd<TF>(pc[1][2]), wm::rnd<TF>(pc[1][3]), ih1, il1);
        const uint32_t nh0 = ih0 ^ 0x80008000u, nh1 = ih1 ^ 0x80008000u;  // -P_im
        const uint32_t nl0 = il0 ^ 0x80008000u, nl1 = il1 ^ 0x80008000u;
#pragma unroll
        for (int mt = 0; mt < MZ; ++mt) {
          const uint4* fz = fzf + ((mt * KZ + kz) * 4) * 32 + lane;
          const uint4 arh = fz[0], aih = fz[64];
          float dr[4] = {0.f, 0.f, 0.f, 0.f}, di[4] = {0.f, 0.f, 0.f, 0.f};
          if (SPLIT) {
            const uint4 arl = fz[32], ail = fz[96];
            wm::mma16(dr, arl.x, arl.y, arl.z, arl.w, rh0, rh1);
            wm::mma16(di, arl.x, arl.y, arl.z, arl.w, ih0, ih1);
            wm::mma16(dr, arh.x, arh.y, arh.z, arh.w, rl0, rl1);
            wm::mma16(di, arh.x, arh.y, arh.z, arh.w, il0, il1);
            wm::mma16(dr, ail.x, ail.y, ail.z, ail.w, nh0, nh1);
            wm::mma16(di, ail.x, ail.y, ail.z, ail.w, rh0, rh1);
            wm::mma16(dr, aih.x, aih.y, aih.z, aih.w, nl0, nl1);
            wm::mma16(di, aih.x, aih.y, aih.z, aih.w, rl0, rl1);
          }
          wm::mma16(dr, arh.x, arh.y, arh.z, arh.w, rh0, rh1);
          wm::mma16(di, arh.x, arh.y, arh.z, arh.w, ih0, ih1);
          wm::mma16(dr, aih.x, aih.y, aih.z, aih.w, nh0, nh1);
          wm::mma16(di, aih.x, aih.y, aih.z, aih.w, rh0, rh1);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            tre[mt][q] += dr[q];
            tim[mt][q] += di[q];
          }
        }
        if (++kz == KZ) {
          // T[col][kz][jt]: rows kz = 16 mt + g8 (+8), cols jt = 2 t4 + {0, 1}
          float2* oc = p.out + col * (long long)(p.Jz * p.Jt);
#pragma unroll
          for (int mt = 0; mt < MZ; ++mt)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
              const int r = 16 * mt + g8 + 8 * hh;
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                const int jt = 2 * t4 + e;
                if (r < p.Jz && jt < p.Jt)
                  oc[r * p.Jt + jt] = make_float2(tre[mt][2 * hh + e], tim[mt][2 * hh + e]);
                tre[mt][2 * hh + e] = tim[mt][2 * hh + e] = 0.f;
              }
            }
          kz = 0;
          col += nw;
        }
      }
    }
  }
}

template <int MZ, int KT, bool SPLIT, bool TF>
static cudaError_t launch_tzr_t(const TzR& k, const char* name, cudaStream_t s) {
  const size_t smem = 16 * 32 * ((size_t)MZ * k.KZ * 4 + (KT <= 2 ? 0 : 2 * KT));
  const void* kern = (const void*)k_fwd_tz_reg<MZ, KT, SPLIT, TF>;
  cudaError_t e = allow_smem(kern, smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kTzrWarps, smem) != cudaSuccess || per_sm < 1)
    per_sm = 1;
  const long long need = (k.ncol + kTzrWarps - 1) / kTzrWarps;
  const int grid = (int)std::max<long long>(1, std::min<long long>((long long)per_sm * sm_count(), need));
  FNO_LAUNCH(name, (k_fwd_tz_reg<MZ, KT, SPLIT, TF>), grid, 32 * kTzrWarps, smem, s, k);
  return cudaSuccess;
}

template <int MZ, bool SPLIT, bool TF>
static cudaError_t launch_tzr_k(const TzR& k, const char* name, cudaStream_t s) {
  if (k.KT == 1) return launch_tzr_t<MZ, 1, SPLIT, TF>(k, name, s);
  if (k.KT == 2) return launch_tzr_t<MZ, 2, SPLIT, TF>(k, name, s);
  if (k.KT <= 4) return launch_tzr_t<MZ, 4, SPLIT, TF>(k, name, s);
  if (k.KT <= 6) return launch_tzr_t<MZ, 6, SPLIT, TF>(k, name, s);
  return launch_tzr_t<MZ, 8, SPLIT, TF>(k, name, s);
}

template <bool SPLIT, bool TF>
static cudaError_t launch_tzr_m(const TzR& k, const char* name, cudaStream_t s) {
  if (k.Jz <= 16) return launch_tzr_k<1, SPLIT, TF>(k, name, s);
  return launch_tzr_k<2, SPLIT, TF>(k, name, s);
}

bool fwd_tz_reg_supported(const Dims& d, bool split) {
  if (!split && d.Nt <= 16) return false;  // the ring is faster there (see the top)
  const size_t fz = 16 * 32 * (size_t)(d.Jz <= 16 ? 1 : 2) * (size_t)((d.Nz + 15) / 16) * 4;
  return d.Nt % 2 == 0 && d.Nt <= 128 && d.Jt <= 8 && d.Jz <= 32 && fz + 16 * 32 * 16 <= 110 * 1024;
}

cudaError_t launch_fwd_tz_reg(const float* in, float2* out, int64_t ncol, const Dims& d, const float2* ft,
                              const float2* fz, bool split, bool tf32, cudaStream_t s) {
  if (ncol <= 0) return cudaSuccess;
  TzR k{};
  k.in = in;
  k.out = out;
  k.Ft = ft;
  k.Fz = fz;
  k.ncol = ncol;
  k.Nz = (int)d.Nz;
  k.Nt = (int)d.Nt;
  k.Jz = (int)d.Jz;
  k.Jt = (int)d.Jt;
  k.KT = (int)((d.Nt + 15) / 16);
  k.KZ = (int)((d.Nz + 15) / 16);
  if (tf32) return launch_tzr_m<true, true>(k, "fno_fwd_tz_mma_tf32", s);
  if (split) return launch_tzr_m<true, false>(k, "fno_fwd_tz_mma_bf16x3", s);
  return launch_tzr_m<false, false>(k, "fno_fwd_tz_mma_bf16", s);
}

}  // namespace fno
