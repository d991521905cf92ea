// One 16-token page of attention on mma.sync, shared by the decode kernel and the small-tile extend kernel.
//
// Scores are computed as S^T = K Q^T with tokens in the M dimension of mma.sync.m16n8k16 (one 16-token page per MMA row
// block, 8 query rows in N), so the K fragments are exactly the 16-byte chunks as they lie in the pool and no padding
// of the query rows to 16 is needed; O^T = V^T P^T uses the same trick with byte permutes pairing two tokens.
#pragma once

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace kvattn {

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                               uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(y) : "r"(x));
  return y;
}

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;\n" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// (not .nc: the decode kernel is resident while the append in front of it may still be storing pages)
__device__ __forceinline__ uint4 ldg_stream(const void* p) {
  uint4 v;
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

template <int D>
struct PageRegs {
  uint4 k[2][D / 32];     // [token group][j]   : slot 8g + r, chunk 4j + c
  uint4 v[2][2][D / 64];  // [token group][parity][u]: slot 8g + 2c + parity, chunk 8u + r
};

template <int D>
__device__ __forceinline__ void load_page(PageRegs<D>& pr, const char* kblk, const char* vblk, int r, int c) {
#pragma unroll
  for (int g = 0; g < 2; ++g) {
#pragma unroll
    for (int j = 0; j < D / 32; ++j) {
      const int ch = 4 * j + c;
      pr.k[g][j] = ldg_stream(kblk + g * (D * 16) + (ch >> 3) * 1024 + r * 128 + (((ch & 7) ^ r) << 4));
    }
  }
#pragma unroll
  for (int g = 0; g < 2; ++g) {
#pragma unroll
    for (int par = 0; par < 2; ++par) {
      const int row = 2 * c + par;
#pragma unroll
      for (int u = 0; u < D / 64; ++u)
        pr.v[g][par][u] = ldg_stream(vblk + g * (D * 16) + u * 1024 + row * 128 + ((r ^ row) << 4));
    }
  }
}

// Fragments of one page from a shared-memory slot (K block, then V block).  Within a quarter warp the K loads of the
// lanes with an odd row take the other 64-byte half first (j ^ 1), so that the eight lanes touch eight different
// 16-byte bank groups; the registers are swapped back afterwards.
template <int D>
__device__ __forceinline__ void load_page_smem(PageRegs<D>& pr, uint32_t slot, int r, int c) {
  auto lds = [](uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
  };
  const int flip = r & 1;
#pragma unroll
  for (int g = 0; g < 2; ++g) {
#pragma unroll
    for (int j = 0; j < D / 32; ++j) {
      const int ch = 4 * (j ^ flip) + c;
      pr.k[g][j] = lds(slot + g * (D * 16) + (ch >> 3) * 1024 + r * 128 + (((ch & 7) ^ r) << 4));
    }
    if (flip) {
#pragma unroll
      for (int j = 0; j < D / 32; j += 2) {
        const uint4 t = pr.k[g][j];
        pr.k[g][j] = pr.k[g][j + 1];
        pr.k[g][j + 1] = t;
      }
    }
  }
  const uint32_t vslot = slot + 16 * D * 2;
#pragma unroll
  for (int g = 0; g < 2; ++g) {
#pragma unroll
    for (int par = 0; par < 2; ++par) {
      const int row = 2 * c + par;
#pragma unroll
      for (int u = 0; u < D / 64; ++u)
        pr.v[g][par][u] = lds(vslot + g * (D * 16) + u * 1024 + row * 128 + ((r ^ row) << 4));
    }
  }
}

// Running softmax of a warp's 8 query rows.  Lane (r, c) = (lane / 4, lane % 4) holds the rows n0 = 2c and n1 = 2c + 1:
// their maxima (shared by the lanes of equal c), its own share of their sums (tokens r and r + 8 of every page), and
// acc[u][w][i]: dims 64u + 8r + 2w + {0, 1} of row n0 (i = 0, 2) and n1 (i = 1, 3).
template <int D>
struct RowState {
  float acc[D / 64][4][4];
  float m0, m1, l0, l1;
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int u = 0; u < D / 64; ++u)
#pragma unroll
      for (int w = 0; w < 4; ++w)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[u][w][i] = 0.f;
    m0 = m1 = -INFINITY;
    l0 = l1 = 0.f;
  }
};

// Takes the page of tokens tok0 .. tok0 + 15 into the running softmax.  qf: fragments of the query rows (row r's 16-byte
// chunks 4j + c); limit0 / limit1: keys the rows n0 / n1 see; L: tokens of the sequence (slots at or past it hold
// arbitrary bits).
template <int D>
__device__ __forceinline__ void page_step(RowState<D>& st, PageRegs<D>& pr, const uint4 (&qf)[D / 32], int tok0, int limit0,
                                          int limit1, int L, float scale_log2, int r, int c) {
  constexpr int NJ = D / 32, NU = D / 64;
  // ---- S^T[16 tokens][8 rows] = K Q^T, in two accumulators: the chain of dependent MMAs is what a page's latency starts with
  float s[4] = {0.f, 0.f, 0.f, 0.f}, t[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    mma_bf16_16816(s, pr.k[0][j].x, pr.k[1][j].x, pr.k[0][j].y, pr.k[1][j].y, qf[j].x, qf[j].y);
    mma_bf16_16816(t, pr.k[0][j].z, pr.k[1][j].z, pr.k[0][j].w, pr.k[1][j].w, qf[j].z, qf[j].w);
  }
  // s00: (token r, row n0)  s01: (token r, n1)  s10: (token r+8, n0)  s11: (token r+8, n1)
  const int ta = tok0 + r, tb = tok0 + r + 8;
  const float s00 = ta < limit0 ? (s[0] + t[0]) * scale_log2 : -INFINITY;
  const float s01 = ta < limit1 ? (s[1] + t[1]) * scale_log2 : -INFINITY;
  const float s10 = tb < limit0 ? (s[2] + t[2]) * scale_log2 : -INFINITY;
  const float s11 = tb < limit1 ? (s[3] + t[3]) * scale_log2 : -INFINITY;
  float mx0 = fmaxf(s00, s10), mx1 = fmaxf(s01, s11);
  // Only a page with a larger score pays for the search among the lanes and the rescaling.  The maximum in use is the exact
  // one, so that a row's largest weight is exactly 1 and loses nothing when P is rounded to bf16: with one that may lag by 8
  // binades the error of O (2-norm) on 256 sequences of 1024-4096 tokens is 2.31e-3, this way 2.10e-3.  It costs what the
  // lag saved: 13 sequences of 200-3000 tokens, 64 dims, 13.4 -> 13.8 us, 5 of 8192-16384 42.4 -> 42.9, the 256 390 -> 392.
  if (__any_sync(0xffffffffu, mx0 > st.m0 || mx1 > st.m1)) {
#pragma unroll
    for (int off = 4; off < 32; off <<= 1) {
      mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, off));
      mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, off));
    }
    const float mn0 = fmaxf(st.m0, mx0), mn1 = fmaxf(st.m1, mx1);
    const float al0 = mn0 == -INFINITY ? 1.f : fast_exp2(st.m0 - mn0), al1 = mn1 == -INFINITY ? 1.f : fast_exp2(st.m1 - mn1);
    st.l0 *= al0;
    st.l1 *= al1;
    st.m0 = mn0;
    st.m1 = mn1;
#pragma unroll
    for (int u = 0; u < NU; ++u)
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        st.acc[u][w][0] *= al0; st.acc[u][w][2] *= al0;
        st.acc[u][w][1] *= al1; st.acc[u][w][3] *= al1;
      }
  }
  const float mu0 = st.m0 == -INFINITY ? 0.f : st.m0, mu1 = st.m1 == -INFINITY ? 0.f : st.m1;
  const float p00 = fast_exp2(s00 - mu0), p01 = fast_exp2(s01 - mu1);
  const float p10 = fast_exp2(s10 - mu0), p11 = fast_exp2(s11 - mu1);
  st.l0 += p00 + p10;
  st.l1 += p01 + p11;
  // P^T fragments: transpose the 8x8 (token, row) tiles held as packed bf16 pairs
  const uint32_t pt0 = movmatrix_trans(pack_bf16x2(p00, p01));
  const uint32_t pt1 = movmatrix_trans(pack_bf16x2(p10, p11));

  // stale slots past the sequence end may hold NaN/Inf bits: select them away (0 * NaN != 0)
  if (tok0 + 16 > L) {
#pragma unroll
    for (int g = 0; g < 2; ++g)
#pragma unroll
      for (int par = 0; par < 2; ++par)
        if (tok0 + 8 * g + 2 * c + par >= L) {
#pragma unroll
          for (int u = 0; u < NU; ++u) pr.v[g][par][u] = make_uint4(0, 0, 0, 0);
        }
  }
  // ---- O^T[D][8 rows] += V^T P^T
#pragma unroll
  for (int u = 0; u < NU; ++u) {
    const uint4 va = pr.v[0][0][u], vb = pr.v[0][1][u], vc = pr.v[1][0][u], vd = pr.v[1][1][u];
    const uint32_t wa[4] = {va.x, va.y, va.z, va.w}, wb[4] = {vb.x, vb.y, vb.z, vb.w};
    const uint32_t wc[4] = {vc.x, vc.y, vc.z, vc.w}, wd[4] = {vd.x, vd.y, vd.z, vd.w};
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      mma_bf16_16816(st.acc[u][w], __byte_perm(wa[w], wb[w], 0x5410), __byte_perm(wa[w], wb[w], 0x7632),
                     __byte_perm(wc[w], wd[w], 0x5410), __byte_perm(wc[w], wd[w], 0x7632), pt0, pt1);
    }
  }
}

}  // namespace kvattn
