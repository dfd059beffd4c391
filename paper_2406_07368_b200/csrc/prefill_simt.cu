// Prefill on the CUDA cores in fp32: serves fp32 inputs, head dimension 64, and any shape the tensor-core kernel does
// not take (but for the shortest calls, whose tokens are walked: prefill_walk.cu).  Chunkwise form of the cumulative sum of Sec. 4.1 in plain fp32 multiply-adds (what the fp32 tolerance needs
// and a single-pass tf32/bf16 contraction would not give):
//     O = phi(Q) S_prev + (P o M) V,   den = phi(Q) . z_prev + rowsum(P o M),   S += phi(K)^T V,   z += colsum phi(K)
// with P = phi(Q) phi(K)^T and M causal, per chunk of C tokens (64 at d = 64, 32 at d = 128).
//
// A chain (batch, head) is cut along the sequence over the CTAs of one thread-block cluster.  Every CTA but the last
// first forms the sums of its own segment, leaves them in its shared memory, and adds up those of the CTAs before it
// through distributed shared memory; then all segments run at once.  No workspace, one launch.  Cost: S += phi(K)^T V
// of all but a segment's last chunk is formed twice (d^2 of about 3 d^2 + C d multiply-adds per token).
//
// What bounds it: the latency of the shared-memory loads behind the multiply-adds at 12 warps per SM.  48 chains of 1000
// tokens, d = 64: 64 us in a graph, where its multiply-adds alone need about 22 at the fp32 peak, and where one CTA per chain
// that walked the tokens one by one took 443.  All products are register tiles (8 x 4 per thread at d = 64) fed by 128-bit
// shared-memory loads, three wavefronts per thirty-two multiply-adds of a warp.
#include <cooperative_groups.h>

#include <algorithm>

#include "la_common.cuh"

namespace la {
namespace simt {

namespace cg = cooperative_groups;

constexpr int kMaxCluster = 8;

// Threads stand in a grid of 16 columns (tx) by TY rows (ty).  A thread owns rows ty + TY r and columns 4 tx + 64 g of an
// output tile, rows ty + TY r and columns tx + 16 c of P, rows 4 ty + 4 TY a and columns 4 tx + 64 g of the state: 8 x 4
// values of each at d = 64.
template <int D> struct Shape {
  static constexpr int C = D == 64 ? 64 : 32;                // tokens per chunk
  static constexpr int NT = D == 64 ? 128 : 256, TY = NT / 16;
  static constexpr int QS = D + 4, PS = C + 4;              // row strides: rows a multiple of 4 banks apart
  static constexpr int R = C / TY, CB = C / 16;              // rows and columns of P per thread
  static constexpr int G = D / 64, A = D / (4 * TY);         // groups of 4 columns; groups of 4 state rows
  static constexpr int LPR = NT / C;                         // threads that share a row's denominator
  static constexpr int ZP = NT / D;                          // threads that share a feature of z
  static constexpr int LD = C * D / 4 / NT;                  // 4-element pieces of a chunk per thread
  static constexpr int kResident = D == 64 ? 3 : 1;          // CTAs per SM that shared memory allows at few taps
  static constexpr size_t bytes(int W) {
    return sizeof(float) * ((size_t)2 * C * QS + (size_t)(W - 1 + C) * D + D * D + D + C +
                            ZP * D + (size_t)W * D);
  }
};

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float4 x) { *reinterpret_cast<float4*>(p) = x; }
__device__ __forceinline__ float4 gld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 gld4(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                     __uint_as_float(u.y & 0xffff0000u));
}
__device__ __forceinline__ void gst4(float* p, float4 x) { *reinterpret_cast<float4*>(p) = x; }
__device__ __forceinline__ void gst4(__nv_bfloat16* p, float4 x) {
  __nv_bfloat162 a = __floats2bfloat162_rn(x.x, x.y), b = __floats2bfloat162_rn(x.z, x.w);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<uint32_t*>(&a), *reinterpret_cast<uint32_t*>(&b));
}
// phi with both sides formed always, a select and not a branch per element, for whole chunks at a time (few values, as in
// decode and commit, are faster with the branch: 1024 units of d = 64 decode in 6.2 us with it, 6.9 without).
template <int PHI> __device__ __forceinline__ float phi_both(float x) {
  if (PHI != LA_PHI_ELU1) return phi<PHI>(x);
  const float e = expf(x > 0.f ? 0.f : x);                   // (not fminf, which would drop a NaN)
  return x > 0.f ? x + 1.f : e;
}
template <int PHI> __device__ __forceinline__ float4 phi4(float4 x) {
  return make_float4(phi_both<PHI>(x.x), phi_both<PHI>(x.y), phi_both<PHI>(x.z), phi_both<PHI>(x.w));
}
__device__ __forceinline__ void fma4(float4& acc, float a, float4 b) {
  acc.x = fmaf(a, b.x, acc.x);
  acc.y = fmaf(a, b.y, acc.y);
  acc.z = fmaf(a, b.z, acc.z);
  acc.w = fmaf(a, b.w, acc.w);
}
__device__ __forceinline__ float comp(const float4& x, int i) { return i == 0 ? x.x : i == 1 ? x.y : i == 2 ? x.z : x.w; }

template <typename T, int D, int PHI>
__global__ void __launch_bounds__(Shape<D>::NT, Shape<D>::kResident)
prefill_simt_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                    const float* __restrict__ w, float* __restrict__ S, float* __restrict__ z, T* __restrict__ win,
                    int64_t* __restrict__ pos, T* __restrict__ o, int H, int Tlen, int W, float eps, int init, int seg_len) {
  using Sh = Shape<D>;
  constexpr int C = Sh::C, QS = Sh::QS, PS = Sh::PS, NT = Sh::NT, TY = Sh::TY, R = Sh::R, CB = Sh::CB, G = Sh::G, A = Sh::A,
                LPR = Sh::LPR, ZP = Sh::ZP, LD = Sh::LD;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* sq = reinterpret_cast<float*>(smem_raw);            // [C][QS] phi(q), then [C][PS] the masked P
  float* sk = sq + C * QS;                                   // [C][QS] phi(k)
  float* sS = sk + C * QS;                  // [D][D] the state before the chunk
  float* sz = sS + D * D;                                    // [D] z before the chunk
  float* szp = sz + D;                                       // [ZP][D] parts of the chunk's column sums of phi(k)
  float* sden = szp + ZP * D;                                // [C]
  float* sw = sden + C;                                      // [W][D]
  float* sv = sw + W * D;                                    // [W - 1 + C][D] v, the rows before the chunk first
  float* svc = sv + (W - 1) * D;                             // row 0 of the chunk

  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), nrank = (int)cluster.num_blocks();
  const int bh = blockIdx.x / nrank, h = bh % H, t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int tx = (warp & 1) * 8 + (lane & 7), ty = (warp >> 1) * 4 + (lane >> 3);   // a warp: 4 row groups x 8 column groups
  const size_t base = (size_t)bh * Tlen * D;
  const int seg0 = rank * seg_len, seg1 = min(Tlen, seg0 + seg_len);
  const bool last_rank = rank == nrank - 1;
  float* Sb = S + (size_t)bh * D * D;
  float* zb = z + (size_t)bh * D;
  T* wb = win + (size_t)bh * (W - 1) * D;

  float4 s[A][4][G];                                         // this thread's block of the state
#pragma unroll
  for (int g = 0; g < A; ++g)
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int c = 0; c < G; ++c)
        s[g][i][c] = init && rank == 0 ? ld4(Sb + (size_t)(4 * TY * g + 4 * ty + i) * D + 64 * c + 4 * tx) : make_float4(0.f, 0.f, 0.f, 0.f);
  float zr = t < D && init && rank == 0 ? zb[t] : 0.f;       // z, one feature per thread of the first D
  for (int idx = t; idx < W * D; idx += NT) sw[(idx % W) * D + idx / W] = w[(size_t)h * D * W + idx];

  // A chunk's rows of one tensor, all of a thread's loads in flight together (rows at or beyond n: zeros).
  auto fetch = [&](float4 (&x)[LD], const T* src, int i0, int n) {
#pragma unroll
    for (int it = 0; it < LD; ++it) {
      const int idx = t + it * NT, j = idx / (D / 4), e = idx % (D / 4) * 4;
      x[it] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (j < n) x[it] = gld4(src + base + (size_t)(i0 + j) * D + e);
    }
  };
  auto put_phi = [&](const float4 (&x)[LD], float* dst, int n) {
#pragma unroll
    for (int it = 0; it < LD; ++it) {
      const int idx = t + it * NT, j = idx / (D / 4), e = idx % (D / 4) * 4;
      st4(dst + j * QS + e, j < n ? phi4<PHI>(x[it]) : make_float4(0.f, 0.f, 0.f, 0.f));
    }
  };
  auto put_v = [&](const float4 (&x)[LD]) {
#pragma unroll
    for (int it = 0; it < LD; ++it) {
      const int idx = t + it * NT;
      st4(svc + idx * 4, x[it]);
    }
  };
  auto load_halo = [&](int i0) {                             // the W - 1 rows of v before token i0
    for (int idx = t; idx < (W - 1) * (D / 4); idx += NT) {
      const int i = idx / (D / 4), e = idx % (D / 4) * 4, tok = i0 - (W - 1) + i;
      st4(sv + i * D + e, tok >= 0 ? gld4(v + base + (size_t)tok * D + e)
                          : init   ? gld4(wb + (size_t)(W - 1 + tok) * D + e)
                                   : make_float4(0.f, 0.f, 0.f, 0.f));
    }
  };
  // S += phi(K)^T V of the chunk in shared memory, and the parts of z += colsum phi(K).  (Three loads feed 32 multiply-adds
  // here, and 12 warps per SM do not hide them alone: eight tokens' loads in flight.  48 chains of 2000 tokens, d = 64:
  // 144.9 us with 2, 134.5 with 4, 132.2 with 8, 132.5 with 16; the scores below, four steps instead of two: 131.6.)
  auto absorb = [&]() {
#pragma unroll 8
    for (int j = 0; j < C; ++j) {
      float4 kk[A], vv[G];
#pragma unroll
      for (int g = 0; g < A; ++g) kk[g] = ld4(sk + j * QS + 4 * TY * g + 4 * ty);
#pragma unroll
      for (int g = 0; g < G; ++g) vv[g] = ld4(svc + j * D + 64 * g + 4 * tx);
#pragma unroll
      for (int g = 0; g < A; ++g)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int c = 0; c < G; ++c) fma4(s[g][i][c], comp(kk[g], i), vv[c]);
    }
    float sum = 0.f;
#pragma unroll 8
    for (int j = 0; j < C / ZP; ++j) sum += sk[(t / D * (C / ZP) + j) * QS + t % D];
    szp[t] = sum;
  };
  auto z_total = [&]() {                                     // (after a barrier behind absorb)
    if (t < D)
#pragma unroll
      for (int p = 0; p < ZP; ++p) zr += szp[p * D + t];
  };
  auto publish = [&]() {                                     // state registers -> shared memory
#pragma unroll
    for (int g = 0; g < A; ++g)
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < G; ++c) st4(sS + (4 * TY * g + 4 * ty + i) * D + 64 * c + 4 * tx, s[g][i][c]);
    if (t < D) sz[t] = zr;
  };

  // ---- the sums of this segment, exchanged inside the cluster: the state before it ----
  if (nrank > 1) {
    if (!last_rank) {
      float4 x[LD], y[LD];
      fetch(x, k, seg0, min(C, seg1 - seg0));
      fetch(y, v, seg0, min(C, seg1 - seg0));
      for (int i0 = seg0; i0 < seg1; i0 += C) {
        __syncthreads();
        put_phi(x, sk, min(C, seg1 - i0));
        put_v(y);
        if (i0 + C < seg1) {                                 // in flight beside the products
          fetch(x, k, i0 + C, min(C, seg1 - i0 - C));
          fetch(y, v, i0 + C, min(C, seg1 - i0 - C));
        }
        __syncthreads();
        absorb();
        __syncthreads();
        z_total();
      }
      publish();
    }
    cluster.sync();
    // Rank r turns the r-th slice of everybody's sums into exclusive prefixes, in place: every thread has all of its
    // loads from the other CTAs in flight at once, and a CTA moves one state in and one out whatever its rank.  (Each
    // rank adding up all the states before it took 17 K cycles at rank 7.)
    constexpr int N4 = D * D / 4;
    const int per = (N4 + nrank - 1) / nrank, sl1 = min(N4, (rank + 1) * per);
    for (int i = rank * per + t; i < sl1; i += NT) {
      float4 x[kMaxCluster];
#pragma unroll
      for (int r = 0; r < kMaxCluster; ++r)
        if (r < nrank - 1) x[r] = ld4(cluster.map_shared_rank(sS, r) + 4 * i);
      float4 run = x[0];
#pragma unroll
      for (int r = 1; r < kMaxCluster; ++r)
        if (r < nrank) {
          st4(cluster.map_shared_rank(sS, r) + 4 * i, run);
          if (r < nrank - 1) run.x += x[r].x, run.y += x[r].y, run.z += x[r].z, run.w += x[r].w;
        }
    }
    if (t < D) {
      float part[kMaxCluster];
#pragma unroll
      for (int r = 0; r < kMaxCluster; ++r)
        if (r < rank) part[r] = cluster.map_shared_rank(sz, r)[t];
      if (rank > 0) zr = 0.f;
#pragma unroll
      for (int r = 0; r < kMaxCluster; ++r)
        if (r < rank) zr += part[r];
    }
    load_halo(seg0);                                         // (before anybody stores an output: o may lie on v)
    cluster.sync();                                          // the prefixes are in place
    if (rank > 0) {
#pragma unroll
      for (int g = 0; g < A; ++g)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int c = 0; c < G; ++c) s[g][i][c] = ld4(sS + (4 * TY * g + 4 * ty + i) * D + 64 * c + 4 * tx);
      if (t < D) sz[t] = zr;
    }
    if (rank == 0) {                                         // the first segment starts from the caller's state
#pragma unroll
      for (int g = 0; g < A; ++g)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int c = 0; c < G; ++c)
            s[g][i][c] = init ? ld4(Sb + (size_t)(4 * TY * g + 4 * ty + i) * D + 64 * c + 4 * tx) : make_float4(0.f, 0.f, 0.f, 0.f);
      zr = t < D && init ? zb[t] : 0.f;
    }
  }
  if (rank == 0) publish();

  float4 x[LD];
  {                                                          // the first chunk
    const int n = min(C, seg1 - seg0);
    float4 y[LD];
    fetch(x, k, seg0, n);
    fetch(y, q, seg0, n);
    if (nrank == 1) load_halo(seg0);
    put_phi(x, sk, n);
    fetch(x, v, seg0, n);
    put_phi(y, sq, n);
    put_v(x);
  }
  for (int i0 = seg0; i0 < seg1; i0 += C) {
    const int n = min(C, seg1 - i0), nn = min(C, seg1 - i0 - C);
    const bool more = nn > 0;
    __syncthreads();                                         // the chunk, the state and z before it are in place

    // P = phi(Q) phi(K)^T, the blocks of TY rows x 16 columns that reach the diagonal or lie below it
    float p[R][CB];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int c = 0; c < CB; ++c) p[r][c] = 0.f;
#pragma unroll 4
    for (int a = 0; a < D; a += 4) {
      float4 kk[CB];
#pragma unroll
      for (int c = 0; c < CB; ++c) kk[c] = ld4(sk + (tx + 16 * c) * QS + a);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float4 qq = ld4(sq + (ty + TY * r) * QS + a);
#pragma unroll
        for (int c = 0; c < CB; ++c)
          if (16 * c < TY * (r + 1))
            p[r][c] = fmaf(qq.x, kk[c].x, fmaf(qq.y, kk[c].y, fmaf(qq.z, kk[c].z, fmaf(qq.w, kk[c].w, p[r][c]))));
      }
    }
    // phi(q) . z of row t / LPR, this thread's part
    float den = 0.f;
    {
      const float* qr = sq + (t / LPR) * QS;
#pragma unroll
      for (int m = 0; m < D / LPR / 4; ++m) {
        const int e = 4 * (t % LPR + LPR * m);
        const float4 a = ld4(qr + e), b = ld4(sz + e);
        den = fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, den))));
      }
    }
    // O = phi(Q) S
    float4 acc[R][G];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int g = 0; g < G; ++g) acc[r][g] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (init || i0 > 0) {
#pragma unroll 2
      for (int a = 0; a < D; a += 4) {
        float4 qq[R];
#pragma unroll
        for (int r = 0; r < R; ++r) qq[r] = ld4(sq + (ty + TY * r) * QS + a);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int g = 0; g < G; ++g) {
            const float4 b = ld4(sS + (a + i) * D + 64 * g + 4 * tx);
#pragma unroll
            for (int r = 0; r < R; ++r) fma4(acc[r][g], comp(qq[r], i), b);
          }
      }
    }
    if (more || last_rank) absorb();                         // (nobody needs the sums behind an inner segment)
    __syncthreads();                                         // phi(q), phi(k) and the state copy have been read
#pragma unroll
    for (int r = 0; r < R; ++r)                              // the masked P takes the place of phi(q)
#pragma unroll
      for (int c = 0; c < CB; ++c)
        sq[(ty + TY * r) * PS + tx + 16 * c] = tx + 16 * c <= ty + TY * r ? p[r][c] : 0.f;
    if (more || last_rank) z_total();
    if (more) {
      publish();
      fetch(x, k, i0 + C, nn);                               // in flight beside the product with V
    }
    __syncthreads();
    {
      const float* pr = sq + (t / LPR) * PS;
#pragma unroll
      for (int m = 0; m < C / LPR / 4; ++m) {
        const float4 a = ld4(pr + 4 * (t % LPR + LPR * m));
        den += (a.x + a.y) + (a.z + a.w);
      }
#pragma unroll
      for (int m = LPR / 2; m > 0; m >>= 1) den += __shfl_xor_sync(0xffffffffu, den, m);
      if (t % LPR == 0) sden[t / LPR] = den;
    }
    // O += (P o M) V, TY tokens at a time, which meet TY rows on the diagonal and all those below.  The tokens behind a row are
    // left out, not met with a zero: where v is not finite that would be a NaN in the rows before it.
#pragma unroll
    for (int b = 0; b < R; ++b) {
#pragma unroll 2
      for (int j = 0; j < TY; j += 4) {
        float4 pp[R];
#pragma unroll
        for (int r = b; r < R; ++r) pp[r] = ld4(sq + (ty + TY * r) * PS + TY * b + j);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int g = 0; g < G; ++g) {
            const float4 vv = ld4(svc + (TY * b + j + i) * D + 64 * g + 4 * tx);
            if (j + i <= ty) fma4(acc[b][g], comp(pp[b], i), vv);
#pragma unroll
            for (int r = b + 1; r < R; ++r) fma4(acc[r][g], comp(pp[r], i), vv);
          }
      }
    }
    if (more) {
      put_phi(x, sk, nn);
      fetch(x, q, i0 + C, nn);                               // in flight beside the epilogue
    }
    __syncthreads();                                         // denominators in place, P has been read
    // o = O / (den + eps) + conv
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float d = sden[ty + TY * r] + eps;
#pragma unroll
      for (int g = 0; g < G; ++g)
        acc[r][g] = make_float4(acc[r][g].x / d, acc[r][g].y / d, acc[r][g].z / d, acc[r][g].w / d);
    }
    for (int tap = 0; tap < W; ++tap) {
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const int e = 64 * g + 4 * tx;
        const float4 a = ld4(sw + tap * D + e);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const float4 b = ld4(svc + (ty + TY * r - tap) * D + e);
          acc[r][g].x = fmaf(a.x, b.x, acc[r][g].x);
          acc[r][g].y = fmaf(a.y, b.y, acc[r][g].y);
          acc[r][g].z = fmaf(a.z, b.z, acc[r][g].z);
          acc[r][g].w = fmaf(a.w, b.w, acc[r][g].w);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (ty + TY * r < n)
#pragma unroll
        for (int g = 0; g < G; ++g) gst4(o + base + (size_t)(i0 + ty + TY * r) * D + 64 * g + 4 * tx, acc[r][g]);
    if (more) {
      put_phi(x, sq, nn);
      fetch(x, v, i0 + C, nn);
      // The rows before the next chunk are the last W - 1 of this one: from shared memory, not from v, where the outputs may
      // stand by now (a call in place, o = v).
      constexpr int HP = (LA_MAX_TAPS - 1) * D / 4 / NT + 1; // pieces per thread
      float4 y[HP];
#pragma unroll
      for (int it = 0; it < HP; ++it)
        if (t + it * NT < (W - 1) * (D / 4)) y[it] = ld4(sv + C * D + (t + it * NT) * 4);
      __syncthreads();                                       // v has been read
#pragma unroll
      for (int it = 0; it < HP; ++it)
        if (t + it * NT < (W - 1) * (D / 4)) st4(sv + (t + it * NT) * 4, y[it]);
      put_v(x);
    }
  }

  // The first segment reads the caller's window, the last one overwrites it.
  if (nrank > 1) cluster.sync();
  else __syncthreads();
  if (!last_rank) return;
#pragma unroll
  for (int g = 0; g < A; ++g)
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int c = 0; c < G; ++c) st4(Sb + (size_t)(4 * TY * g + 4 * ty + i) * D + 64 * c + 4 * tx, s[g][i][c]);
  if (t < D) {
    zb[t] = zr;
    const float* tail = sv + ((seg1 - seg0 - 1) % C + 1) * D + t;   // behind the tokens of the last chunk
    for (int i = 0; i < W - 1; ++i) wb[(size_t)i * D + t] = from_f32<T>(tail[i * D]);
  }
  if (h == 0 && t == 0) pos[bh / H] = (init ? pos[bh / H] : 0) + Tlen;
}

template <typename T, int D, int PHI>
static cudaError_t launch_t(la_ctx* ctx, int B, int Tlen, const void* q, const void* k, const void* v, const float* w,
                            int init, const la_state& st, void* o, cudaStream_t s) {
  using Sh = Shape<D>;
  const la_config& c = ctx->cfg;
  auto kern = prefill_simt_kernel<T, D, PHI>;
  const size_t smem = Sh::bytes(c.conv_taps);
  cudaError_t e = allow_smem((const void*)kern, ctx->device);
  if (e != cudaSuccess) return e;
  // CTAs per chain, each a segment of whole chunks: a whole cluster, until the chains alone fill half of the places for
  // CTAs.  (d = 64, 1000 tokens, us by CTAs per chain, as first measured: 48 chains 196 with 1, 126 with 2, 94 with 4, 67 with 8; 192 chains
  // 287, 254, 254, 254; 384 chains 374 and 480-510.  d = 128, 300 tokens: 48 chains 135, 95, 113, 86; 96 chains 135 and
  // 168-188.)
  const int BH = B * c.H, chunks = (Tlen + Sh::C - 1) / Sh::C;
  int n = 2 * BH >= ctx->sm_count * Sh::kResident ? 1 : std::min((int)kMaxCluster, chunks);
  const int per = (chunks + n - 1) / n;
  n = (chunks + per - 1) / per;
  ctx->launches += 1;
  return launch_cluster(n, false, kern, dim3(BH * n), dim3(Sh::NT), smem, s, (const T*)q, (const T*)k, (const T*)v, w, st.S, st.z,
                        (T*)st.win, st.pos, (T*)o, c.H, Tlen, c.conv_taps, c.eps, init, per * Sh::C);
}

template <typename T, int D>
static cudaError_t launch_phi(la_ctx* ctx, int B, int Tlen, const void* q, const void* k, const void* v, const float* w,
                              int init, const la_state& st, void* o, cudaStream_t s) {
  return ctx->cfg.phi == LA_PHI_ELU1 ? launch_t<T, D, LA_PHI_ELU1>(ctx, B, Tlen, q, k, v, w, init, st, o, s)
                                     : launch_t<T, D, LA_PHI_RELU>(ctx, B, Tlen, q, k, v, w, init, st, o, s);
}

}  // namespace simt

// Whether walking the tokens (prefill_walk.cu) is faster: a chunk costs the same however few tokens it holds.  One line per
// number of chunks, in tokens, from both kernels at 50 lengths x 17 numbers of chains (fp32, 3 taps; us walked / in chunks):
//   d = 64    up to one chain per SM: 25 tokens (24 13.4 / 14.0, 26 14.3 / 14.8, 28 15.2 / 14.8; 1 tap: 24 12.5 / 13.1, 26 13.3 /
//             13.2), 22 with ReLU, which is cheap for a whole chunk (22 13.8 / 13.8, 24 14.7 / 13.6).  Up to three, as many
//             blocks as an SM holds: 28 and 25 (256 chains: 26 17 / 18, 30 18.6 / 18; ReLU: 25 17.8 / 17.9, 27 19 / 18.2).  Beyond, blocks wait for a place: 45 tokens per chunk (512 chains: 40
//             tokens 34 / 37, 48 40 / 37; 82 66 / 75, 96 76 / 74; 129 102 / 113; 1024 chains: 40 60 / 58, 76 115 / 120)
//   d = 128   up to one chain per SM, as many chunked blocks as an SM holds: 19.5 per chunk (14 tokens 12.6 / 13.0, 16 13.4 /
//             12.8; 33 24 / 25.6).  Beyond: 28.5 (160 chains: 22 tokens 23.5 / 24, 24 25.6 / 24; 48 46 / 50; 161 144 / 160; 512
//             chains: 48 95 / 102, 136 267 / 277), and 24.5 where the chains of the last pair of chunked waves, which is one
//             wave walked, fill half of it (1024 chains: 18 tokens 85 / 88, 44 183 / 190)
static bool walks(int d, bool relu, int BH, int T, int sms) {
  if (d == 64) return BH <= 3 * sms ? T <= (BH > sms ? (relu ? 25 : 28) : (relu ? 22 : 25)) : T + 4 <= 45 * ((T + 63) / 64);
  const int waves = (BH + sms - 1) / sms;
  return 2 * (T + 5) <= (waves == 1 ? 39 : waves % 2 == 0 ? 57 : 49) * ((T + 31) / 32);
}

cudaError_t launch_prefill_simt(la_ctx* ctx, int B, int Tlen, const void* q, const void* k, const void* v,
                                const float* w, int init, const la_state& st, void* o, cudaStream_t s) {
  const la_config& c = ctx->cfg;
  if (walks(c.d, c.phi == LA_PHI_RELU, B * c.H, Tlen, ctx->sm_count)) return launch_prefill_walk(ctx, B, Tlen, q, k, v, w, init, st, o, s);
  if (c.io_dtype == LA_F32)
    return c.d == 64 ? simt::launch_phi<float, 64>(ctx, B, Tlen, q, k, v, w, init, st, o, s)
                     : simt::launch_phi<float, 128>(ctx, B, Tlen, q, k, v, w, init, st, o, s);
  return c.d == 64 ? simt::launch_phi<__nv_bfloat16, 64>(ctx, B, Tlen, q, k, v, w, init, st, o, s)
                   : simt::launch_phi<__nv_bfloat16, 128>(ctx, B, Tlen, q, k, v, w, init, st, o, s);
}

}  // namespace la
