// Commit of the accepted draft path (Sec. 4.2: later tokens interact with the verified
// tokens of earlier groups).  Per (sequence, head): rebuild the root-to-node path from
// the parent array (integer work, bit-exact), then stream the d x d state once, adding the
// rank-1 updates of all path tokens in order, and advance z, the convolution window and pos.
// The loads of the state are issued first, so that they are in flight while the path is rebuilt and the path
// tokens are gathered.
#include "la_common.cuh"
#include "la_internal.h"

namespace la {

// The d x d state of one (sequence, head) unit is shared out among kCommitSplit CTAs (a band of rows each), so that
// a launch of few units still spreads evenly over the SMs; the first of them also advances z and the window.
constexpr int kCommitSplit = 4;

// Shared memory: phi(k) and v of the path tokens (max_depth rows each), then the integer tables.
struct CommitTables {
  int par[LA_MAX_NODES];
  int path[LA_MAX_NODES];
  int len;
  int bad;
};

// d = 64 keeps to 32 registers, eight blocks per SM: with the 48 that the window's eight rows in flight take, 1024 units took
// 12.8 us instead of 10.6 (3 taps; few units and 32 taps, on the other hand, 5.2 instead of 6.4).
template <typename T, int D, int PHI, int BLOCKS>
__global__ void __launch_bounds__(256, BLOCKS)
commit_kernel(const T* __restrict__ k, const T* __restrict__ v, const int32_t* __restrict__ parent,
              const int32_t* __restrict__ accept, float* __restrict__ S, float* __restrict__ z, T* __restrict__ win,
              int64_t* __restrict__ pos, int32_t* __restrict__ path_out, int32_t* __restrict__ commit_len, int* status,
              int H, int N, int W, int max_depth, int fresh) {
  constexpr int TPR = D / 4, RPP = 256 / TPR, ROWS = D / kCommitSplit, PASSES = ROWS / RPP;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float (*fk)[D] = reinterpret_cast<float (*)[D]>(smem_raw);
  float (*vv)[D] = fk + max_depth;
  CommitTables& sm = *reinterpret_cast<CommitTables*>(vv + max_depth);
  const int bh = blockIdx.x / kCommitSplit, part = blockIdx.x % kCommitSplit, b = bh / H, h = bh % H, t = threadIdx.x;

  pdl_wait();                      // the kernel before this one in the stream may still be running until here
  pdl_trigger();
  // The state is requested before anything else: the loads are in flight while the path is rebuilt.
  const int c4 = (t % TPR) * 4, rg = part * ROWS + t / TPR;   // this CTA's rows of S: part * ROWS .. + ROWS - 1
  float* Sb = S + (size_t)bh * D * D;
  float4 s[PASSES];
#pragma unroll
  for (int m = 0; m < PASSES; ++m) s[m] = __ldcs(reinterpret_cast<const float4*>(Sb + (size_t)(rg + RPP * m) * D + c4));

  if (t < N) sm.par[t] = parent[(size_t)b * N + t];
  __syncthreads();
  if (t == 0) {
    int a = accept[b], L = 0, bad = 0;     // (requested ahead of the tree it cost launches of many units 4 %)
    if (a < -1 || a >= N) bad = 1;
    int m = bad ? -1 : a;
    while (m >= 0) {                       // m strictly decreases: terminates
      if (L >= max_depth) { bad = 1; break; }
      sm.path[L++] = m;
      const int p = sm.par[m];
      if (p < -1 || p >= m) { bad = 1; break; }
      m = p;
    }
    for (int i = 0; i < L / 2; ++i) {      // root first
      const int x = sm.path[i];
      sm.path[i] = sm.path[L - 1 - i];
      sm.path[L - 1 - i] = x;
    }
    sm.len = L;
    sm.bad = bad;
  }
  __syncthreads();
  if (sm.bad) {
    if (t == 0) report(status, LA_ERR_BAD_TREE);
    if (h == 0 && part == 0) {             // buffers whose contents nobody has seen yet
      if (fresh & LA_FRESH_PATH)
        for (int i = t; i < max_depth; i += 256) path_out[(size_t)b * max_depth + i] = -1;
      if ((fresh & LA_FRESH_LEN) && t == 0) commit_len[b] = 0;
    }
    return;
  }
  const int L = sm.len;
  if (h == 0 && part == 0) {
    for (int i = t; i < max_depth; i += 256) path_out[(size_t)b * max_depth + i] = i < L ? sm.path[i] : -1;
    if (t == 0) commit_len[b] = L;
  }
  if (L == 0) return;

  const size_t base = (size_t)bh * N * D;
  for (int idx = t; idx < L * D; idx += 256) {
    const int l = idx / D, e = idx % D;
    const size_t g = base + (size_t)sm.path[l] * D + e;
    fk[l][e] = phi<PHI>(to_f32(k[g]));
    vv[l][e] = to_f32(v[g]);
  }
  __syncthreads();

  for (int l = 0; l < L; ++l) {
    const float4 v4 = *reinterpret_cast<const float4*>(&vv[l][c4]);
#pragma unroll
    for (int m = 0; m < PASSES; ++m) {
      const float a = fk[l][rg + RPP * m];
      s[m].x = fmaf(a, v4.x, s[m].x);
      s[m].y = fmaf(a, v4.y, s[m].y);
      s[m].z = fmaf(a, v4.z, s[m].z);
      s[m].w = fmaf(a, v4.w, s[m].w);
    }
  }
#pragma unroll
  for (int m = 0; m < PASSES; ++m) __stcs(reinterpret_cast<float4*>(Sb + (size_t)(rg + RPP * m) * D + c4), s[m]);

  if (part == 0 && t < D) {
    float zz = z[(size_t)bh * D + t];
    for (int l = 0; l < L; ++l) zz += fk[l][t];
    z[(size_t)bh * D + t] = zz;
    // window <- last W-1 entries of (window ++ v_path); ascending, source index above target.  Eight rows at a time, their
    // loads in flight together (row by row, each waited for the store before it: 4 us at 8 taps).
    T* wb = win + (size_t)bh * (W - 1) * D + t;
    for (int i0 = 0; i0 < W - 1; i0 += 8) {
      T x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int src = L + i0 + i;
        if (i0 + i < W - 1) x[i] = src < W - 1 ? wb[(size_t)src * D] : from_f32<T>(vv[src - (W - 1)][t]);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (i0 + i < W - 1) wb[(size_t)(i0 + i) * D] = x[i];
    }
  }
  if (h == 0 && part == 0 && t == 0) pos[b] += L;
}

template <int D> static size_t commit_smem(const la_config& c) {
  return (size_t)2 * c.max_depth * D * sizeof(float) + sizeof(CommitTables);
}

template <typename T, int D, int PHI, int BLOCKS>
static cudaError_t launch_b(la_ctx* ctx, int B, int N, const void* k, const void* v, const int32_t* parent,
                            const int32_t* accept, const la_state& st, int32_t* path_out, int32_t* commit_len, int fresh,
                            cudaStream_t s) {
  const la_config& c = ctx->cfg;
  auto kern = commit_kernel<T, D, PHI, BLOCKS>;
  const size_t smem = commit_smem<D>(c);
  cudaError_t e = allow_smem((const void*)kern, ctx->device);
  if (e != cudaSuccess) return e;
  ctx->launches += 1;
  return launch_pdl(kern, dim3(B * c.H * kCommitSplit), dim3(256), smem, s, (const T*)k, (const T*)v, parent, accept, st.S,
                    st.z, (T*)st.win, st.pos, path_out, commit_len, ctx->d_status, c.H, N, c.conv_taps, c.max_depth, fresh);
}

template <typename T, int D, int PHI>
static cudaError_t launch_t(la_ctx* ctx, int B, int N, const void* k, const void* v, const int32_t* parent,
                            const int32_t* accept, const la_state& st, int32_t* path_out, int32_t* commit_len, int fresh,
                            cudaStream_t s) {
  if constexpr (D == 64) {
    return launch_b<T, D, PHI, 8>(ctx, B, N, k, v, parent, accept, st, path_out, commit_len, fresh, s);
  } else {
    // Six blocks per SM (40 registers; a ReLU spills 4 bytes, measured with them) or five (48).  Six where the launch then takes one
    // wave instead of two (a few blocks more find room as the first end), and from three waves of five on: 186 ... 228 units
    // 0.89-0.99 of the time of five, 372 ... 1280 units 0.94-0.99 (3 taps, both types, both phi); between them, in two waves either
    // way, 0.99-1.03; 128 ... 184 units are one wave of five, 1.05-1.08 of whose time six took.  And only while six blocks leave most
    // of the SM's memory to the L1, through which everything else goes: 512 and 1024 units 0.97 and 0.94 up to max_depth 24, 0.98 and
    // 0.98 at 26, 0.99 and 1.00 at 28, 1.08 and 1.20 at 32.
    const int blocks = B * ctx->cfg.H * kCommitSplit, sms = ctx->sm_count;
    const bool six = ((blocks > 5 * sms && 5 * blocks <= 31 * sms) || blocks > 10 * sms) && 6 * commit_smem<D>(ctx->cfg) <= 160u * 1024u;
    return six ? launch_b<T, D, PHI, 6>(ctx, B, N, k, v, parent, accept, st, path_out, commit_len, fresh, s)
               : launch_b<T, D, PHI, 5>(ctx, B, N, k, v, parent, accept, st, path_out, commit_len, fresh, s);
  }
}

template <typename T, int D>
static cudaError_t launch_phi(la_ctx* ctx, int B, int N, const void* k, const void* v, const int32_t* parent,
                              const int32_t* accept, const la_state& st, int32_t* path_out, int32_t* commit_len, int fresh,
                              cudaStream_t s) {
  return ctx->cfg.phi == LA_PHI_ELU1
             ? launch_t<T, D, LA_PHI_ELU1>(ctx, B, N, k, v, parent, accept, st, path_out, commit_len, fresh, s)
             : launch_t<T, D, LA_PHI_RELU>(ctx, B, N, k, v, parent, accept, st, path_out, commit_len, fresh, s);
}

cudaError_t launch_commit(la_ctx* ctx, int B, int N, const void* k, const void* v, const int32_t* parent,
                          const int32_t* accept, const la_state& st, int32_t* path_out, int32_t* commit_len, int fresh,
                          cudaStream_t s) {
  const la_config& c = ctx->cfg;
  if (c.io_dtype == LA_F32)
    return c.d == 64 ? launch_phi<float, 64>(ctx, B, N, k, v, parent, accept, st, path_out, commit_len, fresh, s)
                     : launch_phi<float, 128>(ctx, B, N, k, v, parent, accept, st, path_out, commit_len, fresh, s);
  return c.d == 64 ? launch_phi<__nv_bfloat16, 64>(ctx, B, N, k, v, parent, accept, st, path_out, commit_len, fresh, s)
                   : launch_phi<__nv_bfloat16, 128>(ctx, B, N, k, v, parent, accept, st, path_out, commit_len, fresh, s);
}

}  // namespace la
