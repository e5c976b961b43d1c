// Learned warm start for the constant-potential solve (the learned form): a per-electrode-site MLP
// (80 -> 128 -> 128 -> 1, SiLU; FP32 parameters, forward GEMMs on the tensor cores) maps local
// electrolyte descriptors to the unprojected solution
// y = A^-1 (dpsi d + b) of the charge update (Eqs. 9-10), which seeds the PCG iteration.
//
// Descriptors of site j (80 floats):
//   0..31   sum over ions with q > 0 within rc of  |q| exp(-(r - mu_b)^2 / (2 s^2)), mu_b = 0.25 + b / 31 nm
//   32..63  the same for ions with q < 0
//   64..79  Re, Im of exp(-i k_z Z_j) S1(k_z) for k_z = 2 pi m / L_z, m = 1..8 (the lowest k_z modes
//           that the symmetry-preserving set I keeps, Eqs. 15 and 24)
// Inputs and the target are standardised with the training set's mean and spread, which are part of
// the parameter vector.  Training minimises the mean squared error with AdamW; the activations of a
// minibatch come from one kernel, the weight gradients (sums over the rows in a fixed order) and the
// AdamW update from a second.
#include "sfu.cuh"
#include "srbe_internal.cuh"
#include "tc.cuh"

namespace srbe {

constexpr int kIn = 80, kH = 128;
constexpr int kNbasis = 32, kNlow = 8;
constexpr float kRbfSigma = 0.035f;
// parameter layout
constexpr int oW1 = 0, oB1 = oW1 + kH * kIn, oW2 = oB1 + kH, oB2 = oW2 + kH * kH, oW3 = oB2 + kH, oB3 = oW3 + kH,
              oXm = oB3 + 1, oXs = oXm + kIn, oYm = oXs + kIn, oYs = oYm + 1, kNparam = oYs + 1;
constexpr int kNtrain = oXm;     // trainable entries come first

// z / (1 + e^-z); below -87, where it is -5e-36 and less, e^87 keeps the divisor a normal number
__device__ __forceinline__ float silu(float z) {
  const float d = 1.f + exp_n(fminf(-z, 87.f));
  return quotient(z, d, rcp_n(d));
}

// S_low[m] = sum_i q_i exp(i 2 pi m z_i / L_z), m = 1..8: one partial per block of 256 ions (Re, Im of
// the 8 modes), added in block order by the descriptors.  (One block over all ions: 98 us at 8,000.)
constexpr int kLowBlocks = 64;
__global__ void __launch_bounds__(256)
k_low_modes(int64_t n, const double *__restrict__ z, const double *__restrict__ q, double invLz,
            double *__restrict__ part) {
  __shared__ double red[8][2 * kNlow];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  double a[2 * kNlow];
#pragma unroll
  for (int m = 0; m < 2 * kNlow; ++m) a[m] = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * 256 + t; i < n; i += (int64_t)gridDim.x * 256) {
    const uint64_t u = to_turns64(z[i], invLz);
    const double w = q[i];
#pragma unroll
    for (int m = 0; m < kNlow; ++m) {
      float c, s;
      sincos_turns32((uint32_t)((u * (uint64_t)(m + 1)) >> 32), c, s);
      a[2 * m] += w * c;
      a[2 * m + 1] += w * s;
    }
  }
#pragma unroll
  for (int m = 0; m < 2 * kNlow; ++m) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a[m] += __shfl_xor_sync(0xffffffffu, a[m], o);
    if (lane == 0) red[warp][m] = a[m];
  }
  __syncthreads();
  if (t < 2 * kNlow) {
    double s = red[0][t];
    for (int w = 1; w < 8; ++w) s += red[w][t];
    part[blockIdx.x * 2 * kNlow + t] = s;
  }
}

// descriptors, one warp per electrode site; lane b owns basis function b
__global__ void __launch_bounds__(256)
k_descriptors(int64_t ne, const double *__restrict__ ex, const double *__restrict__ ey, const double *__restrict__ ez,
              const float4 *__restrict__ ion_pf, const int32_t *__restrict__ ei, const int32_t *__restrict__ ei_n,
              int cap, float Lx, float Ly, float rc2, const double2 *__restrict__ low, int nlow, double invLz,
              float *__restrict__ D) {
  const int lane = threadIdx.x & 31;
  const int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (j >= ne) return;
  const float X = (float)ex[j], Y = (float)ey[j], Z = (float)ez[j];
  const float mu = 0.25f + lane * (1.0f / 31.0f);
  const float inv2s2 = 1.0f / (2.0f * kRbfSigma * kRbfSigma);
  float pos = 0.f, neg = 0.f;
  const int cnt = min(ei_n[j], cap);
  for (int base = 0; base < cnt; base += 32) {
    const int k = base + lane;
    float r = 0.f, qv = 0.f;
    if (k < cnt) {
      const int32_t e = ei[j * (int64_t)cap + k];
      const int idx = e & 0x7fffff, ix = ((e >> 24) & 15) - 8, iy = ((unsigned)e >> 28) - 8;
      const float4 o = ion_pf[idx];
      const float dx = X - (o.x + ix * Lx), dy = Y - (o.y + iy * Ly), dz = Z - o.z;
      const float r2 = dx * dx + dy * dy + dz * dz;
      if (r2 < rc2) {
        r = sqrtf(r2);
        qv = o.w;
      }
    }
    const int m = min(32, cnt - base);
    for (int l = 0; l < m; ++l) {
      const float rl = __shfl_sync(0xffffffffu, r, l), ql = __shfl_sync(0xffffffffu, qv, l);
      if (ql == 0.f) continue;
      const float g = fabsf(ql) * __expf(-(rl - mu) * (rl - mu) * inv2s2);
      if (ql > 0.f) pos += g;
      else neg += g;
    }
  }
  float *row = D + j * (int64_t)kIn;
  row[lane] = pos;
  row[32 + lane] = neg;
  if (lane < kNlow) {
    // exp(-i k Z) S(k) with k = 2 pi (m + 1) / L_z
    const uint64_t u = to_turns64(ez[j], invLz);
    float c, s;
    sincos_turns32((uint32_t)((u * (uint64_t)(lane + 1)) >> 32), c, s);
    double2 S = make_double2(0.0, 0.0);
#pragma unroll 8
    for (int b = 0; b < nlow; ++b) {
      const double2 v = __ldg(low + b * kNlow + lane);
      S.x += v.x;
      S.y += v.y;
    }
    row[64 + 2 * lane] = (float)(c * S.x + s * S.y);
    row[64 + 2 * lane + 1] = (float)(c * S.y - s * S.x);
  }
}

// ------------------------------------------------------------------------------------------------
// forward pass on the tensor cores (tcgen05): 128 rows per tile, Z1 = X W1^T and Z2 = H1 W2^T as
// kind::f16 MMAs into tensor memory with FP32 accumulation.  Every operand is split into BF16
// (hi, lo) and each product taken as hi hi + hi lo + lo hi, which keeps about 16 significand bits
// (the scalar FP32 path keeps 24; the difference stays below 1e-5 of the output here).
//
// The special-function unit bounds it (two operations per SiLU, 256 SiLUs per row: 2.1 us per tile and
// SM) as long as nothing else waits, so one CTA per SM runs two groups of 8 warps, each with a tile of
// its own: while one group waits for its loads, its MMAs or a barrier the other computes.  A group's
// 40 KB operand buffer holds X and then, since X is dead once Z1 is complete, each half of H1 in turn
// (64 columns: K steps 0-3, then 4-7 of the second layer), so that the weights (104 KB) and both
// groups fit the shared memory.  The next tile's rows are loaded into registers while the first layer
// runs.  The weights come already split and blocked from k_mlp_split.
// 98,304 rows: 33 us; 66 us with one tile in flight per SM, the weights split by every CTA and IEEE divisions in
// the SiLU and the standardisation.  3,072 rows: 26.5 -> 14 us.  The quotients are corrected ones (sfu.cuh): with
// plain products by the reciprocal (30 us) the error against 64 bits was 1.0012 +- 0.0003 of the divisions' over
// 80 networks of 4,000 rows, with the correction 1.0001 +- 0.0001 (6.84e-6, which is the BF16 split's).
// ------------------------------------------------------------------------------------------------
constexpr int kTcK1 = kIn / tc::kKstep;    // 5 K steps of layer 1
constexpr int kTcK2 = kH / tc::kKstep;     // 8 K steps of layer 2
constexpr int kTcWeights = (2 * kTcK1 + 2 * kTcK2) * tc::kBlockElems;               // BF16 elements
constexpr int kTcGroup = 256;              // threads of a group: 8 warps, two per tensor-memory lane quarter
constexpr int kTcThreads = 2 * kTcGroup;
constexpr int kTcBuf = 2 * kTcK1 * tc::kBlockElems;                                  // X (hi, lo); H1 half needs 8 blocks
constexpr size_t kTcSmem = (size_t)(kTcWeights + 2 * kTcBuf) * 2;                    // 184 KB
constexpr int kTcPolls = 1 << 20;          // bounded mbarrier waits
static_assert(kIn % tc::kKstep == 0 && kH == tc::kRows && kTcK2 <= 2 * kTcK1, "MLP sizes must match the MMA tiles");

// W1 and W2 as (hi, lo) BF16 operands in the MMA's blocked layout: W1 hi, W1 lo, W2 hi, W2 lo
__global__ void k_mlp_split(const float *__restrict__ P, __nv_bfloat16 *__restrict__ W) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  __nv_bfloat16 *w1h = W, *w1l = w1h + kTcK1 * tc::kBlockElems, *w2h = w1l + kTcK1 * tc::kBlockElems,
                *w2l = w2h + kTcK2 * tc::kBlockElems;
  if (i < kH * kIn) {
    const int h = i / kIn, k = i - h * kIn;
    tc::split_bf16(P[oW1 + i], w1h[tc::off(h, k)], w1l[tc::off(h, k)]);
  }
  if (i < kH * kH) {
    const int h = i / kH, k = i - h * kH;
    tc::split_bf16(P[oW2 + i], w2h[tc::off(h, k)], w2l[tc::off(h, k)]);
  }
}

// barrier of one group, and with an OR over its threads
__device__ __forceinline__ void group_sync(int g) {
  asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(kTcGroup) : "memory");
}
__device__ __forceinline__ bool group_any(int g, bool v) {
  uint32_t r;
  asm volatile("{\n .reg .pred p, q;\n setp.ne.u32 q, %1, 0;\n bar.red.or.pred p, %2, %3, q;\n selp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(r)
               : "r"(v ? 1u : 0u), "r"(g + 1), "r"(kTcGroup)
               : "memory");
  return r != 0;
}

__global__ void __launch_bounds__(kTcThreads, 1)
k_mlp_forward_tc(int64_t n, const float *__restrict__ D, const float *__restrict__ P,
                 const __nv_bfloat16 *__restrict__ W, float *__restrict__ out, double *__restrict__ out_y,
                 int *__restrict__ status) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __nv_bfloat16 *w1h = reinterpret_cast<__nv_bfloat16 *>(smem);
  const __nv_bfloat16 *w1l = w1h + kTcK1 * tc::kBlockElems, *w2h = w1l + kTcK1 * tc::kBlockElems;
  const __nv_bfloat16 *w2l = w2h + kTcK2 * tc::kBlockElems;
  __shared__ float sb1[kH], sb2[kH], sw3[kH], sxm[kIn], sxs[kIn], sxi[kIn];
  __shared__ float part[2][2][128];            // the output's partial dot products per group and column half
  __shared__ __align__(8) uint64_t mbars[2];
  __shared__ uint32_t tbase;
  const int t = threadIdx.x, g = t / kTcGroup, tg = t - g * kTcGroup, lane = t & 31, w = tg >> 5;
  // warp w of a group reads tensor-memory lanes 32 (w % 4) .. + 31 (rows of the tile) and column half w / 4
  const int quarter = w & 3, half = w >> 2, row_t = 32 * quarter + lane;
  {
    const uint4 *src = reinterpret_cast<const uint4 *>(W);
    uint4 *dst = reinterpret_cast<uint4 *>(smem);
    constexpr int kVec = kTcWeights / 8;
#pragma unroll
    for (int i = 0; i < kVec / kTcThreads; ++i) dst[t + i * kTcThreads] = __ldg(src + t + i * kTcThreads);
    static_assert(kVec % kTcThreads == 0, "the weights are copied in whole rounds");
  }
  if (t < kH) {
    sb1[t] = P[oB1 + t];
    sb2[t] = P[oB2 + t];
    sw3[t] = P[oW3 + t];
  }
  if (t < kIn) {
    sxm[t] = P[oXm + t];
    sxs[t] = P[oXs + t];
    sxi[t] = 1.0f / sxs[t];
  }
  const float b3 = P[oB3], ym = P[oYm], ys = P[oYs];
  if (t < 2) tc::mbar_init(&mbars[t], 1);
  if (t < 32) tc::tmem_alloc(&tbase, 512);
  tc::fence_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  __nv_bfloat16 *bh = w1h + kTcWeights + g * kTcBuf;       // this group's operand buffer
  __nv_bfloat16 *xl = bh + kTcK1 * tc::kBlockElems, *hl = bh + (kTcK2 / 2) * tc::kBlockElems;
  uint64_t *mbar = &mbars[g];
  const uint32_t d1 = tbase + 256u * g, d2 = d1 + 128, lanes = (uint32_t)(32 * quarter) << 16;
  const uint32_t idesc = tc::idesc_bf16(128, 128);
  const int64_t ntiles = (n + 127) / 128, step = 2 * (int64_t)gridDim.x;
  uint32_t phase = 0;
  bool fail = false;
  float4 q[kIn / 8];                            // this thread's part of a tile: row row_t, 8-wide chunks half, half + 2, ...
  auto fetch = [&](int64_t tile) {
    const bool live = tile < ntiles && tile * 128 + row_t < n;
    const float4 *src = reinterpret_cast<const float4 *>(D + (tile * 128 + row_t) * kIn);
#pragma unroll
    for (int c = 0; c < kIn / 16; ++c) {
      const int ch = half + 2 * c;
      q[2 * c] = live ? __ldg(src + 2 * ch) : make_float4(0.f, 0.f, 0.f, 0.f);
      q[2 * c + 1] = live ? __ldg(src + 2 * ch + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  // operands written by this group's threads become visible to the tensor core, then one thread issues
  auto handoff = [&] {
    tc::fence_async_smem();
    tc::fence_before_sync();
    group_sync(g);
    tc::fence_after_sync();
  };
  auto done = [&] {                             // waits for the group's last commit; false at the limit
    fail = group_any(g, !tc::mbar_wait(mbar, phase, kTcPolls));
    if (fail) return false;
    phase ^= 1u;
    tc::fence_after_sync();
    return true;
  };
  auto layer2 = [&](int s0) {                   // K steps s0 .. s0 + 3 from the H1 half in the buffer
    for (int s = 0; s < kTcK2 / 2; ++s) {
      const uint64_t ah = tc::block_desc(bh + s * tc::kBlockElems), al = tc::block_desc(hl + s * tc::kBlockElems);
      const uint64_t wh = tc::block_desc(w2h + (s0 + s) * tc::kBlockElems);
      const uint64_t wl = tc::block_desc(w2l + (s0 + s) * tc::kBlockElems);
      tc::mma_bf16(d2, ah, wh, idesc, s0 + s > 0);
      tc::mma_bf16(d2, ah, wl, idesc, true);
      tc::mma_bf16(d2, al, wh, idesc, true);
    }
    tc::commit(mbar);
  };
  // H1 = SiLU(Z1 + b1), columns 64 h + 32 half .. + 31 of this thread's row
  auto hidden = [&](int h, float *v) {
    const int c0 = 64 * h + 32 * half;
    tc::ld32(d1 + lanes + (uint32_t)c0, v);
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = silu(v[j] + sb1[c0 + j]);
  };
  auto store_hidden = [&](const float *v) {
#pragma unroll
    for (int c = 0; c < 4; ++c) tc::store8_split(bh, hl, row_t, 32 * half + 8 * c, v + 8 * c);
  };
  // tiles blockIdx.x + gridDim.x (g + 2 i): every CTA gets its first tile before any gets a second
  int64_t tile = blockIdx.x + (int64_t)gridDim.x * g;
  fetch(tile);
  for (; tile < ntiles; tile += step) {
    // standardised inputs (rows beyond n are zero)
    {
      const bool live = tile * 128 + row_t < n;
#pragma unroll
      for (int c = 0; c < kIn / 16; ++c) {
        const int k0 = 8 * (half + 2 * c);
        float v[8] = {q[2 * c].x, q[2 * c].y, q[2 * c].z, q[2 * c].w, q[2 * c + 1].x, q[2 * c + 1].y, q[2 * c + 1].z,
                      q[2 * c + 1].w};
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = live ? quotient(v[j] - sxm[k0 + j], sxs[k0 + j], sxi[k0 + j]) : 0.f;
        tc::store8_split(bh, xl, row_t, k0, v);
      }
    }
    handoff();
    if (tg == 0) {
      for (int s = 0; s < kTcK1; ++s) {
        const uint64_t ah = tc::block_desc(bh + s * tc::kBlockElems), al = tc::block_desc(xl + s * tc::kBlockElems);
        const uint64_t wh = tc::block_desc(w1h + s * tc::kBlockElems), wl = tc::block_desc(w1l + s * tc::kBlockElems);
        tc::mma_bf16(d1, ah, wh, idesc, s > 0);
        tc::mma_bf16(d1, ah, wl, idesc, true);
        tc::mma_bf16(d1, al, wh, idesc, true);
      }
      tc::commit(mbar);
    }
    fetch(tile + step);
    if (!done()) break;
    float v[32];
    hidden(0, v);
    store_hidden(v);
    handoff();
    if (tg == 0) layer2(0);
    hidden(1, v);                               // while the first half's MMAs run
    if (!done()) break;
    store_hidden(v);
    handoff();
    if (tg == 0) layer2(kTcK2 / 2);
    if (!done()) break;
    // output = W3 . SiLU(Z2 + b2) + b3: partial sums per column half, added in order
    float acc = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c0 = 64 * half + 32 * h;
      tc::ld32(d2 + lanes + (uint32_t)c0, v);
#pragma unroll
      for (int j = 0; j < 32; ++j) acc = fmaf(sw3[c0 + j], silu(v[j] + sb2[c0 + j]), acc);
    }
    part[g][half][row_t] = acc;
    tc::fence_before_sync();
    group_sync(g);
    if (tg < 128) {
      const int64_t row = tile * 128 + tg;
      if (row < n) {
        const float y = (part[g][0][tg] + part[g][1][tg] + b3) * ys + ym;
        if (out) out[row] = y;
        if (out_y) out_y[row] = (double)y;
      }
    }
  }
  if (fail) {
    // an MMA did not complete within the limit: raise the flag, give it one more bounded wait, then
    // release the tensor memory and return
    if (tg == 0) *(volatile int *)(status + kStatTimeout) = 1;
    tc::mbar_wait(mbar, phase, kTcPolls);
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (t < 32) tc::tmem_dealloc(tbase, 512);
}

// Training pass (forward + backward of the standardised MSE loss), FP32 on the CUDA cores, two kernels:
//
// k_mlp_rows: a block stages W1 and W2 in shared memory once (odd row strides: both the row reads of the
//   forward pass and the column reads of the backward pass are free of bank conflicts) and walks tiles
//   of R rows; thread (h, half) owns hidden unit h and half of each dot product, the R rows of a tile are
//   R independent FMA chains that share every weight read.  It writes the activations the weight
//   gradients need: x, h1, dz1, dz2 and dout a2 per row.
// k_mlp_wgrad: the weight gradients as products over the rows, dz2^T h1 and dz1^T x, one 16 x 16 tile of
//   an output matrix per block, four row groups per block added in order, so that the small reduction
//   (a minibatch) still fills the GPU; bias, W3 and loss sums in blocks of their own.  With one row
//   split the same kernel applies AdamW, else a third kernel adds the splits in order.
//
// One block per row chunk with the gradient in shared memory and the weights read from global memory
// (every thread its own row: uncoalesced, and 32-way bank conflicts on the gradient) took 440 us per
// 512-row minibatch on GB300, host synchronisation included.
constexpr int kTrThreads = 256;
constexpr int kW1s = kIn + 1, kW2s = kH + 1;            // shared-memory row strides (odd)
constexpr int64_t kTrSplit = 1024;                       // rows per split of the weight gradients
// rows whose activations (156 MB) and split gradients (7 MB) are kept at once.  (With 38,912 rows, 92 MB, the gradients
// of 300,000 rows take 4.18 instead of 4.10 ms, with 19,456 rows 4.33, host copies included.)
constexpr int64_t kTrChunk = 65536;
static_assert(kTrChunk % kTrSplit == 0, "a chunk is a whole number of splits");
constexpr int kTrStage = 128;                            // rows staged per step of k_mlp_wgrad
constexpr int kTile = 16;
constexpr int kTilesW2 = (kH / kTile) * (kH / kTile), kTilesW1 = (kH / kTile) * (kIn / kTile);
constexpr int kColBlocks = 3 * kH / 32;                  // b1, b2, W3: 32 columns per block
constexpr int kWgradBlocks = kTilesW2 + kTilesW1 + kColBlocks + 1;
static_assert(kH % 32 == 0 && kIn % kTile == 0 && kTrStage % 8 == 0, "MLP sizes must match the gradient tiles");

struct TrainAct {                                        // per-row activations of one chunk, row-major
  float *x, *h1, *dz1, *dz2, *a3;                        // [n][kIn], [n][kH] x 4 (a3 = dout SiLU(z2))
  float2 *out;                                           // (dout, err)
};

// the training pass takes the correctly scaled exponential (the fast one is 2 ulp and more off): its
// cost is hidden behind the dot products, and the gradients come out closer to their 64-bit values
__device__ __forceinline__ float silu_train(float z) { return z / (1.f + expf(-z)); }
__device__ __forceinline__ float silu_grad_train(float z) {
  const float s = 1.f / (1.f + expf(-z));
  return s * (1.f + z * (1.f - s));
}

template <int R>
__global__ void __launch_bounds__(kTrThreads)
k_mlp_rows(int64_t n, const int32_t *__restrict__ rows, const float *__restrict__ D, const float *__restrict__ T,
           const float *__restrict__ P, float inv_n, TrainAct act) {
  extern __shared__ float tsm[];
  float *w1 = tsm, *w2 = w1 + kH * kW1s;
  float *xs = w2 + kH * kW2s;                            // [kIn][R]
  float *hs = xs + kIn * R, *ds = hs + kH * R;           // [kH][R] each: h1, then dz2
  float *ps = ds + kH * R;                               // [kH][R]: the upper half's partial sums
  __shared__ float wsum[4][R];
  __shared__ float serr[R];
  const int t = threadIdx.x, h = t & (kH - 1), half = t >> 7, lane = t & 31;
  for (int i = t; i < kH * kIn; i += kTrThreads) w1[(i / kIn) * kW1s + i % kIn] = P[oW1 + i];
  for (int i = t; i < kH * kH; i += kTrThreads) w2[(i / kH) * kW2s + i % kH] = P[oW2 + i];
  const float b1 = P[oB1 + h], b2 = P[oB2 + h], w3 = P[oW3 + h], b3 = P[oB3], ym = P[oYm], ys = P[oYs];
  const int64_t ntile = (n + R - 1) / R;
  for (int64_t tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
    const int64_t r0 = tile * R;
    __syncthreads();                                     // weights staged / the last tile's buffers free
    for (int i = t; i < kIn * R; i += kTrThreads) {
      const int r = i / kIn, k = i - r * kIn;
      float v = 0.f;
      if (r0 + r < n) {
        const int64_t row = rows ? rows[r0 + r] : r0 + r;
        v = (D[row * kIn + k] - P[oXm + k]) / P[oXs + k];
        act.x[(r0 + r) * kIn + k] = v;
      }
      xs[k * R + r] = v;
    }
    __syncthreads();
    float z[R], z1[R], z2[R];
    // layer 1
#pragma unroll
    for (int r = 0; r < R; ++r) z[r] = 0.f;
    {
      const int k0 = half * (kIn / 2);
#pragma unroll 8
      for (int k = 0; k < kIn / 2; ++k) {
        const float w = w1[h * kW1s + k0 + k];
#pragma unroll
        for (int r = 0; r < R; ++r) z[r] = fmaf(w, xs[(k0 + k) * R + r], z[r]);
      }
    }
    if (half) {
#pragma unroll
      for (int r = 0; r < R; ++r) ps[h * R + r] = z[r];
    }
    __syncthreads();
    if (!half) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        z1[r] = b1 + (z[r] + ps[h * R + r]);
        hs[h * R + r] = silu_train(z1[r]);
      }
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (r0 + r < n) act.h1[(r0 + r) * kH + h] = hs[h * R + r];
    }
    __syncthreads();
    // layer 2
#pragma unroll
    for (int r = 0; r < R; ++r) z[r] = 0.f;
    {
      const int k0 = half * (kH / 2);
#pragma unroll 8
      for (int k = 0; k < kH / 2; ++k) {
        const float w = w2[h * kW2s + k0 + k];
#pragma unroll
        for (int r = 0; r < R; ++r) z[r] = fmaf(w, hs[(k0 + k) * R + r], z[r]);
      }
    }
    if (half) {
#pragma unroll
      for (int r = 0; r < R; ++r) ps[h * R + r] = z[r];
    }
    __syncthreads();
    if (!half) {
      // output: the four warps of this half add W3 . SiLU(z2) over the hidden units
#pragma unroll
      for (int r = 0; r < R; ++r) {
        z2[r] = b2 + (z[r] + ps[h * R + r]);
        float v = w3 * silu_train(z2[r]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) wsum[h >> 5][r] = v;
      }
    }
    __syncthreads();
    if (t < R) {
      const float o3 = wsum[0][t] + wsum[1][t] + wsum[2][t] + wsum[3][t] + b3;
      float err = 0.f;
      if (r0 + t < n) {
        const int64_t row = rows ? rows[r0 + t] : r0 + t;
        err = o3 - (T[row] - ym) / ys;
        act.out[r0 + t] = make_float2(2.f * err * inv_n, err);
      }
      serr[t] = err;
    }
    __syncthreads();
    if (!half) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float dout = 2.f * serr[r] * inv_n;
        const float d2 = dout * w3 * silu_grad_train(z2[r]);
        ds[h * R + r] = d2;
        if (r0 + r < n) {
          act.dz2[(r0 + r) * kH + h] = d2;
          act.a3[(r0 + r) * kH + h] = dout * silu_train(z2[r]);
        }
      }
    }
    __syncthreads();
    // dh1[h] = sum_k W2[k][h] dz2[k]
#pragma unroll
    for (int r = 0; r < R; ++r) z[r] = 0.f;
    {
      const int k0 = half * (kH / 2);
#pragma unroll 8
      for (int k = 0; k < kH / 2; ++k) {
        const float w = w2[(k0 + k) * kW2s + h];
#pragma unroll
        for (int r = 0; r < R; ++r) z[r] = fmaf(w, ds[(k0 + k) * R + r], z[r]);
      }
    }
    if (half) {
#pragma unroll
      for (int r = 0; r < R; ++r) ps[h * R + r] = z[r];
    }
    __syncthreads();
    if (!half) {
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (r0 + r < n) act.dz1[(r0 + r) * kH + h] = (z[r] + ps[h * R + r]) * silu_grad_train(z1[r]);
    }
  }
}

struct AdamW {
  float *P, *m1, *m2;
  int t;
  float lr, wd;
};
// one AdamW update of parameter i with gradient s
__device__ __forceinline__ void adamw_update(const AdamW &a, int i, float s) {
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float m = b1 * a.m1[i] + (1.f - b1) * s, v = b2 * a.m2[i] + (1.f - b2) * s * s;
  a.m1[i] = m;
  a.m2[i] = v;
  const float mh = m / (1.f - powf(b1, (float)a.t)), vh = v / (1.f - powf(b2, (float)a.t));
  a.P[i] -= a.lr * (mh / (sqrtf(vh) + eps) + a.wd * a.P[i]);
}

// weight gradients over the rows of split blockIdx.y of the chunk; fused: the only split, so each
// gradient goes to grad (if given) and into AdamW (if apply), else to gpart[split]
__global__ void __launch_bounds__(kTrThreads)
k_mlp_wgrad(int64_t n, TrainAct act, float *__restrict__ gpart, double *__restrict__ lpart, int fused,
            float *__restrict__ grad, int apply, AdamW opt) {
  __shared__ __align__(16) float sa[kTrStage][kTile], sb[kTrStage][kTile];
  __shared__ float red[4][kTile * kTile];
  const int t = threadIdx.x, blk = blockIdx.x;
  const int64_t r0 = (int64_t)blockIdx.y * kTrSplit, r1 = min(n, r0 + kTrSplit);
  const int64_t slot = blockIdx.y;
  auto put = [&](int i, float s) {
    if (!fused) {
      gpart[slot * kNtrain + i] = s;
      return;
    }
    if (grad) grad[i] = s;
    if (apply) adamw_update(opt, i, s);
  };
  if (blk < kTilesW2 + kTilesW1) {
    // 16 x 16 outputs: g[h0 + i][k0 + j] = sum_r A[r][h0 + i] B[r][k0 + j]
    const bool second = blk < kTilesW2;
    const int tl = second ? blk : blk - kTilesW2, across = second ? kH / kTile : kIn / kTile;
    const int h0 = (tl / across) * kTile, k0 = (tl % across) * kTile;
    const float *A = second ? act.dz2 : act.dz1, *B = second ? act.h1 : act.x;
    const int ldb = second ? kH : kIn;
    const int grp = t >> 6, i2 = 2 * ((t & 63) >> 3), j2 = 2 * (t & 7);
    float g00 = 0.f, g01 = 0.f, g10 = 0.f, g11 = 0.f;
    // a stage's loads: each thread two rows' 16-byte pieces of A and of B, fetched one stage ahead
    const int lr = t >> 2, lc = 4 * (t & 3);
    float4 pa[2], pb[2];
    auto fetch = [&](int64_t base) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int64_t r = base + lr + 64 * u;
        const bool ok = r < r1;
        pa[u] = ok ? __ldcg(reinterpret_cast<const float4 *>(A + r * kH + h0 + lc)) : make_float4(0.f, 0.f, 0.f, 0.f);
        pb[u] = ok ? __ldcg(reinterpret_cast<const float4 *>(B + r * ldb + k0 + lc)) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    };
    fetch(r0);
    for (int64_t base = r0; base < r1; base += kTrStage) {
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        *reinterpret_cast<float4 *>(&sa[lr + 64 * u][lc]) = pa[u];
        *reinterpret_cast<float4 *>(&sb[lr + 64 * u][lc]) = pb[u];
      }
      __syncthreads();
      if (base + kTrStage < r1) fetch(base + kTrStage);
#pragma unroll 8
      for (int r = grp; r < kTrStage; r += 4) {          // rows beyond r1 are zero
        const float2 a = *reinterpret_cast<const float2 *>(&sa[r][i2]);
        const float2 b = *reinterpret_cast<const float2 *>(&sb[r][j2]);
        g00 = fmaf(a.x, b.x, g00);
        g01 = fmaf(a.x, b.y, g01);
        g10 = fmaf(a.y, b.x, g10);
        g11 = fmaf(a.y, b.y, g11);
      }
    }
    red[grp][i2 * kTile + j2] = g00;
    red[grp][i2 * kTile + j2 + 1] = g01;
    red[grp][(i2 + 1) * kTile + j2] = g10;
    red[grp][(i2 + 1) * kTile + j2 + 1] = g11;
    __syncthreads();
    const float s = ((red[0][t] + red[1][t]) + red[2][t]) + red[3][t];
    put((second ? oW2 : oW1) + (h0 + t / kTile) * (second ? kH : kIn) + k0 + t % kTile, s);
  } else if (blk < kTilesW2 + kTilesW1 + kColBlocks) {
    // column sums: 32 columns x 8 row groups, added in group order
    const int cb = blk - kTilesW2 - kTilesW1, what = cb / (kH / 32), c0 = (cb % (kH / 32)) * 32;
    const float *A = what == 0 ? act.dz1 : (what == 1 ? act.dz2 : act.a3);
    const int col = t & 31, grp = t >> 5;
    float s = 0.f;
#pragma unroll 16
    for (int64_t r = r0 + grp; r < r1; r += 8) s += __ldcg(A + r * kH + c0 + col);
    float *rs = &red[0][0];
    rs[t] = s;
    __syncthreads();
    if (t < 32) {
      float v = rs[t];
#pragma unroll
      for (int g = 1; g < 8; ++g) v += rs[32 * g + t];
      put((what == 0 ? oB1 : (what == 1 ? oB2 : oW3)) + c0 + t, v);
    }
  } else {
    // b3 and the loss
    __shared__ double dred[kTrThreads];
    float s = 0.f;
    double l = 0.0;
    for (int64_t r = r0 + t; r < r1; r += kTrThreads) {
      const float2 o = __ldcg(act.out + r);
      s += o.x;
      l += (double)o.y * (double)o.y;
    }
    float *rs = &red[0][0];
    rs[t] = s;
    dred[t] = l;
    __syncthreads();
    for (int o = kTrThreads / 2; o > 0; o >>= 1) {
      if (t < o) {
        rs[t] += rs[t + o];
        dred[t] += dred[t + o];
      }
      __syncthreads();
    }
    if (t == 0) {
      put(oB3, rs[0]);
      lpart[fused ? 0 : slot] = dred[0];
    }
  }
}

// adds a chunk's split gradients (and squared errors) in order to the sums of the chunks before (first: none); the
// last chunk's call hands the sums on and optionally applies AdamW
__global__ void k_mlp_reduce(int64_t nslot, const float *__restrict__ gpart, const double *__restrict__ lpart,
                             float *__restrict__ gsum, double *__restrict__ loss, float *__restrict__ grad, int first,
                             int last, int apply, AdamW opt) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) {
    double l = first ? 0.0 : *loss;
    for (int64_t b = 0; b < nslot; ++b) l += lpart[b];
    *loss = l;
  }
  if (i >= kNtrain) return;
  float s = first ? 0.f : gsum[i];
#pragma unroll 8
  for (int64_t b = 0; b < nslot; ++b) s += gpart[b * kNtrain + i];
  if (!last) {
    gsum[i] = s;
    return;
  }
  if (grad) grad[i] = s;
  if (apply) adamw_update(opt, i, s);
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
int mlp_param_count() { return kNparam; }
int mlp_input_width() { return kIn; }

void mlp_descriptors(srbe_ctx *c, float *D_dev) {
  const int64_t ne = c->ne;
  const int nlow = (int)std::max<int64_t>(1, std::min<int64_t>(kLowBlocks, (c->ni + 255) / 256));
  c->mlp.Slow.ensure(kNlow * kLowBlocks);
  k_low_modes<<<nlow, 256, 0, c->stream>>>(c->ni, c->z.p, c->q.p, 1.0 / c->L[2],
                                           reinterpret_cast<double *>(c->mlp.Slow.p));
  const float rc = (float)c->rc;
  k_descriptors<<<blocks_for(ne * 32, 256), 256, 0, c->stream>>>(
      ne, c->ex.p, c->ey.p, c->ez.p, c->icells.pf.p, c->nbr.ei.p, c->nbr.ei_n.p, c->nbr.cap, (float)c->L[0],
      (float)c->L[1], rc * rc, c->mlp.Slow.p, nlow, 1.0 / c->L[2], D_dev);
  c->launches += 2;
  SRBE_CUDA(cudaGetLastError());
}

// The forward pass's operands from the parameters: queued by every call that changes them, not by the pass
// itself, so that a prediction captured in a CUDA graph (by a caller, or in a captured step) holds no split
// of its own, allocates nothing and reads the parameters as they are when it is replayed.
void mlp_split(srbe_ctx *c) {
  k_mlp_split<<<blocks_for(kH * kH, 256), 256, 0, c->stream>>>(
      c->mlp.P.p, reinterpret_cast<__nv_bfloat16 *>(c->mlp.split.ensure(kTcWeights)));
  c->launches++;
  SRBE_CUDA(cudaGetLastError());
}

void mlp_forward(srbe_ctx *c, const float *D_dev, int64_t n, float *out_dev, double *out_y_dev) {
  if (n <= 0) return;
  static KernelSetup setup;
  const int nsm = setup.sms([] {
    SRBE_CUDA(cudaFuncSetAttribute(k_mlp_forward_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmem));
  });
  const __nv_bfloat16 *W = reinterpret_cast<const __nv_bfloat16 *>(c->mlp.split.p);
  const unsigned grid = (unsigned)std::min<int64_t>((n + 127) / 128, nsm);
  k_mlp_forward_tc<<<grid, kTcThreads, kTcSmem, c->stream>>>(n, D_dev, c->mlp.P.p, W, out_dev, out_y_dev,
                                                             c->d_status);
  c->launches++;
  SRBE_CUDA(cudaGetLastError());
}

// gradient (and optionally one AdamW step) over rows (all n rows when rows_dev is null); the sum of the
// squared standardised errors goes to *loss_dev.  Queued on the context's stream.
void mlp_grad_step(srbe_ctx *c, const float *D_dev, const float *T_dev, const int32_t *rows_dev, int64_t n,
                   float *grad_dev, bool apply, float lr, float wd, double *loss_dev) {
  auto &m = c->mlp;
  constexpr size_t kRowsSmem4 = sizeof(float) * (kH * (kW1s + kW2s) + 4 * (kIn + 3 * kH));
  constexpr size_t kRowsSmem8 = sizeof(float) * (kH * (kW1s + kW2s) + 8 * (kIn + 3 * kH));
  static KernelSetup setup;
  const int nsm = setup.sms([] {
    SRBE_CUDA(cudaFuncSetAttribute(k_mlp_rows<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRowsSmem4));
    SRBE_CUDA(cudaFuncSetAttribute(k_mlp_rows<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRowsSmem8));
  });
  const int64_t nslot = (n + kTrSplit - 1) / kTrSplit, most = std::min(n, kTrChunk);
  const bool fused = nslot == 1;
  const int64_t rows_max = (most + 3) & ~(int64_t)3;     // keeps every array on a 16-byte boundary
  float *buf = m.act.ensure((size_t)rows_max * (kIn + 4 * kH + 2));
  TrainAct act;
  act.out = reinterpret_cast<float2 *>(buf);
  act.x = buf + 2 * rows_max;
  act.h1 = act.x + kIn * rows_max;
  act.dz1 = act.h1 + kH * rows_max;
  act.dz2 = act.dz1 + kH * rows_max;
  act.a3 = act.dz2 + kH * rows_max;
  const int64_t nslot_chunk = std::min(nslot, kTrChunk / kTrSplit);
  if (!fused) {
    m.gpart.ensure((size_t)(nslot_chunk + 1) * kNtrain);   // the last one: the sums over the chunks
    m.lpart.ensure((size_t)nslot_chunk);
  }
  if (apply) m.t++;
  const AdamW opt{m.P.p, m.m1.p, m.m2.p, m.t, lr, wd};
  for (int64_t b0 = 0; b0 < n; b0 += kTrChunk) {
    const int64_t nb = std::min(kTrChunk, n - b0);
    const int32_t *rows = rows_dev ? rows_dev + b0 : nullptr;
    const float *D = rows_dev ? D_dev : D_dev + b0 * kIn, *T = rows_dev ? T_dev : T_dev + b0;
    // 4 rows per tile while one wave of blocks covers them (a 512-row minibatch: 128 blocks), then 8
    if (nb <= 4 * (int64_t)nsm)
      k_mlp_rows<4><<<(unsigned)((nb + 3) / 4), kTrThreads, kRowsSmem4, c->stream>>>(nb, rows, D, T, m.P.p,
                                                                                    1.0f / (float)n, act);
    else
      k_mlp_rows<8><<<(unsigned)std::min<int64_t>((nb + 7) / 8, nsm), kTrThreads, kRowsSmem8, c->stream>>>(
          nb, rows, D, T, m.P.p, 1.0f / (float)n, act);
    const unsigned splits = (unsigned)((nb + kTrSplit - 1) / kTrSplit);
    k_mlp_wgrad<<<dim3(kWgradBlocks, splits), kTrThreads, 0, c->stream>>>(
        nb, act, m.gpart.p, fused ? loss_dev : m.lpart.p, fused ? 1 : 0, grad_dev, apply ? 1 : 0, opt);
    c->launches += 2;
    if (fused) continue;
    k_mlp_reduce<<<blocks_for(kNtrain, 128), 128, 0, c->stream>>>(
        splits, m.gpart.p, m.lpart.p, m.gpart.p + nslot_chunk * kNtrain, loss_dev, grad_dev, b0 == 0 ? 1 : 0,
        b0 + nb == n ? 1 : 0, apply ? 1 : 0, opt);
    c->launches++;
  }
  SRBE_CUDA(cudaGetLastError());
}

}  // namespace srbe
