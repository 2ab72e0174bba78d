// FP32 path at head_dim 64, hidden 128: register-tiled SIMT kernels.
//
// One CTA (256 threads, one per SM) processes one work item: a token range of
// one chain at one chunk step, in tiles of tokens.  Per tile the products run
// as register-tiled GEMMs out of shared memory, each thread holding a block of
// outputs, on packed float32 pairs (fma.rn.f32x2: the FMA rate is the scalar
// one, 128 a clock and SM, but half the issue slots, which leaves the other
// half to the shared-memory loads).  Two ways to form the pairs, so that every
// weight matrix is read in the layout it has in global memory (no transposed
// copy) and with 16-byte loads:
//   - a product whose operands are both contiguous along the contraction
//     (z = k W^T over d, o = h W2^T over f) pairs the contraction: one lane
//     sums the even terms, one the odd ones, added at the end;
//   - one whose B operand is contiguous along the output (p = e W2, dk = g W1)
//     pairs the outputs and broadcasts the A value to both lanes.
// Shared-memory rows are padded by 16 bytes and the weight rows are stored in
// the order in which consecutive threads read them, so that a warp's 16-byte
// loads (8 different rows, or 4 broadcast token rows) are free of conflicts.
//
// Measured on GB300 (forward + backward of two sequences of 4 frames x 1041
// tokens, 16 heads, chunks of 2 frames): 8.43 ms with the untiled kernels this
// replaced (one output per thread, the backward's weights reloaded twice per
// 8 tokens), 2.56 ms tiled, 2.00 ms with the planner's tail fill (one piece
// per task share left the longest pieces alone for a third of a launch),
// 1.93 ms with the inner loops unrolled four times.  8 chunks of 128 tokens of
// one head, forward: 248 -> 114 us.
//
// What bounds it, with eight warps a SM at 255 registers (ncu, one mixed step of
// that training pass): the forward's FMA pipe is 56 % active and its shared-memory
// pipe 55 %, the backward's 52 and 76 %.  The loads set the backward (short
// scoreboard is its first stall after the fixed waits), neither alone the forward.
// The FMA rate is 74.5 TFLOP/s, measured for independent FMAs, scalar and packed
// alike; the gradient pieces' products take 20 16-byte loads per 96 packed FMAs,
// their token sums 8 per 48.
//
// Forward roles (Sec. 4.2, Eq. 8, Eq. 9, Supp. Sec. A):
//   KEY    gradient partial of the chunk at the pre-chunk weights W, e = -dL/df:
//            z1 = W1 k, z3 = W3 k, a = SiLU(z1), u = a o z3,
//            e = v (dot loss) | v - W2 u (MSE),  p = W2^T e,
//            g1 = r1 p o z3 o SiLU'(z1), g3 = r3 p o a    (rates r1, r3, r2 of W1, W3, W2)
//            A1 += g1 k^T, A3 += g3 k^T, A2t += r2 u e^T  (W += A after the step)
//   APPLY  o = W2 (SiLU(W1 q) o W3 q)                          (Eq. 4)
// Backward roles (reverse-mode differentiation of the forward recurrence):
//   BAPPLY VJP of o = f_W(q): the KEY pass on (q, do) without rates, plus
//          dq = W1^T A1 + W3^T A3 per token.
//   BKEY   VJP of W~ = W - G(W; k, v, lr) given R = dL/dW~ (see run_bkey).
#include <type_traits>

#include "sm100.cuh"
#include "ttt_internal.h"

namespace scal3r {
namespace {

using sm100::f32x2;
using sm100::fma2;
using sm100::x2;
using sm100::x2_hi;
using sm100::x2_lo;

constexpr int D = 64;
constexpr int F = 128;
constexpr int P = 3 * F * D;
constexpr int NTH = 256;
constexpr int LDK = D + 4;     // row strides in shared memory (floats): token rows,
constexpr int LDW = D + 4;     //   W1 / W3 rows,
constexpr int LDF = F + 4;     //   W2 rows and factor rows

__device__ __forceinline__ float sigm(float z) { return 1.f / (1.f + expf(-z)); }

__device__ __forceinline__ void cp16(float* dst, const float* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sm100::smem_u32(dst)), "l"(src),
               "r"(valid ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp4(float* dst, const float* src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(sm100::smem_u32(dst)), "l"(src),
               "r"(valid ? 4 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

struct Pair2 {
  f32x2 a, b;
};
__device__ __forceinline__ Pair2 ld2(const float* p) {   // 16 bytes as two pairs
  const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
  return {v.x, v.y};
}
__device__ __forceinline__ float4 ld4s(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float get(const float4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

// n (<= rows) token rows of head h from token t; the rows past n are zero.
__device__ __forceinline__ void load_rows(float* dst, const float* __restrict__ src, int64_t t, int n, int rows, int H,
                                          int h) {
  for (int c = threadIdx.x; c < rows * (D / 4); c += NTH) {
    const int r = c / (D / 4), q = c % (D / 4);
    const bool ok = r < n;
    cp16(dst + r * LDK + 4 * q, src + ((size_t)(t + (ok ? r : 0)) * H + h) * D + 4 * q, ok);
  }
}
// The tokens' nr rates (one, or one per matrix); zero past n.
__device__ __forceinline__ void load_rates(float* dst, const float* __restrict__ lr, int64_t t, int n, int rows, int H,
                                           int h, int nr) {
  for (int i = threadIdx.x; i < rows * nr; i += NTH) {
    const int r = i / nr;
    const bool ok = r < n;
    cp4(dst + i, lr + ((size_t)(t + (ok ? r : 0)) * H + h) * nr + i % nr, ok);
  }
}

// ---------------------------------------------------------------------------
// the token pass: KEY, APPLY and BAPPLY, whole weight set resident
// ---------------------------------------------------------------------------
// Thread (tx, ty) of the hidden-unit products owns hidden units 4 tx .. 4 tx + 3
// of tokens ty + 8 i; a warp is 8 tx by 4 ty.  W1 / W3 row f sits in row slot
// (f % 4) * 32 + f / 4, W2 row d in slot (d % 4) * 16 + d / 4: the slots that
// consecutive threads read are consecutive.
constexpr int W_FLOATS = 2 * F * LDW + D * LDF;
constexpr int KT = 32;         // KEY / BAPPLY tile (tokens)
constexpr int AT = 64;         // APPLY tile
constexpr int KEY_SMEM = 4 * (W_FLOATS + 4 * KT * LDK + KT * LDK + 3 * KT * LDF + 2 * 3 * KT);
constexpr int APPLY_SMEM = 4 * (W_FLOATS + 2 * AT * LDK + AT * LDF);
constexpr int TOK_SMEM = KEY_SMEM > APPLY_SMEM ? KEY_SMEM : APPLY_SMEM;

__device__ __forceinline__ void load_weights(float* sm, const float* __restrict__ w) {
  for (int c = threadIdx.x; c < 2 * F * (D / 4); c += NTH) {
    const int r = c / (D / 4), q = c % (D / 4), f = r % F;
    cp16(sm + ((r / F) * F + (f % 4) * 32 + f / 4) * LDW + 4 * q, w + (size_t)r * D + 4 * q, true);
  }
  float* w2 = sm + 2 * F * LDW;
  for (int c = threadIdx.x; c < D * (F / 4); c += NTH) {
    const int d = c / (F / 4), q = c % (F / 4);
    cp16(w2 + ((d % 4) * 16 + d / 4) * LDF + 4 * q, w + 2 * (size_t)F * D + (size_t)d * F + 4 * q, true);
  }
}

// z1, z3 of the thread's TM tokens x 4 hidden units (contraction pairs).
template <int TM>
__device__ __forceinline__ void hidden_z(const float* Xs, const float* W1s, int tx, int ty, float (&z1)[TM][4],
                                         float (&z3)[TM][4]) {
  f32x2 a1[TM][4], a3[TM][4];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) a1[i][j] = a3[i][j] = 0ull;
  const float* xp = Xs + ty * LDK;
  const float* wp = W1s + tx * LDW;
#pragma unroll 4
  for (int d = 0; d < D; d += 4) {
    Pair2 x[TM];
#pragma unroll
    for (int i = 0; i < TM; ++i) x[i] = ld2(xp + 8 * i * LDK + d);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const Pair2 w1 = ld2(wp + 32 * j * LDW + d), w3 = ld2(wp + (F + 32 * j) * LDW + d);
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        a1[i][j] = fma2(x[i].b, w1.b, fma2(x[i].a, w1.a, a1[i][j]));
        a3[i][j] = fma2(x[i].b, w3.b, fma2(x[i].a, w3.a, a3[i][j]));
      }
    }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      z1[i][j] = x2_lo(a1[i][j]) + x2_hi(a1[i][j]);
      z3[i][j] = x2_lo(a3[i][j]) + x2_hi(a3[i][j]);
    }
}

// p = W2^T y of the same elements (output pairs).
template <int TM>
__device__ __forceinline__ void hidden_p(const float* Ys, const float* W2s, int tx, int ty, float (&pv)[TM][4]) {
  f32x2 a[TM][2];
#pragma unroll
  for (int i = 0; i < TM; ++i) a[i][0] = a[i][1] = 0ull;
  const float* yp = Ys + ty * LDK;
  const float* wp = W2s + 4 * tx;
#pragma unroll 4
  for (int d = 0; d < D; d += 4) {
    float4 y[TM];
#pragma unroll
    for (int i = 0; i < TM; ++i) y[i] = ld4s(yp + 8 * i * LDK + d);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const Pair2 w = ld2(wp + (16 * c + d / 4) * LDF);
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const f32x2 yd = x2(get(y[i], c));
        a[i][0] = fma2(yd, w.a, a[i][0]);
        a[i][1] = fma2(yd, w.b, a[i][1]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    pv[i][0] = x2_lo(a[i][0]);
    pv[i][1] = x2_hi(a[i][0]);
    pv[i][2] = x2_lo(a[i][1]);
    pv[i][3] = x2_hi(a[i][1]);
  }
}

// y[tok][d] = sum_f h[tok][f] W2[d][f] for tokens ty + 16 i and d = 4 dx ..
// 4 dx + 3 (contraction pairs).
template <int TM>
__device__ __forceinline__ void out_d(const float* Hs, const float* W2s, int dx, int ty, float (&y)[TM][4]) {
  f32x2 a[TM][4];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) a[i][j] = 0ull;
  const float* hp = Hs + ty * LDF;
  const float* wp = W2s + dx * LDF;
#pragma unroll 4
  for (int f = 0; f < F; f += 4) {
    Pair2 hv[TM];
#pragma unroll
    for (int i = 0; i < TM; ++i) hv[i] = ld2(hp + 16 * i * LDF + f);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const Pair2 w = ld2(wp + 16 * j * LDF + f);
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i][j] = fma2(hv[i].b, w.b, fma2(hv[i].a, w.a, a[i][j]));
    }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) y[i][j] = x2_lo(a[i][j]) + x2_hi(a[i][j]);
}

// The three token sums of a piece: thread (fx, dx) owns hidden units 8 fx ..
// 8 fx + 7 by d = 4 dx .. 4 dx + 3 of each (output pairs along d), 96 registers.
struct Sums {
  f32x2 a[3][8][2];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
      for (int b = 0; b < 8; ++b) a[m][b][0] = a[m][b][1] = 0ull;
  }
};

template <int TT>
__device__ __forceinline__ void token_sums(Sums& s, const float* G1, const float* G3, const float* U, const float* Xs,
                                           const float* Ys, int fx, int dx) {
#pragma unroll 4
  for (int t = 0; t < TT; ++t) {
    const Pair2 x = ld2(Xs + t * LDK + 4 * dx), y = ld2(Ys + t * LDK + 4 * dx);
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const float* g = (m == 0 ? G1 : m == 1 ? G3 : U) + t * LDF + 8 * fx;
      const Pair2& r = m < 2 ? x : y;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float4 gv = ld4s(g + 4 * q);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const f32x2 gd = x2(get(gv, c));
          s.a[m][4 * q + c][0] = fma2(gd, r.a, s.a[m][4 * q + c][0]);
          s.a[m][4 * q + c][1] = fma2(gd, r.b, s.a[m][4 * q + c][1]);
        }
      }
    }
  }
}

// The sums into the piece's slot, packed like the weights (the W2 part as [D][F]).
__device__ __forceinline__ void store_sums(float* __restrict__ out, const Sums& s, int fx, int dx) {
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int b = 0; b < 8; ++b)
      *reinterpret_cast<float4*>(out + (size_t)m * F * D + (size_t)(8 * fx + b) * D + 4 * dx) =
          make_float4(x2_lo(s.a[m][b][0]), x2_hi(s.a[m][b][0]), x2_lo(s.a[m][b][1]), x2_hi(s.a[m][b][1]));
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    float v[8];
#pragma unroll
    for (int b = 0; b < 8; ++b) v[b] = (c & 1) ? x2_hi(s.a[2][b][c / 2]) : x2_lo(s.a[2][b][c / 2]);
    float4* o = reinterpret_cast<float4*>(out + 2 * (size_t)F * D + (size_t)(4 * dx + c) * F + 8 * fx);
    o[0] = make_float4(v[0], v[1], v[2], v[3]);
    o[1] = make_float4(v[4], v[5], v[6], v[7]);
  }
}

struct TokTile {   // one tile of the token pass
  const float *x, *y, *rates;   // X and Y rows, the tokens' rates (KEY)
  int64_t t;
  int n;
};

// One tile of TT tokens of a KEY (VJP = false) or BAPPLY (VJP = true) item.
template <int TT, bool VJP>
__device__ __forceinline__ void token_tile(const Params& p, const TokTile& tl, float* sm, float* Es, float* Gs, Sums& s,
                                           int h) {
  constexpr int TM = TT / 8, TM2 = TT / 16;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int tx = (warp & 3) * 8 + (lane & 7), ty = (warp >> 2) * 4 + (lane >> 3);     // hidden products
  const int dx = (warp & 1) * 8 + (lane & 7), fy = (warp >> 1) * 4 + (lane >> 3);     // d products and sums
  const float* W2s = sm + 2 * F * LDW;
  float *G1 = Gs, *G3 = Gs + KT * LDF, *U = Gs + 2 * KT * LDF;
  const bool mse = !VJP && p.loss == SCAL3R_LOSS_MSE;
  float z1[TM][4], z3[TM][4], pv[TM][4];
  hidden_z<TM>(tl.x, sm, tx, ty, z1, z3);
  const float* ys = tl.y;
  if (mse) {   // e = v - W2 u
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      float u[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) u[j] = z1[i][j] * sigm(z1[i][j]) * z3[i][j];
      *reinterpret_cast<float4*>(U + (ty + 8 * i) * LDF + 4 * tx) = make_float4(u[0], u[1], u[2], u[3]);
    }
    __syncthreads();
    float y[TM2][4];
    out_d<TM2>(U, W2s, dx, fy, y);
#pragma unroll
    for (int i = 0; i < TM2; ++i) {
      const float4 v = ld4s(tl.y + (fy + 16 * i) * LDK + 4 * dx);
      *reinterpret_cast<float4*>(Es + (fy + 16 * i) * LDK + 4 * dx) =
          make_float4(v.x - y[i][0], v.y - y[i][1], v.z - y[i][2], v.w - y[i][3]);
    }
    __syncthreads();
    ys = Es;
  }
  hidden_p<TM>(ys, W2s, tx, ty, pv);
  const int nr = p.lr_mat ? 3 : 1;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int tok = ty + 8 * i;
    float r1 = 1.f, r3 = 1.f, r2 = 1.f;
    if (!VJP) {
      r1 = tl.rates[tok * nr];
      r3 = p.lr_mat ? tl.rates[tok * nr + 1] : r1;
      r2 = p.lr_mat ? tl.rates[tok * nr + 2] : r1;
    }
    float g1[4], g3[4], u[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float sg = sigm(z1[i][j]);
      const float a = z1[i][j] * sg;
      g1[j] = r1 * pv[i][j] * z3[i][j] * (sg * (1.f + z1[i][j] * (1.f - sg)));
      g3[j] = r3 * pv[i][j] * a;
      u[j] = r2 * (a * z3[i][j]);
    }
    *reinterpret_cast<float4*>(G1 + tok * LDF + 4 * tx) = make_float4(g1[0], g1[1], g1[2], g1[3]);
    *reinterpret_cast<float4*>(G3 + tok * LDF + 4 * tx) = make_float4(g3[0], g3[1], g3[2], g3[3]);
    *reinterpret_cast<float4*>(U + tok * LDF + 4 * tx) = make_float4(u[0], u[1], u[2], u[3]);
  }
  __syncthreads();
  if (VJP) {   // dq = W1^T A1 + W3^T A3 of tokens fy + 16 i, d = 4 dx .. (output pairs)
    f32x2 a[TM2][2];
#pragma unroll
    for (int i = 0; i < TM2; ++i) a[i][0] = a[i][1] = 0ull;
#pragma unroll 4
    for (int f = 0; f < F; f += 4) {
      float4 v1[TM2], v3[TM2];
#pragma unroll
      for (int i = 0; i < TM2; ++i) {
        v1[i] = ld4s(G1 + (fy + 16 * i) * LDF + f);
        v3[i] = ld4s(G3 + (fy + 16 * i) * LDF + f);
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const Pair2 w1 = ld2(sm + (32 * c + f / 4) * LDW + 4 * dx), w3 = ld2(sm + (F + 32 * c + f / 4) * LDW + 4 * dx);
#pragma unroll
        for (int i = 0; i < TM2; ++i) {
          const f32x2 d1 = x2(get(v1[i], c)), d3 = x2(get(v3[i], c));
          a[i][0] = fma2(d1, w1.a, fma2(d3, w3.a, a[i][0]));
          a[i][1] = fma2(d1, w1.b, fma2(d3, w3.b, a[i][1]));
        }
      }
    }
    float* dq = static_cast<float*>(p.dq);
#pragma unroll
    for (int i = 0; i < TM2; ++i) {
      const int r = fy + 16 * i;
      if (r < tl.n)
        *reinterpret_cast<float4*>(dq + ((size_t)(tl.t + r) * p.H + h) * D + 4 * dx) =
            make_float4(x2_lo(a[i][0]), x2_hi(a[i][0]), x2_lo(a[i][1]), x2_hi(a[i][1]));
    }
  }
  token_sums<TT>(s, G1, G3, U, tl.x, ys, fy, dx);
}

// KEY (X = k, Y = v) and BAPPLY (X = q, Y = d_o) items: tiles of 32 tokens, a
// last one of at most 16 as a 16-token tile; the next tile's rows are copied
// while this one is computed.
template <bool VJP>
__device__ void run_token_pass(const Params& p, const WorkItem& it, const float* w, float* sm) {
  float* Xs = sm + W_FLOATS;            // two buffers of X rows | Y rows
  float* Es = Xs + 4 * KT * LDK;        // MSE: e
  float* Gs = Es + KT * LDK;            // the three factors
  float* rates = Gs + 3 * KT * LDF;     // two buffers
  const int H = p.H, h = it.chain % H, nr = p.lr_mat ? 3 : 1;
  const float* x = static_cast<const float*>(VJP ? p.q : p.k);
  const float* y = static_cast<const float*>(VJP ? p.d_o : p.v);
  Sums s;
  s.zero();
  auto load = [&](int64_t t, int buf) {
    if (t >= it.t1) return;
    const int n = (int)min((int64_t)KT, it.t1 - t), rows = n > 16 ? KT : 16;
    load_rows(Xs + 2 * buf * KT * LDK, x, t, n, rows, H, h);
    load_rows(Xs + (2 * buf + 1) * KT * LDK, y, t, n, rows, H, h);
    if (!VJP) load_rates(rates + buf * 3 * KT, p.lr, t, n, rows, H, h, nr);
  };
  load_weights(sm, w);
  load(it.t0, 0);
  cp_commit();
  int buf = 0;
  for (int64_t t = it.t0; t < it.t1; t += KT, buf ^= 1) {
    load(t + KT, buf ^ 1);
    cp_commit();
    cp_wait<1>();
    __syncthreads();
    const TokTile tl{Xs + 2 * buf * KT * LDK, Xs + (2 * buf + 1) * KT * LDK, rates + buf * 3 * KT, t,
                     (int)min((int64_t)KT, it.t1 - t)};
    if (tl.n > 16) token_tile<KT, VJP>(p, tl, sm, Es, Gs, s, h);
    else token_tile<16, VJP>(p, tl, sm, Es, Gs, s, h);
    __syncthreads();   // the factors and this buffer are read
  }
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  store_sums(p.part + (size_t)it.slot * P, s, (warp >> 1) * 4 + (lane >> 3), (warp & 1) * 8 + (lane & 7));
}

// One APPLY tile of TT tokens.
template <int TT>
__device__ __forceinline__ void apply_tile(const Params& p, const float* Qs, int64_t t, int n, float* sm, float* Hs,
                                           int h) {
  constexpr int TM = TT / 8, TM2 = TT / 16;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int tx = (warp & 3) * 8 + (lane & 7), ty = (warp >> 2) * 4 + (lane >> 3);
  const int dx = (warp & 1) * 8 + (lane & 7), fy = (warp >> 1) * 4 + (lane >> 3);
  {
    float z1[TM][4], z3[TM][4];
    hidden_z<TM>(Qs, sm, tx, ty, z1, z3);
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      float u[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) u[j] = z1[i][j] * sigm(z1[i][j]) * z3[i][j];
      *reinterpret_cast<float4*>(Hs + (ty + 8 * i) * LDF + 4 * tx) = make_float4(u[0], u[1], u[2], u[3]);
    }
  }
  __syncthreads();
  float y[TM2][4];
  out_d<TM2>(Hs, sm + 2 * F * LDW, dx, fy, y);
  float* o = static_cast<float*>(p.o);
#pragma unroll
  for (int i = 0; i < TM2; ++i) {
    const int r = fy + 16 * i;
    if (r < n)
      *reinterpret_cast<float4*>(o + ((size_t)(t + r) * p.H + h) * D + 4 * dx) =
          make_float4(y[i][0], y[i][1], y[i][2], y[i][3]);
  }
}

__device__ void run_apply(const Params& p, const WorkItem& it, const float* w, float* sm) {
  float* Qs = sm + W_FLOATS;
  float* Hs = Qs + 2 * AT * LDK;
  const int H = p.H, h = it.chain % H;
  const float* q = static_cast<const float*>(p.q);
  auto load = [&](int64_t t, int buf) {
    if (t >= it.t1) return;
    const int n = (int)min((int64_t)AT, it.t1 - t);
    load_rows(Qs + buf * AT * LDK, q, t, n, n > 32 ? AT : n > 16 ? 32 : 16, H, h);
  };
  load_weights(sm, w);
  load(it.t0, 0);
  cp_commit();
  int buf = 0;
  for (int64_t t = it.t0; t < it.t1; t += AT, buf ^= 1) {
    load(t + AT, buf ^ 1);
    cp_commit();
    cp_wait<1>();
    __syncthreads();
    const int n = (int)min((int64_t)AT, it.t1 - t);
    const float* qs = Qs + buf * AT * LDK;
    if (n > 32) apply_tile<AT>(p, qs, t, n, sm, Hs, h);
    else if (n > 16) apply_tile<32>(p, qs, t, n, sm, Hs, h);
    else apply_tile<16>(p, qs, t, n, sm, Hs, h);
    __syncthreads();
  }
}

__global__ void __launch_bounds__(NTH, 1) fp32_tiled_sweep(Params p, const WorkItem* __restrict__ items, int step) {
  extern __shared__ __align__(16) float smf[];
  pdl_wait();   // the step's weights come from the kernel ahead of this one
  const WorkItem it = items[blockIdx.x];
  const float* w = p.w_items ? p.w0 + (size_t)(it.chain / p.H) * p.w0_seq_stride + (size_t)(it.chain % p.H) * P
                             : p.wm + ((size_t)(step & 1) * p.S * p.H + it.chain) * P;
  if (it.role == ROLE_APPLY) run_apply(p, it, w, smf);
  else run_token_pass<false>(p, it, w, smf);
}

// ---------------------------------------------------------------------------
// BKEY: the VJP of a chunk update
// ---------------------------------------------------------------------------
// Per token, with e = dL/df without its rate (-v | W2 u - v), rates r1, r3, r2:
//   pp = W2^T e,  du = -r2 R2^T e,  h1 = -R1 k, h3 = -R3 k,
//   dp = r3 h3 a + r1 h1 z3 s',  da = r3 h3 pp + du z3,
//   dz3 = r1 h1 pp s' + du a,  dz1 = r1 h1 pp z3 s'' + da s',
//   de = W2 dp - r2 R2 u,  dv = -de,
//   dk = W1^T dz1 + W3^T dz3 - R1^T g1 - R3^T g3   (g1 = r1 pp z3 s', g3 = r3 pp a),
//   dlr = sum over hidden units of pp z3 s' h1 (W1), pp a h3 (W3), u (-R2^T e) (W2),
//   L1 += dz1 k^T, L3 += dz3 k^T, L2t += dp e^T;
// the squared error adds du += W2^T de (into da, dz3) and L2t += u de^T.
// The six matrices (192 KB) do not fit beside the tiles, so the hidden units
// go in blocks of 32 whose slices stream from L2 through two buffers (53 KB
// each) while the block before is computed: 192 KB per 64 tokens, 3 bytes a
// clock and SM, against 8 million FMAs.  dk, de and the three sums stay in
// registers over the blocks.  The squared error runs the blocks three times
// (y, then de, then the rest), as each of the three needs the one before over
// all hidden units.
constexpr int FB = 32, NB = F / FB;
constexpr int LDB = FB + 4;                                // rows of the W2 / R2 slices and of the factors
constexpr int BT = 64;                                     // tile (tokens)
constexpr int BLK_FLOATS = 4 * FB * LDW + 2 * D * LDB;     // W1, W3, R1, R3 rows | W2, R2 slices
constexpr int BKEY_SMEM = 4 * (2 * BLK_FLOATS + 4 * BT * LDK + 6 * BT * LDB + 3 * BT);
static_assert(BKEY_SMEM <= 232448 && TOK_SMEM <= 232448, "shared memory");

// Rows: W1, W3, R1, R3 row f of the block in slot (f % 2) * 16 + f / 2; W2, R2
// row d in slot (d % 4) * 16 + d / 4 (the order consecutive threads read).
__device__ __forceinline__ void load_block(float* dst, const float* __restrict__ w, const float* __restrict__ r, int fb) {
  for (int c = threadIdx.x; c < 4 * FB * (D / 4); c += NTH) {
    const int row = c / (D / 4), q = c % (D / 4), m = row / FB, f = row % FB;
    const float* src = (m < 2 ? w : r) + ((size_t)(m & 1) * F + fb * FB + f) * D + 4 * q;
    cp16(dst + (m * FB + (f % 2) * 16 + f / 2) * LDW + 4 * q, src, true);
  }
  float* d2 = dst + 4 * FB * LDW;
  for (int c = threadIdx.x; c < 2 * D * (FB / 4); c += NTH) {
    const int row = c / (FB / 4), q = c % (FB / 4), m = row / D, d = row % D;
    const float* src = (m ? r : w) + 2 * (size_t)F * D + (size_t)d * F + fb * FB + 4 * q;
    cp16(d2 + (m * D + (d % 4) * 16 + d / 4) * LDB + 4 * q, src, true);
  }
}

struct BSums {   // thread (fx, dx): hidden units 2 fx, 2 fx + 1 of every block by d = 4 dx .. 4 dx + 3
  f32x2 a[NB][3][2][2];
};

enum Stage { FULL, MSE_Y, MSE_DE, MSE_REST };   // FULL: the dot loss in one sweep over the blocks

struct BTile {
  const float *k, *e;   // K rows; E rows: v (dot, the sign follows), or e = y - v
  const float* dy;      // MSE_REST: de rows
  float *fac, *rates;
  int pm;
};

// Products of a thread's TM tokens (ty + 16 i) x 2 hidden units with two row
// matrices (slots m0 and m0 + 1 of the block): contraction pairs over d.
template <int TM>
__device__ __forceinline__ void block_z(const float* X, const float* B, int m0, int tx, int ty, float (&o0)[TM][2],
                                        float (&o1)[TM][2]) {
  f32x2 a[2][TM][2];
#pragma unroll
  for (int i = 0; i < TM; ++i) a[0][i][0] = a[0][i][1] = a[1][i][0] = a[1][i][1] = 0ull;
#pragma unroll 4
  for (int d = 0; d < D; d += 4) {
    Pair2 x[TM];
#pragma unroll
    for (int i = 0; i < TM; ++i) x[i] = ld2(X + (ty + 16 * i) * LDK + d);
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const Pair2 w = ld2(B + ((m0 + m) * FB + 16 * j + tx) * LDW + d);
#pragma unroll
        for (int i = 0; i < TM; ++i) a[m][i][j] = fma2(x[i].b, w.b, fma2(x[i].a, w.a, a[m][i][j]));
      }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      o0[i][j] = x2_lo(a[0][i][j]) + x2_hi(a[0][i][j]);
      o1[i][j] = x2_lo(a[1][i][j]) + x2_hi(a[1][i][j]);
    }
}

// W2^T y (and R2^T y) of the same elements: output pairs.
template <int TM, bool BOTH>
__device__ __forceinline__ void block_p(const float* Y, const float* B2, int tx, int ty, f32x2 (&o0)[TM],
                                        f32x2 (&o1)[TM]) {
#pragma unroll
  for (int i = 0; i < TM; ++i) o0[i] = o1[i] = 0ull;
#pragma unroll 4
  for (int d = 0; d < D; d += 4) {
    float4 y[TM];
#pragma unroll
    for (int i = 0; i < TM; ++i) y[i] = ld4s(Y + (ty + 16 * i) * LDK + d);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int slot = 16 * c + d / 4;
      const f32x2 w = *reinterpret_cast<const f32x2*>(B2 + slot * LDB + 2 * tx);
      f32x2 r = 0ull;
      if (BOTH) r = *reinterpret_cast<const f32x2*>(B2 + (D + slot) * LDB + 2 * tx);
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const f32x2 yd = x2(get(y[i], c));
        o0[i] = fma2(yd, w, o0[i]);
        if (BOTH) o1[i] = fma2(yd, r, o1[i]);
      }
    }
  }
}

// One block of one tile.  acc_k: dk of tokens ty + 16 i, d = 4 dx .. (FULL,
// MSE_REST); acc_e: de (FULL, MSE_DE) or y (MSE_Y); dl: the tokens' dlr terms.
template <int TM, Stage ST>
__device__ __forceinline__ void bkey_block(const BTile& tl, const float* B, int fb, f32x2 (&acc_k)[TM][2],
                                           float (&acc_e)[TM][4], float (&dl)[TM][3], BSums& L) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int tx = (warp & 1) * 8 + (lane & 7), ty = (warp >> 1) * 4 + (lane >> 3);
  const float* B2 = B + 4 * FB * LDW;
  float* fac = tl.fac;
  constexpr int FT = BT * LDB;   // floats of one factor tile: dz1, dz3, -g1, -g3, dp, -r2 u (MSE: u)
  constexpr bool mse = ST != FULL;
  {
    float z1[TM][2], z3[TM][2];
    block_z<TM>(tl.k, B, 0, tx, ty, z1, z3);
    float h1[TM][2], h3[TM][2];
    f32x2 pq[TM], rq[TM], wq[TM];
    if (ST != MSE_Y) {
      block_z<TM>(tl.k, B, 2, tx, ty, h1, h3);
      block_p<TM, true>(tl.e, B2, tx, ty, pq, rq);
      if (ST == MSE_REST) {
        f32x2 un[TM];
        block_p<TM, false>(tl.dy, B2, tx, ty, wq, un);
      }
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int tok = ty + 16 * i;
      const int nr = tl.pm ? 3 : 1;
      float r1 = 0.f, r3 = 0.f, r2 = 0.f;
      if (ST != MSE_Y) {
        r1 = tl.rates[tok * nr];
        r3 = tl.pm ? tl.rates[tok * nr + 1] : r1;
        r2 = tl.pm ? tl.rates[tok * nr + 2] : r1;
      }
      float o[6][2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float sg = sigm(z1[i][j]);
        const float a = z1[i][j] * sg, u = a * z3[i][j];
        if (ST == MSE_Y) {
          o[5][j] = u;
          continue;
        }
        const float sgn = mse ? 1.f : -1.f;   // dot: the E rows hold v, e = -v
        const float pp = sgn * (j ? x2_hi(pq[i]) : x2_lo(pq[i])), du0 = -sgn * (j ? x2_hi(rq[i]) : x2_lo(rq[i]));
        const float sp = sg * (1.f + z1[i][j] * (1.f - sg));
        const float spp = sg * (1.f - sg) * (2.f + z1[i][j] * (1.f - 2.f * sg));
        const float d1 = -h1[i][j], d3 = -h3[i][j], z3sp = z3[i][j] * sp;
        const float t1 = d1 * z3sp, t3 = d3 * a;
        if (ST != MSE_DE) {
          dl[i][0] = fmaf(pp, t1, dl[i][0]);
          dl[i][1] = fmaf(pp, t3, dl[i][1]);
          dl[i][2] = fmaf(u, du0, dl[i][2]);
        }
        o[4][j] = r3 * t3 + r1 * t1;                           // dp
        o[5][j] = ST == MSE_REST ? u : -r2 * u;
        if (ST == MSE_DE) continue;
        float du = r2 * du0;
        if (ST == MSE_REST) du += j ? x2_hi(wq[i]) : x2_lo(wq[i]);
        const float q1 = r1 * d1 * pp;
        const float da = r3 * d3 * pp + du * z3[i][j];
        o[0][j] = q1 * z3[i][j] * spp + da * sp;               // dz1
        o[1][j] = q1 * sp + du * a;                            // dz3
        o[2][j] = -r1 * pp * z3sp;                             // -g1
        o[3][j] = -r3 * pp * a;                                // -g3
      }
#pragma unroll
      for (int m = 0; m < 6; ++m) {
        if (m < 4 && (ST == MSE_Y || ST == MSE_DE)) continue;
        if (m == 4 && ST == MSE_Y) continue;
        *reinterpret_cast<float2*>(fac + m * FT + tok * LDB + 2 * tx) = make_float2(o[m][0], o[m][1]);
      }
    }
  }
  __syncthreads();
  const int dx = tx;   // the d products and the sums use the same thread grid
  if (ST == FULL || ST == MSE_REST) {   // dk: output pairs over d
#pragma unroll 4
    for (int f = 0; f < FB; f += 4) {
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        float4 g[TM];
#pragma unroll
        for (int i = 0; i < TM; ++i) g[i] = ld4s(fac + m * FT + (ty + 16 * i) * LDB + f);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const Pair2 w = ld2(B + (m * FB + 16 * (c & 1) + f / 2 + c / 2) * LDW + 4 * dx);
#pragma unroll
          for (int i = 0; i < TM; ++i) {
            const f32x2 gd = x2(get(g[i], c));
            acc_k[i][0] = fma2(gd, w.a, acc_k[i][0]);
            acc_k[i][1] = fma2(gd, w.b, acc_k[i][1]);
          }
        }
      }
    }
  }
  if (ST != MSE_REST) {   // de (or y): contraction pairs over f
    f32x2 a[TM][4];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) a[i][j] = 0ull;
#pragma unroll 4
    for (int f = 0; f < FB; f += 4) {
#pragma unroll
      for (int m = (ST == MSE_Y ? 1 : 0); m < 2; ++m) {
        Pair2 g[TM];
#pragma unroll
        for (int i = 0; i < TM; ++i) g[i] = ld2(fac + (4 + m) * FT + (ty + 16 * i) * LDB + f);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const Pair2 w = ld2(B2 + ((ST == MSE_Y ? 0 : m * D) + 16 * j + dx) * LDB + f);
#pragma unroll
          for (int i = 0; i < TM; ++i) a[i][j] = fma2(g[i].b, w.b, fma2(g[i].a, w.a, a[i][j]));
        }
      }
    }
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc_e[i][j] += x2_lo(a[i][j]) + x2_hi(a[i][j]);
  }
  if (ST == FULL || ST == MSE_REST) {   // the sums over tokens
    const int fx = ty;
    auto sums = [&](f32x2 (&s)[3][2][2]) {
#pragma unroll 4
      for (int t = 0; t < 16 * TM; ++t) {
        const Pair2 x = ld2(tl.k + t * LDK + 4 * dx), y = ld2(tl.e + t * LDK + 4 * dx);
        const float* g = fac + t * LDB + 2 * fx;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          const float2 gv = *reinterpret_cast<const float2*>(g + (m < 2 ? m : 4) * FT);
          const Pair2& r = m < 2 ? x : y;
          const f32x2 g0 = x2(gv.x), g1 = x2(gv.y);
          s[m][0][0] = fma2(g0, r.a, s[m][0][0]);
          s[m][0][1] = fma2(g0, r.b, s[m][0][1]);
          s[m][1][0] = fma2(g1, r.a, s[m][1][0]);
          s[m][1][1] = fma2(g1, r.b, s[m][1][1]);
        }
        if (mse) {   // + u de^T
          const float2 gv = *reinterpret_cast<const float2*>(g + 5 * FT);
          const Pair2 r = ld2(tl.dy + t * LDK + 4 * dx);
          const f32x2 g0 = x2(gv.x), g1 = x2(gv.y);
          s[2][0][0] = fma2(g0, r.a, s[2][0][0]);
          s[2][0][1] = fma2(g0, r.b, s[2][0][1]);
          s[2][1][0] = fma2(g1, r.a, s[2][1][0]);
          s[2][1][1] = fma2(g1, r.b, s[2][1][1]);
        }
      }
    };
    if (fb == 0) sums(L.a[0]);   // constant indices: the sums stay in registers
    else if (fb == 1) sums(L.a[1]);
    else if (fb == 2) sums(L.a[2]);
    else sums(L.a[3]);
  }
}

struct BkeyMem {
  float *blk, *Ks, *Vs, *Es, *Ys, *fac, *rates;
};

// One tile of 16 TM tokens; `cur` is the block buffer that holds (or is being
// filled with) block 0, and each block's successor is copied while it is computed.
template <int TM, bool MSE>
__device__ __forceinline__ void bkey_tile(const Params& p, const WorkItem& it, const float* w, const float* r,
                                          const BkeyMem& m, int64_t t, int& cur, BSums& L) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int dx = (warp & 1) * 8 + (lane & 7), ty = (warp >> 1) * 4 + (lane >> 3);
  const int H = p.H, h = it.chain % H, nr = p.lr_mat ? 3 : 1;
  constexpr int TT = 16 * TM;
  const int n = (int)min((int64_t)TT, it.t1 - t);
  load_rows(m.Ks, static_cast<const float*>(p.k), t, n, TT, H, h);
  load_rows(m.Vs, static_cast<const float*>(p.v), t, n, TT, H, h);
  load_rates(m.rates, p.lr, t, n, TT, H, h, nr);
  cp_commit();
  f32x2 acc_k[TM][2];
  float acc_e[TM][4], dl[TM][3];
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    acc_k[i][0] = acc_k[i][1] = 0ull;
    dl[i][0] = dl[i][1] = dl[i][2] = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) acc_e[i][j] = 0.f;
  }
  BTile tl{m.Ks, MSE ? m.Es : m.Vs, m.Ys, m.fac, m.rates, p.lr_mat};
  // the sweep over the blocks; the block after the last one is the next
  // sweep's (or tile's) first
  auto sweep = [&](auto stage) {
#pragma unroll 1
    for (int fb = 0; fb < NB; ++fb) {
      cp_wait<0>();
      __syncthreads();   // the block is here; everyone is done with the one before
      load_block(m.blk + (cur ^ 1) * BLK_FLOATS, w, r, (fb + 1) % NB);
      cp_commit();
      bkey_block<TM, decltype(stage)::value>(tl, m.blk + cur * BLK_FLOATS, fb, acc_k, acc_e, dl, L);
      cur ^= 1;
    }
  };
  // a thread's elements of a [token][d] tile
  auto each = [&](auto fn) {
#pragma unroll
    for (int i = 0; i < TM; ++i) fn(i, ty + 16 * i);
  };
  float* dv = static_cast<float*>(p.dv);
  auto store_dv = [&]() {
    each([&](int i, int tok) {
      if (tok < n)
        *reinterpret_cast<float4*>(dv + ((size_t)(t + tok) * H + h) * D + 4 * dx) =
            make_float4(-acc_e[i][0], -acc_e[i][1], -acc_e[i][2], -acc_e[i][3]);
    });
  };
  if (MSE) {
    sweep(std::integral_constant<Stage, MSE_Y>{});
    each([&](int i, int tok) {   // e = y - v
      const float4 v = ld4s(m.Vs + tok * LDK + 4 * dx);
      *reinterpret_cast<float4*>(m.Es + tok * LDK + 4 * dx) =
          make_float4(acc_e[i][0] - v.x, acc_e[i][1] - v.y, acc_e[i][2] - v.z, acc_e[i][3] - v.w);
      acc_e[i][0] = acc_e[i][1] = acc_e[i][2] = acc_e[i][3] = 0.f;
    });
    sweep(std::integral_constant<Stage, MSE_DE>{});
    each([&](int i, int tok) {
      *reinterpret_cast<float4*>(m.Ys + tok * LDK + 4 * dx) =
          make_float4(acc_e[i][0], acc_e[i][1], acc_e[i][2], acc_e[i][3]);
    });
    store_dv();
    sweep(std::integral_constant<Stage, MSE_REST>{});
  } else {
    sweep(std::integral_constant<Stage, FULL>{});
    store_dv();
  }
  float* dk = static_cast<float*>(p.dk);
  each([&](int i, int tok) {
    if (tok < n)
      *reinterpret_cast<float4*>(dk + ((size_t)(t + tok) * H + h) * D + 4 * dx) =
          make_float4(x2_lo(acc_k[i][0]), x2_hi(acc_k[i][0]), x2_lo(acc_k[i][1]), x2_hi(acc_k[i][1]));
  });
  __syncthreads();   // the factors are read: their place takes the dlr partials
  // dlr: a token's 16 threads' terms, 8 lanes by shuffles, the two warps through shared memory
  float* red = m.fac;
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      float v = dl[i][j];
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if ((lane & 7) == 0) red[((warp & 1) * TT + ty + 16 * i) * 3 + j] = v;
    }
  __syncthreads();
  if ((int)threadIdx.x < n) {
    const int tok = threadIdx.x;
    float s[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) s[j] = red[tok * 3 + j] + red[(TT + tok) * 3 + j];
    float* out = p.dlr + ((size_t)(t + tok) * H + h) * nr;
    if (p.lr_mat) {
      out[0] = s[0];
      out[1] = s[1];
      out[2] = s[2];
    } else {
      out[0] = s[0] + s[1] + s[2];
    }
  }
  __syncthreads();   // before the next tile's rows and factors
}

template <bool MSE>
__device__ void run_bkey(const Params& p, const WorkItem& it, const float* w, const float* r, float* sm) {
  BkeyMem m;
  m.blk = sm;
  m.Ks = m.blk + 2 * BLK_FLOATS;
  m.Vs = m.Ks + BT * LDK;
  m.Es = m.Vs + BT * LDK;
  m.Ys = m.Es + BT * LDK;
  m.fac = m.Ys + BT * LDK;
  m.rates = m.fac + 6 * BT * LDB;
  BSums L;
#pragma unroll
  for (int b = 0; b < NB; ++b)
#pragma unroll
    for (int q = 0; q < 3; ++q) L.a[b][q][0][0] = L.a[b][q][0][1] = L.a[b][q][1][0] = L.a[b][q][1][1] = 0ull;
  int cur = 0;
  load_block(m.blk, w, r, 0);
  cp_commit();
  for (int64_t t = it.t0; t < it.t1;) {
    if (it.t1 - t > 16) {
      bkey_tile<4, MSE>(p, it, w, r, m, t, cur, L);
      t += BT;
    } else {
      bkey_tile<1, MSE>(p, it, w, r, m, t, cur, L);
      t += 16;
    }
  }
  cp_wait<0>();   // the block copied ahead of a tile that does not come
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int dx = (warp & 1) * 8 + (lane & 7), fx = (warp >> 1) * 4 + (lane >> 3);
  float* out = p.part + (size_t)it.slot * P;
  const float sgn = MSE ? 1.f : -1.f;   // dot: the sum ran on v = -e
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int f = b * FB + 2 * fx;
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int j = 0; j < 2; ++j)
        *reinterpret_cast<float4*>(out + (size_t)q * F * D + (size_t)(f + j) * D + 4 * dx) =
            make_float4(x2_lo(L.a[b][q][j][0]), x2_hi(L.a[b][q][j][0]), x2_lo(L.a[b][q][j][1]),
                        x2_hi(L.a[b][q][j][1]));
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const f32x2 s0 = L.a[b][2][0][c / 2], s1 = L.a[b][2][1][c / 2];
      *reinterpret_cast<float2*>(out + 2 * (size_t)F * D + (size_t)(4 * dx + c) * F + f) =
          (c & 1) ? make_float2(sgn * x2_hi(s0), sgn * x2_hi(s1)) : make_float2(sgn * x2_lo(s0), sgn * x2_lo(s1));
    }
  }
}

__global__ void __launch_bounds__(NTH, 1) fp32_tiled_bsweep(Params p, const WorkItem* __restrict__ items) {
  extern __shared__ __align__(16) float smf[];
  pdl_wait();
  const WorkItem it = items[blockIdx.x];
  const int H = p.H, h = it.chain % H, s = it.chain / H;
  const float* w = (it.wchunk >= 0) ? p.w_ckpt_in + ((size_t)it.wchunk * H + h) * P
                                    : p.w0 + (size_t)s * p.w0_seq_stride + (size_t)h * P;
  if (it.role == ROLE_BAPPLY) {
    run_token_pass<true>(p, it, w, smf);
    return;
  }
  const float* r = p.rbuf + (size_t)it.chain * P;
  if (p.loss == SCAL3R_LOSS_MSE) run_bkey<true>(p, it, w, r, smf);
  else run_bkey<false>(p, it, w, r, smf);
}

constexpr int BWD_SMEM = BKEY_SMEM > TOK_SMEM ? BKEY_SMEM : TOK_SMEM;

}  // namespace

bool fp32_tiled_shape(int Dd, int Ff) { return Dd == D && Ff == F; }

cudaError_t prepare_fp32_tiled() {
  cudaError_t e = cudaFuncSetAttribute(fp32_tiled_sweep, cudaFuncAttributeMaxDynamicSharedMemorySize, TOK_SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fp32_tiled_bsweep, cudaFuncAttributeMaxDynamicSharedMemorySize, BWD_SMEM);
  return e;
}

cudaError_t launch_fp32_tiled_sweep(const Params& prm, const WorkItem* items, int n, int step, cudaStream_t st) {
  return launch_pdl(fp32_tiled_sweep, dim3(n), dim3(NTH), TOK_SMEM, st, prm, items, step);
}

cudaError_t launch_fp32_tiled_bsweep(const Params& prm, const WorkItem* items, int n, cudaStream_t st) {
  return launch_pdl(fp32_tiled_bsweep, dim3(n), dim3(NTH), BWD_SMEM, st, prm, items);
}

}  // namespace scal3r
