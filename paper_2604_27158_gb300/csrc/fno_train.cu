// FNO training kernels (Sec. 2.2 forward with saved activations, and its exact
// reverse mode) for GB300 (sm_103a) and their C ABI.
//
// The training path keeps FP32 master parameters and FP32 activations: the forward
// pass saves, per layer, the latent field theta_n, the derivative sigma'(z_n) of its
// activation (zpre below) and the kept spectral coefficients X_n = F(theta_n); the backward pass is the chain rule
// through the same operators, with the spectral layer's adjoint written out:
//   z = W theta + b + F^-1(R . F(theta)),   theta' = sigma(z)
//   dz      = dtheta' * sigma'(z)
//   dW      = sum_pixels dz theta^T,  db = sum_pixels dz
//   dY[k]   = (c_kx / (H W)) * F(dz)[k]           (transpose of the real inverse)
//   dR[k]   = sum_batch conj(X[k]) dY[k]          (per-mode complex channel mixing)
//   dX[k]   = dY[k] conj(R[k])^T
//   dtheta  = W^T dz + Re sum_k dX[k] e^{+i phi_k}  (transpose of the forward DFT)
// with F the truncated forward DFT over ky in [0, m) U [H-m, H), kx in [0, m),
// c_0 = 1, c_kx = 2 for kx > 0, phi_k = 2 pi (ky y / H + kx x / W).
//
// Layout: latent fields channels-last, [B][H][W][C] FP32 (pixel p = (b H + y) W + x);
// spectral buffers [B][rows][m][C] float2.  Every reduction is in a fixed order (block
// partials, then one ordered pass), so gradients are deterministic.
#include <math.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "gelu_train_poly.cuh"

namespace lbmfno {

namespace {

inline cudaStream_t TS(void* s) { return reinterpret_cast<cudaStream_t>(s); }

constexpr int kTrModesMax = 32;
constexpr int kTrSms = 152;
__host__ __device__ constexpr int pw_ctas(int threads) { return 512 / threads; }  // 128 registers
constexpr int kWgThreads = 256;  // threads of the weight-gradient kernel
constexpr int kWgTile = 64;      // pixels of one of its stages
constexpr int kDftM = 128;       // (row, channel) pairs of an x-DFT block
constexpr int kDftX = 32;        // columns of one of its stages
constexpr int kDftYA = 8;        // kept rows of a forward y-DFT thread
constexpr int kDftYC = 64;       // rows of one of its stages
constexpr int kInvY = 8;         // rows of an inverse y-DFT thread
__host__ __device__ constexpr int y_chunks(int mc) { return (mc + 63) / 64; }  // blocks of an item's m C columns

struct TrOff {
  size_t lift0_w, lift0_b, lift1_w, lift1_b;
  std::vector<size_t> r1re, r1im, r2re, r2im, w, b, dec_w, dec_b;
  size_t out_w, out_b, n;
};

int tr_offsets(const fno_config& c, TrOff* o) {
  LBM_REQUIRE(c.c_in >= 1 && c.c_in <= 16 && c.c_out >= 1 && c.c_out <= 16,
              "fno_train: channel counts out of range");
  LBM_REQUIRE(c.width >= 2 && c.width <= 64 && c.width % 2 == 0,
              "fno_train: width must be even, <= 64");
  LBM_REQUIRE(c.layers >= 1 && c.layers <= 16 && c.modes >= 1 && c.modes <= kTrModesMax,
              "fno_train: layers in 1..16, modes in 1..%d", kTrModesMax);
  LBM_REQUIRE(c.dec_layers >= 1 && c.dec_layers <= 8 && c.dec_size >= 1 && c.dec_size <= 64,
              "fno_train: decoder shape out of range");
  LBM_REQUIRE(c.activation == FNO_ACT_GELU || c.activation == FNO_ACT_RELU,
              "fno_train: unknown activation");
  LBM_REQUIRE(c.padding == 0, "fno_train: padding is not supported by the training path");
  const size_t C = c.width, h = C / 2, m = c.modes, cin2 = c.c_in + 2;
  size_t p = 0;
  auto take = [&](size_t n) {
    const size_t at = p;
    p += n;
    return at;
  };
  o->lift0_w = take(h * cin2);
  o->lift0_b = take(h);
  o->lift1_w = take(C * h);
  o->lift1_b = take(C);
  for (int n = 0; n < c.layers; ++n) {
    o->r1re.push_back(take(C * C * m * m));
    o->r1im.push_back(take(C * C * m * m));
    o->r2re.push_back(take(C * C * m * m));
    o->r2im.push_back(take(C * C * m * m));
    o->w.push_back(take(C * C));
    o->b.push_back(take(C));
  }
  size_t fan = C;
  for (int l = 0; l < c.dec_layers; ++l) {
    o->dec_w.push_back(take((size_t)c.dec_size * fan));
    o->dec_b.push_back(take(c.dec_size));
    fan = c.dec_size;
  }
  o->out_w = take((size_t)c.c_out * fan);
  o->out_b = take(c.c_out);
  o->n = p;
  return LBM_OK;
}

// Saved activations (floats) and workspace (bytes) of one (config, B, H, W).
struct TrPlan {
  size_t P, C, S, h, cin2, m;
  // saved, in floats
  size_t xin, h1pre, theta, zpre, xh, hdpre, saved_floats;
  // workspace, in bytes
  size_t rt, x1, yh, dyh, z, ta, tb, part, ex, ey, ycl, ws_bytes;
  size_t s, twx, twy;  // ReLU forward pass
  int wg_blocks;
  int np, ng, ep;  // x-DFT: kx pairs a thread, thread groups, floats a row of the table
};

TrPlan tr_plan(const fno_config& c, int B, int H, int W) {
  TrPlan t{};
  t.P = (size_t)B * H * W;
  t.C = c.width;
  t.S = c.dec_size;
  t.h = c.width / 2;
  t.cin2 = c.c_in + 2;
  t.m = c.modes;
  const size_t N = c.layers, L = c.dec_layers, P = t.P, C = t.C, m = t.m;
  const size_t spec = (size_t)B * 2 * m * m * C;  // float2 per layer
  size_t f = 0;
  auto takef = [&](size_t n) {
    const size_t at = f;
    f += (n + 63) / 64 * 64;
    return at;
  };
  t.xin = takef(P * t.cin2);
  t.h1pre = takef(P * t.h);
  t.theta = takef((N + 1) * P * C);
  t.zpre = takef(N * P * C);
  t.xh = takef(N * spec * 2);
  t.hdpre = takef(L * P * t.S);
  t.saved_floats = f;
  size_t b = 0;
  auto take = [&](size_t bytes) {
    const size_t at = b;
    b = align_up(b + bytes, 256);
    return at;
  };
  const size_t wide = std::max(std::max(C, t.S), std::max(t.cin2, (size_t)c.c_out));
  t.rt = take(N * 2 * m * m * C * C * sizeof(float2));
  t.x1 = take((size_t)B * H * m * C * sizeof(float2));
  t.yh = take(spec * sizeof(float2));
  t.dyh = take(spec * sizeof(float2));
  t.z = take((size_t)B * H * m * C * sizeof(float2));
  t.ta = take(P * wide * sizeof(float));
  t.tb = take(P * wide * sizeof(float));
  t.wg_blocks = (int)std::min<size_t>(2 * kTrSms, (P + 4 * kWgTile - 1) / (4 * kWgTile));
  t.part = take((size_t)t.wg_blocks * 64 * 65 * sizeof(float));
  // kx pairs a thread of the x-DFT: the split with the fewest padded pairs
  t.np = 4;
  for (int np : {6, 7, 8})
    if ((m + np - 1) / np * np < (m + t.np - 1) / t.np * t.np ||
        ((m + np - 1) / np * np == (m + t.np - 1) / t.np * t.np && np > t.np))
      t.np = np;
  t.ng = (int)((m + t.np - 1) / t.np);
  t.ep = (2 * t.np * t.ng + 3) / 4 * 4;
  t.ex = take((size_t)W * t.ep * sizeof(float));
  t.ey = take((size_t)H * 2 * m * sizeof(float4));
  t.ycl = take(P * c.c_out * sizeof(float));
  if (c.activation == FNO_ACT_RELU) {
    t.s = take(P * C * sizeof(float));
    t.twx = take((size_t)W * sizeof(float2));
    t.twy = take((size_t)H * sizeof(float2));
  }
  t.ws_bytes = b;
  return t;
}

// sigma(v) and sigma'(v) of two values: GELU v Phi(v) and Phi(v) + v phi(v), or ReLU and the
// step function.  With a = |v|, e = exp(-a^2 / 2) and Q = Phi(-a) = e S(a) (gelu_train_poly.cuh):
//   v Phi(v) = max(v, 0) - a Q,   sigma'(v) = 1 - r for v >= 0, r else, r = e (S - a / sqrt(2 pi)).
// Packed FP32, one ex2.approx a value; as accurate as the erf form in FP32 (2.4e-7 at most, 1.8e-8
// rms on normal values, against 4.5e-7 and 2.4e-8; the derivative 2.6e-8 rms, against 2.6e-8).  The
// erf form took as many issue slots as the 64-channel layer it follows.  NaN propagates.
__device__ __forceinline__ void tr_gelu2(float2 v, float2* g, float2* d) {
  constexpr float c[GELU_T_DEG + 1] = GELU_T_COEFFS;
  // |v|; positive values are clamped to 64, where the tail is 0, so that a Q is 0 for +inf; -inf
  // and the derivative of both infinities are NaN, as in the erf form
  const float2 a = make_float2(fmaxf(-v.x, fminf(v.x, 64.0f)), fmaxf(-v.y, fminf(v.y, 64.0f)));
  const float2 u = __ffma2_rn(make_float2(fminf(a.x, 6.0f), fminf(a.y, 6.0f)),
                              make_float2(1.0f / 3.0f, 1.0f / 3.0f), make_float2(-1.0f, -1.0f));
  float2 p = make_float2(c[GELU_T_DEG], c[GELU_T_DEG]);
#pragma unroll
  for (int k = GELU_T_DEG - 1; k >= 0; --k) p = __ffma2_rn(p, u, make_float2(c[k], c[k]));
  const float2 t = __fmul2_rn(__fmul2_rn(a, a), make_float2(-0.72134752044448170f, -0.72134752044448170f));
  float2 e;  // 2^t = exp(-a^2 / 2)
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.x) : "f"(t.x));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.y) : "f"(t.y));
  float2 h;
  asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(h.x) : "f"(v.x));
  asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(h.y) : "f"(v.y));
  if (g) *g = __ffma2_rn(make_float2(-a.x, -a.y), __fmul2_rn(e, p), h);
  if (d) {
    const float2 nv = make_float2(-fabsf(v.x), -fabsf(v.y));
    const float2 r = __fmul2_rn(e, __ffma2_rn(nv, make_float2(0.39894228040143268f, 0.39894228040143268f), p));
    // a NaN compares false with both: v itself
    *d = make_float2(v.x >= 0.0f ? 1.0f - r.x : (v.x < 0.0f ? r.x : v.x),
                     v.y >= 0.0f ? 1.0f - r.y : (v.y < 0.0f ? r.y : v.y));
  }
}
__device__ __forceinline__ float2 tr_act2(float2 v, int act) {
  if (act != FNO_ACT_GELU) return make_float2(fmaxf(v.x, 0.0f), fmaxf(v.y, 0.0f));
  float2 g;
  tr_gelu2(v, &g, nullptr);
  return g;
}
__device__ __forceinline__ float2 tr_dact2(float2 v, int act) {
  if (act != FNO_ACT_GELU) return make_float2(v.x > 0.0f ? 1.0f : 0.0f, v.y > 0.0f ? 1.0f : 0.0f);
  float2 d;
  tr_gelu2(v, nullptr, &d);
  return d;
}
__device__ __forceinline__ float4 tr_act4(float4 v, int act) {
  const float2 a = tr_act2(make_float2(v.x, v.y), act), b = tr_act2(make_float2(v.z, v.w), act);
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float tr_act(float v, int act) { return tr_act2(make_float2(v, v), act).x; }
__device__ __forceinline__ float bf16r(float v) {
  return __bfloat162float(__float2bfloat16_rn(v));
}

// ex[x][2 kx] = (cos, -sin)(2 pi kx x / W), 0 for kx >= m.
__global__ void k_tr_ex(float* __restrict__ ex, int W, int m, int ep) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= W * (ep / 2)) return;
  const int x = t / (ep / 2), kx = t - x * (ep / 2);
  double s = 0.0, c = 0.0;
  if (kx < m) sincospi(2.0 * (double)((long long)kx * x % W) / (double)W, &s, &c);
  ex[x * ep + 2 * kx] = (float)c;
  ex[x * ep + 2 * kx + 1] = (float)-s;
}
// ey[y][a] = (cos, -sin, sin, cos)(2 pi ky(a) y / H), ky(a) = a (a < m) or H - 2m + a: a
// complex product with e^{-i phi} is two packed multiply-adds.
__global__ void k_tr_ey(float4* __restrict__ ey, int H, int m) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= H * 2 * m) return;
  const int y = t / (2 * m), a = t - y * (2 * m);
  const int ky = a < m ? a : H - 2 * m + a;
  double s, c;
  sincospi(2.0 * (double)((long long)ky * y % H) / (double)H, &s, &c);
  ey[t] = make_float4((float)c, (float)-s, (float)s, (float)c);
}

// Rt[layer][mode][i][o] = R[i][o][ky][kx] (mode = a m + kx; a < m: r1 at ky = a,
// a >= m: r2 at ky = a - m).
struct RtOffs {
  unsigned long long v[4 * 16];  // r1re, r1im, r2re, r2im of each layer
};
__global__ void k_tr_rt(const float* __restrict__ params, const RtOffs offs,
                        float2* __restrict__ rt, int layers, int C, int m) {
  const size_t per = (size_t)2 * m * m * C * C;
  const size_t n = per * layers;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n;
       t += (size_t)gridDim.x * blockDim.x) {
    const int layer = (int)(t / per);
    const size_t r = t - layer * per;
    const int o = (int)(r % C);
    const int i = (int)((r / C) % C);
    const int mode = (int)(r / ((size_t)C * C));
    const int a = mode / m, kx = mode % m;
    const bool lo = a < m;
    const int ky = lo ? a : a - m;
    const size_t src = (((size_t)i * C + o) * m + ky) * m + kx;
    const unsigned long long* ol = offs.v + 4 * layer;
    rt[t] = lo ? make_float2(params[ol[0] + src], params[ol[1] + src])
               : make_float2(params[ol[2] + src], params[ol[3] + src]);
  }
}

// Lifting network input: xin[p] = (in channels, x/(W-1), y/(H-1)) with the coordinate
// channels rounded to bfloat16 as in the inference path.
__global__ void k_tr_xin(const float* __restrict__ in, float* __restrict__ xin, int B, int H,
                         int W, int cin) {
  const size_t P = (size_t)B * H * W;
  const size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (p >= P) return;
  const int x = (int)(p % W);
  const int y = (int)((p / W) % H);
  const int b = (int)(p / ((size_t)W * H));
  const int cin2 = cin + 2;
  for (int c = 0; c < cin; ++c) xin[p * cin2 + c] = in[(((size_t)b * cin + c) * H + y) * W + x];
  xin[p * cin2 + cin] = bf16r((float)x / (float)max(W - 1, 1));
  xin[p * cin2 + cin + 1] = bf16r((float)y / (float)max(H - 1, 1));
}

__device__ __forceinline__ void cpa16(float* s, const float* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(s)),
               "l"(g)
               : "memory");
}
__device__ __forceinline__ void cpa8(float* s, const float* g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(s)),
               "l"(g)
               : "memory");
}
__device__ __forceinline__ void cpa4(float* s, const float* g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(s)),
               "l"(g)
               : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cpa_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// Walks j = threadIdx.x, + n, ... over rows of `len` items as (row r, item c) with one division.
struct Walk {
  int r, c, dr, dc, len;
  __device__ __forceinline__ Walk(int n, int len_) : len(len_) {
    r = (int)threadIdx.x / len;
    c = (int)threadIdx.x - r * len;
    dr = n / len;
    dc = n - dr * len;
  }
  __device__ __forceinline__ void next() {
    r += dr;
    c += dc;
    if (c >= len) {
      c -= len;
      ++r;
    }
  }
};
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }

// Pointwise linear layer, with the inverse x-DFT of a row's coefficients added:
//   v[p][o] = bias[o] + sum_i Wm(o, i) A(in[p][i]) + sum_kx Re(z[row][kx][o] e^{+2 pi i kx x / W}),
//   Wm(o, i) = trans ? w[i * cout + o] : w[o * cin + i],  A = sigma if in_act else identity;
//   pre[p][o] = sigma'(v) (if pre);  out[p][o] = sigma(v) if out_act, v * d[p][o] if d,
//   v * sigma'(dz[p][o]) if dz, else v
// (planar: out is [b][cout][hw]).  One contraction over cin + 2m terms: the columns of A are
// the inputs and the (cos, -sin) table of the pixel's column, those of B the weights and the
// row's coefficients (Re, Im).
//
// FP32 multiply-adds bound it (64 channels, 13 modes: 92 terms an output against 16 bytes).  A
// thread owns PPT pixels x 4 outputs and packs its accumulators over pairs of terms, so both
// operands are plain 16-byte shared loads of four terms; row pitches are an odd number of
// 16-byte units (no bank conflicts) and weights are stored with the rows of the four outputs
// of a thread G apart.  A block walks a contiguous range of tiles; the next tile (and row's
// coefficients) is copied while the current one is summed.
struct PwArgs {
  const float* in;
  const float* w;
  const float* bias;
  const float2* z;   // [row][m][cout], or null
  const float* ex;
  const float* d;
  const float* dz;
  float* pre;
  float* out;
  size_t P, hw;
  int cin, cout, trans, in_act, out_act, act, planar;
  int in_vec, out_vec;  // pixels of `in`, and of every array of cout channels, are whole 16-byte units
  int W, m, ep;      // row length; modes and table pitch (z)
  int ap, wp, zp;    // row pitches: inputs, weights, coefficients
  int ntiles, tpr;   // tiles; tiles a row (z)
};
template <int OP, int PT, int NT>
__global__ void __launch_bounds__(NT, pw_ctas(NT)) k_tr_pw(const PwArgs a) {
  constexpr int G = OP / 4, NPG = NT / G, PPT = PT / NPG;
  static_assert(PPT >= 1 && NPG * PPT == PT, "pixels a thread");
  extern __shared__ __align__(16) float sm[];
  float* As = sm;                       // [2][PT][ap]: inputs, then the table's columns
  float* Ws = As + 2 * PT * a.ap;       // [OP][wp], output o in row (o % 4) * G + o / 4
  float* Zs = Ws + OP * a.wp;           // [2][OP][zp], rows as Ws
  const int ap = a.ap, wp = a.wp, zp = a.zp, cin = a.cin, cout = a.cout;
  const int cin4 = (cin + 3) & ~3, m2 = a.z ? 2 * a.m : 0, m24 = (m2 + 3) & ~3;
  for (int j = threadIdx.x; j < 2 * PT * ap + OP * (wp + 2 * zp); j += NT) sm[j] = 0.0f;
  __syncthreads();
  for (int j = threadIdx.x; j < cout * cin; j += NT) {
    const int o = a.trans ? j % cout : j / cin, i = a.trans ? j / cout : j - o * cin;
    Ws[((o & 3) * G + (o >> 2)) * wp + i] = a.w[j];
  }
  const int og = threadIdx.x % G, pg = threadIdx.x / G;
  float bias[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) bias[j] = a.bias && og * 4 + j < cout ? a.bias[og * 4 + j] : 0.0f;
  const int t0 = (int)((long long)a.ntiles * blockIdx.x / gridDim.x);
  const int t1 = (int)((long long)a.ntiles * (blockIdx.x + 1) / gridDim.x);
  // first pixel and pixels of tile t (x0: its column, z)
  auto place = [&](int t, size_t& p0, int& np, int& x0) {
    if (m2) {
      const int row = t / a.tpr;
      x0 = (t - row * a.tpr) * PT;
      p0 = (size_t)row * a.W + x0;
      np = min(PT, a.W - x0);
    } else {
      x0 = 0;
      p0 = (size_t)t * PT;
      np = (int)min((size_t)PT, a.P - p0);
    }
  };
  // items of a pixel's inputs as they are copied: four channels, or one
  const bool quad = a.in_vec;
  const Walk wa(NT, quad ? cin >> 2 : cin), we(NT, max(a.m, 1)),
      wz(NT, cout);
  auto load = [&](int t, int buf, bool zrow) {
    size_t p0;
    int np, x0;
    place(t, p0, np, x0);
    float* A = As + buf * PT * ap;
    const float* src = a.in + p0 * cin;
    if (quad) {
      for (Walk w = wa; w.r < np; w.next()) cpa16(A + w.r * ap + 4 * w.c, src + w.r * cin + 4 * w.c);
    } else {
      for (Walk w = wa; w.r < np; w.next()) cpa4(A + w.r * ap + w.c, src + w.r * cin + w.c);
    }
    if (m2) {
      for (Walk w = we; w.r < np; w.next())
        cpa8(A + w.r * ap + cin4 + 2 * w.c, a.ex + (x0 + w.r) * a.ep + 2 * w.c);
      if (zrow) {
        const int row = t / a.tpr;
        float* Z = Zs + (row & 1) * OP * zp;
        const float* zr = reinterpret_cast<const float*>(a.z + (size_t)row * a.m * cout);
        for (Walk w = wz; w.r < a.m; w.next())
          cpa8(Z + ((w.c & 3) * G + (w.c >> 2)) * zp + 2 * w.r, zr + 2 * (w.r * cout + w.c));
      }
    }
  };
  if (t0 < t1) load(t0, 0, true);
  cpa_commit();
  for (int t = t0; t < t1; ++t) {
    const int buf = (t - t0) & 1;
    size_t p0;
    int np, x0;
    place(t, p0, np, x0);
    if (t + 1 < t1) load(t + 1, buf ^ 1, m2 && (t + 1) % a.tpr == 0);
    cpa_commit();
    cpa_wait<1>();
    float* A = As + buf * PT * ap;
    if (a.in_act) {  // each thread the elements it copied
      if (quad) {
        for (Walk w = wa; w.r < np; w.next()) {
          float4* e = reinterpret_cast<float4*>(A + w.r * ap + 4 * w.c);
          *e = tr_act4(*e, a.act);
        }
      } else {
        for (Walk w = wa; w.r < np; w.next()) {
          float* e = A + w.r * ap + w.c;
          *e = tr_act(*e, a.act);
        }
      }
    }
    __syncthreads();
    float2 acc[PPT][4];
#pragma unroll
    for (int i = 0; i < PPT; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
    auto sums = [&](const float* ar, const float* br, int bp, int n) {
      const float *pa[PPT], *pb[4];  // running pointers: no address arithmetic but their steps
#pragma unroll
      for (int i = 0; i < PPT; ++i) pa[i] = ar + i * NPG * ap;
#pragma unroll
      for (int j = 0; j < 4; ++j) pb[j] = br + j * G * bp;
      auto term4 = [&](int at) {
        float4 b[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4*>(pb[j] + at);
#pragma unroll
        for (int i = 0; i < PPT; ++i) {
          const float4 v = *reinterpret_cast<const float4*>(pa[i] + at);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            acc[i][j] = __ffma2_rn(make_float2(v.x, v.y), make_float2(b[j].x, b[j].y), acc[i][j]);
            acc[i][j] = __ffma2_rn(make_float2(v.z, v.w), make_float2(b[j].z, b[j].w), acc[i][j]);
          }
        }
      };
      int k = 0;
#pragma unroll 1
      for (; k + 8 <= n; k += 8) {
        term4(0);
        term4(4);
#pragma unroll
        for (int i = 0; i < PPT; ++i) pa[i] += 8;
#pragma unroll
        for (int j = 0; j < 4; ++j) pb[j] += 8;
      }
      if (k < n) term4(0);
    };
    sums(A + pg * ap, Ws + og * wp, wp, cin4);
    if (m2) sums(A + pg * ap + cin4, Zs + ((t / a.tpr) & 1) * OP * zp + og * zp, zp, m24);
    __syncthreads();  // the buffers may be refilled
    if (og * 4 < cout) {
#pragma unroll
      for (int i = 0; i < PPT; ++i) {
        const int p = pg + i * NPG;
        if (p >= np) continue;
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = (acc[i][j].x + acc[i][j].y) + bias[j];
        const size_t at = (p0 + p) * cout + og * 4;
        if (a.planar) {
          const size_t b = (p0 + p) / a.hw, q = (p0 + p) - b * a.hw;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (og * 4 + j < cout) a.out[(b * cout + og * 4 + j) * a.hw + q] = v[j];
        } else {
          // derivative of the activation (pre) or of the one whose argument dz holds, and value
          const bool quad_out = a.out_vec;
          float2 w0 = make_float2(v[0], v[1]), w1 = make_float2(v[2], v[3]);
          float2 f0 = w0, f1 = w1;
          if (a.dz || a.d) {
            float q[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            const float* from = (a.d ? a.d : a.dz) + at;
            if (quad_out) {
              const float4 q4 = *reinterpret_cast<const float4*>(from);
              q[0] = q4.x;
              q[1] = q4.y;
              q[2] = q4.z;
              q[3] = q4.w;
            } else {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (og * 4 + j < cout) q[j] = from[j];
            }
            float2 q0 = make_float2(q[0], q[1]), q1 = make_float2(q[2], q[3]);
            if (!a.d) {
              q0 = tr_dact2(q0, a.act);
              q1 = tr_dact2(q1, a.act);
            }
            w0 = __fmul2_rn(w0, q0);
            w1 = __fmul2_rn(w1, q1);
          } else if (a.out_act) {
            if (a.act == FNO_ACT_GELU) {
              tr_gelu2(f0, &w0, &f0);
              tr_gelu2(f1, &w1, &f1);
            } else {
              w0 = tr_act2(f0, a.act);
              w1 = tr_act2(f1, a.act);
              f0 = tr_dact2(f0, a.act);
              f1 = tr_dact2(f1, a.act);
            }
          }
          if (quad_out) {
            if (a.pre) *reinterpret_cast<float4*>(a.pre + at) = make_float4(f0.x, f0.y, f1.x, f1.y);
            *reinterpret_cast<float4*>(a.out + at) = make_float4(w0.x, w0.y, w1.x, w1.y);
          } else {
            const float f[4] = {f0.x, f0.y, f1.x, f1.y}, w[4] = {w0.x, w0.y, w1.x, w1.y};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              if (og * 4 + j >= cout) continue;
              if (a.pre) a.pre[at + j] = f[j];
              a.out[at + j] = w[j];
            }
          }
        }
      }
    }
  }
}

// Block partials of dW[o][i] = sum_p dz[p][o] A(in[p][i]) and db[o] = sum_p dz[p][o] (pair
// (o, cin) of the partial is db).  Block k covers a contiguous range of pixel tiles; a thread
// owns 8 x 8 pairs (two quads along each axis) and one pixel in `groups`, the groups' sums are
// added in order at the end.  FP32 multiply-adds bound it (32 packed ones for four shared loads);
// stages are copied one ahead of use.
struct WgArgs {
  const float* dz;
  const float* in;
  float* part;
  size_t P;
  int cout, cin, in_act, act;
  int dz_vec, in_vec;  // pixels are whole 16-byte units
};
__device__ __forceinline__ void wg_load(const float* src, int n, int c, int vec, int pitch,
                                        float* dst, const Walk& from) {
  if (vec) {
    for (Walk w = from; w.r < n; w.next()) cpa16(dst + w.r * pitch + 4 * w.c, src + w.r * c + 4 * w.c);
  } else {
    for (Walk w = from; w.r < n; w.next()) cpa4(dst + w.r * pitch + w.c, src + w.r * c + w.c);
  }
}
__global__ void __launch_bounds__(kWgThreads, 2) k_tr_wgrad(const WgArgs a) {
  extern __shared__ __align__(16) float sm[];
  const int nto = (a.cout + 7) / 8, nti = (a.cin + 7) / 8;
  const int dp = nto * 8, ip = nti * 8;             // row pitches
  const int stage = kWgTile * (dp + ip);
  const int tpg = nto * nti, groups = kWgThreads / tpg;
  const int g = threadIdx.x / tpg, tg = threadIdx.x - g * tpg;
  const int og = tg / nti, ig = tg - og * nti;
  const int nbs = kWgThreads / dp, bo = threadIdx.x % dp, bs = threadIdx.x / dp;  // bias sums
  const int npairs = a.cout * (a.cin + 1);
  const int sd = groups * dp, si = groups * ip;  // steps of a group's pixels
  for (int j = threadIdx.x; j < 2 * stage; j += kWgThreads) sm[j] = 0.0f;  // pads stay 0
  __syncthreads();
  const size_t tiles = (a.P + kWgTile - 1) / kWgTile;
  const size_t ta = tiles * blockIdx.x / gridDim.x, tb = tiles * (blockIdx.x + 1) / gridDim.x;
  const Walk wd(kWgThreads, a.dz_vec ? a.cout >> 2 : a.cout),
      wi(kWgThreads, a.in_vec ? a.cin >> 2 : a.cin);
  auto load = [&](size_t t, float* st) {
    const size_t p0 = t * kWgTile;
    const int n = (int)min((size_t)kWgTile, a.P - p0);
    wg_load(a.dz + p0 * a.cout, n, a.cout, a.dz_vec, dp, st, wd);
    wg_load(a.in + p0 * a.cin, n, a.cin, a.in_vec, ip, st + kWgTile * dp, wi);
  };
  float2 acc[8][4];
  float db = 0.0f;
#pragma unroll
  for (int o = 0; o < 8; ++o)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[o][i] = make_float2(0.0f, 0.0f);
  if (ta < tb) load(ta, sm);
  cpa_commit();
  for (size_t t = ta; t < tb; ++t) {
    float* st = sm + (t - ta & 1) * stage;
    if (t + 1 < tb) load(t + 1, sm + ((t - ta + 1) & 1) * stage);
    cpa_commit();
    cpa_wait<1>();
    __syncthreads();
    const int n = (int)min((size_t)kWgTile, a.P - t * kWgTile);
    float* is = st + kWgTile * dp;
    if (a.in_act) {
      for (int j = threadIdx.x; j < n * ip / 4; j += kWgThreads) {
        float4* e = reinterpret_cast<float4*>(is) + j;
        *e = tr_act4(*e, a.act);
      }
      __syncthreads();
    }
    if (g < groups) {
      const float *pd = st + g * dp + og * 4, *pe = pd + nto * 4;
      const float *pv = is + g * ip + ig * 4, *pw = pv + nti * 4;
#pragma unroll 2
      for (int p = g; p < n; p += groups) {
        const float4 d0 = *reinterpret_cast<const float4*>(pd);
        const float4 d1 = *reinterpret_cast<const float4*>(pe);
        const float4 v0 = *reinterpret_cast<const float4*>(pv);
        const float4 v1 = *reinterpret_cast<const float4*>(pw);
        pd += sd;
        pe += sd;
        pv += si;
        pw += si;
        const float dd[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
        const float2 vv[4] = {make_float2(v0.x, v0.y), make_float2(v0.z, v0.w),
                              make_float2(v1.x, v1.y), make_float2(v1.z, v1.w)};
#pragma unroll
        for (int o = 0; o < 8; ++o)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[o][i] = __ffma2_rn(dup2(dd[o]), vv[i], acc[o][i]);
      }
    }
    if (bs < nbs)
      for (int p = bs; p < n; p += nbs) db += st[p * dp + bo];
    __syncthreads();
  }
  cpa_wait<0>();
  __syncthreads();
  // The groups' sums, in order: as many groups at a time as the stages' memory holds write their
  // accumulators, then each pair's are added by one thread.  (One group after the other, a
  // barrier each: 93 us a launch on layers of 8 x 8 channels and 22,000 pixels, now 9.)
  float* red = sm;  // [dp][ip + 1]
  const int rp = ip + 1;
  float* slot = sm + (dp * rp + 1) / 2 * 2;  // [nslot][dp][ip]
  const int nslot = (2 * stage - (dp * rp + 1)) / (dp * ip), have = min(groups, kWgTile);
  for (int j = threadIdx.x; j < dp * rp; j += kWgThreads) red[j] = 0.0f;
  for (int q = 0; q < have; q += nslot) {
    __syncthreads();
    if (g >= q && g < min(q + nslot, have)) {
      float* to = slot + (g - q) * dp * ip;
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        const int oo = (o >> 2) * nto * 4 + og * 4 + (o & 3);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          *reinterpret_cast<float2*>(to + oo * ip + (i >> 1) * nti * 4 + ig * 4 + (i & 1) * 2) =
              acc[o][i];
      }
    }
    __syncthreads();
    const int n = min(nslot, have - q);
    for (int j = threadIdx.x; j < dp * ip; j += kWgThreads) {
      const int oo = j / ip;
      float v = red[oo * rp + j - oo * ip];
      for (int k = 0; k < n; ++k) v += slot[k * dp * ip + j];
      red[oo * rp + j - oo * ip] = v;
    }
  }
  __syncthreads();
  if (bs < nbs) slot[bs * dp + bo] = db;
  __syncthreads();
  if (threadIdx.x < dp) {
    float v = 0.0f;
    for (int q = 0; q < nbs; ++q) v += slot[q * dp + threadIdx.x];
    red[threadIdx.x * rp + ip] = v;
  }
  __syncthreads();
  float* out = a.part + (size_t)blockIdx.x * npairs;
  for (int j = threadIdx.x; j < npairs; j += kWgThreads) {
    const int o = j / (a.cin + 1), i = j - o * (a.cin + 1);
    out[j] = red[o * rp + (i == a.cin ? ip : i)];
  }
}

// Ordered sum of the block partials into dW (cout x cin) and db (cout): 32 pairs a block,
// eight interleaved slices of the partials, in FP64.
__global__ void __launch_bounds__(256) k_tr_wgrad_reduce(const float* __restrict__ part, int nblk,
                                                         int cout, int cin, float* __restrict__ dw,
                                                         float* __restrict__ db) {
  __shared__ double red[8][32];
  const int npairs = cout * (cin + 1);
  const int l = threadIdx.x & 31, s = threadIdx.x >> 5;
  const int pr = blockIdx.x * 32 + l;
  double v = 0.0;
  if (pr < npairs)
    for (int k = s; k < nblk; k += 8) v += (double)part[(size_t)k * npairs + pr];
  red[s][l] = v;
  __syncthreads();
  if (s == 0 && pr < npairs) {
    for (int q = 1; q < 8; ++q) v += red[q][l];
    const int o = pr / (cin + 1), i = pr - o * (cin + 1);
    if (i == cin)
      db[o] = (float)v;
    else
      dw[o * cin + i] = (float)v;
  }
}

// Forward x-DFT: X1[row][kx][c] = sum_x f[row][x][c] e^{-2 pi i kx x / W}.  A block takes
// kDftM (row, channel) pairs (whole rows' channels, padded to cp); a thread four channels x NP
// frequencies (accumulators (Re, Im) packed) of every ks-th column; the column slices are
// added in order.  Bound by FP32 multiply-adds and the one read of f; stages are double
// buffered.
// Where its blocks leave multiprocessors idle it takes fewer rows, and 16 warps instead of 8, that is
// more and shorter column slices: its time is then one block's.  (Eight channels, 29 modes, one item
// of 100 x 1000, a training pass: 1.00 -> 0.71 ms.)
template <int NP>
__global__ void __launch_bounds__(512, 1) k_tr_dft_x(const float* __restrict__ f,
                                                     float2* __restrict__ x1,
                                                     const float* __restrict__ ex, size_t rows,
                                                     int W, int C, int cp, int rpb, int m, int ng,
                                                     int ks, int ep, int vec) {
  extern __shared__ __align__(16) float sm[];
  const int stage = kDftX * (kDftM + ep);
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int kg = wp % ng, sl = wp / ng;
  const size_t row0 = (size_t)blockIdx.x * rpb;
  const int nr = (int)min((size_t)rpb, rows - row0);
  const int nthr = blockDim.x;
  const bool quad = vec;
  const Walk wf(nthr, quad ? C >> 2 : C);
  auto load = [&](int x0, float* st) {
    const int n = min(kDftX, W - x0);
    for (int r = 0; r < nr; ++r) {
      const float* src = f + ((row0 + r) * W + x0) * C;
      float* d = st + r * cp;
      if (quad) {
        for (Walk w = wf; w.r < n; w.next()) cpa16(d + w.r * kDftM + 4 * w.c, src + w.r * C + 4 * w.c);
      } else {
        for (Walk w = wf; w.r < n; w.next()) cpa4(d + w.r * kDftM + w.c, src + w.r * C + w.c);
      }
    }
    float* es = st + kDftX * kDftM;
    for (int j = threadIdx.x; j < n * (ep >> 2); j += nthr) cpa16(es + 4 * j, ex + x0 * ep + 4 * j);
  };
  float2 acc[4][NP];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int k = 0; k < NP; ++k) acc[j][k] = make_float2(0.0f, 0.0f);
  load(0, sm);
  cpa_commit();
  int it = 0;
  for (int x0 = 0; x0 < W; x0 += kDftX, it ^= 1) {
    if (x0 + kDftX < W) load(x0 + kDftX, sm + (it ^ 1) * stage);
    cpa_commit();
    cpa_wait<1>();
    __syncthreads();
    const float* st = sm + it * stage;
    const float* es = st + kDftX * kDftM + kg * 2 * NP;
    const int n = min(kDftX, W - x0);
    const float *pv = st + sl * kDftM + 4 * lane, *pe = es + sl * ep;
#pragma unroll 2
    for (int x = sl; x < n; x += ks) {
      const float4 v = *reinterpret_cast<const float4*>(pv);
      const float2 d[4] = {dup2(v.x), dup2(v.y), dup2(v.z), dup2(v.w)};
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        const float2 e = *reinterpret_cast<const float2*>(pe + 2 * k);
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[j][k] = __ffma2_rn(d[j], e, acc[j][k]);
      }
      pv += ks * kDftM;
      pe += ks * ep;
    }
    __syncthreads();
  }
  cpa_wait<0>();
  // the column slices, in order: slice q adds into (or starts) the block's sums
  float2* red = reinterpret_cast<float2*>(sm);  // [NP ng][kDftM]
  for (int q = 0; q < ks; ++q) {
    if (sl == q) {
#pragma unroll
      for (int k = 0; k < NP; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float2* r = red + (kg * NP + k) * kDftM + 4 * lane + j;
          if (q == 0)
            *r = acc[j][k];
          else
            *r = make_float2(r->x + acc[j][k].x, r->y + acc[j][k].y);
        }
    }
    __syncthreads();
  }
  for (int j = threadIdx.x; j < nr * m * C; j += nthr) {
    const int r = j / (m * C), kx = j / C - r * m, c = j % C;
    x1[((row0 + r) * m + kx) * C + c] = red[kx * kDftM + r * cp + c];
  }
}

// Forward y-DFT over the kept rows: Xh[b][a][kx][c] = scale(kx) sum_y X1[b][y][kx][c]
// e^{-2 pi i ky(a) y / H}, ky(a) = a (a < m) or H - 2m + a; scale = 1, or c_kx / (H W)
// for the adjoint of the real inverse transform.  A block takes 32 pairs of a batch item's m C
// columns (kx, c), a lane one pair, and kDftYA kept rows; a warp every eighth y; the warps' sums
// are added in order.  (With one kx a block, networks of 8 channels used four lanes of a warp and
// the same table rows in eight blocks: 32 items of 64 x 58, 29 modes, took 1.66 ms a training pass,
// now 0.91.)
__global__ void __launch_bounds__(256) k_tr_dft_y(const float2* __restrict__ x1,
                                                  float2* __restrict__ xh,
                                                  const float4* __restrict__ ey, int H, int W,
                                                  int C, int m, int adjoint_scale, int vec) {
  __shared__ float4 es[kDftYC][kDftYA];
  __shared__ float4 red[kDftYA][32];
  const int mc = m * C, nch = y_chunks(mc);
  const int b = blockIdx.x / nch, a0 = blockIdx.y * kDftYA;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int at = 2 * (32 * (int)(blockIdx.x % nch) + lane);  // the lane's first column
  const bool on = at < mc;
  float2 acc[kDftYA][2];
#pragma unroll
  for (int a = 0; a < kDftYA; ++a) acc[a][0] = acc[a][1] = make_float2(0.0f, 0.0f);
  for (int y0 = 0; y0 < H; y0 += kDftYC) {
    __syncthreads();
    for (int j = threadIdx.x; j < kDftYC * kDftYA; j += 256) {
      const int y = y0 + j / kDftYA, a = a0 + j % kDftYA;
      es[j / kDftYA][j % kDftYA] =
          y < H && a < 2 * m ? ey[(size_t)y * 2 * m + a] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    const int n = min(kDftYC, H - y0);
    if (on) {
#pragma unroll 4
      for (int y = wp; y < n; y += 8) {
        const float4 v = *reinterpret_cast<const float4*>(
            x1 + ((size_t)b * H + y0 + y) * mc + at);
#pragma unroll
        for (int a = 0; a < kDftYA; ++a) {
          const float4 e = es[y][a];
          acc[a][0] = __ffma2_rn(dup2(v.x), make_float2(e.x, e.y), acc[a][0]);
          acc[a][0] = __ffma2_rn(dup2(v.y), make_float2(e.z, e.w), acc[a][0]);
          acc[a][1] = __ffma2_rn(dup2(v.z), make_float2(e.x, e.y), acc[a][1]);
          acc[a][1] = __ffma2_rn(dup2(v.w), make_float2(e.z, e.w), acc[a][1]);
        }
      }
    }
  }
  for (int q = 0; q < 8; ++q) {
    if (wp == q) {
#pragma unroll
      for (int a = 0; a < kDftYA; ++a) {
        float4 r = q ? red[a][lane] : make_float4(0.f, 0.f, 0.f, 0.f);
        red[a][lane] = make_float4(r.x + acc[a][0].x, r.y + acc[a][0].y, r.z + acc[a][1].x,
                                   r.w + acc[a][1].y);
      }
    }
    __syncthreads();
  }
  const float sc = adjoint_scale ? (at < C ? 1.0f : 2.0f) / ((float)H * (float)W) : 1.0f;
  const int a = wp;  // kDftYA == 8 warps
  if (on && a0 + a < 2 * m) {
    const float4 r = red[a][lane];
    float2* o = xh + ((size_t)b * 2 * m + a0 + a) * mc + at;
    if (vec) {
      *reinterpret_cast<float4*>(o) = make_float4(r.x * sc, r.y * sc, r.z * sc, r.w * sc);
    } else {
      o[0] = make_float2(r.x * sc, r.y * sc);
      o[1] = make_float2(r.z * sc, r.w * sc);
    }
  }
}

// ---- forward pass of ReLU networks -----------------------------------------------------------
// ReLU's derivative jumps at 0.  Sums in another order move the pre-activations that lie within
// rounding of 0 across it, and one pixel that changes sides changes a gradient, a sum over pixels
// with random signs, by 1e-4 of its norm or more, with the same error against 64 bits.  So the
// forward pass of ReLU networks keeps the order their results have always had: every sum runs over
// its terms one after the other (the kernels below, one output a thread and term loop).  The tiled
// kernels do not: their packed accumulators hold pairs of terms.  (Tiles whose accumulators hold
// pairs of outputs would keep this order; there are none yet.)  The backward pass, which takes
// the signs as saved, uses the tiled kernels.
constexpr int kSqPix = 128;      // pixels a block of the pointwise kernel
constexpr int kSqThreads = 256;
constexpr int kSqAcc = 16;       // spectral accumulators a thread

__global__ void k_sq_twiddle(float2* __restrict__ tw, int N) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < N) {
    double s, c;
    sincospi(2.0 * (double)t / (double)N, &s, &c);
    tw[t] = make_float2((float)c, (float)s);
  }
}

// Pointwise linear layer over kSqPix pixels per block:
//   v[p][o] = add[p][o] + bias[o] + sum_i w[o * cin + i] * in[p][i];
//   pre[p][o] = v (if pre != null);  out[p][o] = out_act ? max(v, 0) : v.
__global__ void __launch_bounds__(kSqPix) k_sq_pw(const float* __restrict__ in, int cin,
                                                  const float* __restrict__ w,
                                                  const float* __restrict__ bias,
                                                  const float* __restrict__ add, int cout,
                                                  float* __restrict__ pre, float* __restrict__ out,
                                                  int out_act, size_t P) {
  extern __shared__ float sm[];
  float* ws = sm;                               // [cout][cin]
  float* is = ws + cout * cin;                  // [kSqPix][cin + 1]
  float* os = is + kSqPix * (cin + 1);          // [kSqPix][cout + 1]
  const size_t p0 = (size_t)blockIdx.x * kSqPix;
  const int np = (int)min((size_t)kSqPix, P - p0);
  for (int j = threadIdx.x; j < cout * cin; j += kSqPix) ws[j] = w[j];
  for (int j = threadIdx.x; j < np * cin; j += kSqPix) {
    const int t = j / cin, i = j - t * cin;
    is[t * (cin + 1) + i] = in[p0 * cin + j];
  }
  for (int j = threadIdx.x; j < np * cout; j += kSqPix) {
    const int t = j / cout, o = j - t * cout;
    os[t * (cout + 1) + o] = (add ? add[p0 * cout + j] : 0.0f) + (bias ? bias[o] : 0.0f);
  }
  __syncthreads();
  const int t = threadIdx.x;
  if (t < np) {
    const float* ir = is + t * (cin + 1);
    float* orow = os + t * (cout + 1);
    for (int o = 0; o < cout; ++o) {
      const float* wr = ws + o * cin;
      float acc = 0.0f;
      for (int i = 0; i < cin; ++i) acc = fmaf(wr[i], ir[i], acc);
      orow[o] += acc;
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < np * cout; j += kSqPix) {
    const int tt = j / cout, o = j - tt * cout;
    const float v = os[tt * (cout + 1) + o];
    if (pre) pre[p0 * cout + j] = v;
    out[p0 * cout + j] = out_act ? fmaxf(v, 0.0f) : v;
  }
}

// Forward x-DFT of each row: X1[row][kx][c] = sum_x f[row][x][c] e^{-2 pi i kx x / W}.
__global__ void __launch_bounds__(kSqThreads) k_sq_dft_x(const float* __restrict__ f,
                                                           float2* __restrict__ x1,
                                                           const float2* __restrict__ twx,
                                                           int W, int C, int m) {
  extern __shared__ float sm[];
  float2* tw = reinterpret_cast<float2*>(sm);  // W
  float* tile = sm + 2 * W;                     // [32][C]
  const size_t row = blockIdx.x;
  for (int t = threadIdx.x; t < W; t += kSqThreads) tw[t] = twx[t];
  const int G = kSqThreads / C;
  const int c = threadIdx.x % C, g = threadIdx.x / C;
  float2 acc[kSqAcc];
#pragma unroll
  for (int k = 0; k < kSqAcc; ++k) acc[k] = make_float2(0.f, 0.f);
  for (int x0 = 0; x0 < W; x0 += 32) {
    const int nx = min(32, W - x0);
    __syncthreads();
    for (int j = threadIdx.x; j < nx * C; j += kSqThreads)
      tile[j] = f[(row * W + x0) * C + j];
    __syncthreads();
    if (g < G) {
#pragma unroll
      for (int k = 0; k < kSqAcc; ++k) {
        const int kx = g + k * G;
        if (kx < m) {
          int idx = (kx * x0) % W;  // phase index (kx x) mod W, advanced by kx per x
          for (int xx = 0; xx < nx; ++xx) {
            const float2 e = tw[idx];
            const float v = tile[xx * C + c];
            acc[k].x = fmaf(v, e.x, acc[k].x);
            acc[k].y = fmaf(-v, e.y, acc[k].y);
            idx += kx;
            if (idx >= W) idx -= W;
          }
        }
      }
    }
  }
  if (g < G) {
#pragma unroll
    for (int k = 0; k < kSqAcc; ++k) {
      const int kx = g + k * G;
      if (kx < m) x1[(row * m + kx) * C + c] = acc[k];
    }
  }
}

// Forward y-DFT over the kept rows: Xh[b][a][kx][c] = sum_y X1[b][y][kx][c]
// e^{-2 pi i ky(a) y / H}, ky(a) = a (a < m) or H - 2m + a.
__global__ void __launch_bounds__(kSqThreads) k_sq_dft_y(const float2* __restrict__ x1,
                                                           float2* __restrict__ xh,
                                                           const float2* __restrict__ twy,
                                                           int H, int C, int m) {
  extern __shared__ float sm[];
  float2* tw = reinterpret_cast<float2*>(sm);  // H
  float2* tile = tw + H;                        // [32][C]
  const int b = blockIdx.x / m, kx = blockIdx.x % m;
  for (int t = threadIdx.x; t < H; t += kSqThreads) tw[t] = twy[t];
  const int G = kSqThreads / C;
  const int c = threadIdx.x % C, g = threadIdx.x / C;
  float2 acc[kSqAcc];
#pragma unroll
  for (int k = 0; k < kSqAcc; ++k) acc[k] = make_float2(0.f, 0.f);
  for (int y0 = 0; y0 < H; y0 += 32) {
    const int ny = min(32, H - y0);
    __syncthreads();
    for (int j = threadIdx.x; j < ny * C; j += kSqThreads) {
      const int yy = j / C, cc = j - yy * C;
      tile[j] = x1[(((size_t)b * H + y0 + yy) * m + kx) * C + cc];
    }
    __syncthreads();
    if (g < G) {
#pragma unroll
      for (int k = 0; k < kSqAcc; ++k) {
        const int a = g + k * G;
        if (a < 2 * m) {
          const int ky = a < m ? a : H - 2 * m + a;
          int idx = (int)(((long long)ky * y0) % H);  // (ky y) mod H, advanced by ky per y
          for (int yy = 0; yy < ny; ++yy) {
            const float2 e = tw[idx];  // e^{+i}: use conj
            idx += ky;
            if (idx >= H) idx -= H;
            const float2 v = tile[yy * C + c];
            // v * conj(e)
            acc[k].x = fmaf(v.x, e.x, fmaf(v.y, e.y, acc[k].x));
            acc[k].y = fmaf(v.y, e.x, fmaf(-v.x, e.y, acc[k].y));
          }
        }
      }
    }
  }
  if (g < G) {
#pragma unroll
    for (int k = 0; k < kSqAcc; ++k) {
      const int a = g + k * G;
      if (a < 2 * m) xh[(((size_t)b * 2 * m + a) * m + kx) * C + c] = acc[k];
    }
  }
}

// Inverse y-DFT: Z[b][y][kx][c] = sum_a Yh[b][a][kx][c] e^{+2 pi i ky(a) y / H}.
__global__ void __launch_bounds__(kSqThreads) k_sq_inv_y(const float2* __restrict__ yh,
                                                           float2* __restrict__ z,
                                                           const float2* __restrict__ twy,
                                                           int H, int C, int m) {
  extern __shared__ float sm[];
  float2* tw = reinterpret_cast<float2*>(sm);  // H
  float2* col = tw + H;                         // [2m][C]
  const int b = blockIdx.x / m, kx = blockIdx.x % m;
  for (int t = threadIdx.x; t < H; t += kSqThreads) tw[t] = twy[t];
  for (int j = threadIdx.x; j < 2 * m * C; j += kSqThreads) {
    const int a = j / C, c = j - a * C;
    col[j] = yh[(((size_t)b * 2 * m + a) * m + kx) * C + c];
  }
  __syncthreads();
  const int G = kSqThreads / C;
  const int c = threadIdx.x % C, g = threadIdx.x / C;
  if (g >= G) return;
  for (int y = g; y < H; y += G) {
    float re = 0.f, im = 0.f;
    int idx = 0;  // (ky y) mod H for ky = 0 .. m-1, then H-m .. H-1
    for (int a = 0; a < 2 * m; ++a) {
      if (a == m) idx = (int)(((long long)(H - m) * y) % H);
      const float2 e = tw[idx];
      idx += y;
      if (idx >= H) idx -= H;
      const float2 v = col[a * C + c];
      re = fmaf(v.x, e.x, fmaf(-v.y, e.y, re));
      im = fmaf(v.x, e.y, fmaf(v.y, e.x, im));
    }
    z[(((size_t)b * H + y) * m + kx) * C + c] = make_float2(re, im);
  }
}

// Inverse x-DFT with real output: S[row][x][c] = scale sum_kx c_kx Re(Z[row][kx][c]
// e^{+2 pi i kx x / W}).
__global__ void __launch_bounds__(kSqThreads) k_sq_inv_x(const float2* __restrict__ z,
                                                           float* __restrict__ s,
                                                           const float2* __restrict__ twx,
                                                           int W, int C, int m, float scale) {
  extern __shared__ float sm[];
  float2* tw = reinterpret_cast<float2*>(sm);  // W
  float2* zr = tw + W;                          // [m][C]
  const size_t row = blockIdx.x;
  for (int t = threadIdx.x; t < W; t += kSqThreads) tw[t] = twx[t];
  for (int j = threadIdx.x; j < m * C; j += kSqThreads) {
    const int kx = j / C;
    float2 v = z[row * m * C + j];
    const float wk = kx > 0 ? 2.0f * scale : scale;
    zr[j] = make_float2(v.x * wk, v.y * wk);
  }
  __syncthreads();
  const int G = kSqThreads / C;
  const int c = threadIdx.x % C, g = threadIdx.x / C;
  if (g >= G) return;
  for (int x = g; x < W; x += G) {
    float acc = 0.f;
    int idx = 0;  // (kx x) mod W
    for (int kx = 0; kx < m; ++kx) {
      const float2 e = tw[idx];
      idx += x;
      if (idx >= W) idx -= W;
      const float2 v = zr[kx * C + c];
      acc = fmaf(v.x, e.x, fmaf(-v.y, e.y, acc));
    }
    s[(row * W + x) * C + c] = acc;
  }
}

// ---- both -------------------------------------------------------------------------------------
// Per-mode channel mixing and its two adjoints (modes = 2 m m, Rt[mode][i][o]).
__global__ void k_tr_mix(const float2* __restrict__ xh, const float2* __restrict__ rt,
                         float2* __restrict__ yh, int B, int C, int modes) {
  const size_t n = (size_t)B * modes * C;
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int o = (int)(t % C);
  const size_t bm = t / C;  // b * modes + mode
  const int mode = (int)(bm % modes);
  const float2* xr = xh + bm * C;
  const float2* rr = rt + (size_t)mode * C * C + o;
  float re = 0.f, im = 0.f;
  for (int i = 0; i < C; ++i) {
    const float2 x = xr[i], r = rr[(size_t)i * C];
    re = fmaf(x.x, r.x, fmaf(-x.y, r.y, re));
    im = fmaf(x.x, r.y, fmaf(x.y, r.x, im));
  }
  yh[t] = make_float2(re, im);
}
__global__ void k_tr_mix_bwd_x(const float2* __restrict__ dyh, const float2* __restrict__ rt,
                               float2* __restrict__ dxh, int B, int C, int modes) {
  const size_t n = (size_t)B * modes * C;
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int i = (int)(t % C);
  const size_t bm = t / C;
  const int mode = (int)(bm % modes);
  const float2* dy = dyh + bm * C;
  const float2* rr = rt + ((size_t)mode * C + i) * C;
  float re = 0.f, im = 0.f;
  for (int o = 0; o < C; ++o) {  // dy * conj(r)
    const float2 d = dy[o], r = rr[o];
    re = fmaf(d.x, r.x, fmaf(d.y, r.y, re));
    im = fmaf(d.y, r.x, fmaf(-d.x, r.y, im));
  }
  dxh[t] = make_float2(re, im);
}
// dR[i][o][ky][kx] (re into r?re, im into r?im) = sum_b conj(X[b][mode][i]) dY[b][mode][o]
__global__ void k_tr_mix_bwd_r(const float2* __restrict__ xh, const float2* __restrict__ dyh,
                               float* __restrict__ dparams, size_t r1re, size_t r1im, size_t r2re,
                               size_t r2im, int B, int C, int m) {
  const int modes = 2 * m * m;
  const size_t n = (size_t)modes * C * C;
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int o = (int)(t % C);
  const int i = (int)((t / C) % C);
  const int mode = (int)(t / ((size_t)C * C));
  float re = 0.f, im = 0.f;
  for (int b = 0; b < B; ++b) {
    const float2 x = xh[((size_t)b * modes + mode) * C + i];
    const float2 d = dyh[((size_t)b * modes + mode) * C + o];
    re = fmaf(x.x, d.x, fmaf(x.y, d.y, re));
    im = fmaf(x.x, d.y, fmaf(-x.y, d.x, im));
  }
  const int a = mode / m, kx = mode % m;
  const bool lo = a < m;
  const int ky = lo ? a : a - m;
  const size_t dst = (((size_t)i * C + o) * m + ky) * m + kx;
  dparams[(lo ? r1re : r2re) + dst] = re;
  dparams[(lo ? r1im : r2im) + dst] = im;
}

// Inverse y-DFT: Z[b][y][kx][c] = w(kx) scale sum_a Yh[b][a][kx][c] e^{+2 pi i ky(a) y / H},
// w(kx) = c_kx (forward) or 1 (adjoint of the forward DFT), ready for the pointwise kernel.  A
// block takes 32 pairs of an item's columns (kx, c), as k_tr_dft_y, and 8 warps x kInvY rows.
__global__ void __launch_bounds__(256) k_tr_inv_y(const float2* __restrict__ yh,
                                                  float2* __restrict__ z,
                                                  const float4* __restrict__ ey, int H, int C,
                                                  int m, float scale, int hermitian) {
  extern __shared__ __align__(16) float sm[];
  constexpr int YB = 8 * kInvY, EP = YB + 1;
  float4* es = reinterpret_cast<float4*>(sm);       // [2m][EP]
  float4* col = es + 2 * m * EP;                    // [2m][32]
  const int mc = m * C, nch = y_chunks(mc);
  const int b = blockIdx.x / nch, y0 = blockIdx.y * YB;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int at0 = 64 * (int)(blockIdx.x % nch), at = at0 + 2 * lane;  // first columns: block, lane
  const bool on = at < mc;
  for (int j = threadIdx.x; j < 2 * m * YB; j += 256) {
    const int y = j / (2 * m), a = j - y * (2 * m);
    es[a * EP + y] = y0 + y < H ? ey[(size_t)(y0 + y) * 2 * m + a] : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  for (int j = threadIdx.x; j < 2 * m * 32; j += 256) {
    const int a = j >> 5, l = j & 31;
    if (at0 + 2 * l < mc)
      col[j] = *reinterpret_cast<const float4*>(yh + ((size_t)b * 2 * m + a) * mc + at0 + 2 * l);
  }
  __syncthreads();
  if (!on) return;
  float2 acc[kInvY][2];
#pragma unroll
  for (int y = 0; y < kInvY; ++y) acc[y][0] = acc[y][1] = make_float2(0.0f, 0.0f);
#pragma unroll 2
  for (int a = 0; a < 2 * m; ++a) {
    const float4 v = col[a * 32 + lane];
#pragma unroll
    for (int y = 0; y < kInvY; ++y) {
      const float4 e = es[a * EP + wp * kInvY + y];  // (c, -s, s, c); e^{+i phi}: (c, s, -s, c)
      acc[y][0] = __ffma2_rn(dup2(v.x), make_float2(e.x, e.z), acc[y][0]);
      acc[y][0] = __ffma2_rn(dup2(v.y), make_float2(e.y, e.w), acc[y][0]);
      acc[y][1] = __ffma2_rn(dup2(v.z), make_float2(e.x, e.z), acc[y][1]);
      acc[y][1] = __ffma2_rn(dup2(v.w), make_float2(e.y, e.w), acc[y][1]);
    }
  }
  const float w = (hermitian && at >= C) ? 2.0f * scale : scale;
#pragma unroll
  for (int y = 0; y < kInvY; ++y) {
    const int yy = y0 + wp * kInvY + y;
    if (yy < H)
      *reinterpret_cast<float4*>(z + ((size_t)b * H + yy) * mc + at) =
          make_float4(acc[y][0].x * w, acc[y][0].y * w, acc[y][1].x * w, acc[y][1].y * w);
  }
}

__global__ void k_sq_cl_to_nchw(const float* __restrict__ cl, float* __restrict__ out, int B,
                                int H, int W, int C) {
  const size_t n = (size_t)B * C * H * W;
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  const size_t hw = (size_t)H * W;
  const int b = (int)(t / (C * hw));
  const int c = (int)((t / hw) % C);
  const size_t q = t % hw;
  out[t] = cl[((size_t)b * hw + q) * C + c];
}
// planar -> channels-last for the gradient of the output
__global__ void k_tr_nchw_to_cl(const float* __restrict__ in, float* __restrict__ cl, int B, int H,
                                int W, int C) {
  const size_t n = (size_t)B * C * H * W;
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  const size_t hw = (size_t)H * W;
  const int b = (int)(t / (C * hw));
  const int c = (int)((t / hw) % C);
  const size_t q = t % hw;
  cl[((size_t)b * hw + q) * C + c] = in[t];
}
// din[b][c][y][x] = dxin[p][c] for the physical input channels
__global__ void k_tr_din(const float* __restrict__ dxin, float* __restrict__ din, int B, int H,
                         int W, int cin) {
  const size_t n = (size_t)B * cin * H * W;
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  const size_t hw = (size_t)H * W;
  const int b = (int)(t / (cin * hw));
  const int c = (int)((t / hw) % cin);
  const size_t q = t % hw;
  din[t] = dxin[((size_t)b * hw + q) * (cin + 2) + c];
}

inline unsigned nb(size_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

struct TrCtx {
  const fno_config* c;
  TrOff off;
  TrPlan pl;
  int B, H, W;
  cudaStream_t st;
  unsigned char* ws;
};

// Whether pixels of c channels at p are whole 16-byte units: the caller's saved_d may be 8-byte
// aligned only, and its arrays are then copied a value at a time.
int vec_of(const void* p, int c) {
  return c % 4 == 0 && (reinterpret_cast<uintptr_t>(p) & 15) == 0;
}

// A row pitch of at least n floats: an odd number of 16-byte units.
int odd_pitch(int n) { return 4 * (((n + 3) / 4) | 1); }
constexpr size_t kPwSmemMax = 227u << 10;
struct PwSmem {
  int ap, wp, zp;
  size_t bytes;
};
PwSmem pw_smem(int op, int pt, int cin, int m) {
  PwSmem r;
  r.ap = odd_pitch((cin + 3) / 4 * 4 + 2 * m);
  r.wp = odd_pitch(cin);
  r.zp = m ? odd_pitch(2 * m) : 0;
  r.bytes = sizeof(float) * ((size_t)2 * pt * r.ap + (size_t)op * (r.wp + 2 * r.zp));
  return r;
}
template <int OP, int PT, int NT>
int pw_run(const TrCtx& x, PwArgs a) {
  const PwSmem sm = pw_smem(OP, PT, a.cin, a.z ? a.m : 0);
  a.ap = sm.ap;
  a.wp = sm.wp;
  a.zp = sm.zp;
  a.tpr = (a.W + PT - 1) / PT;
  a.ntiles = a.z ? x.B * x.H * a.tpr : (int)((a.P + PT - 1) / PT);
  const int ctas = std::max(1, std::min<int>(pw_ctas(NT), (int)((227 << 10) / (sm.bytes + 1024))));
  k_tr_pw<OP, PT, NT><<<std::min(a.ntiles, ctas * kTrSms), NT, sm.bytes, x.st>>>(a);
  LBM_CHECK_LAUNCH();
  return LBM_OK;
}
// What one pointwise launch does besides its layer (PwArgs).
struct PwOpt {
  const float2* z = nullptr;
  const float* d = nullptr;
  const float* dz = nullptr;
  float* pre = nullptr;
  int in_act = 0, out_act = 0, planar = 0;
};
int pw(const TrCtx& x, const float* in, int cin, const float* w, int trans, const float* bias,
       int cout, float* out, const PwOpt& o = PwOpt{}) {
  PwArgs a{};
  a.in = in;
  a.w = w;
  a.bias = bias;
  a.z = o.z;
  a.ex = reinterpret_cast<const float*>(x.ws + x.pl.ex);
  a.d = o.d;
  a.dz = o.dz;
  a.pre = o.pre;
  a.out = out;
  a.P = x.pl.P;
  a.hw = (size_t)x.H * x.W;
  a.cin = cin;
  a.cout = cout;
  a.trans = trans;
  a.in_act = o.in_act;
  a.out_act = o.out_act;
  a.act = x.c->activation;
  a.planar = o.planar;
  a.in_vec = vec_of(in, cin);
  a.out_vec = vec_of(out, cout) && vec_of(o.d, cout) && vec_of(o.dz, cout) && vec_of(o.pre, cout);
  a.W = x.W;
  a.m = x.c->modes;
  a.ep = x.pl.ep;
  // Output columns of a block: the smallest tile that holds them.  64 columns: 256 pixels,
  // eight a thread (fewest shared loads a sum), when the stages fit and rows fill the tile.
  if (cout > 32) {
    if (pw_smem(64, 256, a.cin, a.z ? a.m : 0).bytes <= kPwSmemMax &&
        (a.z ? (a.W + 255) / 256 * 256 <= a.W + a.W / 4 : a.P >= (size_t)256 * kTrSms))
      return pw_run<64, 256, 512>(x, a);
    return pw_run<64, 64, 256>(x, a);
  }
  return cout > 16 ? pw_run<32, 128, 256>(x, a) : pw_run<16, 128, 256>(x, a);
}

size_t wg_smem(int cout, int cin) {
  const size_t dp = (cout + 7) / 8 * 8, ip = (cin + 7) / 8 * 8;
  return sizeof(float) * std::max(2 * kWgTile * (dp + ip), dp * (ip + 1));
}
int wgrad(const TrCtx& x, const float* dz, int cout, const float* in, int cin, int in_act,
          float* dw, float* db) {
  float* part = reinterpret_cast<float*>(x.ws + x.pl.part);
  const WgArgs a{dz, in, part, x.pl.P, cout, cin, in_act, x.c->activation, vec_of(dz, cout),
                 vec_of(in, cin)};
  k_tr_wgrad<<<x.pl.wg_blocks, kWgThreads, wg_smem(cout, cin), x.st>>>(a);
  LBM_CHECK_LAUNCH();
  k_tr_wgrad_reduce<<<nb((size_t)cout * (cin + 1), 32), 256, 0, x.st>>>(part, x.pl.wg_blocks, cout,
                                                                        cin, dw, db);
  LBM_CHECK_LAUNCH();
  return LBM_OK;
}

// X (or the adjoint-scaled dY) of a field: forward x-DFT then y-DFT over the kept rows.
size_t dft_x_smem(int ep, int np, int ng) {
  return std::max(sizeof(float) * 2 * kDftX * (kDftM + ep), sizeof(float2) * kDftM * np * ng);
}
int spectral_fwd(const TrCtx& x, const float* f, float2* out, int adjoint_scale) {
  const int C = x.c->width, m = x.c->modes, np = x.pl.np, ng = x.pl.ng, ep = x.pl.ep;
  float2* x1 = reinterpret_cast<float2*>(x.ws + x.pl.x1);
  const int cp = C <= 8 ? 8 : (C <= 16 ? 16 : (C <= 32 ? 32 : 64));
  const size_t rows = (size_t)x.B * x.H;
  int rpb = kDftM / cp;  // rows a block
  const int ks = std::max(1, (nb(rows, rpb) < (unsigned)kTrSms ? 16 : 8) / ng);
  while (rpb > 1 && nb(rows, rpb) < (unsigned)kTrSms) rpb /= 2;
  auto kernel = np == 4 ? k_tr_dft_x<4> : (np == 6 ? k_tr_dft_x<6> : (np == 7 ? k_tr_dft_x<7>
                                                                              : k_tr_dft_x<8>));
  kernel<<<nb(rows, rpb), 32 * ng * ks, dft_x_smem(ep, np, ng), x.st>>>(
      f, x1, reinterpret_cast<const float*>(x.ws + x.pl.ex), rows, x.W, C, cp, rpb, m, ng, ks, ep,
      vec_of(f, C));
  LBM_CHECK_LAUNCH();
  k_tr_dft_y<<<dim3(x.B * y_chunks(m * C), nb(2 * m, kDftYA)), 256, 0, x.st>>>(
      x1, out, reinterpret_cast<const float4*>(x.ws + x.pl.ey), x.H, x.W, C, m, adjoint_scale,
      vec_of(out, 4));
  LBM_CHECK_LAUNCH();
  return LBM_OK;
}

// Row coefficients from kept coefficients: the inverse y-DFT (the pointwise kernel does the
// rest of the inverse).
size_t inv_y_smem(int m) { return sizeof(float4) * 2 * m * (8 * kInvY + 1 + 32); }
int spectral_inv(const TrCtx& x, const float2* coef, float scale, int hermitian) {
  const int C = x.c->width, m = x.c->modes;
  k_tr_inv_y<<<dim3(x.B * y_chunks(m * C), nb(x.H, 8 * kInvY)), 256, inv_y_smem(m), x.st>>>(
      coef, reinterpret_cast<float2*>(x.ws + x.pl.z),
      reinterpret_cast<const float4*>(x.ws + x.pl.ey), x.H, C, m, scale, hermitian);
  LBM_CHECK_LAUNCH();
  return LBM_OK;
}

// The ReLU forward pass.
size_t sq_pw_smem(int cin, int cout) {
  return sizeof(float) * ((size_t)cout * cin + (size_t)kSqPix * (cin + 1) + (size_t)kSqPix * (cout + 1));
}

int sq_pw(const TrCtx& x, const float* in, int cin, const float* w, const float* bias,
          const float* add, int cout, float* pre, float* out, int out_act) {
  const size_t smem = sq_pw_smem(cin, cout);
  k_sq_pw<<<nb(x.pl.P, kSqPix), kSqPix, smem, x.st>>>(in, cin, w, bias, add, cout, pre, out,
                                                      out_act, x.pl.P);
  LBM_CHECK_LAUNCH();
  return LBM_OK;
}

// X of a field: forward x-DFT then y-DFT over the kept rows.
int sq_spectral_fwd(const TrCtx& x, const float* f, float2* out) {
  const int C = x.c->width, m = x.c->modes;
  float2* x1 = reinterpret_cast<float2*>(x.ws + x.pl.x1);
  const float2* twx = reinterpret_cast<const float2*>(x.ws + x.pl.twx);
  const float2* twy = reinterpret_cast<const float2*>(x.ws + x.pl.twy);
  k_sq_dft_x<<<x.B * x.H, kSqThreads, (2 * x.W + 32 * C) * sizeof(float), x.st>>>(f, x1, twx, x.W,
                                                                                    C, m);
  LBM_CHECK_LAUNCH();
  k_sq_dft_y<<<x.B * m, kSqThreads, (x.H + 32 * C) * sizeof(float2), x.st>>>(
      x1, out, twy, x.H, C, m);
  LBM_CHECK_LAUNCH();
  return LBM_OK;
}

// Real field from kept coefficients: inverse y-DFT then inverse x-DFT.
int sq_spectral_inv(const TrCtx& x, const float2* coef, float* s, float scale) {
  const int C = x.c->width, m = x.c->modes;
  float2* z = reinterpret_cast<float2*>(x.ws + x.pl.z);
  const float2* twx = reinterpret_cast<const float2*>(x.ws + x.pl.twx);
  const float2* twy = reinterpret_cast<const float2*>(x.ws + x.pl.twy);
  k_sq_inv_y<<<x.B * m, kSqThreads, (x.H + 2 * m * C) * sizeof(float2), x.st>>>(coef, z, twy,
                                                                                  x.H, C, m);
  LBM_CHECK_LAUNCH();
  k_sq_inv_x<<<x.B * x.H, kSqThreads, (x.W + m * C) * sizeof(float2), x.st>>>(z, s, twx, x.W, C, m,
                                                                                scale);
  LBM_CHECK_LAUNCH();
  return LBM_OK;
}


int sq_forward(const TrCtx& x, const float* params, const float* xin, float* saved, float* out_d) {
  const fno_config& c = *x.c;
  const TrPlan& pl = x.pl;
  const TrOff& o = x.off;
  const int B = x.B, C = c.width, h = C / 2, S = c.dec_size, m = c.modes;
  const size_t P = pl.P, spec = (size_t)B * 2 * m * m * C;
  float* ta = reinterpret_cast<float*>(x.ws + pl.ta);
  float* tb = reinterpret_cast<float*>(x.ws + pl.tb);
  float* s = reinterpret_cast<float*>(x.ws + pl.s);
  float* ycl = reinterpret_cast<float*>(x.ws + pl.ycl);
  float2* yh = reinterpret_cast<float2*>(x.ws + pl.yh);
  const float2* rt = reinterpret_cast<const float2*>(x.ws + pl.rt);
  const float* p = params;
  auto theta = [&](int n) { return saved + pl.theta + (size_t)n * P * C; };
  k_sq_twiddle<<<nb(x.W), 256, 0, x.st>>>(reinterpret_cast<float2*>(x.ws + pl.twx), x.W);
  LBM_CHECK_LAUNCH();
  k_sq_twiddle<<<nb(x.H), 256, 0, x.st>>>(reinterpret_cast<float2*>(x.ws + pl.twy), x.H);
  LBM_CHECK_LAUNCH();
  LBM_TRY(sq_pw(x, xin, c.c_in + 2, p + o.lift0_w, p + o.lift0_b, nullptr, h, saved + pl.h1pre,
                ta, 1));
  LBM_TRY(sq_pw(x, ta, h, p + o.lift1_w, p + o.lift1_b, nullptr, C, nullptr, theta(0), 0));
  for (int n = 0; n < c.layers; ++n) {
    float2* xh = reinterpret_cast<float2*>(saved + pl.xh) + (size_t)n * spec;
    LBM_TRY(sq_spectral_fwd(x, theta(n), xh));
    k_tr_mix<<<nb(spec), 256, 0, x.st>>>(xh, rt + (size_t)n * 2 * m * m * C * C, yh, B, C, 2 * m * m);
    LBM_CHECK_LAUNCH();
    LBM_TRY(sq_spectral_inv(x, yh, s, 1.0f / ((float)x.H * (float)x.W)));
    LBM_TRY(sq_pw(x, theta(n), C, p + o.w[n], p + o.b[n], s, C, saved + pl.zpre + (size_t)n * P * C,
                  theta(n + 1), 1));
  }
  const float* hin = theta(c.layers);
  int fan = C;
  for (int l = 0; l < c.dec_layers; ++l) {
    float* hout = (l % 2 == 0) ? ta : tb;
    LBM_TRY(sq_pw(x, hin, fan, p + o.dec_w[l], p + o.dec_b[l], nullptr, S,
                  saved + pl.hdpre + (size_t)l * P * S, hout, 1));
    hin = hout;
    fan = S;
  }
  LBM_TRY(sq_pw(x, hin, fan, p + o.out_w, p + o.out_b, nullptr, c.c_out, nullptr, ycl, 0));
  k_sq_cl_to_nchw<<<nb(P * c.c_out), 256, 0, x.st>>>(ycl, out_d, B, x.H, x.W, c.c_out);
  LBM_CHECK_LAUNCH();
  return LBM_OK;
}

template <typename K>
cudaError_t smem_limit(K k, size_t bytes) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
int set_smem_limits() {
  static bool done = false;
  if (done) return LBM_OK;
  LBM_CHECK_CUDA(smem_limit(k_tr_pw<64, 256, 512>, kPwSmemMax));
  LBM_CHECK_CUDA(smem_limit(k_tr_pw<64, 64, 256>, pw_smem(64, 64, 64, kTrModesMax).bytes));
  LBM_CHECK_CUDA(smem_limit(k_tr_pw<32, 128, 256>, pw_smem(32, 128, 64, kTrModesMax).bytes));
  LBM_CHECK_CUDA(smem_limit(k_tr_pw<16, 128, 256>, pw_smem(16, 128, 64, kTrModesMax).bytes));
  LBM_CHECK_CUDA(smem_limit(k_tr_wgrad, wg_smem(64, 64)));
  LBM_CHECK_CUDA(smem_limit(k_tr_dft_x<4>, dft_x_smem(64, 8, 4)));
  LBM_CHECK_CUDA(smem_limit(k_tr_dft_x<6>, dft_x_smem(72, 8, 5)));
  LBM_CHECK_CUDA(smem_limit(k_tr_dft_x<7>, dft_x_smem(72, 8, 5)));
  LBM_CHECK_CUDA(smem_limit(k_tr_dft_x<8>, dft_x_smem(64, 8, 4)));
  LBM_CHECK_CUDA(smem_limit(k_tr_inv_y, inv_y_smem(kTrModesMax)));
  LBM_CHECK_CUDA(cudaFuncSetAttribute(k_sq_pw, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)sq_pw_smem(64, 64)));
  LBM_CHECK_CUDA(cudaFuncSetAttribute(k_sq_dft_x, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)((2 * 2048 + 32 * 64) * sizeof(float))));
  LBM_CHECK_CUDA(cudaFuncSetAttribute(k_sq_dft_y, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)((8192 + 32 * 64) * sizeof(float2))));
  LBM_CHECK_CUDA(cudaFuncSetAttribute(k_sq_inv_y, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)((8192 + 2 * kTrModesMax * 64) * sizeof(float2))));
  LBM_CHECK_CUDA(cudaFuncSetAttribute(k_sq_inv_x, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)((2048 + kTrModesMax * 64) * sizeof(float2))));
  done = true;
  return LBM_OK;
}

int tr_setup(const fno_config* cfg, const float* params, const float* saved, int B, int H, int W,
             void* ws, void* stream, TrCtx* x) {
  LBM_REQUIRE(cfg != nullptr && params != nullptr && ws != nullptr, "fno_train: null argument");
  LBM_TRY(tr_offsets(*cfg, &x->off));
  LBM_REQUIRE(B >= 1 && H >= 2 && W >= 2 && H <= 8192 && W <= 2048,
              "fno_train: need B >= 1, 2 <= H <= 8192, 2 <= W <= 2048");
  LBM_REQUIRE(2 * cfg->modes <= H && cfg->modes <= W / 2, "fno_train: need 2m <= H and m <= W/2");
  LBM_REQUIRE((reinterpret_cast<uintptr_t>(ws) & 255) == 0, "fno_train: ws must be 256-byte aligned");
  LBM_REQUIRE((reinterpret_cast<uintptr_t>(saved) & 7) == 0,
              "fno_train: saved_d must be 8-byte aligned");
  LBM_TRY(set_smem_limits());
  x->c = cfg;
  x->pl = tr_plan(*cfg, B, H, W);
  x->B = B;
  x->H = H;
  x->W = W;
  x->st = TS(stream);
  x->ws = static_cast<unsigned char*>(ws);
  k_tr_ex<<<nb((size_t)W * x->pl.ep / 2), 256, 0, x->st>>>(
      reinterpret_cast<float*>(x->ws + x->pl.ex), W, cfg->modes, x->pl.ep);
  LBM_CHECK_LAUNCH();
  k_tr_ey<<<nb((size_t)H * 2 * cfg->modes), 256, 0, x->st>>>(
      reinterpret_cast<float4*>(x->ws + x->pl.ey), H, cfg->modes);
  LBM_CHECK_LAUNCH();
  // spectral filters per layer, transposed to [mode][i][o]
  RtOffs offs{};
  for (int n = 0; n < cfg->layers; ++n) {
    offs.v[4 * n + 0] = x->off.r1re[n];
    offs.v[4 * n + 1] = x->off.r1im[n];
    offs.v[4 * n + 2] = x->off.r2re[n];
    offs.v[4 * n + 3] = x->off.r2im[n];
  }
  const size_t nrt = (size_t)cfg->layers * 2 * cfg->modes * cfg->modes * cfg->width * cfg->width;
  k_tr_rt<<<(unsigned)std::min<size_t>(nb(nrt), 65535), 256, 0, x->st>>>(
      params, offs, reinterpret_cast<float2*>(x->ws + x->pl.rt), cfg->layers, cfg->width,
      cfg->modes);
  LBM_CHECK_LAUNCH();
  return LBM_OK;
}

}  // namespace

}  // namespace lbmfno

using namespace lbmfno;

extern "C" {

int fno_train_query(const fno_config* cfg_h, int B, int H, int W, fno_train_sizes* out_h) {
  LBM_REQUIRE(cfg_h != nullptr && out_h != nullptr, "fno_train_query: null argument");
  TrOff off;
  LBM_TRY(tr_offsets(*cfg_h, &off));
  LBM_REQUIRE(B >= 1 && H >= 2 && W >= 2, "fno_train_query: bad shape");
  const TrPlan pl = tr_plan(*cfg_h, B, H, W);
  out_h->n_params = off.n;
  out_h->saved_bytes = pl.saved_floats * sizeof(float);
  out_h->ws_bytes = pl.ws_bytes;
  return LBM_OK;
}

int fno_train_forward(const fno_config* cfg_h, const float* params_d, const float* in_d,
                      float* out_d, int B, int H, int W, float* saved_d, void* ws_d,
                      void* stream) {
  LBM_REQUIRE(in_d != nullptr && out_d != nullptr && saved_d != nullptr,
              "fno_train_forward: null argument");
  TrCtx x;
  LBM_TRY(tr_setup(cfg_h, params_d, saved_d, B, H, W, ws_d, stream, &x));
  const fno_config& c = *cfg_h;
  const TrPlan& pl = x.pl;
  const TrOff& o = x.off;
  const int C = c.width, h = C / 2, S = c.dec_size, m = c.modes;
  const size_t P = pl.P, spec = (size_t)B * 2 * m * m * C;
  float* xin = saved_d + pl.xin;
  float* h1pre = saved_d + pl.h1pre;
  auto theta = [&](int n) { return saved_d + pl.theta + (size_t)n * P * C; };
  auto zpre = [&](int n) { return saved_d + pl.zpre + (size_t)n * P * C; };
  auto xh = [&](int n) { return reinterpret_cast<float2*>(saved_d + pl.xh) + (size_t)n * spec; };
  auto hdpre = [&](int l) { return saved_d + pl.hdpre + (size_t)l * P * S; };
  float2* yh = reinterpret_cast<float2*>(x.ws + pl.yh);
  const float2* z = reinterpret_cast<const float2*>(x.ws + pl.z);
  const float2* rt = reinterpret_cast<const float2*>(x.ws + pl.rt);
  const float* p = params_d;

  k_tr_xin<<<nb(P), 256, 0, x.st>>>(in_d, xin, B, H, W, c.c_in);
  LBM_CHECK_LAUNCH();
  if (c.activation == FNO_ACT_RELU) return sq_forward(x, p, xin, saved_d, out_d);
  // hidden layers store their pre-activations only; the next layer applies sigma as it reads
  LBM_TRY(pw(x, xin, c.c_in + 2, p + o.lift0_w, 0, p + o.lift0_b, h, h1pre));
  PwOpt act_in;
  act_in.in_act = 1;
  LBM_TRY(pw(x, h1pre, h, p + o.lift1_w, 0, p + o.lift1_b, C, theta(0), act_in));
  for (int n = 0; n < c.layers; ++n) {
    LBM_TRY(spectral_fwd(x, theta(n), xh(n), 0));
    k_tr_mix<<<nb(spec), 256, 0, x.st>>>(xh(n), rt + (size_t)n * 2 * m * m * C * C, yh, B, C,
                                         2 * m * m);
    LBM_CHECK_LAUNCH();
    LBM_TRY(spectral_inv(x, yh, 1.0f / ((float)H * (float)W), 1));
    PwOpt opt;
    opt.z = z;
    opt.pre = zpre(n);
    opt.out_act = 1;
    LBM_TRY(pw(x, theta(n), C, p + o.w[n], 0, p + o.b[n], C, theta(n + 1), opt));
  }
  for (int l = 0; l < c.dec_layers; ++l)
    LBM_TRY(pw(x, l == 0 ? theta(c.layers) : hdpre(l - 1), l == 0 ? C : S, p + o.dec_w[l], 0,
               p + o.dec_b[l], S, hdpre(l), l == 0 ? PwOpt{} : act_in));
  act_in.planar = 1;
  LBM_TRY(pw(x, hdpre(c.dec_layers - 1), S, p + o.out_w, 0, p + o.out_b, c.c_out, out_d, act_in));
  return LBM_OK;
}

int fno_train_backward(const fno_config* cfg_h, const float* params_d, const float* dout_d,
                       const float* saved_d, float* dparams_d, float* din_d, int B, int H, int W,
                       void* ws_d, void* stream) {
  LBM_REQUIRE(dout_d != nullptr && saved_d != nullptr && dparams_d != nullptr,
              "fno_train_backward: null argument");
  TrCtx x;
  LBM_TRY(tr_setup(cfg_h, params_d, saved_d, B, H, W, ws_d, stream, &x));
  const fno_config& c = *cfg_h;
  const TrPlan& pl = x.pl;
  const TrOff& o = x.off;
  const int C = c.width, h = C / 2, S = c.dec_size, m = c.modes;
  const size_t P = pl.P, spec = (size_t)B * 2 * m * m * C;
  const float* xin = saved_d + pl.xin;
  const float* h1pre = saved_d + pl.h1pre;
  auto theta = [&](int n) { return saved_d + pl.theta + (size_t)n * P * C; };
  auto zpre = [&](int n) { return saved_d + pl.zpre + (size_t)n * P * C; };
  auto xh = [&](int n) {
    return reinterpret_cast<const float2*>(saved_d + pl.xh) + (size_t)n * spec;
  };
  auto hdpre = [&](int l) { return saved_d + pl.hdpre + (size_t)l * P * S; };
  float* ta = reinterpret_cast<float*>(x.ws + pl.ta);
  float* tb = reinterpret_cast<float*>(x.ws + pl.tb);
  float2* dyh = reinterpret_cast<float2*>(x.ws + pl.dyh);
  float2* dxh = reinterpret_cast<float2*>(x.ws + pl.yh);
  const float2* rt = reinterpret_cast<const float2*>(x.ws + pl.rt);
  const float* p = params_d;
  float* dp = dparams_d;

  // decoder: output layer, then the hidden layers in reverse
  float* ycl = reinterpret_cast<float*>(x.ws + pl.ycl);
  k_tr_nchw_to_cl<<<nb(P * c.c_out), 256, 0, x.st>>>(dout_d, ycl, B, H, W, c.c_out);
  LBM_CHECK_LAUNCH();
  const int L = c.dec_layers;
  const bool relu = c.activation == FNO_ACT_RELU;  // zpre holds z, not sigma'(z)
  // g: gradient with respect to the pre-activation of the layer at hand, in ta or tb
  LBM_TRY(wgrad(x, ycl, c.c_out, hdpre(L - 1), S, 1, dp + o.out_w, dp + o.out_b));
  PwOpt opt;
  opt.dz = hdpre(L - 1);
  LBM_TRY(pw(x, ycl, c.c_out, p + o.out_w, 1, nullptr, S, ta, opt));
  float* g = ta;
  for (int l = L - 1; l >= 0; --l) {
    const float* lin = (l == 0) ? theta(c.layers) : hdpre(l - 1);
    const int fan = (l == 0) ? C : S;
    LBM_TRY(wgrad(x, g, S, lin, fan, l == 0 ? 0 : 1, dp + o.dec_w[l], dp + o.dec_b[l]));
    float* gn = (g == ta) ? tb : ta;
    opt.d = (l == 0 && !relu) ? zpre(c.layers - 1) : nullptr;
    opt.dz = (l == 0) ? zpre(c.layers - 1) : hdpre(l - 1);
    LBM_TRY(pw(x, g, S, p + o.dec_w[l], 1, nullptr, fan, gn, opt));
    g = gn;
  }
  // Fourier layers in reverse: g = dz_n
  for (int n = c.layers - 1; n >= 0; --n) {
    LBM_TRY(wgrad(x, g, C, theta(n), C, 0, dp + o.w[n], dp + o.b[n]));
    LBM_TRY(spectral_fwd(x, g, dyh, 1));
    k_tr_mix_bwd_r<<<nb((size_t)2 * m * m * C * C), 256, 0, x.st>>>(
        xh(n), dyh, dp, o.r1re[n], o.r1im[n], o.r2re[n], o.r2im[n], B, C, m);
    LBM_CHECK_LAUNCH();
    k_tr_mix_bwd_x<<<nb(spec), 256, 0, x.st>>>(dyh, rt + (size_t)n * 2 * m * m * C * C, dxh, B, C,
                                               2 * m * m);
    LBM_CHECK_LAUNCH();
    LBM_TRY(spectral_inv(x, dxh, 1.0f, 0));
    float* gn = (g == ta) ? tb : ta;
    PwOpt lo;
    lo.z = reinterpret_cast<const float2*>(x.ws + pl.z);
    lo.d = n > 0 && !relu ? zpre(n - 1) : nullptr;
    lo.dz = n > 0 ? zpre(n - 1) : nullptr;
    LBM_TRY(pw(x, g, C, p + o.w[n], 1, nullptr, C, gn, lo));
    g = gn;
  }
  // lifting network: g = dL/dtheta_0
  LBM_TRY(wgrad(x, g, C, h1pre, h, 1, dp + o.lift1_w, dp + o.lift1_b));
  float* gh = (g == ta) ? tb : ta;
  opt.d = nullptr;
  opt.dz = h1pre;
  LBM_TRY(pw(x, g, C, p + o.lift1_w, 1, nullptr, h, gh, opt));
  LBM_TRY(wgrad(x, gh, h, xin, c.c_in + 2, 0, dp + o.lift0_w, dp + o.lift0_b));
  if (din_d) {
    float* gx = (gh == ta) ? tb : ta;
    LBM_TRY(pw(x, gh, h, p + o.lift0_w, 1, nullptr, c.c_in + 2, gx));
    k_tr_din<<<nb(P * c.c_in), 256, 0, x.st>>>(gx, din_d, B, H, W, c.c_in);
    LBM_CHECK_LAUNCH();
  }
  return LBM_OK;
}

}  // extern "C"
