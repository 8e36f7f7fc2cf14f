// NeuralODE object poses (Sec. 3.2, Eqs. 3-4): the object state
// z(t) = [position, rotation vector] evolves as dz/dt = f(z, t, c), f a
// two-hidden-layer tanh perceptron of width 64 and c the object's instance
// embedding; z at the output times comes from classical fourth-order
// Runge-Kutta steps from z(t0) (`substeps` equal steps between consecutive
// output times), and the pose at each output time is the rotation exp(r) as
// a unit quaternion with the translation z[0:3] (the instance pose of
// Sec. 3.3, local -> world).
//
// An instance's time steps are a chain of dependent evaluations of f, so the
// kernels are bound by the latency of one evaluation, not by throughput. One
// evaluation is spread over a group of two warps, thread u owning hidden unit
// u with its rows of the weights in registers; the 64-wide hidden vectors are
// exchanged through shared memory (one store, one 64-thread barrier, sixteen
// broadcast 128-bit loads) and the dot products are packed f32x2 FMAs in four
// chains. The six outputs are taken by four lanes each and broadcast with
// shuffles. With one warp per instance, two units per lane and the weights read
// from shared memory, an evaluation took about 2,200 cycles.
//
// The backward walks an instance's steps in reverse from the stored states. Its
// chain is only the adjoint: recomputing a step's four stages does not depend on
// it, nor do the parameter sums feed it. So a CTA (one instance) runs four
// groups side by side, two steps per tick: two groups recompute the stages of
// the tick's two steps, a third walks the adjoint through the two steps
// recomputed one tick earlier, a fourth adds the parameter adjoints of the two
// steps walked before those, its rows of the sums in registers, and a ninth warp
// takes the pose adjoints (sines and cosines) that enter the walk. They meet at
// one CTA barrier per tick and pass the activations through a ring of three
// ticks in shared memory.
//
// At 120 instances, 400 times, 2 substeps and embedding width 8 the forward
// takes 0.89 ms (570 cycles per evaluation) and the backward 0.98 ms, together
// 1.88 ms against 15.1 ms. The backward is bound by the adjoint's walk (545
// cycles per stage): without the ninth warp, its sines and cosines in the
// recomputing groups, it took 1.37 ms.
#include "s3r_internal.cuh"

namespace s3r {
namespace {

constexpr int kH = S3R_ODE_HIDDEN;     // hidden width
constexpr int kMaxD = S3R_ODE_MAX_EMBED;
constexpr int kGroup = kH;             // threads of a group: one per hidden unit
static_assert(kGroup == 64, "a group is two warps");

struct OdeLayout {
  int D, I;
  int64_t oW1, ob1, oW2, ob2, oW3, ob3, count;   // offsets in the flat parameter vector
};
__host__ __device__ inline OdeLayout ode_layout(int D) {
  OdeLayout L;
  L.D = D;
  L.I = 7 + D;
  L.oW1 = 0;
  L.ob1 = L.oW1 + (int64_t)kH * L.I;
  L.oW2 = L.ob1 + kH;
  L.ob2 = L.oW2 + (int64_t)kH * kH;
  L.oW3 = L.ob2 + kH;
  L.ob3 = L.oW3 + 6 * kH;
  L.count = L.ob3 + 6;
  return L;
}

// Barrier of one group (two warps); ids 1..4, 0 is the CTA's.
__device__ __forceinline__ void group_sync(int id) {
  asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory");
}

// Sum over the 64 entries of `v` (shared memory, 16-byte aligned) of v[m] w[m],
// w as consecutive pairs in registers.
__device__ __forceinline__ float dot64(const float* v, const f2 (&w)[kH / 2]) {
  const float4* v4 = reinterpret_cast<const float4*>(v);
  f2 acc[4];
#pragma unroll
  for (int i = 0; i < kH / 4; ++i) {
    const float4 x = v4[i];
    const int q = 2 * (i & 1);
    const f2 lo = pk(x.x, x.y), hi = pk(x.z, x.w);
    acc[q] = i < 2 ? mul2(lo, w[2 * i]) : fma2(lo, w[2 * i], acc[q]);
    acc[q + 1] = i < 2 ? mul2(hi, w[2 * i + 1]) : fma2(hi, w[2 * i + 1], acc[q + 1]);
  }
  float a, b;
  upk(add2(add2(acc[0], acc[1]), add2(acc[2], acc[3])), a, b);
  return a + b;
}

// Six 64-term sums at once: lane 4 o + q (o < 6) takes the 16 terms of output o
// in the float4s q, q + 4, q + 8, q + 12 of v; two shuffles add the quarters and
// six broadcast the outputs to every lane. `first` is added to output o.
__device__ __forceinline__ void six_sums(const float* v, const f2 (&w)[8], float first, uint32_t lane,
                                         float (&out)[6]) {
  const float4* v4 = reinterpret_cast<const float4*>(v) + (lane & 3u);
  f2 acc[2];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float4 x = v4[4 * i];
    acc[0] = i == 0 ? mul2(pk(x.x, x.y), w[0]) : fma2(pk(x.x, x.y), w[2 * i], acc[0]);
    acc[1] = i == 0 ? mul2(pk(x.z, x.w), w[1]) : fma2(pk(x.z, x.w), w[2 * i + 1], acc[1]);
  }
  float a, b;
  upk(add2(acc[0], acc[1]), a, b);
  a += b;
  a += __shfl_xor_sync(0xffffffffu, a, 1);
  a += __shfl_xor_sync(0xffffffffu, a, 2);
  a += first;
#pragma unroll
  for (int o = 0; o < 6; ++o) out[o] = __shfl_sync(0xffffffffu, a, 4 * o);
}

// Weights of one evaluation of f that thread u of a group keeps in registers.
struct EvalWeights {
  f2 w2[kH / 2];        // row u of W2
  f2 w3[8];             // its lane's quarter of row lane / 4 of W3 (see six_sums)
  float w1[6], wt;      // row u of W1: z and t
  float base;           // b1[u] + W1[u, 7:] c
  float b2, b3;
};
__device__ __forceinline__ void load_eval_weights(EvalWeights& e, const float* __restrict__ p,
                                                  const OdeLayout& L, const float* c, int u) {
  const uint32_t lane = (uint32_t)u & 31u;
  const float* W1 = p + L.oW1 + (int64_t)u * L.I;
#pragma unroll
  for (int i = 0; i < 6; ++i) e.w1[i] = W1[i];
  e.wt = W1[6];
  e.base = p[L.ob1 + u];
  for (int d = 0; d < L.D; ++d) e.base = fmaf(W1[7 + d], c[d], e.base);
  const float* W2 = p + L.oW2 + (int64_t)u * kH;
#pragma unroll
  for (int m = 0; m < kH / 2; ++m) e.w2[m] = pk(W2[2 * m], W2[2 * m + 1]);
  e.b2 = p[L.ob2 + u];
  const int o = (int)(lane >> 2);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = 4 * ((int)(lane & 3u) + 4 * (i >> 1)) + 2 * (i & 1);
    e.w3[i] = o < 6 ? pk(p[L.oW3 + o * kH + m], p[L.oW3 + o * kH + m + 1]) : pk(0.f, 0.f);
  }
  e.b3 = o < 6 ? p[L.ob3 + o] : 0.f;
}

// f(z, t, c) (Eq. 3) by one group: `out` in every thread; the hidden activations
// go to h1 and h2 (64 floats of shared memory each). h1 may be rewritten by the
// next evaluation and h2 after the next evaluation's first barrier, which is
// where this function writes them, so evaluations follow each other freely.
__device__ __forceinline__ void hidden(const EvalWeights& e, const float (&z)[6], float t, int u,
                                       int bar, float* h1, float* h2) {
  const float a = fmaf(e.w1[2], z[2], fmaf(e.w1[1], z[1], fmaf(e.w1[0], z[0], fmaf(e.wt, t, e.base))));
  const float b = fmaf(e.w1[5], z[5], fmaf(e.w1[4], z[4], e.w1[3] * z[3]));
  h1[u] = tanhf(a + b);
  group_sync(bar);
  h2[u] = tanhf(dot64(h1, e.w2) + e.b2);
}
__device__ __forceinline__ void eval_f(const EvalWeights& e, const float (&z)[6], float t, int u,
                                       int bar, float* h1, float* h2, float (&out)[6]) {
  hidden(e, z, t, u, bar, h1, h2);
  group_sync(bar);
  six_sums(h2, e.w3, e.b3, (uint32_t)u & 31u, out);
}

// exp(r) as a unit quaternion (w, x, y, z); a series below |r| = 1e-4.
__device__ __forceinline__ float4 quat_from_rotvec(float rx, float ry, float rz) {
  const float th2 = rx * rx + ry * ry + rz * rz;
  float cw, s;
  if (th2 < 1e-8f) {
    cw = 1.f - th2 * 0.125f;
    s = 0.5f - th2 * (1.f / 48.f);
  } else {
    const float th = sqrtf(th2);
    float sn, cs;
    sincosf(0.5f * th, &sn, &cs);
    cw = cs;
    s = sn / th;
  }
  return make_float4(cw, s * rx, s * ry, s * rz);
}

// Adjoint of r for the adjoint g of quat_from_rotvec(r).
__device__ __forceinline__ void quat_from_rotvec_vjp(const float r[3], float4 g, float out[3]) {
  const float th2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2];
  const float gv[3] = {g.y, g.z, g.w};
  if (th2 < 1e-8f) {
    // w = 1 - th^2/8, v = (1/2 - th^2/48) r to second order
    const float dot = r[0] * gv[0] + r[1] * gv[1] + r[2] * gv[2];
    for (int i = 0; i < 3; ++i)
      out[i] = -0.25f * r[i] * g.x + (0.5f - th2 * (1.f / 48.f)) * gv[i] - (1.f / 24.f) * r[i] * dot;
    return;
  }
  const float th = sqrtf(th2);
  float sn, cs;
  sincosf(0.5f * th, &sn, &cs);
  const float s = sn / th;
  const float ds = (0.5f * cs * th - sn) / th2;   // d s / d th
  const float dot = r[0] * gv[0] + r[1] * gv[1] + r[2] * gv[2];
  for (int i = 0; i < 3; ++i)
    out[i] = -0.5f * s * r[i] * g.x + s * gv[i] + r[i] * (ds / th) * dot;
}

struct OdeArgs {
  const float* params;
  const float* embed;
  int D, n_inst, n_times, substeps;
  const float* times;
  const float* z0;          // forward
  float* states;            // [(n_times - 1) * substeps + 1][n_inst][6]
  float* quat;              // [n_times][n_inst][4]
  float* trans;             // [n_times][n_inst][3]
  const float* g_quat;      // backward
  const float* g_trans;
  float* g_params;
  float* g_embed;
  float* g_z0;
};

// One group per instance. The poses come from the stored states once the chain
// is done, all output times in parallel, so that no sine or cosine sits in it.
__global__ void __launch_bounds__(kGroup) k_ode_fwd(OdeArgs a) {
  __shared__ __align__(16) float s_h1[kH], s_h2[kH];
  const OdeLayout L = ode_layout(a.D);
  const int u = threadIdx.x, k = blockIdx.x, K = a.n_inst;
  EvalWeights w;
  load_eval_weights(w, a.params, L, a.embed + (size_t)k * a.D, u);
  float z[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) z[i] = a.z0[6 * (size_t)k + i];
  if (u < 6) a.states[6 * (size_t)k + u] = a.z0[6 * (size_t)k + u];
  float* dst = a.states + 6 * ((size_t)K + k);
  float t0 = a.times[0];
  for (int j = 0; j + 1 < a.n_times; ++j) {
    const float t1 = a.times[j + 1];
    const float h = (t1 - t0) / (float)a.substeps;
    for (int s = 0; s < a.substeps; ++s) {
      const float t = t0 + (float)s * h;
      float k1[6], k2[6], k3[6], k4[6], v[6];
      eval_f(w, z, t, u, 1, s_h1, s_h2, k1);
#pragma unroll
      for (int i = 0; i < 6; ++i) v[i] = fmaf(0.5f * h, k1[i], z[i]);
      eval_f(w, v, t + 0.5f * h, u, 1, s_h1, s_h2, k2);
#pragma unroll
      for (int i = 0; i < 6; ++i) v[i] = fmaf(0.5f * h, k2[i], z[i]);
      eval_f(w, v, t + 0.5f * h, u, 1, s_h1, s_h2, k3);
#pragma unroll
      for (int i = 0; i < 6; ++i) v[i] = fmaf(h, k3[i], z[i]);
      eval_f(w, v, t + h, u, 1, s_h1, s_h2, k4);
      float mine = 0.f;
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        z[i] = fmaf(h * (1.f / 6.f), k1[i] + 2.f * k2[i] + 2.f * k3[i] + k4[i], z[i]);
        mine = u == i ? z[i] : mine;
      }
      if (u < 6) dst[u] = mine;
      dst += 6 * (size_t)K;
    }
    t0 = t1;
  }
  __syncthreads();   // the states of this instance are written
  for (int j = u; j < a.n_times; j += kGroup) {
    const float* zs = a.states + 6 * ((size_t)j * a.substeps * K + k);
    const size_t row = (size_t)j * K + k;
    *reinterpret_cast<float4*>(a.quat + 4 * row) = quat_from_rotvec(zs[3], zs[4], zs[5]);
#pragma unroll
    for (int i = 0; i < 3; ++i) a.trans[3 * row + i] = zs[i];
  }
}

// What the backward's groups hand to each other for one step: the stages'
// inputs, activations and times, the adjoints of their outputs and hidden
// units, and the pose adjoint that enters at the step's end.
struct __align__(16) StepSlot {
  float h1[4][kH], h2[4][kH], p1[4][kH], p2[4][kH];
  float x[4][8];     // z at the stage, then t
  float yb[4][8];    // adjoint of the stage's output
  float inj[8];
  float h;
};
static_assert(sizeof(StepSlot) % 16 == 0, "the slots' vectors are read as float4");
constexpr int kRing = 3, kTickSteps = 2;
constexpr int kBwdThreads = 4 * kGroup + 32;

// The pose adjoints of state index i (an output time iff i is a multiple of the
// substeps), for the state's six components.
__device__ __forceinline__ void pose_adjoint(const OdeArgs& a, int i, int k, float (&g)[6]) {
#pragma unroll
  for (int q = 0; q < 6; ++q) g[q] = 0.f;
  if (i % a.substeps != 0) return;
  const size_t row = (size_t)(i / a.substeps) * a.n_inst + k;
  const float* zs = a.states + 6 * ((size_t)i * a.n_inst + k);
  const float r[3] = {zs[3], zs[4], zs[5]};
  float gr[3];
  quat_from_rotvec_vjp(r, *reinterpret_cast<const float4*>(a.g_quat + 4 * row), gr);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    g[q] = a.g_trans[3 * row + q];
    g[3 + q] = gr[q];
  }
}

// What the recomputation of step i (from state i - 1 to state i) starts from,
// loaded one tick ahead.
struct StepStart {
  float z[6], t0, t1;
  int sub;
};
__device__ __forceinline__ void load_start(const OdeArgs& a, int i, int k, StepStart& s) {
  const int jj = (i - 1) / a.substeps;
  s.sub = (i - 1) - jj * a.substeps;
  const float* zs = a.states + 6 * ((size_t)(i - 1) * a.n_inst + k);
#pragma unroll
  for (int q = 0; q < 6; ++q) s.z[q] = zs[q];
  s.t0 = a.times[jj];
  s.t1 = a.times[jj + 1];
}

// Recomputes a step's stages into its slot.
__device__ __forceinline__ void recompute_step(const EvalWeights& w, int substeps, const StepStart& b, int u,
                                               int bar, StepSlot& s) {
  const float h = (b.t1 - b.t0) / (float)substeps;
  const float t = b.t0 + (float)b.sub * h;
  float v[6], kk[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) v[q] = b.z[q];
#pragma unroll
  for (int st = 0; st < 4; ++st) {
    const float ts = st == 0 ? t : (st == 3 ? t + h : t + 0.5f * h);
    if (u < 8) {
      float mine = ts;
#pragma unroll
      for (int q = 0; q < 6; ++q) mine = u == q ? v[q] : mine;
      s.x[st][u] = mine;
    }
    if (st == 3) {   // the last stage's output feeds nothing
      hidden(w, v, ts, u, bar, s.h1[st], s.h2[st]);
      break;
    }
    eval_f(w, v, ts, u, bar, s.h1[st], s.h2[st], kk);
    const float step = st == 2 ? h : 0.5f * h;
#pragma unroll
    for (int q = 0; q < 6; ++q) v[q] = fmaf(step, kk[q], b.z[q]);
  }
  if (u == 0) s.h = h;
}

// Walks the adjoint `ab` of state i back through step i: per stage the reverse
// of f, hidden layer by hidden layer, with the same exchanges as eval_f.
struct AdjointWeights {
  f2 w2[kH / 2];      // column u of W2
  f2 w1[8];           // its lane's quarter of column lane / 4 of W1 (see six_sums)
  float w3[6];        // column u of W3
};
__device__ __forceinline__ void walk_step(const AdjointWeights& w, int u, int bar, StepSlot& s,
                                          float (&ab)[6]) {
  const uint32_t lane = (uint32_t)u & 31u;
  const float h = s.h;
#pragma unroll
  for (int q = 0; q < 6; ++q) ab[q] += s.inj[q];
  // z' = z + h/6 (k1 + 2 k2 + 2 k3 + k4), stages in reverse
  float zb[6], kb[6], xb[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    zb[q] = ab[q];
    kb[q] = h * (1.f / 6.f) * ab[q];
  }
#pragma unroll
  for (int st = 3; st >= 0; --st) {
    const float h1 = s.h1[st][u], h2 = s.h2[st][u];
    const float ga = fmaf(w.w3[2], kb[2], fmaf(w.w3[1], kb[1], w.w3[0] * kb[0]));
    const float gb = fmaf(w.w3[5], kb[5], fmaf(w.w3[4], kb[4], w.w3[3] * kb[3]));
    s.p2[st][u] = (ga + gb) * (1.f - h2 * h2);
    if (u < 6) {
      float mine = 0.f;
#pragma unroll
      for (int q = 0; q < 6; ++q) mine = u == q ? kb[q] : mine;
      s.yb[st][u] = mine;
    }
    group_sync(bar);
    s.p1[st][u] = dot64(s.p2[st], w.w2) * (1.f - h1 * h1);
    group_sync(bar);
    six_sums(s.p1[st], w.w1, 0.f, lane, xb);
    // the next stage's output adjoint: k_st fed the following stage with the
    // factor `step` and the step's sum with `share`
    const float step = st == 3 ? h : 0.5f * h;
    const float share = st == 1 ? h * (1.f / 6.f) : h * (1.f / 3.f);
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      zb[q] += xb[q];
      kb[q] = fmaf(step, xb[q], share * ab[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < 6; ++q) ab[q] = zb[q];
}

// Row u of every parameter adjoint, summed over the instance's steps. The
// embedding is constant along the trajectory, so its terms need only the sum
// of p1.
struct ParamSums {
  f2 w2[kH / 2];
  float w1[7], w3[6], p1, p2, yb;
};
__device__ __forceinline__ void add_step(ParamSums& g, int u, const StepSlot& s) {
#pragma unroll
  for (int st = 3; st >= 0; --st) {
    const float p1 = s.p1[st][u], p2 = s.p2[st][u], h2 = s.h2[st][u];
    const f2 p22 = pk(p2, p2);
    const float4* h1 = reinterpret_cast<const float4*>(s.h1[st]);
#pragma unroll
    for (int m = 0; m < kH / 4; ++m) {
      const float4 x = h1[m];
      g.w2[2 * m] = fma2(pk(x.x, x.y), p22, g.w2[2 * m]);
      g.w2[2 * m + 1] = fma2(pk(x.z, x.w), p22, g.w2[2 * m + 1]);
    }
#pragma unroll
    for (int i = 0; i < 7; ++i) g.w1[i] = fmaf(p1, s.x[st][i], g.w1[i]);
#pragma unroll
    for (int o = 0; o < 6; ++o) g.w3[o] = fmaf(h2, s.yb[st][o], g.w3[o]);
    g.p1 += p1;
    g.p2 += p2;
    if (u < 6) g.yb += s.yb[st][u];
  }
}

__global__ void __launch_bounds__(kBwdThreads) k_ode_bwd(OdeArgs a) {
  __shared__ __align__(16) StepSlot s_ring[kRing][kTickSteps];
  __shared__ float s_p1[kH];
  const OdeLayout L = ode_layout(a.D);
  const int u = threadIdx.x & (kGroup - 1), role = threadIdx.x / kGroup;   // warp-uniform
  const int k = blockIdx.x;
  const int n_steps = (a.n_times - 1) * a.substeps;
  const int ticks = (n_steps + kTickSteps - 1) / kTickSteps + 2;
  const float* c = a.embed + (size_t)k * a.D;
  const float* p = a.params;
  // tick n: groups 0 and 1 recompute the steps of tick n, the ninth warp takes
  // their pose adjoints, group 2 walks the steps of tick n - 1 and group 3 sums
  // those of tick n - 2. Every group runs the same number of ticks, one CTA
  // barrier each; step s counts from the end.
  if (role < kTickSteps) {
    EvalWeights w;
    load_eval_weights(w, p, L, c, u);
    StepStart now, next;
    if (role < n_steps) load_start(a, n_steps - role, k, next);
    for (int n = 0; n < ticks; ++n) {
      const int s = n * kTickSteps + role;
      now = next;
      if (s + kTickSteps < n_steps) load_start(a, n_steps - s - kTickSteps, k, next);
      if (s < n_steps) recompute_step(w, a.substeps, now, u, 1 + role, s_ring[n % kRing][role]);
      __syncthreads();
    }
  } else if (role == 4) {
    for (int n = 0; n < ticks; ++n) {
      const int s = n * kTickSteps + u;
      if (u < kTickSteps && s < n_steps) {
        float g[6];
        pose_adjoint(a, n_steps - s, k, g);
#pragma unroll
        for (int q = 0; q < 6; ++q) s_ring[n % kRing][u].inj[q] = g[q];
      }
      __syncthreads();
    }
  } else if (role == 2) {
    AdjointWeights w;
#pragma unroll
    for (int m = 0; m < kH / 2; ++m)
      w.w2[m] = pk(p[L.oW2 + (int64_t)(2 * m) * kH + u], p[L.oW2 + (int64_t)(2 * m + 1) * kH + u]);
    const int i = (u & 31) >> 2;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int m = 4 * ((u & 3) + 4 * (q >> 1)) + 2 * (q & 1);
      w.w1[q] = i < 6 ? pk(p[L.oW1 + (int64_t)m * L.I + i], p[L.oW1 + (int64_t)(m + 1) * L.I + i])
                      : pk(0.f, 0.f);
    }
#pragma unroll
    for (int o = 0; o < 6; ++o) w.w3[o] = p[L.oW3 + o * kH + u];
    float ab[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int n = 0; n < ticks; ++n) {
      if (n > 0)
        for (int q = 0; q < kTickSteps; ++q)
          if ((n - 1) * kTickSteps + q < n_steps) walk_step(w, u, 3, s_ring[(n - 1) % kRing][q], ab);
      __syncthreads();
    }
    if (u == 0) {
      float g[6];
      pose_adjoint(a, 0, k, g);
#pragma unroll
      for (int q = 0; q < 6; ++q) a.g_z0[6 * (size_t)k + q] += ab[q] + g[q];
    }
  } else {
    ParamSums g = {};
    for (int n = 0; n < ticks; ++n) {
      if (n > 1)
        for (int q = 0; q < kTickSteps; ++q)
          if ((n - 2) * kTickSteps + q < n_steps) add_step(g, u, s_ring[(n - 2) % kRing][q]);
      __syncthreads();
    }
    float* out = a.g_params;
    float* W1 = out + L.oW1 + (int64_t)u * L.I;
#pragma unroll
    for (int i = 0; i < 7; ++i) atomicAdd(W1 + i, g.w1[i]);
    for (int d = 0; d < a.D; ++d) atomicAdd(W1 + 7 + d, g.p1 * c[d]);
    atomicAdd(out + L.ob1 + u, g.p1);
    atomicAdd(out + L.ob2 + u, g.p2);
#pragma unroll
    for (int m = 0; m < kH / 2; ++m) {
      float x, y;
      upk(g.w2[m], x, y);
      atomicAdd(out + L.oW2 + (int64_t)u * kH + 2 * m, x);
      atomicAdd(out + L.oW2 + (int64_t)u * kH + 2 * m + 1, y);
    }
#pragma unroll
    for (int o = 0; o < 6; ++o) atomicAdd(out + L.oW3 + o * kH + u, g.w3[o]);
    if (u < 6) atomicAdd(out + L.ob3 + u, g.yb);
    // dL/dc = W1[:, 7:]^T sum p1
    s_p1[u] = g.p1;
    group_sync(4);
    if (u < a.D) {
      float v = 0.f;
      for (int m = 0; m < kH; ++m) v = fmaf(p[L.oW1 + (int64_t)m * L.I + 7 + u], s_p1[m], v);
      a.g_embed[(size_t)k * a.D + u] += v;
    }
  }
}

}  // namespace

int64_t ode_param_count(int embed_dim) { return ode_layout(embed_dim).count; }

cudaError_t launch_ode_fwd(const s3r_ode_net* net, int n_inst, const float* z0, const float* times,
                           int n_times, int substeps, float* states, float* quat, float* trans,
                           cudaStream_t st) {
  OdeArgs a = {};
  a.params = net->params;
  a.embed = net->embed;
  a.D = net->embed_dim;
  a.n_inst = n_inst;
  a.n_times = n_times;
  a.substeps = substeps;
  a.times = times;
  a.z0 = z0;
  a.states = states;
  a.quat = quat;
  a.trans = trans;
  k_ode_fwd<<<n_inst, kGroup, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_ode_bwd(const s3r_ode_net* net, int n_inst, const float* times, int n_times,
                           int substeps, const float* states, const float* g_quat,
                           const float* g_trans, float* g_params, float* g_embed, float* g_z0,
                           cudaStream_t st) {
  OdeArgs a = {};
  a.params = net->params;
  a.embed = net->embed;
  a.D = net->embed_dim;
  a.n_inst = n_inst;
  a.n_times = n_times;
  a.substeps = substeps;
  a.times = times;
  a.states = const_cast<float*>(states);
  a.g_quat = g_quat;
  a.g_trans = g_trans;
  a.g_params = g_params;
  a.g_embed = g_embed;
  a.g_z0 = g_z0;
  k_ode_bwd<<<n_inst, kBwdThreads, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace s3r
