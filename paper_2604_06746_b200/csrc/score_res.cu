// Host side of the resident scorer (score_res.cuh): which calls take it, and how a sequence is shared out.
#include "score_res.cuh"

#include <algorithm>
#include <cmath>

namespace skv {
namespace {

// Common references of a launch's rows (their largest logit over kRefKeys keys that all of them see), and clean summed
// words.  One CTA per unit, a thread per row.
struct RefArgs {
  struct { const __nv_bfloat16 *q, *k; int n_keys; float c2; } prob[kMaxBatch];   // c2 with the scale's sign
  long long k_stride_head, k_stride_token;
  int n_kv, group, window, w_pad;
  unsigned long long* sums;
  float* refs;
};
template <int D>
__global__ void __launch_bounds__(kResRows) res_refs(const __grid_constant__ RefArgs a) {
  __shared__ alignas(16) float ks[kRefKeys][D];
  const int unit = blockIdx.x, pi = unit / a.n_kv, g = unit - pi * a.n_kv;
  const int row = threadIdx.x, head = row / a.w_pad, i = row - head * a.w_pad;
  pdl_trigger();
  pdl_wait();
  const auto& pb = a.prob[pi];
  const int open = pb.n_keys - a.window;                   // the last key every window row sees
  for (int e = threadIdx.x; e < kRefKeys * D; e += kResRows) {
    const int s = e / D, j = s < kRefKeys / 2 ? min(s, open) : max(0, open - (s - kRefKeys / 2));
    ks[s][e % D] = __bfloat162float(pb.k[g * a.k_stride_head + j * a.k_stride_token + e % D]);
  }
  __syncthreads();
  float ref = 0.f;
  if (head < a.group && i < a.window) {
    const uint4* q = reinterpret_cast<const uint4*>(pb.q + ((size_t)(g * a.group + head) * a.window + i) * D);
    float dot[kRefKeys] = {};
#pragma unroll 4
    for (int c = 0; c < D / 8; ++c) {
      const uint4 v = q[c];
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int s = 0; s < kRefKeys; ++s)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 k4 = *reinterpret_cast<const float4*>(&ks[s][c * 8 + 4 * h]);
          dot[s] = fmaf(__uint_as_float(w[2 * h] << 16), k4.x, dot[s]);
          dot[s] = fmaf(__uint_as_float(w[2 * h] & 0xffff0000u), k4.y, dot[s]);
          dot[s] = fmaf(__uint_as_float(w[2 * h + 1] << 16), k4.z, dot[s]);
          dot[s] = fmaf(__uint_as_float(w[2 * h + 1] & 0xffff0000u), k4.w, dot[s]);
        }
    }
    ref = -INFINITY;
#pragma unroll
    for (int s = 0; s < kRefKeys; ++s) ref = fmaxf(ref, dot[s] * pb.c2);
    if (!(fabsf(ref) < 3.0e38f)) ref = 0.f;
  }
  a.refs[(size_t)unit * kResRows + row] = ref;
  reinterpret_cast<ulonglong2*>(a.sums)[(size_t)unit * kResRows + row] = make_ulonglong2(0, 0);
}

struct Plan { int teams, team; };             // team = 0: does not fit

// How `sms` CTAs form teams for the KV groups of a sequence.  A function of the shape alone, so that a layer gives the
// same bits by itself and among others.  As many teams as KV groups, so that one layer runs at once, while a CTA's
// share takes up to half of its tensor memory (two units in flight); else half as many, twice as large.
Plan plan_of(int n_keys, int n_kv, int sms) {
  const int chunks = (n_keys + kResChunk - 1) / kResChunk;
  constexpr int kSlots = ResSmem<128, 1>::kSlots;
  Plan best{0, 0};
  for (int teams = std::min(n_kv, sms); teams >= 1; teams /= 2) {
    const int team = std::min(sms / teams, chunks), tiles = ((chunks + team - 1) / team + 3) / 4;
    if (tiles > kSlots) continue;
    best = Plan{teams, team};
    if (tiles <= kSlots / 2) break;
  }
  return best;
}
// Shorter sequences stay with the general scorer, which has less to do per unit (see score_res.cuh).
constexpr int kResFrom = 4096;

template <int MAXP>
cudaError_t launch_problems(const Ctx& ctx, const ScoreCall& a, int first, int n, cudaStream_t st) {
  ResParams<MAXP> p;
  const structkv_config& cfg = ctx.cfg;
  const int sms = std::min(ctx.sm_count, kMaxSms);
  const Plan plan = plan_of(a.n_keys, cfg.n_kv_heads, sms);
  const cuuint64_t row = (cuuint64_t)cfg.head_dim * 2;
  for (int i = 0; i < n; ++i) {
    const cuuint64_t s_tok = (cuuint64_t)a.k_stride_token * 2;
    const cuuint64_t s_head = cfg.n_kv_heads == 1 ? s_tok * (cuuint64_t)a.n_keys : (cuuint64_t)a.k_stride_head * 2;
    if (!tc_encode3(ctx, &p.map_q[i], a.q[first + i], cfg.window, (cuuint64_t)cfg.n_q_heads, row, row * cfg.window, ctx.w_pad,
                    kResRows / ctx.w_pad) ||
        !tc_encode3(ctx, &p.map_k[i], a.k[first + i], a.n_keys, cfg.n_kv_heads, s_tok, s_head, kResChunk, 1))
      return cudaErrorInvalidValue;
    ResProblem& pb = p.prob[i];
    pb.n_keys = a.n_keys;
    pb.cols = a.cols + (size_t)(first + i) * a.cols_layer_stride;
    const float c2 = a.scale[first + i] * kLog2e;
    pb.negate = c2 < 0.f;
    pb.c2 = std::max(std::fabs(c2), 1e-30f);
  }
  p.n_prob = n;
  p.n_kv = cfg.n_kv_heads;
  p.team = plan.team;
  p.teams = std::min(plan.teams, n * cfg.n_kv_heads);
  p.window = cfg.window;
  p.group = cfg.n_q_heads / cfg.n_kv_heads;
  p.rows_pg = p.group * ctx.w_pad;
  p.w_pad = ctx.w_pad;
  p.ctl = ctx.ws.ctl;
  p.xch = ctx.ws.xch;
  p.sums = nullptr;
  p.refs = nullptr;
  if (plan.team > kDirectTeam) {
    const int units = n * cfg.n_kv_heads;
    p.sums = reinterpret_cast<unsigned long long*>(a.part);
    p.refs = reinterpret_cast<const float*>(p.sums + 2 * (size_t)units * kResRows);
    RefArgs r = {};
    for (int i = 0; i < n; ++i)
      r.prob[i] = {(const __nv_bfloat16*)a.q[first + i], (const __nv_bfloat16*)a.k[first + i], a.n_keys,
                   p.prob[i].negate ? -p.prob[i].c2 : p.prob[i].c2};
    r.k_stride_head = a.k_stride_head;
    r.k_stride_token = a.k_stride_token;
    r.n_kv = cfg.n_kv_heads; r.group = p.group; r.window = cfg.window; r.w_pad = ctx.w_pad;
    r.sums = p.sums;
    r.refs = const_cast<float*>(p.refs);
    const cudaError_t e = cfg.head_dim == 128 ? launch_pdl(res_refs<128>, dim3(units), dim3(kResRows), 0, st, r)
                                              : launch_pdl(res_refs<64>, dim3(units), dim3(kResRows), 0, st, r);
    if (e != cudaSuccess) return e;
  }
  p.row_ent = a.row_ent + (size_t)first * ctx.rows_pad;
  p.col_stride = a.col_stride;
  p.status = ctx.ws.status;
  return cfg.head_dim == 128 ? res_launch_128(p, ctx.device, st) : res_launch_64(p, ctx.device, st);
}

}  // namespace

bool res_supported(const Ctx& ctx, const ScoreCall& a) {
  return !a.cu_seqlens && a.n_keys >= kResFrom && ctx.cfg.n_q_heads / ctx.cfg.n_kv_heads * ctx.w_pad <= kResRows &&
         plan_of(a.n_keys, ctx.cfg.n_kv_heads, std::min(ctx.sm_count, kMaxSms)).team > 0;
}

cudaError_t launch_score_res(const Ctx& ctx, const ScoreCall& a, int first, int n, cudaStream_t st) {
  return n == 1 ? launch_problems<1>(ctx, a, first, n, st) : launch_problems<kMaxBatch>(ctx, a, first, n, st);
}

}  // namespace skv
