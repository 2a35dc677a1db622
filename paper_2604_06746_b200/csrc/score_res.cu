// Host side of the resident scorer (score_res.cuh): which calls take it, and how a sequence is shared out.
#include "score_res.cuh"

#include <algorithm>
#include <cmath>

namespace skv {
namespace {

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
// Shorter sequences stay with the general scorer: however short, a team takes 2.6 us for a unit among many and has its way
// through the exchange in one by itself, and as many units follow one another as a team has KV groups.  us per layer,
// general / this one, one layer | one of 32: one KV head 4096 keys 14.7 / 17.7 | 1.8 / 2.6, 9001 keys 15.0 / 18.6 | 2.4 / 2.6,
// 16000 keys 17.1 / 18.5 | 2.9 / 2.6, 20000 keys 19.3 / 18.5 | 3.4 / 3.0; two 4096 keys 15.8 / 18.5 | 2.0 / 2.6, 7500
// keys 17.4 / 18.5 | 2.7 / 2.6, 9001 keys 18.6 / 18.5 | 3.2 / 2.7; four 4096 keys 18.5 / 18.5 | 2.9 / 2.7; eight 2500
// keys 21.4 / 18.9 | 3.2 / 3.5, 4096 keys 21.3 / 20.3 | 4.5 / 3.4.
constexpr int kResFrom = 4096, kResKeys = 16384;           // keys; keys of all KV heads

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
    pb.q = (const __nv_bfloat16*)a.q[first + i];
    pb.k = (const __nv_bfloat16*)a.k[first + i];
    pb.n_keys = a.n_keys;
    pb.cols = a.cols + (size_t)(first + i) * a.cols_layer_stride;
    const float c2 = a.scale[first + i] * kLog2e;
    pb.negate = c2 < 0.f;
    pb.c2 = std::max(std::fabs(c2), 1e-30f);
  }
  p.n_prob = n;
  p.k_stride_head = a.k_stride_head;
  p.k_stride_token = a.k_stride_token;
  p.n_kv = cfg.n_kv_heads;
  p.team = plan.team;
  p.teams = std::min(plan.teams, n * cfg.n_kv_heads);
  p.window = cfg.window;
  p.group = cfg.n_q_heads / cfg.n_kv_heads;
  p.rows_pg = p.group * ctx.w_pad;
  p.w_pad = ctx.w_pad;
  p.ctl = ctx.ws.ctl;
  p.xch = ctx.ws.xch;
  p.sums = plan.team > kDirectTeam ? reinterpret_cast<unsigned long long*>(a.part) : nullptr;
  p.row_ent = a.row_ent + (size_t)first * ctx.rows_pad;
  p.col_stride = a.col_stride;
  p.status = ctx.ws.status;
  return cfg.head_dim == 128 ? res_launch_128(p, ctx.device, st) : res_launch_64(p, ctx.device, st);
}

}  // namespace

bool res_supported(const Ctx& ctx, const ScoreCall& a) {
  return !a.cu_seqlens && a.n_keys >= kResFrom && (long long)a.n_keys * ctx.cfg.n_kv_heads >= kResKeys &&
         ctx.cfg.n_q_heads / ctx.cfg.n_kv_heads * ctx.w_pad <= kResRows && plan_of(a.n_keys, ctx.cfg.n_kv_heads, std::min(ctx.sm_count, kMaxSms)).team > 0;
}

cudaError_t launch_score_res(const Ctx& ctx, const ScoreCall& a, int first, int n, cudaStream_t st) {
  return n == 1 ? launch_problems<1>(ctx, a, first, n, st) : launch_problems<kMaxBatch>(ctx, a, first, n, st);
}

}  // namespace skv
