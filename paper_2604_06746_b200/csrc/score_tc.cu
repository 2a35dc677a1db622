// Host side of the tensor-core scorer (score_tc.cuh): tensor maps, how a call's work is cut into
// tasks and in which order they are drawn.
#include "score_short.cuh"

#include <algorithm>
#include <cmath>

namespace skv {
namespace {

struct TcState {
  PFN_cuTensorMapEncodeTiled_v12000 encode;
};

// Self-test of the bounded wait: one thread waits, with the scorer's own helper, on a barrier
// that nothing will ever arrive on.  No copy, MMA or tensor-memory allocation is involved, so
// when the bound expires the kernel simply records STRUCTKV_ERR_TIMEOUT and returns.
__global__ void wait_expiry_probe(unsigned long long limit_cycles, int* status) {
  __shared__ __align__(8) unsigned long long bar;
  __shared__ int abort_word;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    abort_word = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (!mbar_wait(smem_u32(&bar), 0, &abort_word, limit_cycles))
      atomicCAS(status, 0, (int)STRUCTKV_ERR_TIMEOUT);
  }
}

// How a configuration's score rows are laid out and weighted.
struct Layout {
  int group, rows_pg, n_rb, units, shape, unit_rows, w_last, w_group, w_total;
};
Layout layout_of(const structkv_config& cfg) {
  Layout l;
  const int w_pad = tc_window_pad(cfg.window);
  l.group = cfg.n_q_heads / cfg.n_kv_heads;
  l.rows_pg = l.group * w_pad;
  if (l.rows_pg <= 64) {
    // up to 64 rows the wide layout would leave at least half of the lanes to padding
    l.unit_rows = l.rows_pg <= 32 ? 32 : 64;
    l.shape = l.rows_pg <= 32 ? kNarrow32 : kNarrow64;
  } else {
    l.unit_rows = kRowBlock;
    l.shape = w_pad <= 16 ? kWide16 : w_pad == 32 ? kWide32 : w_pad == 64 ? kWide64 : w_pad == 128 ? kWide128 : kWide256;
  }
  l.n_rb = (l.rows_pg + l.unit_rows - 1) / l.unit_rows;
  l.units = cfg.n_kv_heads * l.n_rb;
  // equal units need no weights
  l.w_last = l.n_rb > 1 && l.rows_pg - (l.n_rb - 1) * kRowBlock <= 128 ? 13 : kFullWeight;
  l.w_group = (l.n_rb - 1) * kFullWeight + l.w_last;
  l.w_total = cfg.n_kv_heads * l.w_group;
  return l;
}
// Tasks of one pass: about `target`, at least one for every unit, and no more than one per item of a
// unit.
int clamp_tasks(const Layout& l, int target, int items) {
  const int lo = (l.w_total + l.w_last - 1) / l.w_last;
  const int hi = std::max(lo, (int)std::min(60000ll, (long long)items * l.w_total / kFullWeight));
  return std::min(std::max(target, lo), hi);
}

// Key segments of pass 1 for a sequence that is due `share` of the SMs: at least two pairs of tiles each, unless
// all of them run at once anyway.
int segments(const Layout& l, int share, int tiles, int sms) {
  const int pairs = (tiles + 1) / 2;
  return clamp_tasks(l, share, (long long)l.units * pairs <= sms ? pairs : (pairs + 1) / 2);
}
int batch_share(const ScoreCall& a, int i, int sms) {
  return std::max(1, (int)((long long)sms * (a.cu_seqlens[i + 1] - a.cu_seqlens[i]) / a.cu_seqlens[a.n]));
}
// How finely a batch's pass 1 is cut: one segment per SM in all (1), or two (2).  A sequence's segments are whole
// numbers per unit, so with one per SM the longest can be far above the average (40000 + 20000 + 50000
// + 21072 keys: 39.5 pairs of tiles against 27.8); with two the SMs even out, for one more hand-over
// (worth a pair) and part of a segment at the end.  Measured with one / two, us: those four 205 / 181, six
// of 1001 to 12000 keys 84 / 79; but 50000 + 1000 94 / 98 and 30001 + 1500 65 / 71.
int batch_cut(const Layout& l, const ScoreCall& a, int sms) {
  if (a.n == 1) return 1;                                  // the bits of the plain call
  float longest[2] = {0.f, 0.f}, all = 0.f;
  for (int i = 0; i < a.n; ++i) {
    const int tiles = (a.cu_seqlens[i + 1] - a.cu_seqlens[i] + kKeyTile - 1) / kKeyTile, pairs = (tiles + 1) / 2;
    for (int c = 0; c < 2; ++c) {
      const int per_unit = std::max(1, segments(l, (c + 1) * batch_share(a, i, sms), tiles, sms) * kFullWeight / l.w_total);
      longest[c] = std::max(longest[c], (float)((pairs + per_unit - 1) / per_unit));
    }
    all += (float)pairs * l.w_total / kFullWeight / sms;
  }
  return longest[0] <= all + 0.25f * longest[1] + 1.f ? 1 : 2;
}

// The form for one layer whose segments all run at once, two pairs of tiles each at most (score_short.cuh).  False: not this call.
bool launch_short(const Ctx& ctx, const ScoreCall& a, int first, cudaStream_t st, cudaError_t* e) {
  const structkv_config& cfg = ctx.cfg;
  const Layout l = layout_of(cfg);
  const int sms = std::min(ctx.sm_count, kMaxSms);
  const int n_keys = a.cu_seqlens ? a.cu_seqlens[1] : a.n_keys;
  const int tiles = (n_keys + kKeyTile - 1) / kKeyTile, pairs = (tiles + 1) / 2, s1 = segments(l, sms, tiles, sms);
  // (units of equal weight have equally many segments; the exchange words of a context of one call hold anything)
  if (l.shape >= kNarrow32 || l.w_last != kFullWeight || s1 % l.units != 0 || s1 > sms || ctx.old_words) return false;
  ShortParams p;
  p.n_seg = s1 / l.units;
  if (2 * ((pairs + p.n_seg - 1) / p.n_seg) > kShortTiles) return false;
  p.n_pairs = pairs;
  p.split = p.n_seg == pairs && 2 * s1 <= sms && l.rows_pg - (l.n_rb - 1) * kRowBlock > kRowBlock / 2;
  p.n_tasks = s1 << p.split;
  const cuuint64_t row = (cuuint64_t)cfg.head_dim * 2, s_tok = (cuuint64_t)a.k_stride_token * 2;
  const cuuint64_t s_head = cfg.n_kv_heads == 1 ? s_tok * (cuuint64_t)n_keys : (cuuint64_t)a.k_stride_head * 2;
  *e = cudaErrorInvalidValue;
  if (!tc_encode3(ctx, &p.map_q, a.q[first], cfg.window, (cuuint64_t)cfg.n_q_heads, row, row * cfg.window,
                  std::min(ctx.w_pad, kRowBlock / 2), std::max(1, kRowBlock / 2 / ctx.w_pad)) ||
      !tc_encode3(ctx, &p.map_k, a.k[first], n_keys, cfg.n_kv_heads, s_tok, s_head, kKeyTile, 1))
    return true;
  p.cols = a.cols + (size_t)first * a.cols_layer_stride;
  p.row_ent = a.row_ent + (size_t)first * ctx.rows_pad;
  p.xch = ctx.ws.xch;
  p.ctl = ctx.ws.ctl;
  p.status = ctx.ws.status;
  p.col_stride = a.col_stride;
  const float c2 = a.scale[first] * kLog2e;
  p.negate = c2 < 0.f;
  p.c2 = std::max(std::fabs(c2), 1e-30f);
  p.inv_c2 = 1.f / p.c2;
  p.v_min = -125.f / p.c2;
  p.n_keys = n_keys;
  p.window = cfg.window;
  p.w_pad = ctx.w_pad;
  p.w_shift = 0;
  while ((1 << p.w_shift) < ctx.w_pad) ++p.w_shift;
  p.group = l.group;
  p.rows_pg = l.rows_pg;
  p.n_rb = l.n_rb;
  const int grid = ctx.short_ctas > 0 ? std::min(ctx.short_ctas, p.n_tasks) : p.n_tasks;
  *e = cfg.head_dim == 128 ? short_launch_128(l.shape, p, grid, ctx.device, st) : short_launch_64(l.shape, p, grid, ctx.device, st);
  return true;
}

template <int MAXP>
cudaError_t launch_problems(const Ctx& ctx, const ScoreCall& a, int first, int n, cudaStream_t st) {
  TcParams<MAXP> p;
  const structkv_config& cfg = ctx.cfg;
  const Layout l = layout_of(cfg);
  const bool batch = a.cu_seqlens != nullptr;
  const int sms = std::min(ctx.sm_count, kMaxSms);
  const int total_keys = batch ? a.cu_seqlens[n] : a.n_keys;
  const int box_rows = l.unit_rows == kRowBlock ? kRowBlock / 2 : l.unit_rows;    // Q is loaded in halves of a wide block
  const cuuint64_t row = (cuuint64_t)cfg.head_dim * 2;
  const int n_maps = batch ? 1 : n;
  for (int i = 0; i < n_maps; ++i) {
    if (!tc_encode3(ctx, &p.map_q[i], a.q[first + i], cfg.window, (cuuint64_t)cfg.n_q_heads * (batch ? n : 1), row,
                 row * cfg.window, std::min(ctx.w_pad, box_rows), std::max(1, box_rows / ctx.w_pad)))
      return cudaErrorInvalidValue;
    const cuuint64_t s_tok = (cuuint64_t)a.k_stride_token * 2;
    const cuuint64_t s_head = cfg.n_kv_heads == 1 ? s_tok * (cuuint64_t)total_keys : (cuuint64_t)a.k_stride_head * 2;
    if (!tc_encode3(ctx, &p.map_k[i], a.k[first + i], total_keys, cfg.n_kv_heads, s_tok, s_head, kKeyTile, 1))
      return cudaErrorInvalidValue;
  }
  const int cut = batch ? batch_cut(l, a, sms) : 1;
  int part0 = 0;
  for (int i = 0; i < n; ++i) {
    TcProblem& pb = p.prob[i];
    pb.key0 = batch ? a.cu_seqlens[i] : 0;
    pb.n_keys = batch ? a.cu_seqlens[i + 1] - pb.key0 : a.n_keys;
    pb.map = batch ? 0 : i;
    pb.head0 = batch ? i * cfg.n_q_heads : 0;
    pb.cols = a.cols + (batch ? (size_t)pb.key0 : (size_t)(first + i) * a.cols_layer_stride);
    const float c2 = (batch ? a.scale[0] : a.scale[first + i]) * kLog2e;
    pb.negate = c2 < 0.f;
    pb.c2 = std::max(std::fabs(c2), 1e-30f);
    pb.inv_c2 = 1.f / pb.c2;
    pb.v_min = -125.f / pb.c2;
    const int tiles = (pb.n_keys + kKeyTile - 1) / kKeyTile;
    // Pass 1 leaves one partial per key segment: as many segments as SMs, or twice as many, shared out over the
    // sequences of a batch by their lengths.  That depends on the shape alone, so that a layer gives the same
    // bits by itself and among others.
    const int share = batch ? batch_share(a, i, sms) : sms;
    const int pairs = (tiles + 1) / 2;
    pb.s1 = segments(l, cut * share, tiles, sms);
    // A task by itself runs one segment; with other layers to fill the SMs it runs as many as make five pairs:
    // the way from task to task costs as much as one (32 layers of 5003 keys: 302 us with two pairs a
    // task, 253 with four or more).  The same in pass 2, which leaves no partial results.
    const bool alone = batch || n == 1;
    const long long work = (long long)l.units * pairs;
    const int run = alone ? 1 : (int)std::max(1ll, (10ll * pb.s1 + work) / (2 * work));
    pb.t1 = run == 1 ? pb.s1 : clamp_tasks(l, pb.s1 / run, pb.s1);
    // The pass nothing follows is cut finer: its tasks end closer together.
    // (Not below eight tiles a task, each of which merges its unit's statistics first.)
    const bool last = batch || i == n - 1;
    if (!last) pb.t2 = clamp_tasks(l, share, run > 1 ? (tiles + 9) / 10 : (tiles + 3) / 4);
    else pb.t2 = clamp_tasks(l, (long long)l.units * tiles >= 16ll * share ? 2 * share : share, tiles);
    pb.part0 = part0;
    part0 += pb.s1;
  }
  // ticket order
  int n_ph = 0, tickets = 0;
  auto phase = [&](int i, int pass) {
    p.phase[n_ph++] = TcPhase{tickets, (unsigned char)i, (unsigned char)pass};
    tickets += pass == 1 ? p.prob[i].t1 : p.prob[i].t2;
  };
  if (batch) {
    for (int pass = 1; pass <= 2; ++pass)
      for (int i = 0; i < n; ++i) phase(i, pass);
  } else {
    // Pass 1 runs `ahead` layers in front of pass 2, far enough to cover the way from a unit's last
    // pass-1 task to its merged statistics (10 to 15 us) with other work: one layer where a layer's
    // pass 1 is at least twelve pairs of key tiles (1.2 us each) per SM, more for shorter sequences.
    const long long pairs = (long long)l.units * ((p.prob[0].n_keys + 2 * kKeyTile - 1) / (2 * kKeyTile));
    const int ahead = (int)std::min<long long>(std::min(n - 1, 20), std::max(1ll, (12ll * sms + pairs - 1) / pairs));
    for (int i = 0; i < n + ahead; ++i) {
      if (i < n) phase(i, 1);
      if (i >= ahead) phase(i - ahead, 2);
    }
  }
  p.phase[n_ph] = TcPhase{tickets, 0, 0};
  p.n_phase = n_ph;
  p.n_prob = n;
  p.window = cfg.window;
  p.w_pad = ctx.w_pad;
  p.w_shift = 0;
  while ((1 << p.w_shift) < ctx.w_pad) ++p.w_shift;
  p.group = l.group;
  p.rows_pg = l.rows_pg;
  p.n_rb = l.n_rb;
  p.n_units = l.units;
  p.w_group = l.w_group;
  p.w_total = l.w_total;
  p.w_last = l.w_last;
  p.ctl = ctx.ws.ctl;
  p.part = a.part;
  p.nlse = a.nlse;
  p.row_ent = a.row_ent + (size_t)first * ctx.rows_pad;
  p.col_stride = a.col_stride;
  p.status = ctx.ws.status;
  const long long pairs0 = (long long)l.units * ((p.prob[0].n_keys + 2 * kKeyTile - 1) / (2 * kKeyTile));
  p.form = n == 1 || batch ? kHurry : pairs0 <= kBriefPairs ? kBrief : kAmong;
  const int grid = std::min(sms, tickets);
  return cfg.head_dim == 128 ? tc_launch_128(l.shape, p, grid, ctx.device, st) : tc_launch_64(l.shape, p, grid, ctx.device, st);
}

}  // namespace

cudaError_t launch_wait_probe(unsigned long long limit_cycles, int* status, cudaStream_t st) {
  wait_expiry_probe<<<1, 32, 0, st>>>(limit_cycles, status);
  return cudaGetLastError();
}

bool tc_encode3(const Ctx& ctx, CUtensorMap* m, const void* base, cuuint64_t d1, cuuint64_t d2, cuuint64_t s1,
                cuuint64_t s2, cuuint32_t b1, cuuint32_t b2) {
  const cuuint64_t dims[3] = {(cuuint64_t)ctx.cfg.head_dim, d1, d2};
  const cuuint64_t strides[2] = {s1, s2};
  const cuuint32_t box[3] = {64, b1, b2}, estr[3] = {1, 1, 1};
  return ((TcState*)ctx.tc)->encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
                                    estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int tc_window_pad(int window) {
  int w = 8;
  while (w < window) w *= 2;
  return w;
}

size_t tc_part_tasks(const structkv_config& cfg, int n, bool batch) {
  const size_t units = (size_t)layout_of(cfg).units;
  const size_t m = (size_t)std::min(n, kMaxBatch);
  return batch ? 2 * kMaxSms + 2 * units * m : (kMaxSms + 2 * units) * m;
}

bool tc_supported(const Ctx& ctx, long long k_stride_head, long long k_stride_token) {
  if (!ctx.tc || ctx.cfg.dtype != STRUCTKV_BF16) return false;
  if (ctx.cfg.head_dim != 64 && ctx.cfg.head_dim != 128) return false;
  // tensor-map limits: strides below 2^40 bytes, multiples of 16 bytes (checked by the caller)
  if (k_stride_token * 2 >= (1ll << 40) || k_stride_head * 2 >= (1ll << 40)) return false;
  if (ctx.cfg.n_kv_heads > 1 && k_stride_head == 0) return false;
  return layout_of(ctx.cfg).units <= kQueueUnits;
}

structkv_status tc_create(Ctx& ctx) {
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess ||
      qres != cudaDriverEntryPointSuccess || !fn)
    return STRUCTKV_ERR_CUDA;
  TcState* s = new TcState();
  s->encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
  ctx.tc = s;
  return STRUCTKV_OK;
}

void tc_destroy(Ctx& ctx) {
  delete (TcState*)ctx.tc;
  ctx.tc = nullptr;
}

cudaError_t launch_score_tc(const Ctx& ctx, const ScoreCall& a, cudaStream_t st) {
  if (res_supported(ctx, a)) {
    cudaError_t e = clean_words(ctx, st);
    for (int l = 0; l < a.n && e == cudaSuccess; l += kMaxBatch) e = launch_score_res(ctx, a, l, std::min(kMaxBatch, a.n - l), st);
    // where the device does not give this process all of its SMs at once, the general scorer does it
    if (e != cudaErrorCooperativeLaunchTooLarge) return e;
    cudaGetLastError();
  }
  cudaError_t e = cudaSuccess;
  if (a.n == 1 && launch_short(ctx, a, 0, st, &e)) return e;
  if (a.cu_seqlens) return a.n == 1 ? launch_problems<1>(ctx, a, 0, 1, st) : launch_problems<kMaxBatch>(ctx, a, 0, a.n, st);
  for (int l = 0; l < a.n; l += kMaxBatch) {
    const int n = std::min(kMaxBatch, a.n - l);
    e = n == 1 ? launch_problems<1>(ctx, a, l, 1, st) : launch_problems<kMaxBatch>(ctx, a, l, n, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace skv
