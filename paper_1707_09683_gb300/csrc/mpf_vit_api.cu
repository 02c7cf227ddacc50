// mpf_vit_api.cu -- host side of the P7Viterbi calls of the C ABI
// (mpf_vit_profile_create / _destroy, mpf_viterbi_scan, mpf_viterbi_rescore):
// profile tables, launch grouping and the MSV -> Viterbi hand-off.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <new>
#include <tuple>
#include <utility>
#include <vector>

#include "../../include/mpf.h"
#include "mpf_handles.h"
#include "mpf_internal.h"

using namespace mpf;
using namespace mpf::host;

struct mpf_vprofile {
  mpf_ctx *ctx = nullptr;
  int M = 0, K = 0, Mpad = 0;
  bool fast = false;            // every transition and special score <= 0
  bool packed = false;          // the packed kernel may score it, in these shapes (warps 0: none)
  VitPackShape pack_solo, pack_team;
  int pk_emax = 0, pk_bm = 0, pk_rebase = 0;
  uint32_t pk_split = 0;
  const uint32_t *d_solo = nullptr, *d_team = nullptr;   // its tables, in d_msc's allocation
  int16_t *d_msc = nullptr;     // kVitRows x Mpad, striped; the one allocation of all tables
  int16_t *d_trans = nullptr;   // Mpad x kVitTrans, striped (in the same allocation)
  int sp[kVitSpecial] = {};
  int base = 0;
  float scale = 1.f;
};

namespace {

enum VitMove { VT_BM, VT_MM, VT_IM, VT_DM, VT_MI, VT_II, VT_MD, VT_DD };   // rows of `trans`

// Moves out of or into states that do not exist (node 0, D_1, I_M): in the
// packed kernel their source holds the floor, or nothing reads their target.
bool vit_move_unused(int t, int k, int M) {
  if (t == VT_MI || t == VT_II) return k == M - 1;
  return k == 0 || (k == 1 && (t == VT_DM || t == VT_DD));
}

// Whether the packed kernel may score a profile whose moves are all <= 0
// (conditions: mpf_vit_packed.cu), and its constants.
bool packable(mpf_vprofile *v, const int16_t *msc, const int16_t *trans) {
  const int M = v->M, K = v->K;
  v->pack_solo = vit_pack_solo(M);
  v->pack_team = vit_pack_team(M);
  if (!v->fast || (!v->pack_solo.warps && !v->pack_team.warps)) return false;
  auto tr = [&](int t, int k) { return (int)trans[(size_t)t * M + k]; };
  const int sink = std::max(-v->sp[0], -v->sp[6]);   // xB falls by at most this per row (NN, JJ)
  v->pk_rebase = 1;
  for (int k = 0; k < M; ++k) {
    if (tr(VT_BM, k) != tr(VT_BM, 0)) return false;
    for (int t = VT_MM; t <= VT_DD; ++t) {
      if (vit_move_unused(t, k, M)) continue;
      if (tr(t, k) < -kVitPackReach) return false;
      if ((t == VT_MI || t == VT_II) && tr(t, k) > -sink) v->pk_rebase = 0;
    }
  }
  for (const VitPackShape &s : {v->pack_solo, v->pack_team})
    for (int k0 = s.qh; s.warps && s.qh <= kVitPackShortQH && k0 + s.qh < M; k0 += s.qh) {   // through the D states of a whole segment
      int c = tr(VT_MD, k0);
      for (int k = k0 + 1; k < k0 + s.qh; ++k) c += vit_move_unused(VT_DD, k, M) ? 0 : tr(VT_DD, k);
      if (c < -kVitPackReach) return false;
    }
  v->pk_emax = 1;
  v->pk_split = 0;
  for (int x = 0; x < kVitRows; ++x) {
    int low = x < K ? 0 : -32768, high = 0;
    for (int k = 0; x < K && k < M; ++k) {
      const int s = msc[(size_t)x * M + k];
      low = std::min(low, s);
      high = std::max(high, s);
    }
    v->pk_emax = std::max(v->pk_emax, high);
    if (low < -kVitPackReach) v->pk_split |= 1u << x;
  }
  v->pk_bm = tr(VT_BM, 0);
  const int floor = -32768 + kVitPackReach;
  const int lo = std::max(v->base + v->sp[1], -32768) + v->pk_bm - (v->pk_emax - 1);
  // A match state is at most the entry score plus pk_emax: it has to fit 16 bits.
  return sink <= 1024 && v->pk_emax <= kVitPackReach && lo >= floor + 2048 && lo + v->pk_emax <= 32767;
}

// The packed tables of a shape, appended to *out; returns their offset.
size_t append_packed(const mpf_vprofile *v, const int16_t *msc, const int16_t *trans, VitPackShape s,
                     std::vector<int16_t> *out) {
  static const int order[kVitPackPlanes] = {VT_MD, VT_DD, VT_MM, VT_IM, VT_DM, VT_MI, VT_II};
  const int M = v->M, K = v->K, QH = s.qh, words = s.warps * QH;
  const size_t row = (size_t)words * 32, base = (out->size() + 127) & ~(size_t)127;
  out->resize(base + 2 * (kVitPackPlanes + 2 * (size_t)kVitRows) * row);
  int16_t *h = out->data() + base;   // half 0 is the low one
  std::vector<uint32_t> at((size_t)M);   // each node's place in a row
  for (int k = 0; k < M; ++k) {
    const int seg = k / QH, lane = seg / 2;    // lane over the team
    at[(size_t)k] = (uint32_t)(2 * ((lane / 32 * QH + k % QH) * 32 + lane % 32) + seg % 2);
  }
  // Plane by plane, filled with the value of the nodes past M; the second step
  // of a code whose scores need none stays 0.
  for (int n = 0; n < kVitPackPlanes; ++n) {
    int16_t *d = h + 2 * (size_t)n * row;
    std::fill(d, d + 2 * row, (int16_t)-kVitPackReach);
    const int16_t *t = trans + (size_t)order[n] * M;
    for (int k = 0; k < M; ++k)
      if (!vit_move_unused(order[n], k, M)) d[at[(size_t)k]] = t[k];
  }
  for (int x = 0; x < kVitRows; ++x) {
    int16_t *d = h + 2 * (kVitPackPlanes + (size_t)x) * row, *d2 = d + 2 * kVitRows * row;
    std::fill(d, d + 2 * row, (int16_t)-kVitPackReach);
    const int16_t *sc = msc + (size_t)x * M;
    const bool split = (v->pk_split >> x) & 1u;
    if (split) std::fill(d2, d2 + 2 * row, (int16_t)(-32768 + kVitPackReach));
    for (int k = 0; x < K && k < M; ++k) {
      const int first = std::max((int)sc[k], -kVitPackReach);
      d[at[(size_t)k]] = (int16_t)first;
      if (split) d2[at[(size_t)k]] = (int16_t)(sc[k] - first);
    }
  }
  return base;
}

void fill_query(VitQuery *d, const mpf_vprofile *v, uint64_t q, uint64_t n, int16_t *score, uint8_t *flag,
                float *nat) {
  memset(d, 0, sizeof(*d));
  d->msc = v->d_msc;
  d->trans = v->d_trans;
  for (int i = 0; i < kVitSpecial; ++i) d->sp[i] = v->sp[i];
  d->M = v->M;
  d->Mpad = v->Mpad;
  d->base = v->base;
  d->scale = v->scale;
  d->score = score + q * n;
  d->flag = flag + q * n;
  d->nat = nat ? nat + q * n : nullptr;
  if (v->packed) {
    if (v->pack_solo.warps) d->pk_solo = VitPackTables{v->d_solo, v->pack_solo.qh};
    if (v->pack_team.warps) d->pk_team = VitPackTables{v->d_team, v->pack_team.warps * v->pack_team.qh};
    d->pk_bm = v->pk_bm;
    d->pk_emax = v->pk_emax;
    d->pk_off = v->pk_emax - 1;
    d->pk_split = v->pk_split;
    d->pk_rebase = v->pk_rebase;
  }
}

VitParams scan_params(const mpf_ctx *ctx, const mpf_db *db) {
  VitParams p;
  memset(&p, 0, sizeof(p));
  p.residues = db->d_words;
  p.n_words = db->n_words;
  p.status = ctx->d_status;
  p.seq_word = db->d_seq_word;
  p.seq_len = db->d_seq_len;
  p.seq_orig = db->d_seq_orig;
  p.n_seqs = (uint32_t)db->n_seqs;
  return p;
}

// Streams for n_groups launch groups that run concurrently: event[i] closes
// group i, the last event opens all.
int fork_open(mpf_ctx *ctx, size_t n_groups, std::vector<cudaEvent_t> *evs) {
  while (ctx->n_fork < 8 && (size_t)ctx->n_fork < n_groups) {
    if (cudaStreamCreateWithFlags(&ctx->fork[ctx->n_fork], cudaStreamNonBlocking) != cudaSuccess) break;
    ++ctx->n_fork;
  }
  if (ctx->n_fork < 1) return MPF_ECUDA;
  for (size_t i = 0; i <= n_groups; ++i) {
    cudaEvent_t ev;
    if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) return MPF_ECUDA;
    evs->push_back(ev);
  }
  return cudaEventRecord(evs->back(), ctx->stream) == cudaSuccess ? MPF_OK : MPF_ECUDA;
}

// Join every fork stream that may have work queued, then release the events.
int fork_close(mpf_ctx *ctx, size_t n_groups, const std::vector<cudaEvent_t> &evs) {
  int rc = MPF_OK;
  for (size_t gi = 0; gi < n_groups && gi + 1 < evs.size(); ++gi)
    if (cudaStreamWaitEvent(ctx->stream, evs[gi], 0) != cudaSuccess) rc = MPF_ECUDA;
  for (cudaEvent_t ev : evs) cudaEventDestroy(ev);
  return rc;
}

// Largest number of sequences for which teams are ahead of one warp per
// sequence: 2.5 per warp that an SM holds.  Measured (one query, the first N
// sequences of a database, ms teams / one warp): M = 1200 N = 500 1.07 /
// 1.51, 3,000 1.61 / 2.28, 6,000 2.24 / 2.68, 12,000 4.31 / 3.05; M = 2405
// 500 1.23 / 2.62, 3,000 2.44 / 3.98, 6,000 4.84 / 4.46, 12,000 9.56 / 5.15; M
// = 600 within 10% up to 6,000, then 2.10 / 1.84 at 12,000.
int64_t pack_team_max(const mpf_vprofile *v, int num_sms) {
  if (!v->pack_solo.warps) return INT64_MAX;
  if (!v->pack_team.warps) return -1;
  return (int64_t)num_sms * 16 * 5 / 2;
}

// Launch the packed kernel over the queries that qualify (one launch per
// shape).  *buf: a stream-ordered allocation that the caller frees after the
// launches that read the lists of sequences left to the 32-bit kernels:
// query i's list at fb_ranks[i], its count at fb_count[i] (null: not packed).
// MPF_ENOMEM: nothing was launched and both are null throughout.
int packed_enqueue(mpf_ctx *ctx, const mpf_vprofile *const *vps, int n_q, const mpf_db *db, int16_t *score,
                   uint8_t *flag, float *nat, const uint32_t *ranks, const uint32_t *n_ranks, uint8_t **buf,
                   std::vector<uint32_t *> *fb_ranks, std::vector<uint32_t *> *fb_count) {
  const uint64_t n = db->n_seqs;
  // (warps, words per lane) -> queries; a query whose number of sequences
  // only the device knows is in both its groups, and one of them scores it.
  std::map<std::pair<int, int>, std::vector<int>> groups;
  size_t np = 0, nd = 0;
  for (int q = 0; q < n_q; ++q) {
    const mpf_vprofile *v = vps[q];
    if (!v->packed) continue;
    ++np;
    const int64_t tmax = pack_team_max(v, ctx->num_sms);
    if (tmax >= 0 && (ranks || (int64_t)n <= tmax))
      groups[{v->pack_team.warps, v->pack_team.qh}].push_back(q), ++nd;
    if (tmax < INT64_MAX && (ranks || (int64_t)n > tmax))
      groups[{v->pack_solo.warps, v->pack_solo.qh}].push_back(q), ++nd;
  }
  fb_ranks->assign((size_t)n_q, nullptr);
  fb_count->assign((size_t)n_q, nullptr);
  if (!np) return MPF_OK;
  // Descriptors, work counters, list counts, lists.
  const size_t desc = sizeof(VitQuery) * nd, head = (desc + 4 * (nd + np) + 255) & ~(size_t)255;
  MPF_CUDA(cudaMallocAsync((void **)buf, head + 4 * np * (size_t)n, ctx->stream));
  uint32_t *counters = reinterpret_cast<uint32_t *>(*buf + desc);
  size_t i = 0;
  for (int q = 0; q < n_q; ++q)
    if (vps[q]->packed) {
      (*fb_count)[(size_t)q] = counters + nd + i;
      (*fb_ranks)[(size_t)q] = reinterpret_cast<uint32_t *>(*buf + head) + i * (size_t)n;
      ++i;
    }
  // Longest models first: the last tail is a short one.
  std::vector<std::pair<std::pair<int, int>, std::vector<int>>> order(groups.begin(), groups.end());
  std::stable_sort(order.begin(), order.end(), [](const auto &a, const auto &b) {
    return a.first.first * a.first.second > b.first.first * b.first.second;
  });
  std::vector<VitQuery> qs;
  qs.reserve(nd);
  for (const auto &g : order)
    for (int q : g.second) {
      VitQuery d;
      fill_query(&d, vps[q], (uint64_t)q, n, score, flag, nat);
      d.ranks = ranks ? ranks + (uint64_t)q * n : nullptr;
      d.n_ranks = n_ranks ? n_ranks + q : nullptr;
      d.pk_team_max = pack_team_max(vps[q], ctx->num_sms);
      d.fb_count = (*fb_count)[(size_t)q];
      d.fb_ranks = (*fb_ranks)[(size_t)q];
      qs.push_back(d);
    }
  cudaError_t e = cudaMemcpyAsync(*buf, qs.data(), desc, cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(counters, 0, 4 * (nd + np), ctx->stream);
  int rc = e == cudaSuccess ? MPF_OK : MPF_ECUDA;
  const bool fork = order.size() > 1;
  std::vector<cudaEvent_t> evs;
  if (fork && rc == MPF_OK) rc = fork_open(ctx, order.size(), &evs);
  size_t first = 0;
  for (size_t gi = 0; gi < order.size() && rc == MPF_OK; ++gi) {
    cudaStream_t st = ctx->stream;
    if (fork) {
      st = ctx->fork[gi % (size_t)ctx->n_fork];
      if (cudaStreamWaitEvent(st, evs.back(), 0) != cudaSuccess) rc = MPF_ECUDA;
    }
    VitParams p = scan_params(ctx, db);
    p.n_queries = (uint32_t)order[gi].second.size();
    p.queries = reinterpret_cast<const VitQuery *>(*buf) + first;
    p.counters = counters + first;
    first += order[gi].second.size();
    VitPackShape s;
    s.warps = order[gi].first.first;
    s.qh = order[gi].first.second;
    if (rc == MPF_OK && launch_viterbi_packed(p, s, ctx->max_smem, ctx->num_sms, st) != 0) rc = MPF_ECUDA;
    if (fork && cudaEventRecord(evs[gi], st) != cudaSuccess) rc = MPF_ECUDA;
  }
  if (fork && fork_close(ctx, order.size(), evs) != MPF_OK) rc = MPF_ECUDA;
  return rc;
}

// Launch the 32-bit Viterbi kernels over n_q queries: the general kernel for the
// profiles with a positive move, the fast kernel for the others, one launch
// per group of queries that share a kernel and launch shape (queries of one
// launch are scored one after the other by every block).  Query q scores the
// length ranks listed at ranks[q], n_ranks[q] of them (device), or all where
// ranks[q] is null.
int wide_enqueue(mpf_ctx *ctx, const mpf_vprofile *const *vps, int n_q, const mpf_db *db, int16_t *score,
                 uint8_t *flag, float *nat, const std::vector<const uint32_t *> &ranks,
                 const std::vector<const uint32_t *> &n_ranks) {
  const uint64_t n = db->n_seqs;
  // Group by kernel and launch shape (the key), then order by length.
  std::vector<std::tuple<int, int, int>> order;   // (key, Mpad, query)
  std::map<int, int> group_max;                    // key -> longest model of the group
  for (int q = 0; q < n_q; ++q) {
    const mpf_vprofile *v = vps[q];
    const int key = viterbi_shape_key(v->fast, v->Mpad, db->n_codes, ctx->max_smem, ctx->num_sms,
                                      ranks[(size_t)q] ? 0 : n);
    if (key < 0) return MPF_EUNSUPPORTED;
    order.emplace_back(key, v->Mpad, q);
    group_max[key] = std::max(group_max[key], v->Mpad);
  }
  // Groups with the longest models first (the launches are persistent and
  // fill the GPU in launch order, so the short-model groups finish last and
  // the final tail is short); within a group, longest models first.
  std::stable_sort(order.begin(), order.end(), [&](const std::tuple<int, int, int> &a,
                                                   const std::tuple<int, int, int> &b) {
    const int ga = group_max[std::get<0>(a)], gb = group_max[std::get<0>(b)];
    if (ga != gb) return ga > gb;
    if (std::get<0>(a) != std::get<0>(b)) return std::get<0>(a) < std::get<0>(b);
    return std::get<1>(a) > std::get<1>(b);
  });
  std::vector<VitQuery> qs;
  qs.reserve((size_t)n_q);
  for (const auto &o : order) {
    const int q = std::get<2>(o);
    const mpf_vprofile *v = vps[q];
    VitQuery d;
    fill_query(&d, v, (uint64_t)q, n, score, flag, nat);
    d.ranks = ranks[(size_t)q];
    d.n_ranks = n_ranks[(size_t)q];
    d.team_max = viterbi_team_max(std::get<0>(o), v->Mpad, db->n_codes, ctx->max_smem, ctx->num_sms);
    qs.push_back(d);
  }
  // Groups run concurrently on the context's fork streams, so that one
  // group's tail overlaps the others' work.  Groups of models longer than
  // the shared-memory rows hold get their own slice of device scratch.
  std::vector<std::pair<int, int>> groups;
  std::vector<size_t> state_off, state_len;
  const size_t desc_bytes = sizeof(VitQuery) * (size_t)n_q;
  size_t total = (desc_bytes + 4 * (size_t)n_q + 255) & ~(size_t)255;
  for (int first = 0; first < n_q;) {
    int last = first;
    int max_Mpad = 32;
    while (last < n_q && std::get<0>(order[(size_t)last]) == std::get<0>(order[(size_t)first])) {
      max_Mpad = std::max(max_Mpad, std::get<1>(order[(size_t)last]));
      ++last;
    }
    const mpf_vprofile *v0 = vps[std::get<2>(order[(size_t)first])];
    const size_t len = vit_key_device_rows(std::get<0>(order[(size_t)first]))
                           ? viterbi_state_bytes(v0->fast, max_Mpad, ctx->num_sms)
                           : 0;
    groups.emplace_back(first, last);
    state_off.push_back(total);
    state_len.push_back(len);
    total += (len + 255) & ~(size_t)255;
    first = last;
  }
  uint8_t *dev = nullptr;
  MPF_CUDA(cudaMallocAsync((void **)&dev, total, ctx->stream));
  cudaError_t e = cudaMemcpyAsync(dev, qs.data(), desc_bytes, cudaMemcpyHostToDevice, ctx->stream);
  uint32_t *counters = reinterpret_cast<uint32_t *>(dev + desc_bytes);
  if (e == cudaSuccess) e = cudaMemsetAsync(counters, 0, 4 * (size_t)n_q, ctx->stream);
  int rc = e == cudaSuccess ? MPF_OK : MPF_ECUDA;
  const bool fork = groups.size() > 1;
  std::vector<cudaEvent_t> evs;
  if (fork && rc == MPF_OK) {
    rc = fork_open(ctx, groups.size(), &evs);
  }
  for (size_t gi = 0; gi < groups.size() && rc == MPF_OK; ++gi) {
    const int first = groups[gi].first, last = groups[gi].second;
    const int key = std::get<0>(order[(size_t)first]);
    int max_Mpad = 32;
    for (int i = first; i < last; ++i) max_Mpad = std::max(max_Mpad, std::get<1>(order[(size_t)i]));
    cudaStream_t st = ctx->stream;
    if (fork) {
      st = ctx->fork[gi % (size_t)ctx->n_fork];
      if (cudaStreamWaitEvent(st, evs.back(), 0) != cudaSuccess) {
        rc = MPF_ECUDA;
        break;
      }
    }
    VitParams p = scan_params(ctx, db);
    p.n_queries = (uint32_t)(last - first);
    p.max_Mpad = max_Mpad;
    p.queries = reinterpret_cast<const VitQuery *>(dev) + first;
    p.counters = counters + first;
    p.state = state_len[gi] ? reinterpret_cast<uint2 *>(dev + state_off[gi]) : nullptr;
    p.state_bytes = state_len[gi];
    const int lr = launch_viterbi(p, key, db->n_codes, ctx->max_smem, ctx->num_sms, st);
    if (lr) rc = lr == 2 ? MPF_EUNSUPPORTED : MPF_ECUDA;
    if (fork && cudaEventRecord(evs[gi], st) != cudaSuccess) rc = MPF_ECUDA;
  }
  if (fork && fork_close(ctx, groups.size(), evs) != MPF_OK) rc = MPF_ECUDA;
  cudaFreeAsync(dev, ctx->stream);
  (void)cudaGetLastError();
  return rc;
}

// Launch the Viterbi kernels over n_q queries: the packed kernel for the
// profiles that qualify, then the 32-bit kernels for the other profiles and
// for the few sequences that the packed kernel leaves to them.  ranks /
// n_ranks (nullable) are [n_q][n_seqs] and [n_q] device arrays of selected
// length ranks.
int viterbi_enqueue(mpf_ctx *ctx, const mpf_vprofile *const *vps, int n_q, const mpf_db *db,
                    int16_t *score, uint8_t *flag, float *nat, const uint32_t *ranks,
                    const uint32_t *n_ranks) {
  uint8_t *buf = nullptr;
  std::vector<uint32_t *> fb_ranks, fb_count;
  int rc = packed_enqueue(ctx, vps, n_q, db, score, flag, nat, ranks, n_ranks, &buf, &fb_ranks, &fb_count);
  // No room for the lists: the 32-bit kernels, which need none, score them all.
  if (rc == MPF_ENOMEM) rc = MPF_OK;
  if (rc == MPF_OK) {
    std::vector<const uint32_t *> rk((size_t)n_q), nr((size_t)n_q);
    for (size_t q = 0; q < (size_t)n_q; ++q) {
      rk[q] = fb_ranks[q] ? fb_ranks[q] : ranks ? ranks + q * db->n_seqs : nullptr;
      nr[q] = fb_count[q] ? fb_count[q] : n_ranks ? n_ranks + q : nullptr;
    }
    rc = wide_enqueue(ctx, vps, n_q, db, score, flag, nat, rk, nr);
  }
  if (buf) cudaFreeAsync(buf, ctx->stream);
  (void)cudaGetLastError();
  return rc;
}

bool vit_args_ok(mpf_ctx *ctx, const mpf_vprofile *const *vps, int n_q, const mpf_db *db) {
  if (!ctx || !vps || n_q < 1 || !db || db->ctx->device != ctx->device) return false;
  for (int q = 0; q < n_q; ++q)
    if (!vps[q] || vps[q]->ctx->device != ctx->device) return false;
  return true;
}

}  // namespace

extern "C" {

int mpf_vit_profile_create(mpf_ctx *ctx, int M, int K, const int16_t *msc, const int16_t *trans,
                           const int16_t *special, int base, float scale, mpf_vprofile **out) {
  if (!out) return MPF_EINVAL;
  *out = nullptr;
  if (!ctx || !msc || !trans || !special || M < 1 || K < 1 || K > kVitRows) return MPF_EINVAL;
  if (base < -32768 || base > 32767 || !isfinite(scale) || !(scale > 0.f)) return MPF_EINVAL;
  if (M > kMaxLongM) return MPF_EUNSUPPORTED;
  const int Mpad = (M + 31) & ~31, Q = Mpad / 32;
  bool fast = true;
  for (size_t i = 0; i < (size_t)kVitTrans * M; ++i) fast = fast && trans[i] <= 0;
  for (int i = 0; i < kVitSpecial; ++i) fast = fast && special[i] <= 0;
  std::vector<int16_t> hm((size_t)kVitRows * Mpad, (int16_t)-32768);
  std::vector<int16_t> ht((size_t)kVitTrans * Mpad, (int16_t)-32768);
  // Striped: node k = l*Q + j in slot j*32 + l; transitions 8 per slot.
  for (int k = 0; k < M; ++k) {
    const size_t slot = (size_t)(k % Q) * 32 + (size_t)(k / Q);
    for (int x = 0; x < K; ++x) hm[(size_t)x * Mpad + slot] = msc[(size_t)x * M + k];
    for (int t = 0; t < kVitTrans; ++t) ht[slot * kVitTrans + t] = trans[(size_t)t * M + k];
  }
  mpf_vprofile *v = new (std::nothrow) mpf_vprofile;
  if (!v) return MPF_ENOMEM;
  v->fast = fast;
  v->ctx = ctx;
  v->M = M;
  v->K = K;
  v->Mpad = Mpad;
  for (int i = 0; i < kVitSpecial; ++i) v->sp[i] = special[i];
  v->base = base;
  v->scale = scale;
  DeviceGuard dg(ctx->device);
  // One allocation and one copy: match scores, transitions, packed tables.
  v->packed = packable(v, msc, trans);
  const size_t hm_n = hm.size();
  size_t total = hm.size() + ht.size();
  for (const VitPackShape &s : {v->pack_solo, v->pack_team})
    total += v->packed ? 128 + 2 * (kVitPackPlanes + 2 * (size_t)kVitRows) * (size_t)(s.warps * s.qh) * 32 : 0;
  hm.reserve(total);
  hm.insert(hm.end(), ht.begin(), ht.end());
  size_t solo = 0, team = 0;
  if (v->packed && v->pack_solo.warps) solo = append_packed(v, msc, trans, v->pack_solo, &hm);
  if (v->packed && v->pack_team.warps) team = append_packed(v, msc, trans, v->pack_team, &hm);
  cudaError_t e = cudaMalloc(&v->d_msc, hm.size() * sizeof(int16_t));
  if (e == cudaSuccess) e = cudaMemcpy(v->d_msc, hm.data(), hm.size() * sizeof(int16_t), cudaMemcpyHostToDevice);
  v->d_trans = v->d_msc + hm_n;   // 16-byte aligned: whole rows of Mpad (a multiple of 32) int16
  v->d_solo = reinterpret_cast<uint32_t *>(v->d_msc + solo);
  v->d_team = reinterpret_cast<uint32_t *>(v->d_msc + team);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    mpf_vit_profile_destroy(v);
    return e == cudaErrorMemoryAllocation ? MPF_ENOMEM : MPF_ECUDA;
  }
  *out = v;
  return MPF_OK;
}

void mpf_vit_profile_destroy(mpf_vprofile *v) {
  if (!v) return;
  DeviceGuard dg(v->ctx->device);
  cudaStreamSynchronize(v->ctx->stream);
  cudaFree(v->d_msc);
  (void)cudaGetLastError();
  delete v;
}

int mpf_viterbi_scan(mpf_ctx *ctx, const mpf_vprofile *const *vps, int n_q, const mpf_db *db,
                     int16_t *score, uint8_t *overflow, float *nat) {
  if (!vit_args_ok(ctx, vps, n_q, db) || !score || !overflow) return MPF_EINVAL;
  DeviceGuard dg(ctx->device);
  const uint64_t n = (uint64_t)n_q * db->n_seqs;
  if (db->n_seqs == 0) return MPF_OK;
  const bool device_out = is_device_ptr(score) && is_device_ptr(overflow) && (!nat || is_device_ptr(nat));
  if (device_out) return viterbi_enqueue(ctx, vps, n_q, db, score, overflow, nat, nullptr, nullptr);
  int rc = ensure_out_scratch(ctx, (size_t)n * 7 + 64);
  if (rc) return rc;
  uint8_t *base = (uint8_t *)ctx->d_out;
  float *k_nat = nat ? (float *)base : nullptr;
  int16_t *k_score = reinterpret_cast<int16_t *>(base + (size_t)n * 4);
  uint8_t *k_flag = base + (size_t)n * 6;
  rc = viterbi_enqueue(ctx, vps, n_q, db, k_score, k_flag, k_nat, nullptr, nullptr);
  if (rc == MPF_OK) {
    cudaError_t e = cudaMemcpyAsync(score, k_score, n * 2, cudaMemcpyDefault, ctx->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(overflow, k_flag, n, cudaMemcpyDefault, ctx->stream);
    if (e == cudaSuccess && nat) e = cudaMemcpyAsync(nat, k_nat, n * 4, cudaMemcpyDefault, ctx->stream);
    if (e != cudaSuccess) rc = MPF_ECUDA;
  }
  if (cudaStreamSynchronize(ctx->stream) != cudaSuccess && rc == MPF_OK) rc = MPF_ECUDA;
  (void)cudaGetLastError();
  return rc;
}

int mpf_viterbi_rescore(mpf_ctx *ctx, const mpf_vprofile *const *vps, int n_q, const mpf_db *db,
                        const uint8_t *msv_flag, const float *msv_nat, float msv_min_nat,
                        int16_t *score, uint8_t *overflow, float *nat, uint32_t *n_pass) {
  if (!vit_args_ok(ctx, vps, n_q, db) || !msv_flag || !msv_nat || !score || !overflow || !n_pass ||
      isnan(msv_min_nat))
    return MPF_EINVAL;
  DeviceGuard dg(ctx->device);
  for (const void *ptr : {(const void *)msv_flag, (const void *)msv_nat, (const void *)score,
                          (const void *)overflow, (const void *)n_pass})
    if (!is_device_ptr(ptr)) return MPF_EINVAL;
  if (nat && !is_device_ptr(nat)) return MPF_EINVAL;
  const uint64_t n = db->n_seqs;
  {  // The hand-off reads the MSV outputs while it writes the Viterbi ones: no two may share memory.
    const uint64_t nq = (uint64_t)n_q * n;
    const void *ptr[6] = {msv_flag, msv_nat, score, overflow, nat, n_pass};
    const uint64_t bytes[6] = {nq, 4 * nq, 2 * nq, nq, nat ? 4 * nq : 0, 4 * (uint64_t)n_q};
    if (ranges_overlap(ptr, bytes, 6)) return MPF_EINVAL;
  }
  const uint64_t n_chunks = (n + kSelectChunk - 1) / kSelectChunk;
  uint32_t *ranks = nullptr, *n_ranks = nullptr, *chunk = nullptr;
  cudaError_t e = cudaMallocAsync((void **)&ranks, std::max<uint64_t>(1, (uint64_t)n_q * n) * 4, ctx->stream);
  if (e == cudaSuccess) e = cudaMallocAsync((void **)&n_ranks, (size_t)n_q * 4, ctx->stream);
  if (e == cudaSuccess) e = cudaMallocAsync((void **)&chunk, std::max<uint64_t>(1, 2 * (uint64_t)n_q * n_chunks) * 4, ctx->stream);
  int rc = e == cudaSuccess ? MPF_OK : (e == cudaErrorMemoryAllocation ? MPF_ENOMEM : MPF_ECUDA);
  if (rc == MPF_OK && launch_select(db->d_seq_orig, n, n_q, msv_flag, msv_nat, msv_min_nat, score, 2,
                                    overflow, nat, chunk, chunk + (uint64_t)n_q * n_chunks, ranks,
                                    n_ranks, ctx->stream) != 0)
    rc = MPF_ECUDA;
  if (rc == MPF_OK && n > 0) rc = viterbi_enqueue(ctx, vps, n_q, db, score, overflow, nat, ranks, n_ranks);
  if (rc == MPF_OK && cudaMemcpyAsync(n_pass, n_ranks, (size_t)n_q * 4, cudaMemcpyDeviceToDevice, ctx->stream) != cudaSuccess)
    rc = MPF_ECUDA;
  if (ranks) cudaFreeAsync(ranks, ctx->stream);
  if (n_ranks) cudaFreeAsync(n_ranks, ctx->stream);
  if (chunk) cudaFreeAsync(chunk, ctx->stream);
  (void)cudaGetLastError();
  return rc;
}

}  // extern "C"

