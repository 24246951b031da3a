// Host side of the direct split path (direct_kernel.cuh): which calls take it,
// with which tiles and k slices, and the launch.
#include <algorithm>
#include <cmath>

#include "direct.h"

namespace gbg {
namespace {

int load_mode(bool kcontig, const float* x, int64_t ld, int64_t stride) {
  if (!kcontig) return kRows;
  return (ld & 3) == 0 && (stride & 3) == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0 ? kVec : kScalar;
}

}  // namespace

size_t direct_workspace_bytes(int64_t m, int64_t n, const DirectPlan& plan) {
  if (plan.slices <= 1 || plan.in_cluster) return 0;
  return (size_t)plan.slices * (size_t)((m + 127) / 128) * (size_t)((n + plan.bn - 1) / plan.bn) *
         ((size_t)128 * plan.bn + kDirectExpInts) * 4;
}

namespace {

// Estimated time (us) of a call on the packed path, as its launch chooses
// tiles, pairs and k slices (split.cu, default_schedule): the launches and the
// packing, rounds of tiles at a time per 32-deep chunk, the accumulators' way
// out, and the split-K reduction.  The constants here and in direct_us are
// fitted to measured calls, three sets of operands in turn (m, n log-uniform
// in 64 .. 6000, k in 128 .. 65536, batches to 96): this to 1000 calls, within
// 10% of nearly all, up to 40% too little where pair tiles wait for packed
// panels (k just above 512); that to 3384 plans of 450 calls.
double packed_us(int64_t m, int64_t n, int64_t k, int64_t batch, int num_sms, bool three) {
  const double nkc = (double)panel_k_chunks(k);
  const int64_t tm = (m + 127) / 128;
  auto tiles = [&](int bn) { return (double)(tm * ((n + bn - 1) / bn) * batch); };
  int bn = tiles(256) >= num_sms / 2 ? 256 : tiles(128) >= num_sms / 2 ? 128 : 64;
  int s = batch == 1 ? choose_splitk((int64_t)tiles(256), k, num_sms) : 1;
  if (s > 1) bn = 256;
  double t = 11.6 + (three ? 2.33e-6 : 1.87e-6) * (double)k * (double)(m + n) * (double)batch;
  if (s > 1) t += 3.5;
  const double chunks = std::ceil(nkc / s);
  if (bn == 256 && tm >= 2 && (!three || nkc >= 8)) {
    if (s == 1) return t + choose_pair_tiles(m, n, batch, panel_k_chunks(k), three, num_sms / 2).us;
    const double items = (double)((tm + 1) / 2 * ((n + 255) / 256) * batch) * s;
    return t + std::ceil(items / (num_sms / 2)) * (chunks * (three ? 1.0 : 0.5) + 4.0);
  }
  const double per = bn == 256 ? 0.6 : bn == 128 ? 0.44 : 0.37;
  return t + std::ceil(tiles(bn) * s / num_sms) * (chunks * per * (three ? 1.8 : 1.0) + 1.5);
}

// The same for a plan of the direct path.  Two parts: per 64-deep step 1.25 /
// 1.36 / 1.61 us of a 64 / 128 / 256 wide tile; three parts: per 32-deep step
// 1.0 / 1.32, and 1.63 times that for two CTAs on an SM.  1.2 times that with
// one operand whose rows are not 16-byte aligned, 1.3 with two.  The sum of
// slices in a cluster goes by rounds of four columns a thread.  A CTA serves
// one tile: every further round of CTAs starts anew.  Of the 450 calls, the
// plan this and packed_us choose takes 1.008 times the best one's time in the
// geometric mean, at most 1.29, and at most 1.02 of the packed path's.
double direct_us(const DirectPlan& p, int64_t m, int64_t n, int64_t k, int64_t batch, int num_sms, bool three,
                 int scalars) {
  const int bm = p.pair ? 256 : 128;
  const double ctas = (double)((m + bm - 1) / bm * ((n + p.bn - 1) / p.bn) * batch) * p.slices * (p.pair ? 2 : 1);
  const double chunks = std::ceil((double)panel_k_chunks(k) / p.slices);
  const double steps = three ? chunks : std::ceil(chunks / 2);
  double step = three ? (p.bn == 64 ? 1.0 : 1.32) : p.bn == 64 ? 1.25 : p.bn == 128 ? 1.36 : 1.61;
  step *= scalars == 2 ? (three ? 1.3 : 1.35) : scalars == 1 ? 1.2 : 1.0;
  // Clusters do not fill the GPU's groups of SMs: of 152, clusters of 4, 8 and
  // 16 CTAs reach 144, 120 and 112 (cudaOccupancyMaxActiveClusters on GB300).
  const int size = direct_cluster_ctas(p);
  double slots = num_sms * (size <= 2 ? 1.0 : size == 4 ? 144.0 / 152 : size == 8 ? 120.0 / 152 : 112.0 / 152);
  double again = three ? 3.0 : 5.8;
  if (three && ctas > slots) {  // two CTAs share an SM
    slots *= 2;
    step *= 1.63;
    again = 4.0;
  }
  const double waves = std::ceil(ctas / slots);
  const double out = three ? 0.0 : p.bn * 0.018;  // a tile's way out: not hidden behind the next one
  double t = (three ? 6.7 : 5.2) + waves * (steps * step + out) + (waves - 1) * again;
  if (p.slices > 1)
    t += !p.in_cluster ? 7.0
         : three       ? 0.9 * ((p.bn / p.slices + 7) / 8) + 0.2 * p.slices
                       : 1.15 * ((p.bn / p.slices + 15) / 16);
  return t;
}

// The plan that serves the call best, of clusters of at most max_cluster CTAs.
bool choose_plan(const SplitCall& c, int num_sms, int max_cluster, DirectPlan* plan, double* us = nullptr) {
  const int64_t m = c.m, n = c.n, k = c.k, batch = c.batch;
  if (c.lda >= (1 << 22) || c.ldb >= (1 << 22)) return false;  // offsets within a tile are 32 bits
  const bool three = split_parts(k) == 2;
  const int64_t nkc = panel_k_chunks(k);
  const int scalars = (load_mode(c.ta == 1, c.A, c.lda, batch > 1 ? c.sa : 0) == kScalar) +
                      (load_mode(c.tb == 0, c.B, c.ldb, batch > 1 ? c.sb : 0) == kScalar);
  // In favour of the packed path, for the estimates' error.  Over 1500 further
  // calls drawn alike, path AUTO then takes 0.738 times the packed path's time
  // in the geometric mean, four of them more than 1.02 times, the worst 1.07.
  const double packed = packed_us(m, n, k, batch, num_sms, three);
  double best = (three ? 0.9 : 0.94) * packed;
  bool found = false;
  const size_t packed_bytes = split_layout(m, n, k, batch, 1, 256).total;
  auto offer = [&](int bn, bool pair, int64_t slices, bool in_cluster) {
    if (slices > 1) {  // steps of two chunks; no slice may be empty
      const int64_t unit = three ? 1 : 2;
      const int64_t per = ((nkc + slices - 1) / slices + unit - 1) / unit * unit;
      const int64_t s = (nkc + per - 1) / per;
      if (in_cluster ? s != slices || (nkc + slices - 1) / slices * (slices - 1) >= nkc : s < 2) return;
      slices = s;
      if ((nkc + slices - 1) / slices * (slices - 1) >= nkc) return;
    }
    DirectPlan p;
    p.bn = bn; p.pair = pair; p.slices = (int)slices; p.in_cluster = in_cluster;
    if (direct_cluster_ctas(p) > max_cluster) return;
    const int64_t bm = pair ? 256 : 128;
    if ((m + bm - 1) / bm * ((n + bn - 1) / bn) * batch * slices > 0xFFFFFF) return;
    // never more workspace than the packed path's, which callers may have reserved
    if (direct_workspace_bytes(m, n, p) > packed_bytes) return;
    const double t = direct_us(p, m, n, k, batch, num_sms, three, scalars);
    if (t < best) {
      best = t;
      *plan = p;
      found = true;
    }
  };
  for (int s = 1; s <= 16; s *= 2) offer(64, false, s, true);
  for (int s = 1; s <= 8; s *= 2) offer(128, true, s, true);
  if (!three) {
    offer(256, true, 1, true);
    const int64_t tiles = (m + 255) / 256 * ((n + 255) / 256);
    if (batch == 1 && tiles * 4 <= num_sms) offer(256, true, std::min<int64_t>(num_sms / (2 * tiles), 64), false);
  }
  if (us) us[0] = best, us[1] = packed;
  return found;
}

}  // namespace

// A cluster that the device cannot place (16 CTAs are beyond the portable
// size, and a partition of a GPU may have fewer SMs together) gives way to a
// smaller one, and in the end to the packed path.
bool direct_plan(const SplitCall& c, int num_sms, DirectPlan* plan) {
  const bool three = split_parts(c.k) == 2;
  const int ma = load_mode(c.ta == 1, c.A, c.lda, c.batch > 1 ? c.sa : 0);
  const int mb = load_mode(c.tb == 0, c.B, c.ldb, c.batch > 1 ? c.sb : 0);
  auto fits = three ? (ma == kRows  ? direct_mode_fits<3, kRows>
                       : ma == kVec ? direct_mode_fits<3, kVec>
                                    : direct_mode_fits<3, kScalar>)
                    : (ma == kRows  ? direct_mode_fits<2, kRows>
                       : ma == kVec ? direct_mode_fits<2, kVec>
                                    : direct_mode_fits<2, kScalar>);
  for (int max_cluster = kDirectMaxCluster; max_cluster > 0; max_cluster = direct_cluster_ctas(*plan) / 2) {
    if (!choose_plan(c, num_sms, max_cluster, plan)) return false;
    if (fits(*plan, mb)) return true;
  }
  return false;
}

extern "C" int gbgemm_internal_direct_plan(char transa, char transb, int64_t m, int64_t n, int64_t k, int64_t batch,
                                           int64_t lda, int64_t ldb, int num_sms, int max_cluster, int* plan) {
  SplitCall c;
  c.ta = transa != 'N'; c.tb = transb != 'N';
  c.m = m; c.n = n; c.k = k; c.batch = batch; c.lda = lda; c.ldb = ldb;
  c.sa = batch > 1 ? lda * (c.ta ? m : k) : 0;
  c.sb = batch > 1 ? ldb * (c.tb ? k : n) : 0;
  DirectPlan p;
  double us[2];
  if (!choose_plan(c, num_sms, max_cluster, &p, us)) return 0;
  plan[4] = (int)(1000.0 * us[0]); plan[5] = (int)(1000.0 * us[1]);
  plan[0] = p.bn; plan[1] = p.pair; plan[2] = p.slices; plan[3] = p.in_cluster;
  return 1;
}

cudaError_t launch_direct(const SplitCall& c, const DirectPlan& plan, cudaStream_t s) {
  DirectArgs S{};
  S.A = c.A; S.B = c.B; S.lda = c.lda; S.ldb = c.ldb; S.sa = c.sa; S.sb = c.sb;
  S.m = c.m; S.n = c.n; S.k = c.k;
  S.alpha = c.alpha; S.beta = c.beta;
  S.C = c.C; S.ldc = c.ldc; S.sc = c.sc;
  const int bm = plan.pair ? 256 : 128;
  const int64_t tm = (c.m + bm - 1) / bm, tn = (c.n + plan.bn - 1) / plan.bn;
  const int64_t items = tm * tn * c.batch * plan.slices;
  if (items <= 0 || items > 0x3FFFFFFF) return cudaErrorInvalidValue;
  S.tiles_m = (int)tm;
  S.tiles_n = (int)tn;
  S.nkc = (int)panel_k_chunks(c.k);
  S.slices = plan.slices;
  S.slice_chunks = (S.nkc + plan.slices - 1) / plan.slices;
  if ((int64_t)(S.slices - 1) * S.slice_chunks >= S.nkc) return cudaErrorInvalidValue;  // no empty slice
  S.cluster_slices = plan.in_cluster ? plan.slices : 1;
  if (plan.in_cluster && plan.slices > 1 &&
      (plan.bn % plan.slices || direct_cluster_ctas(plan) > kDirectMaxCluster || plan.bn > 128))
    return cudaErrorInvalidValue;
  S.partial = plan.slices > 1 && !plan.in_cluster ? static_cast<float*>(c.ws) : nullptr;
  if (plan.slices > 1 && !plan.in_cluster && (c.batch != 1 || !c.ws)) return cudaErrorInvalidValue;
  if (S.partial)
    S.partial_exp = reinterpret_cast<int*>(S.partial + (size_t)plan.slices * ((c.m + 127) / 128) * tn * 128 * plan.bn);
  S.status = c.status;
  const int ma = load_mode(c.ta == 1, c.A, c.lda, c.batch > 1 ? c.sa : 0);
  const int mb = load_mode(c.tb == 0, c.B, c.ldb, c.batch > 1 ? c.sb : 0);
  const bool timed = c.gemm_begin && c.gemm_end;
  cudaError_t e = timed ? cudaEventRecord(c.gemm_begin, s) : cudaSuccess;
  if (e != cudaSuccess) return e;
  auto launch = split_parts(c.k) == 2 ? (ma == kRows  ? launch_direct_mode<3, kRows>
                                         : ma == kVec ? launch_direct_mode<3, kVec>
                                                      : launch_direct_mode<3, kScalar>)
                                      : (ma == kRows  ? launch_direct_mode<2, kRows>
                                         : ma == kVec ? launch_direct_mode<2, kVec>
                                                      : launch_direct_mode<2, kScalar>);
  e = launch(plan, mb, S, items, s);
  if (e == cudaSuccess && timed) e = cudaEventRecord(c.gemm_end, s);
  if (e != cudaSuccess || !S.partial) return e;
  SplitGemmArgs a;
  a.m = c.m; a.n = c.n; a.k = c.k; a.alpha = c.alpha; a.beta = c.beta; a.C = c.C; a.ldc = c.ldc;
  a.amaxA = nullptr; a.amaxB = nullptr; a.partial_exp = S.partial_exp;  // every slice has its own exponents
  a.num_sms = c.num_sms; a.bn = plan.bn; a.splitk = plan.slices;
  a.partial = S.partial;
  return launch_splitk_reduce(a, s);
}

}  // namespace gbg
