// Host planner and C entry points for the pattern FFT (setup is host-side,
// exact integers; every transform step runs in the kernels of fft_kernels.cu).
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <cstring>
#include <new>
#include <map>
#include <string>
#include <vector>

#include "../../include/pfft.h"
#include "fft_mixed.hpp"
#include "fft_plan.hpp"
#include "fft_tc.cuh"
#include "lattice.hpp"
#include "plan_common.hpp"
#include "plan_internal.hpp"

using namespace pfft;

namespace {

// Radices for a cycle length: primes from 11 up first (direct stages, up to
// kMaxDirectRadix), then 16s, the rest of the power of two and 3, 5, 7 -- the
// execution order of the stage regions (split-precision plans).  Returns false
// if a prime factor is not supported.
bool factor_radices(int n, std::vector<int>& out, bool tc = false) {
  out.clear();
  for (int p = kMinDirectRadix; p <= kMaxDirectRadix && p <= n; p += 2) {
    bool prime = true;
    for (int q = 3; q * q <= p; q += 2)
      if (p % q == 0) {
        prime = false;
        break;
      }
    if (!prime) continue;
    while (n % p == 0) {
      out.push_back(p);
      n /= p;
    }
  }
  int p2 = 0;
  while (n % 2 == 0) {
    n /= 2;
    ++p2;
  }
  while (tc && p2 >= 5) {  // tensor-core passes: radix-32 stages first
    out.push_back(32);
    p2 -= 5;
  }
  while (p2 >= 4) {
    out.push_back(16);
    p2 -= 4;
  }
  while (p2 >= 3) {
    out.push_back(8);
    p2 -= 3;
  }
  if (p2 == 2) out.push_back(4);
  if (p2 == 1) out.push_back(2);
  static const int primes[] = {3, 5, 7};
  for (int p : primes)
    while (n % p == 0) {
      out.push_back(p);
      n /= p;
    }
  return n == 1;
}

void set_box(BoxDesc& B, const IMat& H) {
  std::memset(&B, 0, sizeof(B));
  B.d = H.d;
  for (int i = 0; i < H.d; ++i)
    for (int j = 0; j < H.d; ++j) B.H[i][j] = int(H(i, j));
  int s = 1;
  for (int r = H.d - 1; r >= 0; --r) {
    B.stride[r] = s;
    s *= int(H(r, r));
  }
}

// Stages of a Stockham DFT along one pencil axis of length a and stride
// sigma, in the radix order of kRadixOrder (Ns accumulates in that order);
// twiddles come from a table of order nD (a multiple of a).
// Smallest primitive root of the prime p (g^((p-1)/f) != 1 for every prime f | p - 1).
int primitive_root(int p) {
  std::vector<int> fs;
  int n = p - 1;
  for (int f = 2; f * f <= n; ++f)
    if (n % f == 0) {
      fs.push_back(f);
      while (n % f == 0) n /= f;
    }
  if (n > 1) fs.push_back(n);
  auto powmod = [p](int b, int e) {
    long long r = 1, x = b;
    while (e) {
      if (e & 1) r = r * x % p;
      x = x * x % p;
      e >>= 1;
    }
    return int(r);
  };
  for (int g = 2; g < p; ++g) {
    bool ok = true;
    for (int f : fs)
      if (powmod(g, (p - 1) / f) == 1) {
        ok = false;
        break;
      }
    if (ok) return g;
  }
  return 0;
}

bool axis_stages(std::vector<StageDesc>& out, int a, int sigma, int nD, bool tc) {
  std::vector<int> rad;
  if (!factor_radices(a, rad, tc)) return false;
  int Ns = 1;
  for (int R : rad) {
    StageDesc s;
    std::memset(&s, 0, sizeof(s));
    s.R = R;
    s.a = a;
    s.aR = a / R;
    s.sigma = sigma;
    s.Ns = Ns;
    s.twstep = nD / (Ns * R);
    s.gen = R >= kMinDirectRadix ? primitive_root(R) : 0;
    s.div_aR.init(uint32_t(s.aR));
    s.div_sigma.init(uint32_t(sigma));
    s.div_Ns.init(uint32_t(Ns));
    out.push_back(s);
    Ns *= R;
  }
  return true;
}

int radix_region(int R) {
  for (int i = 0; i < kDirectRegion; ++i)
    if (kRadixOrder[i] == R) return i;
  if (R == 32) return kTC32Region;
  return R >= kMinDirectRadix && R <= kMaxDirectRadix ? kDirectRegion : -1;
}

// Execution order of the regions: direct prime stages first, then radix 32.
int region_rank(int R) {
  const int reg = radix_region(R);
  return reg == kDirectRegion ? -2 : reg == kTC32Region ? -1 : reg;
}

// Merge the stages of all axes, grouped by radix region (stable, so each
// axis keeps its own order), and fill the per-region counts.
bool set_stages(PassArgs& p, std::vector<StageDesc> all) {
  std::stable_sort(all.begin(), all.end(), [](const StageDesc& x, const StageDesc& y) {
    return region_rank(x.R) < region_rank(y.R);
  });
  if (all.size() > size_t(kMaxStages)) return false;
  p.nstages = int(all.size());
  std::memset(p.cnt, 0, sizeof(p.cnt));
  p.pow2 = 1;
  for (size_t i = 0; i < all.size(); ++i) {
    const int reg = radix_region(all[i].R);
    if (reg < 0) return false;
    p.st[i] = all[i];
    p.cnt[reg] += 1;
    if (reg > 3 && reg != kTC32Region) p.pow2 = 0;  // radix 32 (tensor-core plans) is a power of two
  }
  return true;
}

// Threads needed so that every stage fits its per-thread register budget.
int threads_for(const PassArgs& p, int ept) {
  int need = (p.T * p.L + ept - 1) / ept;
  for (int i = 0; i < p.nstages; ++i) {
    const int R = p.st[i].R;
    if (radix_region(R) == kDirectRegion) {  // the phases of run_direct_stage
      const int nbfly = p.T * (p.L / R), h = (R - 1) / 2;
      const int Q = R >= kDirectQ4MinRadix ? 4 : 2;
      const int cap_main = ept / 8 + (Q == 4 ? 1 : 2);  // kDirectQ4Items / kDirectQ2Items
      const int items = nbfly * ((h + Q - 1) / Q);
      need = std::max(need, (nbfly * h + ept / 2 - 1) / (ept / 2));  // kDirectPre
      need = std::max(need, (items + cap_main - 1) / cap_main);
      need = std::max(need, (nbfly + kDirectZero - 1) / kDirectZero);
      continue;
    }
    const int nb = std::max(1, ept / R);
    const int bfly = p.T * p.L / R;
    need = std::max(need, (bfly + nb - 1) / nb);
  }
  need = ((need + 31) / 32) * 32;
  return need;
}

size_t elem_bytes(int dtype) { return dtype == PFFT_C64 ? 8 : 16; }

// Whether one pencil of length L fits a CTA of the split-precision plans'
// shared-memory kernels: at most `row_max` elements and kMaxThreads threads.
bool tc_tile_fits(int L, int row_max) {
  if (L > row_max) return false;
  std::vector<int> rad;
  if (!factor_radices(L, rad)) return false;
  PassArgs p;
  std::memset(&p, 0, sizeof(p));
  p.T = 1;
  p.L = L;
  p.nstages = int(rad.size());
  if (p.nstages > kMaxStages) return false;
  for (int i = 0; i < p.nstages; ++i) p.st[i].R = rad[i];
  return threads_for(p, 32) <= kMaxThreads;
}

// ------------------------------------------------ mixed-radix passes (fft_mixed.cuh)
int mix_max_threads(const pfft_plan_s& P) {
  return std::min(P.max_threads, P.dtype == PFFT_C64 ? kMixThreadsC64 : kMixThreadsC128);
}
int mix_points(int R) { return R * std::max(1, kMixPoints / R); }  // points a thread takes in a radix-R stage

// Instructions a point costs in one stage: 8 for the shared-memory round trip,
// about 40 per butterfly for its indices, the butterfly and the twiddles
// (operation counts of fft_mixed.cuh); a direct stage about 1.2 per unit of R
// on top of its pre-pass.
double radix_cost(int R, bool direct = false) {
  static const double flops[17] = {0, 0, 4, 6.7, 8, 11.2, 11, 14.4, 13, 15.6, 15.2, 19.6, 14.3, 21.7, 17.7, 17.6, 16.8};
  return direct ? 40 + 1.2 * R : 8 + 40.0 / R + flops[R];
}

// A radix and how its stages run: as register butterflies or as direct sums.
struct Radix {
  int R;
  bool direct;
};

// Cheapest radices covering n (factors 2, 3, 5, 7, 11, 13 through the register
// butterflies, larger primes as direct stages, smallest first and before all
// others), every register radix taking at least min_points points per thread.
// small_direct: 11 and 13, whose butterflies are 11 and 13 points, run as direct
// stages where min_points is more: complex128 pencils of more than 5632 and 6656
// points (512 threads), such as the columns of diag(77, 77, 77).  cost: the sum of
// radix_cost.  False when n has no such cover.
struct RadixCover {
  double cost;
  int R;  // first radix (0: none)
};
RadixCover cover_smooth(int n, int min_points, int max2, std::map<int, RadixCover>& memo) {
  if (n == 1) return {0, 1};
  auto it = memo.find(n);
  if (it != memo.end()) return it->second;
  RadixCover best{1e30, 0};
  for (int R = 16; R >= 2; --R) {
    if (n % R || mix_points(R) < min_points || (R == 16 && max2 < 16)) continue;
    const RadixCover rest = cover_smooth(n / R, min_points, max2, memo);
    if (rest.R && rest.cost + radix_cost(R) < best.cost) best = {rest.cost + radix_cost(R), R};
  }
  memo[n] = best;
  return best;
}
bool mixed_radices(int n, int min_points, int max2, bool small_direct, std::vector<Radix>& out, double* cost = nullptr) {
  out.clear();
  double c = 0;
  for (int p = 11; p <= kMaxDirectRadix && p <= n; p += 2) {
    if (p < kMixMinDirect && !(small_direct && mix_points(p) < min_points)) continue;
    bool prime = p % 3 && p % 5 && p % 7 && (p == 11 || p % 11) && (p == 13 || p % 13);
    for (int q = 17; prime && q * q <= p; q += 2) prime = p % q != 0;
    if (!prime) continue;
    for (; n % p == 0; n /= p) {
      out.push_back({p, true});
      c += radix_cost(p, true);
    }
  }
  std::map<int, RadixCover> memo;
  for (int x = n; x > 1;) {
    const RadixCover r = cover_smooth(x, min_points, max2, memo);
    if (!r.R) return false;
    out.push_back({r.R, false});
    c += radix_cost(r.R);
    x /= r.R;
  }
  if (cost) *cost = c;
  return true;
}

// Points per thread that every stage of a pencil of L points must reach.
int mix_min_points(int L, const pfft_plan_s& P) { return (L + mix_max_threads(P) - 1) / mix_max_threads(P); }

// Time of the direct stages of a complex128 tile of n points with t threads, per
// SM: their multiply-adds bound it, so it is the turns that the busiest of the
// SM's four schedulers gives to warps with items, over the tiles resident at a time
// (128 registers a thread).  Tiles of a multiple of four warps put the warps of a
// last, partial turn on the same schedulers, others spread them.  A tile alone on
// its SM loads and stores beside no other's sums (4%).
double direct_time(const std::vector<Radix>& radices, int n, int t, bool alone = false) {
  const int tiles = alone ? 1 : kMixThreadsC128 / t, per_tile = t / 32;
  double time = 0;
  for (const Radix& r : radices) {
    if (!r.direct) continue;
    const int h = (r.R - 1) / 2, items = n / r.R * ((h + kMixNarrow - 1) / kMixNarrow);
    for (int left = items; left > 0; left -= t) {
      const int warps = (std::min(left, t) + 31) / 32;
      time += double(h) * (per_tile % 4 ? (tiles * warps + 3) / 4 : tiles * ((warps + 3) / 4));
    }
  }
  return time / tiles * (tiles == 1 && !alone ? 1.04 : 1.0);
}

// Threads of a mixed-radix tile of n points (alone: no other tile shares its SM).
int mix_threads(const std::vector<Radix>& radices, int n, int max_threads, int dtype, bool alone = false) {
  int need = (n + kMixPoints - 1) / kMixPoints;
  bool sums = false;
  for (const Radix& r : radices) {
    const int R = r.R, nbf = n / R;
    if (r.direct) {  // pre-pass pairs, then wide items or up to kMixItems narrow ones (mix_direct)
      const int h = (R - 1) / 2;
      const int wide = nbf * ((h + kMixWide - 1) / kMixWide), narrow = nbf * ((h + kMixNarrow - 1) / kMixNarrow);
      need = std::max(need, (nbf * h + kMixPoints / 2 - 1) / (kMixPoints / 2));
      need = std::max(need, dtype == PFFT_C64 && wide <= max_threads ? wide : (narrow + kMixItems - 1) / kMixItems);
      sums = true;
    } else {
      const int nb = std::max(1, kMixPoints / R);
      need = std::max(need, (nbf + nb - 1) / nb);
    }
  }
  need = (need + 31) / 32 * 32;
  if (dtype == PFFT_C64 || !sums) return need;
  // level ones: the fewest turns, then the fewest threads
  auto turns = [&](int t) {
    int u = 0;
    for (const Radix& r : radices)
      if (r.direct) u += (n / r.R * (((r.R - 1) / 2 + kMixNarrow - 1) / kMixNarrow) + t - 1) / t;
    return u;
  };
  int best = need;
  for (int t = need; t <= max_threads; t += 32) {
    const double a = direct_time(radices, n, t, alone), b = direct_time(radices, n, best, alone);
    if (a < b || (a == b && turns(t) < turns(best))) best = t;
  }
  return best;
}

// Whether a pencil of L points (one axis, or the axes of a column) fits a tile.
bool mix_fits(const pfft_plan_s& P, const std::vector<int>& axes, int L, bool small_direct = false,
              double* cost = nullptr) {
  if (L > (P.dtype == PFFT_C64 ? 16384 : 8192)) return false;
  std::vector<Radix> all, rad;
  double c = 0, ca = 0;
  for (int a : axes) {
    if (!mixed_radices(a, mix_min_points(L, P), 16, small_direct, rad, &ca)) return false;
    all.insert(all.end(), rad.begin(), rad.end());
    c += ca;
  }
  if (cost) *cost = c;
  return int(all.size()) <= kMixMaxStages && mix_threads(all, L, mix_max_threads(P), P.dtype) <= mix_max_threads(P);
}

// Pad unit u (element x at x + x / u) under which a walk over the elements in the
// order pos meets the fewest banks twice, of `lanes` banks per wavefront: a divisor
// of run, or the unit at hand (0: none).  A step of 40 elements, as the column
// order of M = [[1200, 240], [0, 1080]] takes, is eight-way without padding and
// free of conflicts with u = 8 (0.401 -> 0.388 ms there and back, batch 8).
int pad_unit(const std::vector<int>& pos, int run, int at_hand, int lanes) {
  const int n = int(std::min<size_t>(pos.size(), 2048)) / lanes * lanes;
  auto conflicts = [&](int u) {
    int total = 0;
    for (int i = 0; i < n; i += lanes) {
      int hits[16] = {}, worst = 0;
      for (int k = 0; k < lanes; ++k) {
        const int x = pos[i + k];
        worst = std::max(worst, ++hits[(x + (u ? x / u : 0)) % lanes]);
      }
      total += worst;
    }
    return total;
  };
  int best = 0, least = conflicts(at_hand);
  for (int u = 64; u >= 8; --u) {  // large ones first: they need less room
    if (run % u || u == at_hand) continue;
    const int c = conflicts(u);
    if (10 * c < 8 * least) {
      least = c;
      best = u;
    }
  }
  return best;
}

// The stages of a kind of tile (everything that does not depend on T) and
// their tables.
pfft_status mix_stages(pfft_plan_s& P, int kind) {
  MixStages& S = P.stages[P.max2 == 16 ? 0 : 1][kind];
  if (S.ready) return PFFT_OK;
  const int L = kind == MIX_ROW ? P.nD : kind == MIX_COL ? P.LB : int(P.m);
  const int tw_n = kind == MIX_COL && P.tw_col ? P.col_n : P.nD;
  struct Axis {
    int a, sigma, Ns;
  };
  std::vector<Axis> axes;
  int sigma = 1;
  if (kind != MIX_COL) {
    axes.push_back({P.nD, 1, 1});
    sigma = P.nD;
  }
  if (kind != MIX_ROW)
    for (int s = int(P.pen.size()) - 1; s >= 0; --s) {
      axes.push_back({P.pen[s], sigma, 1});
      sigma *= P.pen[s];
    }
  std::vector<std::pair<Radix, int>> order;  // (radix, axis)
  std::vector<Radix> rad;
  for (size_t i = 0; i < axes.size(); ++i) {
    if (!mixed_radices(axes[i].a, mix_min_points(L, P), P.max2, P.dtype == PFFT_C128, rad)) return PFFT_ERR_UNSUPPORTED;
    for (const Radix& r : rad) order.push_back({r, int(i)});
  }
  if (order.size() > size_t(kMixMaxStages)) return PFFT_ERR_UNSUPPORTED;
  std::stable_sort(order.begin(), order.end(), [](const std::pair<Radix, int>& x, const std::pair<Radix, int>& y) {
    const Radix &a = x.first, &b = y.first;
    if (a.direct || b.direct) return a.direct != b.direct ? a.direct : a.R < b.R;
    auto rank = [](int R) { return std::find(kMixOrder, kMixOrder + 15, R) - kMixOrder; };
    return rank(a.R) < rank(b.R);
  });
  MixTableArgs t;
  std::memset(&t, 0, sizeof(t));
  std::vector<int> g;
  for (auto& o : order) {
    Axis& ax = axes[o.second];
    MixStage s;
    std::memset(&s, 0, sizeof(s));
    s.R = o.first.R;
    s.aR = ax.a / s.R;
    s.sig = ax.sigma;
    s.Ns = ax.Ns;
    s.twstep = tw_n / (s.Ns * s.R);
    s.div_aR.init(uint32_t(s.aR));
    s.div_Ns.init(uint32_t(s.Ns));
    if (o.first.direct) {
      ++S.ndirect;
      s.gen = int(g.size());
      const int r = primitive_root(s.R);
      for (int e = 0, x = 1; e < s.R - 1; ++e, x = x * r % s.R) g.push_back(x);
    } else if (s.Ns > 1) {
      s.tw = t.total;
      const bool fused = P.dtype == PFFT_C128 && (s.R & (s.R - 1)) == 0;
      t.R[t.n] = s.R;
      t.Ns[t.n] = s.Ns;
      t.fused[t.n] = fused;
      t.off[t.n++] = t.total;
      t.total += s.Ns * (fused ? s.R / 2 : s.R > 8 ? 4 : s.R > 4 ? 3 : s.R > 2 ? 2 : 1);
      t.off[t.n] = t.total;
    }
    ax.Ns *= s.R;
    S.st.push_back(s);
  }
  if (t.total) {
    if (int e = P.alloc(&S.stw, size_t(t.total) * elem_bytes(P.dtype))) return pfft_status(e);
    if (launch_mixed_tables(S.stw, t, P.dtype, 0) != 0) return PFFT_ERR_CUDA;
  }
  if (!g.empty()) {
    if (int e = P.alloc((void**)&S.gtab, g.size() * sizeof(int))) return pfft_status(e);
    if (cudaMemcpy(S.gtab, g.data(), g.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess)
      return PFFT_ERR_CUDA;
  }
  if (kind == MIX_ROW) {
    int R1 = 0;  // unit of the padding that the first register stage starts
    for (auto& s : S.st)
      if (s.Ns == 1 && s.R % 2 == 0) R1 = s.R;
    if (P.fs_na == 1 && !S.st.empty()) {
      const int lanes = 128 / int(elem_bytes(P.dtype));
      if (S.ndirect == 0) S.ws_in = pad_unit(P.PIinv, S.st[0].aR, 0, lanes);
      const MixStage& z = S.st.back();
      if (S.ndirect < int(S.st.size())) S.ws_out = pad_unit(P.PIinv, z.Ns, R1, lanes);
    }
    auto padded = [&](int unit, int** out) {
      if (!unit) return 0;
      std::vector<int> ps(P.PIinv);
      for (int& x : ps) x += x / unit;
      if (int e = P.alloc((void**)out, ps.size() * sizeof(int))) return e;
      return cudaMemcpy(*out, ps.data(), ps.size() * sizeof(int), cudaMemcpyHostToDevice) == cudaSuccess
                 ? 0
                 : int(PFFT_ERR_CUDA);
    };
    if (int e = padded(S.ws_in, &S.psin)) return pfft_status(e);
    if (int e = padded(S.ws_out ? S.ws_out : R1, &S.psout)) return pfft_status(e);
  }
  S.ready = true;
  return PFFT_OK;
}

// Points per thread of a launch that does not fill the chip.  [[64, 16], [-16,
// 64]] x 1 there and back, called from Python: 28.7 us with 16, 24.6 with 8, 29.7 with 5; [[300, 60],
// [0, 240]] x 1: 31.1 and 28.2 us; [[60, 24], [0, 72]] x 1 in complex128: 62 and 50.6 us.
constexpr int kMixFewPoints = 8;

// The descriptor of a kind of tile with T pencils (T a power of two; any T for
// row tiles in [row][element] order and whole tiles).
pfft_status mix_configure(pfft_plan_s& P, int kind, int T) {
  MixDesc& a = P.mix[kind];  // its plan-wide fields are set (plan_device)
  const MixStages& S = P.stages[P.max2 == 16 ? 0 : 1][kind];
  const int max_threads = mix_max_threads(P);
  a.kind = kind;
  a.lay = kind == MIX_ROW && P.fs_na > 1 ? 1 : 0;
  a.L = kind == MIX_ROW ? P.nD : kind == MIX_COL ? P.LB : int(P.m);
  a.T = T;
  a.logT = 0;
  while ((1 << a.logT) < T) ++a.logT;
  a.n = T * a.L;
  const int count = kind == MIX_ROW ? P.LB : kind == MIX_COL ? P.nD : int(P.batch);
  a.groups = (count + T - 1) / T;
  a.divnD.init(uint32_t(P.nD));
  a.divL.init(uint32_t(a.L));
  a.stw = S.stw;
  a.gtab = S.gtab;
  a.tw = kind == MIX_COL && P.tw_col ? P.tw_col : P.tw;
  a.tw_n = kind == MIX_COL && P.tw_col ? P.col_n : P.nD;
  const int tstride = kind == MIX_COL || a.lay ? T : 1;  // stride of the pencil index in the tile
  a.nstages = int(S.st.size());
  std::vector<Radix> rad;
  int rmax = 0;
  int unit = 0;  // pad unit, once padded
  for (int i = 0; i < a.nstages; ++i) {
    MixStage s = S.st[i];
    const bool first = s.sig == 1 && s.Ns == 1 && s.R % 2 == 0 && tstride < 16;
    s.sig *= tstride;
    s.blk = s.aR * s.R * s.sig;
    s.istep = s.aR * s.sig;
    s.ostep = s.Ns * s.sig;
    const int unit_in = unit;
    if (unit) {
      s.ipad = tstride;
      s.istep += s.istep / unit * tstride;
    }
    if (first) unit = s.R * tstride;
    if (unit) {
      s.opad = tstride;
      if (!first) s.ostep += s.ostep / unit * tstride;
    }
    s.div_in.init(uint32_t(s.ipad ? unit_in : 1 << 30));
    s.div_out.init(uint32_t(s.opad ? unit : 1 << 30));
    s.div_sig.init(uint32_t(s.sig));
    s.div_nb.init(uint32_t(std::max(1, a.n / s.R)));
    rad.push_back({s.R, i < S.ndirect});
    if (i < S.ndirect) {
      rmax = std::max(rmax, s.R);
      s.tw = s.R;
      if (s.R < kMixMinDirect) s.R += kMixDirect;
    }
    a.st[i] = s;
  }
  const i64 ctas = i64(a.groups) * (kind == MIX_WHOLE ? 1 : P.batch);
  a.nthreads = mix_threads(rad, a.n, max_threads, P.dtype, !P.generic_only && ctas <= P.nsm);
  // a launch that leaves the chip idle gets twice the threads that its stages ask
  // for, as long as all of it stays resident: half the turns of every load and store
  const int more = (a.n + kMixFewPoints - 1) / kMixFewPoints;
  if (!P.generic_only && more <= max_threads && ctas * more <= i64(P.nsm) * max_threads)
    a.nthreads = std::max(a.nthreads, (more + 31) / 32 * 32);
  // each thread keeps one column (or, of a [element][row] tile, one row in turns of four elements)
  const int keep = a.lay ? 4 * T : tstride;
  if (a.nthreads % keep) a.nthreads = (a.nthreads + keep - 1) / keep * keep;
  if (a.nthreads > max_threads) return PFFT_ERR_UNSUPPORTED;
  a.pad = unit ? tstride : 0;
  a.div_pad.init(uint32_t(unit ? unit : 1 << 30));
  a.dir_off = a.n + (unit ? a.n / unit * tstride : 0);
  a.ws_in = a.ws_out = 0;
  a.pitch_in = a.pitch_out = a.L;
  a.psin = a.psout = a.PIinv;
  if (kind == MIX_ROW) {
    if (S.ws_in) {
      a.ws_in = S.ws_in;
      a.psin = S.psin;
      a.pitch_in += a.L / S.ws_in;
      a.dir_off = std::max(a.dir_off, T * a.pitch_in);
    }
    if (S.ws_out) {
      a.ws_out = S.ws_out;
      a.psout = S.psout;
      a.pitch_out += a.L / S.ws_out;
      a.dir_off = std::max(a.dir_off, T * a.pitch_out);
    } else if (unit) {
      a.psout = S.psout;
      a.pitch_out += a.L / (unit / tstride);
    }
  }
  // roots (R - 1 + kMixWide) and powers (R - 1 ints) of a direct stage
  const int extra = rmax ? rmax + kMixWide + (rmax + 1) / 2 : 0;
  a.smem_bytes = int(size_t(a.dir_off + extra) * elem_bytes(P.dtype));
  return a.smem_bytes <= (P.generic_only ? kMixGroupedSmem : 227 * 1024) ? PFFT_OK : PFFT_ERR_UNSUPPORTED;
}

// Pencils per tile: as many as `budget` points hold (at most `cap`), up to
// `lanes` of them (the adjacent pencils that fill a 32-byte sector) even when
// that takes `most` points; but no more than leave `ctas` tiles for the launch
// once those lanes are there.  A tile of more than half the threads of an SM has
// it alone, every phase waiting for the one before: half the pencils are then the
// better tile, and half of the last 16 bytes of a sector if that puts a quarter more
// threads on the SM (there and back, columns of 1728 points in 576 threads, [[1728,
// 1472], [0, 2048]] x 3: 0.414 and 0.365 ms; [[96, 87, 0], [0, 375, 201], [0, 0,
// 243]] x 7, two columns of 3240 points in 544 threads: 3.60 and 3.24; a mix of 512
// patterns: 2.14 and 2.11; but two of 3850 points in 704 threads lose 7%).
// Complex128 tiles with direct sums hold another number of pencils, up to `most`
// points, where the launch is at least 3% shorter for it.
pfft_status mix_choose(pfft_plan_s& P, int kind, int cap, int budget, int most, int lanes, int ctas) {
  pfft_status st = mix_stages(P, kind);
  if (st != PFFT_OK) return st;
  const int L = kind == MIX_ROW ? P.nD : kind == MIX_COL ? P.LB : int(P.m);
  const i64 count = kind == MIX_ROW ? P.LB : kind == MIX_COL ? P.nD : P.batch;
  const i64 signals = kind == MIX_WHOLE ? 1 : P.batch;
  int T = 1;
  while (2 * T <= cap && 2 * T <= count) {
    const i64 n = 2 * i64(T) * L;
    const bool few = (count + 2 * T - 1) / (2 * T) * signals < ctas;
    if (n > (2 * T <= lanes ? std::max(most, budget) : budget) || (few && 2 * T > lanes && n > 256)) break;
    T *= 2;
  }
  for (;; T /= 2) {
    st = mix_configure(P, kind, T);
    const int max = P.dtype == PFFT_C64 ? kMixThreadsC64 : kMixThreadsC128, t = P.mix[kind].nthreads, half = (t / 2 + 31) / 32 * 32;
    if (T == 1) break;
    if (st != PFFT_OK) continue;
    if (t <= max / 2 || (T * elem_bytes(P.dtype) <= 16 && 4 * (max / half * half) < 5 * t)) break;
  }
  const MixStages& S = P.stages[P.max2 == 16 ? 0 : 1][kind];
  if (st != PFFT_OK || P.dtype == PFFT_C64 || !S.ndirect) return st;
  std::vector<Radix> rad;
  for (int i = 0; i < int(S.st.size()); ++i) rad.push_back({S.st[i].R, i < S.ndirect});
  // Clocks of the launch on its busiest SM (grouped tiles: on average): 16 multiply-adds
  // of a warp a step at half a lane a clock and scheduler, and 5000 that a tile takes
  // besides ([[16336]] x 8: 0.67 ms a direction, 1.09 with pencils for a full chip).
  auto time = [&](int x) {
    if (mix_configure(P, kind, x) != PFFT_OK) return 1e30;
    const double tiles = double((count + x - 1) / x) * signals / P.nsm;
    if (P.generic_only) return (1024 * direct_time(rad, x * L, P.mix[kind].nthreads) + 5000) * tiles;
    return (1024 * direct_time(rad, x * L, P.mix[kind].nthreads, tiles <= 1) + 5000) * std::ceil(tiles);
  };
  double least = 0.97 * time(T);
  for (int x = 16; x >= 1; x /= 2) {
    if (x > cap || x > count || (x > 1 && i64(x) * L > most)) continue;
    const double c = time(x);
    if (c < least) {
      least = c;
      T = x;
    }
  }
  return mix_configure(P, kind, T);
}

// Register-resident column pass over two pencil axes (fft_fast2.cuh): the
// 2-D DFT of sizes top x low (top the slower axis of the row index) is the
// 1-D Stockham DFT of length L = top low without the twiddles that couple the
// axes, provided the first stages' radices multiply to top -- a radix-32
// complex64 pass of L = t 32^s (tail t first) has those products t 32^j,
// j < s.  Box layout, complex64, no split-precision stages, no four-step
// split, both axes powers of two.
bool fast2_axes(const pfft_plan_s& P, int top, int low) {
  if (P.dtype != PFFT_C64 || P.tc || P.generic_only || P.fs_na != 1 || P.pen.size() != 2) return false;
  if (top < 2 || low < 2 || (top & (top - 1)) || (low & (low - 1))) return false;
  const int L = top * low;
  if (L < 64 || L > 16384) return false;
  int lg = 0;
  while ((1 << lg) < L) ++lg;
  const int nmain = lg / 5;
  int b = 1 << (lg - 5 * nmain);
  for (int j = 0; j < nmain; ++j, b *= 32)
    if (b == top) return true;
  return false;
}

// The register-resident pass of a power-of-two length with T pencils per CTA,
// or, in split-precision plans, the shared-memory one.  PFFT_ERR_UNSUPPORTED
// where neither applies.
pfft_status configure_pass(PassArgs& p, const pfft_plan_s& P, bool cols, int T) {
  p.cols = cols;
  p.T = T;
  std::vector<StageDesc> stg;
  if (!cols) {
    p.L = P.nD;
    if (!axis_stages(stg, P.nD, 1, P.nD, P.tc)) return PFFT_ERR_UNSUPPORTED;
    p.groups = (P.LB + T - 1) / T;
  } else {
    p.L = P.LB;
    int sigma = 1;
    for (int s = int(P.pen.size()) - 1; s >= 0; --s) {  // pencil axes, last fastest
      if (!axis_stages(stg, P.pen[s], sigma, p.tw_n, P.tc)) return PFFT_ERR_UNSUPPORTED;
      sigma *= P.pen[s];
    }
    p.groups = (P.nD + T - 1) / T;
  }
  if (!set_stages(p, stg)) return PFFT_ERR_UNSUPPORTED;
  p.divT.init(uint32_t(T));
  p.divnD.init(uint32_t(P.nD));
  p.logT = 0;
  while ((1 << p.logT) < T) ++p.logT;
  // register-resident power-of-two kernels (fft_fast.cuh)
  {
    const int Rm = P.dtype == PFFT_C64 ? 32 : 16;
    const int L = p.L;
    const bool pow2L = L >= Rm && (L & (L - 1)) == 0 && (T & (T - 1)) == 0;
    // split-precision plans use them too, their radix-32 main stages on the tensor cores
    const bool tc_fast = P.tc && P.dtype == PFFT_C64 && p.tw_n % 32 == 0;
    // (a column tile of the register-resident pass holds T whole columns: T divides nD)
    p.fast = ((!P.generic_only || tc_fast) && p.tw_n == P.nD && p.pow2 && pow2L && P.d <= 3 && (!cols || P.pen.size() == 1 || fast2_axes(P, P.pen[0], P.pen[1])) && (!cols || P.nD % T == 0) && T * L <= (P.dtype == PFFT_C64 ? 16384 : 8192)) ? 1 : 0;
    if (p.fast) {
      int lg = 0, lr = 0;
      while ((1 << lg) < L) ++lg;
      while ((1 << lr) < Rm) ++lr;
      p.fast_nmain = lg / lr;
      p.fast_tail = 1 << (lg - p.fast_nmain * lr);
      p.nthreads = T * L / Rm;
      // stage twiddle table: for main stage s (span Ns) and k < Ns, w^(2^b), b < log2 R
      // (complex64), or the R / 2 factors of fused_dft (complex128)
      const int per = P.dtype == PFFT_C64 ? lr : Rm / 2;
      int off = 0, Ns = p.fast_tail;
      for (int s = 0; s < p.fast_nmain; ++s) {
        p.stw_off[s] = off;
        off += Ns * per;
        Ns *= Rm;
      }
      p.stw_n = (off + 1) & ~1;
      const int nel = T * L;
      p.stw_smem_off = (nel + (nel >> 5) + 1) & ~1;
      p.smem_bytes = int(size_t(p.stw_smem_off + p.stw_n) * elem_bytes(P.dtype));
      bool ok = true;
      if (P.tc) {  // W (radix 32), mbarrier and tensor-memory address after the stage table (fft_tc.cuh)
        p.tc = 1;
        p.tc_off = (p.smem_bytes + 15) & ~15;
        p.smem_bytes = p.tc_off + tc_regs_extra_bytes();
        ok = p.nthreads % 128 == 0 && p.fast_nmain >= 1;
      }
      if (ok && p.nthreads <= kMaxThreads && p.smem_bytes <= 227 * 1024 && p.fast_nmain <= 4) return PFFT_OK;
      p.fast = 0;
      p.tc = 0;
    }
  }
  if (!P.tc) return PFFT_ERR_UNSUPPORTED;  // the mixed-radix passes take it
  // shared-memory kernels of split-precision plans: 32 points per thread
  p.ept = 32;
  p.nthreads = threads_for(p, p.ept);
  if (cols && T > 32) p.nthreads = (p.nthreads + T - 1) / T * T;  // each thread keeps one column
  if (p.nthreads > kMaxThreads) return PFFT_ERR_UNSUPPORTED;
  const int nel = T * p.L;
  int rmax = 0;  // omega_R table of the direct stages, after the tile
  for (int i = 0; i < p.nstages; ++i)
    if (radix_region(p.st[i].R) == kDirectRegion) rmax = std::max(rmax, p.st[i].R);
  p.pad = rmax ? 0 : 1;
  p.dir_off = p.pad ? (nel - 1) + ((nel - 1) >> 4) + 1 : nel;
  // direct-stage tables: omega_R^{g^t} (R - 1 complex) and g^t (R - 1 int), with slack
  p.smem_bytes = int(size_t(p.dir_off + 2 * rmax) * elem_bytes(P.dtype));
  p.tc = 1;
  p.tc_off = (p.smem_bytes + 15) & ~15;
  {  // tensor-core stages (fft_tc.cuh)
    // the hi / lo rows of a stage's 128-butterfly chunks overwrite the tile
    for (int i = 0; i < p.nstages; ++i) {
      const int R = p.st[i].R;
      if (R != 16 && R != 32) continue;
      const int nch = (T * p.L / R + 127) / 128;
      p.tc_off = std::max(p.tc_off, nch * tc_chunk_bytes(R));
    }
    p.tc_off = (p.tc_off + 15) & ~15;
    p.smem_bytes = tc_layout(p.tc_off, p.cnt[kTC32Region] > 0, p.cnt[0] > 0, T * p.L / 16).end;
    // every warp of a lane quarter reads its rows of the accumulator: whole warp quadruples
    p.nthreads = (p.nthreads + 127) / 128 * 128;
    if (p.nthreads > kMaxThreads || tc_tmem_cols(T * p.L, p.cnt[kTC32Region] > 0, p.cnt[0] > 0) > 256)
      return PFFT_ERR_UNSUPPORTED;
  }
  if (p.smem_bytes > 227 * 1024) return PFFT_ERR_UNSUPPORTED;
  return PFFT_OK;
}

// Choose the pencils-per-CTA count: the largest power of two (<= cap) whose
// tile fits `budget` elements and the thread limit.  PFFT_ERR_UNSUPPORTED when
// the pass is one for the mixed-radix kernels.
pfft_status choose_and_configure(PassArgs& p, const pfft_plan_s& P, bool cols, int cap, int budget) {
  const int L = cols ? P.LB : P.nD;
  const int limit = cols ? P.nD : P.LB;
  int T = 1;
  while (T * 2 <= cap && T * 2 <= limit && T * 2 * L <= budget) T *= 2;
  for (;;) {
    pfft_status st = configure_pass(p, P, cols, T);
    if (st == PFFT_OK || !P.tc) return st;
    if (T == 1) return st;
    T /= 2;
  }
}

}  // namespace

// ----------------------------------------------------------------- planning
pfft_status pfft::plan_host(pfft_plan_s& P, int d, const int64_t* Mv) {
  if (d < 1 || d > 4) return PFFT_ERR_ARG;
  P.d = d;
  P.M = IMat(d);
  for (int i = 0; i < d * d; ++i) {
    if (Mv[i] >= (int64_t(1) << 24) || Mv[i] <= -(int64_t(1) << 24)) return PFFT_ERR_OVERFLOW;
    P.M.a[i] = Mv[i];
  }
  const i64 det = determinant(P.M);
  if (det == 0) return PFFT_ERR_SINGULAR;
  P.m = det < 0 ? -det : det;
  if (P.m >= (i64(1) << 31)) return PFFT_ERR_OVERFLOW;
  P.H = hermite_normal_form(P.M);
  P.G = hermite_normal_form(P.M.transpose());
  IMat Q, R, U, V;
  smith_normal_form(P.M, Q, P.eps, R, U, V);
  // lambda = Q^{-1} y = U y mod eps ;  mu = R^{-T} k = V^T k mod eps
  std::vector<std::vector<i64>> LAM(d, std::vector<i64>(d)), MU(d, std::vector<i64>(d));
  for (int j = 0; j < d; ++j)
    for (int c = 0; c < d; ++c) {
      LAM[j][c] = posmod(U(j, c), P.eps[j]);
      MU[j][c] = posmod(V(c, j), P.eps[j]);
    }
  // Remark 2: any biorthogonal pair of bases works.  If the fastest input
  // coordinate e_f generates a cycle of maximal length, re-base so that it is
  // the generator of the last cycle; then the row pass reads contiguous runs.
  {
    const int f = d - 1;
    const i64 E = P.eps[d - 1];
    int j0 = -1;
    for (int j = d - 1; j >= 0; --j)
      if (P.eps[j] == E && gcd64(LAM[j][f], E) == 1) {
        j0 = j;
        break;
      }
    if (j0 >= 0 && E > 1) {
      std::vector<i64> v(d);
      for (int j = 0; j < d; ++j) v[j] = LAM[j][f] % P.eps[j];
      const i64 u = modinv(v[j0], E);
      auto L2 = LAM, M2 = MU;
      for (int c = 0; c < d; ++c) L2[j0][c] = posmod(i64((i128)u * LAM[j0][c] % E), E);
      for (int j = 0; j < d; ++j) {
        if (j == j0) continue;
        for (int c = 0; c < d; ++c) {
          i128 t = (i128)LAM[j][c] - (i128)v[j] * u % P.eps[j] * LAM[j0][c];
          L2[j][c] = posmod(i64(t % P.eps[j]), P.eps[j]);
        }
      }
      for (int c = 0; c < d; ++c) {
        i128 s = 0;
        for (int i = 0; i < d; ++i) s += (i128)v[i] * (E / P.eps[i]) % E * MU[i][c];
        M2[j0][c] = posmod(i64(s % E), E);
      }
      std::swap(L2[j0], L2[d - 1]);
      std::swap(M2[j0], M2[d - 1]);
      LAM = L2;
      MU = M2;
    }
  }
  P.D = 0;
  P.n.clear();
  P.LAM.clear();
  P.MU.clear();
  for (int j = 0; j < d; ++j)
    if (P.eps[j] > 1) {
      P.n.push_back(int(P.eps[j]));
      P.LAM.push_back(LAM[j]);
      P.MU.push_back(MU[j]);
      ++P.D;
    }
  if (P.D > 3) return PFFT_ERR_UNSUPPORTED;
  P.fs_N = P.D ? P.n[P.D - 1] : 1;
  P.fs_na = 1;
  P.nD = int(P.fs_N);
  P.pen.assign(P.n.begin(), P.n.end() - (P.D ? 1 : 0));
  // A last cycle longer than one row tile is split four-step style,
  // n = n_a n_b with lambda = lambda_a + n_a lambda_b: the row pass runs the
  // length-n_b DFTs (twiddle exp(-2 pi i lambda_a mu_b / n) between the passes)
  // and lambda_a becomes one more pencil axis of the column pass.
  const int row_max = P.dtype == PFFT_C64 ? 16384 : 8192;
  const i64 n = P.fs_N;
  // A cycle that fits only with radices 11 or 13 as direct stages is split if it
  // can be without them, and stays whole if not; splits that need them come last.
  const bool whole = n <= row_max && (P.tc ? tc_tile_fits(int(n), row_max) : mix_fits(P, {int(n)}, int(n)));
  const bool small_direct = P.dtype == PFFT_C128;
  const bool whole_direct = small_direct && !whole && n <= row_max && mix_fits(P, {int(n)}, int(n), true);
  auto split_cycle = [&](bool direct) {
    const i64 other = P.m / n;
    int best = 0;
    double best_cost = 1e30;
    for (i64 nb = std::min<i64>(row_max, n - 1); nb >= 2; --nb) {
      if (n % nb) continue;
      const i64 na = n / nb, lb = other * na;
      if (lb > row_max) break;  // only grows as nb falls
      if (P.tc) {  // the longest row
        if (!tc_tile_fits(int(nb), row_max) || !tc_tile_fits(int(lb), row_max)) continue;
        best = int(nb);
        break;
      }
      // Stages of both passes, and what a tile loses when it cannot hold eight
      // pencils: above 2048 points eight adjacent pencils (64-byte accesses) no
      // longer leave room for a second tile on the SM, above 4096 the accesses
      // fall to 16 bytes, and fewer than eight rows lambda_a are not eight
      // adjacent slots.  A long complex64 column costs three times what a long row
      // does: its lanes are all the adjacent accesses it has on either side ([[4096,
      // 1024], [0, 8192]] x 1, cycles 1024 and 32768, forward / inverse: 745 / 815 us with
      // rows of 4096 and columns of 8192, 602 / 669 with 8192 and 4096, 780 / 742 before
      // the mixed-radix tiles; in complex128 they are nearly level, [[1024, 256], [0,
      // 4096]] x 1 with rows or columns of 4096: 630 and 650 us).  Weights measured with the passes' own times: 10800 =
      // 16 15 15 3 runs at 28 instructions a point and stage.
      double cr = 0, cc = 0;
      std::vector<int> pen(P.pen.begin(), P.pen.end());
      pen.push_back(int(na));
      if (!mix_fits(P, {int(nb)}, int(nb), direct, &cr) || !mix_fits(P, pen, int(lb), direct, &cc)) continue;
      const int unit = P.dtype == PFFT_C64 ? 1024 : 512;
      auto long_tile = [&](i64 L) { return L > 8 * unit ? 60.0 : L > 4 * unit ? 30.0 : L > 2 * unit ? 12.0 : L > unit ? 3.0 : 0.0; };
      const double column = P.dtype == PFFT_C64 && lb > 4 * unit ? 3.0 : 1.0;
      const double c = cr + cc + long_tile(nb) + column * long_tile(lb) + 3.0 * std::max<i64>(0, 8 - na);
      if (c < best_cost) {
        best_cost = c;
        best = int(nb);
      }
    }
    return best;
  };
  if (n > 1 && !whole) {
    int best = split_cycle(false);
    if (!best && !whole_direct && small_direct) best = split_cycle(true);
    if (!best && !whole_direct) return PFFT_ERR_UNSUPPORTED;
    if (best) {
      P.nD = best;
      P.fs_na = int(n / best);
      P.pen.push_back(P.fs_na);
    }
  }
  if (P.pen.size() > size_t(kMaxSub)) return PFFT_ERR_UNSUPPORTED;
  P.LB = int(P.m / P.nD);
  return PFFT_OK;
}

namespace {
// g_j = M MU_j^T / n_j  (in box(H));  h_j = M^T LAM_j^T / n_j  (in box(G)).
std::vector<i64> generator(const IMat& A, const std::vector<i64>& row, i64 nj, const IMat& box) {
  const int d = A.d;
  std::vector<i64> g(d);
  for (int i = 0; i < d; ++i) {
    i128 s = 0;
    for (int c = 0; c < d; ++c) s += (i128)A(i, c) * row[c];
    if (s % nj != 0) throw LatticeError{PFFT_ERR_OVERFLOW, "generator is not integral"};
    g[i] = i64(s / nj);
  }
  box_reduce(box, g.data());
  return g;
}

std::vector<i64> combo(const std::vector<std::vector<i64>>& gens, const std::vector<i64>& coef,
                       const IMat& box) {
  const int d = box.d;
  std::vector<i64> y(d, 0);
  for (size_t j = 0; j < gens.size(); ++j)
    for (int r = 0; r < d; ++r) y[r] += coef[j] * gens[j][r];  // < 2^62: coef, gens < 2^31
  box_reduce(box, y.data());
  return y;
}
}  // namespace

// The tile of one kind for a points budget: whole and plain row tiles need no
// adjacent pencils, the others four.  Small tiles are the faster ones, several
// of them filling an SM's 1024 threads in different phases (M = [[1200, 240],
// [0, 1080]] x 8 there and back: 0.446 ms with 2048 points, 0.468 with 4096),
// except that four adjacent pencils of a long cycle are worth 8192 points
// ([[2048, 8], [0, 2048]] x 8: 1.03 ms, against 1.17 with two pencils of 2048).
static pfft_status mix_tile(pfft_plan_s& P, int kind, int budget, int ctas) {
  const bool adjacent = kind == MIX_COL || (kind == MIX_ROW && P.fs_na > 1);
  const bool c64 = P.dtype == PFFT_C64;
  return mix_choose(P, kind, kind == MIX_ROW ? 16 : 64, kind == MIX_WHOLE ? (c64 ? 2048 : 1024) : budget, c64 ? 8192 : 4096, adjacent ? 4 : 1,
                    ctas);
}

// Whether whole signals share tiles: one launch, no workspace.  Two tiles of 8192
// complex64 (4096 complex128) points share an SM; one of twice that takes the SM,
// worth it once the batch alone nearly fills the chip, as two passes use more SMs.
// The register-resident passes are the better ones, one direction in us against
// whole tiles,
//   for a single complex64 cycle: 1024 points x 4096 signals 15.0 and 21.6, 4096 x 512
//     12.1 and 13.8, 8192 x 16 8.2 and 10.8 (but 2048 x 64 5.8 and 5.3, 512 x 2048 4%
//     apart), so from 4096 points on, or from 1024 in more than two signals an SM;
//   for a batch that leaves a third of the chip idle, both passes resident: [[128, 0],
//     [0, 128]] x 64 12.5 and 17.1 (x 100: 13% apart, x 152: whole tiles by 6%); in
//     complex128 above 2048 points [[64, 0], [0, 64]] x 1 39 and 47 (x 100: 2% apart);
//   for more than 4096 complex128 points, one such pass being enough: [[64, 0], [0,
//     128]] x 64 54 and 99, x 200 147 and 197, x 512 338 and 406; [[16, 0, 0], [0, 16,
//     0], [0, 0, 32]] x 64 54 and 94, x 512 333 and 383 (x 152 and x 304: whole tiles by
//     5%).
static bool whole_tile(const pfft_plan_s& P, int resident) {
  const bool c64 = P.dtype == PFFT_C64;
  const i64 half = c64 ? 8192 : 4096;
  std::vector<int> axes(P.pen.begin(), P.pen.end());
  axes.push_back(P.nD);
  if (P.m > 2 * half || !mix_fits(P, axes, int(P.m))) return false;
  const i64 most_sms = 2 * i64(P.nsm) / 3;
  if (P.pen.empty()) {
    if (resident && c64 && (P.m >= 4096 || (P.m >= 1024 && P.batch > 2 * i64(P.nsm)))) return false;
  } else if (!c64) {
    if (P.m > half ? resident > 0 : resident == 2 && P.m > half / 2 && P.batch < most_sms) return false;
  }
  return P.m <= half || P.batch >= (resident == 2 ? most_sms : 64);
}

pfft_status pfft::plan_device(pfft_plan_s& P) {
  const int d = P.d, D = P.D;
  if (cudaGetDevice(&P.device) != cudaSuccess) return PFFT_ERR_CUDA;
  if (D == 0) return PFFT_OK;  // m == 1: the transform is the identity
  if (cudaDeviceGetAttribute(&P.nsm, cudaDevAttrMultiProcessorCount, P.device) != cudaSuccess || P.nsm < 1)
    return PFFT_ERR_CUDA;
  // generators of the cycles
  std::vector<std::vector<i64>> g(D), h(D);
  for (int j = 0; j < D; ++j) {
    g[j] = generator(P.M, P.MU[j], P.n[j], P.H);
    h[j] = generator(P.M.transpose(), P.LAM[j], P.n[j], P.G);
  }
  // biorthogonality check (Lemma 1 / Remark 2), exact
  for (int i = 0; i < D; ++i)
    for (int j = 0; j < D; ++j) {
      i128 a = 0, b = 0;
      for (int c = 0; c < d; ++c) {
        a += (i128)P.LAM[i][c] * g[j][c];
        b += (i128)P.MU[i][c] * h[j][c];
      }
      const i64 want = (i == j) ? 1 : 0;
      if (posmod(i64(a % P.n[i]), P.n[i]) != want || posmod(i64(b % P.n[i]), P.n[i]) != want)
        return PFFT_ERR_OVERFLOW;
    }
  const int nD = P.nD, LB = P.LB;
  const int na = P.fs_na;
  const int npen = int(P.pen.size());
  // two pencil axes of which only the faster one starts a register-resident
  // column pass (fast2_axes): make it the slower axis of the row index (the
  // rows then run over (lambda_2, lambda_1); the tables below follow)
  const bool swap2 = npen == 2 && na == 1 && !fast2_axes(P, P.pen[0], P.pen[1]) && fast2_axes(P, P.pen[1], P.pen[0]);
  if (swap2) std::swap(P.pen[0], P.pen[1]);
  // Row (A, B) and column (C, E) generator lists of the logical LB x nD array:
  //   row index  = flatten(lambda_1..lambda_{D-1}[, lambda_a]),  element = lambda_b
  //   col index  = flatten(mu_1..mu_{D-1}[, mu_a]),              position of mu_b
  // with lambda_D = lambda_a + n_a lambda_b and mu_D = mu_b + n_b mu_a when the
  // last cycle is split (n_a > 1); otherwise lambda_b = lambda_D, mu_b = mu_D.
  std::vector<std::vector<i64>> genA(g.begin(), g.end() - 1), genC(h.begin(), h.end() - 1);
  if (swap2) {
    std::swap(genA[0], genA[1]);
    std::swap(genC[0], genC[1]);
  }
  std::vector<i64> gB = g[D - 1], hE = h[D - 1];
  if (na > 1) {
    genA.push_back(g[D - 1]);
    std::vector<i64> hb(d), gb(d);
    for (int k = 0; k < d; ++k) {
      hb[k] = h[D - 1][k] * nD;  // n_b h_D (|h| < 2^31, n_b <= 2^14)
      gb[k] = g[D - 1][k] * na;  // n_a g_D
    }
    box_reduce(P.G, hb.data());
    box_reduce(P.H, gb.data());
    genC.push_back(hb);
    gB = gb;
  }
  // column permutation PI for the column pass (see fft_plan.hpp)
  std::vector<int> PI(nD), PIinv(nD);
  std::vector<int> alpha(3, 0);
  {
    const i64 cf = posmod(P.MU[D - 1][d - 1], P.fs_N);  // mu_D of the fastest output coordinate
    i64 beta = cf % nD;
    for (int j = 0; j + 1 < D; ++j) alpha[j] = int(posmod(P.MU[j][d - 1], P.n[j]));
    if (na > 1) alpha[npen - 1] = int((cf / nD) % na);
    if (swap2) std::swap(alpha[0], alpha[1]);
    const i64 gg = beta == 0 ? nD : gcd64(beta, nD);
    const i64 span = nD / gg;
    const i64 inv = span > 1 ? modinv(beta / gg, span) : 0;
    for (i64 mu = 0; mu < nD; ++mu) {
      const i64 pos = (mu % gg) * span + ((mu / gg) * inv) % span;
      PI[mu] = int(pos);
      PIinv[pos] = int(mu);
    }
  }
  P.PIinv = PIinv;
  // index tables
  const int ts = d <= 2 ? 2 : 4;  // int32 per entry, so that one vector load fetches a point
  std::vector<int> tab(size_t(2 * LB + 2 * nD) * ts + 2 * nD, 0);
  int* Atab = tab.data();
  int* Btab = Atab + size_t(LB) * ts;
  int* Ctab = Btab + size_t(nD) * ts;
  int* Etab = Ctab + size_t(LB) * ts;
  int* PIi = Etab + size_t(nD) * ts;
  int* PIf = PIi + nD;
  std::vector<i64> coef(npen);
  for (int r = 0; r < LB; ++r) {
    int x = r;
    for (int j = npen - 1; j >= 0; --j) {
      coef[j] = x % P.pen[j];
      x /= P.pen[j];
    }
    auto a = combo(genA, coef, P.H);
    auto c = combo(genC, coef, P.G);
    for (int k = 0; k < d; ++k) {
      Atab[size_t(r) * ts + k] = int(a[k]);
      Ctab[size_t(r) * ts + k] = int(c[k]);
    }
  }
  for (int e = 0; e < nD; ++e) {
    auto b = combo({gB}, {e}, P.H);
    auto c = combo({hE}, {PIinv[e]}, P.G);
    for (int k = 0; k < d; ++k) {
      Btab[size_t(e) * ts + k] = int(b[k]);
      Etab[size_t(e) * ts + k] = int(c[k]);
    }
    PIi[e] = PIinv[e];
    PIf[e] = PI[e];
  }
  if (int e_ = P.alloc((void**)&P.dtab, tab.size() * sizeof(int))) return pfft_status(e_);
  if (cudaMemcpy(P.dtab, tab.data(), tab.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess)
    return PFFT_ERR_CUDA;
  const size_t eb = elem_bytes(P.dtype);
  if (int e_ = P.alloc((void**)&P.tw, size_t(nD) * eb)) return pfft_status(e_);
  if (int e_ = P.alloc((void**)&P.status, sizeof(int))) return pfft_status(e_);
  cudaMemset(P.status, 0, sizeof(int));
  if (launch_twiddles(P.tw, nD, P.dtype, 0) != 0) return PFFT_ERR_CUDA;
  // The column pass transforms the pencil axes; their twiddles come from the
  // nD table when every axis divides nD (always, unless the last cycle is
  // split four-step: n_a need not divide n_b), else from a table of order
  // lcm(axes) <= LB.
  int col_n = nD;
  {
    i64 l = 1;
    for (int a : P.pen) l = l / gcd64(l, a) * a;
    if (npen >= 1 && nD % l != 0) {
      col_n = int(l);
      P.col_n = col_n;
      if (int e_ = P.alloc(&P.tw_col, size_t(col_n) * eb)) return pfft_status(e_);
      if (launch_twiddles(P.tw_col, col_n, P.dtype, 0) != 0) return PFFT_ERR_CUDA;
    }
  }
  if (na > 1) {  // exp(-2 pi i t / n) for t < n, as lo[t & 2047] * hi[t >> 11]
    const int nhi = int((P.fs_N + 2047) >> 11);
    if (int e_ = P.alloc(&P.fs_tab, size_t(2048 + nhi) * eb)) return pfft_status(e_);
    if (launch_phase_tables(P.fs_tab, P.fs_N, nhi, P.dtype, 0) != 0) return PFFT_ERR_CUDA;
  }

  // pass descriptors (data pointers and modes are filled per call)
  // arithmetic forms of PI and of the gather table (power-of-two cycles)
  PassArgs arith;
  std::memset(&arith, 0, sizeof(arith));
  {
    const i64 beta = posmod(P.MU[D - 1][d - 1], nD);
    const i64 gg = beta == 0 ? nD : gcd64(beta, nD);
    const i64 span = nD / gg;
    auto lg2 = [](i64 v) { int l = 0; while ((i64(1) << l) < v) ++l; return (i64(1) << l) == v ? l : -1; };
    if (lg2(gg) >= 0 && lg2(span) >= 0) {
      arith.pi_arith = 1;
      arith.pi_lg = lg2(gg);
      arith.pi_lspan = lg2(span);
      arith.pi_inv = int(span > 1 ? modinv(beta / gg, span) : 0);
    }
    // Btab[e] = (Z[e / H_ff], e mod H_ff) when g_D = e_f (the last input coordinate) and H_ff | nD
    const i64 Hff = P.H(d - 1, d - 1);
    bool unit = true;
    std::vector<i64> ef(d, 0);
    ef[d - 1] = 1;
    {
      std::vector<i64> gD = g[D - 1];
      std::vector<i64> e1 = ef;
      box_reduce(P.H, e1.data());
      unit = (gD == e1);
    }
    const int lh = int(lg2(Hff));
    if (unit && lh >= 0 && nD % Hff == 0 && nD / Hff <= 64 && d <= 3) {
      arith.bz_arith = 1;
      arith.bz_lh = lh;
      for (i64 q = 0; q < nD / Hff; ++q) {
        const int* b = Btab + size_t(q * Hff) * ts;
        for (int r = 0; r + 1 < d; ++r) arith.bz[q][r] = b[r];
        if (b[d - 1] != 0) arith.bz_arith = 0;
      }
      for (int e = 0; e < nD && arith.bz_arith; ++e) {  // exact check against the table
        const int* b = Btab + size_t(e) * ts;
        for (int r = 0; r + 1 < d; ++r)
          if (b[r] != arith.bz[e >> lh][r]) arith.bz_arith = 0;
        if (b[d - 1] != (e & ((1 << lh) - 1))) arith.bz_arith = 0;
      }
    }
    if (arith.pi_arith)
      for (int mu = 0; mu < nD; ++mu) {  // exact check against the table
        const int span_i = 1 << arith.pi_lspan;
        const int pos = ((mu & ((1 << arith.pi_lg) - 1)) << arith.pi_lspan) |
                        (((mu >> arith.pi_lg) * arith.pi_inv) & (span_i - 1));
        if (pos != PI[mu]) {
          arith.pi_arith = 0;
          break;
        }
      }
  }
  const int budget = P.dtype == PFFT_C64 ? 8192 : 4096;
  // rows need no adjacent pencils: small CTAs, several of them in different phases
  // on an SM ([[512, 128], [0, 512]] x 16 there and back, rows of 2048: 0.098 ms
  // with 8192 points per CTA, 0.092 with 4096, 0.080 with 2048)
  const int row_budget = P.dtype == PFFT_C64 && !P.tc ? 2048 : budget;
  for (PassArgs* p : {&P.rowp, &P.colp}) {
    std::memset(p, 0, sizeof(PassArgs));
    p->Atab = Atab - tab.data() + P.dtab;
    p->Btab = Btab - tab.data() + P.dtab;
    p->Ctab = Ctab - tab.data() + P.dtab;
    p->Etab = Etab - tab.data() + P.dtab;
    p->PIinv = PIi - tab.data() + P.dtab;
    p->PI = PIf - tab.data() + P.dtab;
    const bool colt = (p == &P.colp) && P.tw_col;
    p->tw = colt ? P.tw_col : P.tw;
    p->tw_n = colt ? col_n : nD;
    p->ts = ts;
    p->cols = p == &P.colp;
    p->nD = nD;
    p->LB = LB;
    p->m = int(P.m);
    p->d = d;
    p->batch = int(P.batch);
    p->status = P.status;
    p->spin_limit = kSpinLimit;
    set_box(p->boxH, P.H);
    set_box(p->boxG, P.G);
    p->pi_arith = arith.pi_arith;
    p->pi_lg = arith.pi_lg;
    p->pi_lspan = arith.pi_lspan;
    p->pi_inv = arith.pi_inv;
    p->bz_arith = arith.bz_arith;
    p->bz_lh = arith.bz_lh;
    std::memcpy(p->bz, arith.bz, sizeof(arith.bz));
    p->nsub = npen;
    for (int s = 0; s < npen; ++s) {
      p->sub_n[s] = P.pen[s];
      p->sub_div[s].init(uint32_t(P.pen[s]));
      p->alpha[s] = alpha[s];
    }
    p->fs_na = na;
    p->fs_div.init(uint32_t(na));
    p->fs_lo = P.fs_tab;
    p->fs_hi = P.fs_tab ? static_cast<const char*>(P.fs_tab) + size_t(2048) * eb : nullptr;
  }
  // The register-resident kernels take power-of-two passes (rows of a cycle that
  // is not split, whose box loads need no lanes across rows); the mixed-radix
  // ones everything else.
  auto no_pass = [](PassArgs& p) { p.fast = p.tc = 0; };
  {
    pfft_status row = PFFT_ERR_UNSUPPORTED, col = PFFT_ERR_UNSUPPORTED;
    if (P.tc || na == 1) row = choose_and_configure(P.rowp, P, false, 64, std::max(row_budget, nD));
    if (npen >= 1) col = choose_and_configure(P.colp, P, true, P.generic_only ? 512 : 16, std::max(budget, LB));
    if (P.tc && row != PFFT_OK) return row;
    if (P.tc && npen >= 1 && col != PFFT_OK) return col;
    const int resident = (row == PFFT_OK) + (col == PFFT_OK);  // register-resident passes
    P.mixed[MIX_WHOLE] = !P.tc && na == 1 && whole_tile(P, resident);
    P.mixed[MIX_ROW] = !P.mixed[MIX_WHOLE] && row != PFFT_OK;
    P.mixed[MIX_COL] = !P.mixed[MIX_WHOLE] && npen >= 1 && col != PFFT_OK;
    if (P.mixed[MIX_WHOLE] || P.mixed[MIX_ROW]) no_pass(P.rowp);
    if (P.mixed[MIX_WHOLE] || P.mixed[MIX_COL]) no_pass(P.colp);
  }
  if (npen >= 1 && P.own_workspace && !P.mixed[MIX_WHOLE])
    if (int e_ = P.alloc(&P.ws, size_t(P.m) * P.batch * eb)) return pfft_status(e_);
  for (int kind = 0; kind < 3; ++kind) {
    if (!P.mixed[kind]) continue;
    MixDesc& a = P.mix[kind];
    std::memset(&a, 0, sizeof(a));
    const PassArgs& p = kind == MIX_COL ? P.colp : P.rowp;
    a.d = d;
    a.ts = ts;
    a.nD = nD;
    a.LB = LB;
    a.m = int(P.m);
    a.batch = int(P.batch);
    a.Atab = p.Atab;
    a.Btab = p.Btab;
    a.Ctab = p.Ctab;
    a.Etab = p.Etab;
    a.PIinv = p.PIinv;
    a.fs_lo = p.fs_lo;
    a.fs_hi = p.fs_hi;
    a.fs_na = na;
    a.fs_div = p.fs_div;
    a.nsub = p.nsub;
    for (int s = 0; s < npen; ++s) {
      a.sub_n[s] = p.sub_n[s];
      a.sub_div[s] = p.sub_div[s];
      a.alpha[s] = p.alpha[s];
    }
    a.boxH = p.boxH;
    a.boxG = p.boxG;
    if (kind == MIX_WHOLE) {
      if (int e_ = P.alloc((void**)&P.maps, 2 * size_t(P.m) * sizeof(int))) return pfft_status(e_);
      a.map_in = P.maps;
      a.map_out = P.maps + P.m;
      if (launch_whole_maps(a, P.rowp.PI, P.maps, P.maps + P.m, 0) != 0) return PFFT_ERR_CUDA;
    }
    // a launch of its own leaves at least two tiles per SM where the lanes of its accesses allow
    const pfft_status st = mix_tile(P, kind, 2048, P.generic_only ? 0 : 2 * P.nsm);
    if (st != PFFT_OK) return st;
  }
  // stage twiddle tables of the register-resident passes, gathered on the
  // device from the FP64-built table: entry (s, k, b) = omega_{Ns R}^(k 2^b)
  std::vector<int> idx;
  std::vector<PassArgs*> fastp;
  for (PassArgs* p : {&P.rowp, &P.colp})
    if (p->fast && (p == &P.rowp || npen >= 1)) fastp.push_back(p);
  std::vector<size_t> base;
  for (PassArgs* p : fastp) {
    const int Rm = P.dtype == PFFT_C64 ? 32 : 16;
    const int lr = Rm == 32 ? 5 : 4;
    base.push_back(idx.size());
    // two pencil axes (fft_fast2.cuh): from span top on, the twiddle of k at
    // span Ns is that of floor(k / top) at span Ns / top (the axes uncoupled)
    const int top = (p == &P.colp && p->nsub == 2) ? p->sub_n[0] : 0;
    int Ns = p->fast_tail;
    for (int s = 0; s < p->fast_nmain; ++s) {
      const bool two = top && Ns >= top;
      const int NsR = (two ? Ns / top : Ns) * Rm;
      for (int k = 0; k < Ns; ++k) {
        const int kk = two ? k / top : k;
        if (P.dtype == PFFT_C64)
          for (int b = 0; b < lr; ++b) idx.push_back(int(((int64_t(kk) << b) % NsR) * (nD / NsR)));
        else
          for (int l = 1; l <= lr; ++l)
            for (int c = 0; c < std::max(1, (1 << l) / 4); ++c)
              idx.push_back(int((Rm >> l) * (int64_t(kk) + int64_t(c) * Ns) % NsR * (nD / NsR)));
      }
      Ns *= Rm;
    }
    while (idx.size() - base.back() < size_t(p->stw_n)) idx.push_back(0);
  }
  // runs of consecutive box slots along each row, for bulk-copy staging
  if (P.rowp.fast && !P.tc && P.rowp.T == 1 && npen >= 1 && (P.m * elem_bytes(P.dtype)) % 16 == 0) {
    std::vector<std::array<int, 4>> runs;
    int maxr = 0;
    bool ok = true;
    std::vector<std::vector<std::array<int, 4>>> per(LB);
    std::vector<i64> y(d);
    auto slot_of = [&](int r, int e) {
      for (int k = 0; k < d; ++k) y[k] = i64(Atab[size_t(r) * ts + k]) + Btab[size_t(e) * ts + k];
      box_reduce(P.H, y.data());
      return box_slot(P.H, y.data());
    };
    const int align = int(16 / elem_bytes(P.dtype));  // elements per 16 bytes
    // maximal element ranges whose gather points differ in the last coordinate
    // alone, by one per element: a row's slots are consecutive along such a range
    // but for one wrap of that coordinate
    std::vector<std::pair<int, int>> ranges;
    for (int e = 0; e < nD; ++e) {
      bool next = e > 0;
      for (int k = 0; next && k < d; ++k)
        next = Btab[size_t(e) * ts + k] == Btab[size_t(e - 1) * ts + k] + (k == d - 1);
      if (next)
        ++ranges.back().second;
      else
        ranges.push_back({e, 1});
    }
    const int Hlast = int(P.H(d - 1, d - 1));
    for (int r = 0; r < LB && ok; ++r) {
      int e0 = 0;  // the run being grown: elements [e0, e) at slots [start, next)
      i64 start = 0, next = -1;
      auto close = [&](int e) {
        const int len = e - e0;
        if (len == 0) return;
        if (e0 % align || start % align || len % align) ok = false;
        per[r].push_back({e0, int(start), len, 0});
      };
      for (const auto& rg : ranges) {
        const int last = (Atab[size_t(r) * ts + d - 1] + Btab[size_t(rg.first) * ts + d - 1]) % Hlast;
        for (int o = 0; o < rg.second;) {  // up to the wrap, then the rest
          const int len = o == 0 ? std::min(rg.second, Hlast - last) : rg.second - o;
          const i64 s = slot_of(r, rg.first + o);
          if (s != next) {
            close(rg.first + o);
            e0 = rg.first + o;
            start = s;
          }
          next = s + len;
          o += len;
        }
      }
      close(nD);
      maxr = std::max<int>(maxr, int(per[r].size()));
      if (maxr > 64 || maxr > P.rowp.nthreads) ok = false;
    }
    if (ok) {
      std::vector<int> flat(size_t(LB) * maxr * 4, 0);
      for (int r = 0; r < LB; ++r)
        for (size_t j = 0; j < per[r].size(); ++j)
          for (int k = 0; k < 4; ++k) flat[(size_t(r) * maxr + j) * 4 + k] = per[r][j][k];
      if (int e_ = P.alloc((void**)&P.runs, flat.size() * sizeof(int))) return pfft_status(e_);
      cudaMemcpy(P.runs, flat.data(), flat.size() * sizeof(int), cudaMemcpyHostToDevice);
      P.rowp.tma = 1;
      // padded workspace-order staging (fft_tma.cuh): 2^lg blocks of one
      // span each, offset so that blocks start 32 / 2^lg banks apart (16-byte
      // multiples for the bulk copies)
      P.rowp.stg_pad = 0;
      if (P.rowp.pi_arith && P.rowp.pi_lg > 0 && P.rowp.pi_lg <= 6 && P.rowp.pi_lspan >= 2) {
        const int esz = int(elem_bytes(P.dtype));
        const int pad = std::max(16, 128 >> P.rowp.pi_lg) / esz;  // elements
        const int nel = P.rowp.T * P.rowp.L;
        const int stage_end = nel + (1 << P.rowp.pi_lg) * pad;
        if (stage_end <= P.rowp.stw_smem_off) P.rowp.stg_pad = pad;  // fits before the stage table
      }
      P.rowp.runs = P.runs;
      P.rowp.nruns = maxr;
      P.rowp.bar_smem_off = (P.rowp.smem_bytes + 15) & ~15;
      P.rowp.smem_bytes = P.rowp.bar_smem_off + 16;
      // rows of 2^14 complex64 elements: the persistent pipelined row pass,
      // shared memory [S: the row + staging pads | X: exchange | stage table | mbarrier]
      if (P.dtype == PFFT_C64 && P.rowp.L == (1 << kPipeLogL) && P.rowp.nthreads == 512 &&
          P.rowp.fast_tail == 16 && P.rowp.fast_nmain == 2) {
        const int nblk = P.rowp.stg_pad ? (1 << P.rowp.pi_lg) : 1;
        const int s_el = P.rowp.L + nblk * P.rowp.stg_pad;
        const int x_off = (s_el + 15) & ~15;
        const int stw_off = (x_off + kPipeX + 15) & ~15;
        const int bar_off = ((stw_off + P.rowp.stw_n) * 8 + 15) & ~15;
        if (bar_off + 16 <= 227 * 1024) {
          // outputs stored from registers: the workspace when the permutation
          // multiplier is 1 and lanes form runs of >= 4 elements (32 B); the
          // box when every row is made of runs of one power-of-two length >= 32
          int direct = 0, lrun = 0;
          if (P.rowp.pi_arith && P.rowp.pi_inv == 1 && P.rowp.pi_lg <= 3) direct |= 1;
          for (int l = 5; l <= kPipeLogL && !(direct & 2); ++l) {
            bool uni = maxr == (1 << (kPipeLogL - l));
            for (int r = 0; r < LB && uni; ++r) {
              uni = per[r].size() == size_t(maxr);
              for (size_t j = 0; j < per[r].size() && uni; ++j)
                uni = per[r][j][0] == int(j) << l && per[r][j][2] == 1 << l;
            }
            if (uni) {
              direct |= 2;
              lrun = l;
            }
          }
          P.rowp.pipe_direct = direct;
          P.rowp.pipe_lrun = lrun;
          P.rowp.pipe = 1;
          P.rowp.pipe_x_off = x_off;
          P.rowp.pipe_grid = P.nsm;
          P.rowp.stw_smem_off = stw_off;
          P.rowp.bar_smem_off = bar_off;
          P.rowp.smem_bytes = bar_off + 16;
        }
      }
    }
  }
  // pencils of 2^10 complex64 points, 8 per tile, or 2^11, 4 per tile (one cycle, or
  // two of 64 x 32; forward only): the persistent pipelined column passes
  const bool cpipe10 = npen == 1 && P.colp.L == (1 << kCPipeLogL) && P.colp.T == 8 && P.colp.fast_tail == 1;
  const bool cpipe11 = (npen == 1 || (npen == 2 && P.pen[0] == 64)) && P.colp.L == 2 << kCPipeLogL && P.colp.T == 4 &&
                       P.colp.fast_tail == 2;
  if ((cpipe10 || cpipe11) && P.dtype == PFFT_C64 && !P.tc && P.colp.fast && P.colp.LB == P.colp.L &&
      P.colp.nthreads == 256 && P.colp.fast_nmain == 2 && (d == 2 || d == 3) && P.nD % P.colp.T == 0) {
    const int e_off = kCPipeS + kCPipeX;  // 2 x 8 column points of up to 4 int32: 32 elements
    const int stw_off = e_off + 32;
    const int bytes = (stw_off + P.colp.stw_n) * 8;
    if (bytes <= 110 * 1024) {
      P.colp.cpipe = 1;
      P.colp.cpipe_x_off = kCPipeS;
      P.colp.cpipe_e_off = e_off;
      P.colp.cpipe_grid = 2 * P.nsm;
      P.colp.stw_smem_off = stw_off;
      P.colp.smem_bytes = bytes;
    }
  }
  int* didx = nullptr;
  int rc = 0;
  if (!idx.empty()) {
    if (int e_ = device_alloc((void**)&didx, idx.size() * sizeof(int))) return pfft_status(e_);
    if (int e_ = P.alloc(&P.stw, idx.size() * eb)) {
      cudaFree(didx);
      return pfft_status(e_);
    }
    cudaMemcpy(didx, idx.data(), idx.size() * sizeof(int), cudaMemcpyHostToDevice);
    rc = launch_twiddle_gather(P.stw, P.tw, didx, int(idx.size()), P.dtype, 0);
    for (size_t i = 0; i < fastp.size(); ++i)
      fastp[i]->stw_g = static_cast<const char*>(P.stw) + base[i] * eb;
  }
  // Every table above is built or copied on the default stream.  The first call
  // may come on a stream that does not wait for that one (cudaStreamNonBlocking),
  // so the host does, after the last of them.
  const cudaError_t ce = cudaDeviceSynchronize();
  if (didx) cudaFree(didx);
  return rc == 0 && ce == cudaSuccess ? PFFT_OK : PFFT_ERR_CUDA;
}

pfft_status pfft::plan_retile(pfft_plan_s& P, int row_budget, int col_budget, int max2) {
  if (!P.generic_only || P.tc || P.D == 0 || (max2 != 16 && max2 != 8)) return PFFT_ERR_ARG;
  P.max2 = max2;
  for (int kind = 0; kind < 3; ++kind) {
    if (!P.mixed[kind]) continue;
    const pfft_status st = mix_tile(P, kind, kind == MIX_COL ? col_budget : row_budget, 0);
    if (st != PFFT_OK) return st;
  }
  return PFFT_OK;
}

void pfft::plan_release(pfft_plan_s* P) {
  if (!P) return;
  if (P->tr) {
    P->tr->ws = nullptr;  // this plan's workspace
    plan_release(P->tr);
  }
  if (!P->arena) {
    for (void* p : {(void*)P->dtab, P->tw, P->tw_col, P->ws, P->stw, P->fs_tab, (void*)P->runs, (void*)P->status,
                    (void*)P->maps})
      if (p) cudaFree(p);
    for (auto& by_max2 : P->stages)
      for (auto& S : by_max2)
        for (void* p : {S.stw, (void*)S.gtab, (void*)S.psin, (void*)S.psout})
          if (p) cudaFree(p);
  }
  delete P;
}
static void release(pfft_plan_s* P) { plan_release(P); }
static pfft_status plan_route(pfft_plan_s& P, int d, const int64_t* M, unsigned flags);

extern "C" pfft_status pfft_plan_create(pfft_plan* out, int d, const int64_t* M, int64_t batch,
                                        int dtype, unsigned flags) {
  if (!out || !M || batch < 1 || batch > 65535 || (dtype != PFFT_C64 && dtype != PFFT_C128) ||
      (flags & ~unsigned(PFFT_FLAG_TC_SPLIT | PFFT_FLAG_LAYOUT_SNF | PFFT_FLAG_AUTOTUNE | PFFT_FLAG_TRANSPOSED)) ||
      d < 1 || d > 4)
    return PFFT_ERR_ARG;
  if ((flags & PFFT_FLAG_TC_SPLIT) && dtype != PFFT_C64) return PFFT_ERR_UNSUPPORTED;
  *out = nullptr;
  pfft_plan_s* P = new (std::nothrow) pfft_plan_s;
  if (!P) return PFFT_ERR_OOM;
  P->batch = batch;
  P->dtype = dtype;
  if (flags & PFFT_FLAG_TC_SPLIT) {
    P->tc = true;
    P->generic_only = true;
  }
  pfft_status st;
  try {
    if (flags & PFFT_FLAG_LAYOUT_SNF) {
      // Smith-coordinate layout: by Theorem 1 the transform of M in Smith
      // coordinates is the plain d-dimensional DFT of sizes eps_1 .. eps_d,
      // i.e. the transform of diag(eps) in the box layout, whose box order is
      // the row-major order of lambda (input) and mu (output).
      IMat A(d), Q, R, U, V;
      std::vector<i64> eps;
      for (int i = 0; i < d * d; ++i) {
        if (M[i] >= (int64_t(1) << 24) || M[i] <= -(int64_t(1) << 24)) throw LatticeError{PFFT_ERR_OVERFLOW, "entry"};
        A.a[i] = M[i];
      }
      if (determinant(A) == 0) throw LatticeError{PFFT_ERR_SINGULAR, "singular"};
      smith_normal_form(A, Q, eps, R, U, V);
      std::vector<int64_t> D(size_t(d) * d, 0);
      for (int i = 0; i < d; ++i) D[size_t(i) * d + i] = eps[i];
      st = plan_host(*P, d, D.data());
    } else {
      st = plan_host(*P, d, M);
    }
    if (st == PFFT_OK && P->m * batch >= (int64_t(1) << 40)) st = PFFT_ERR_OVERFLOW;
    if (st == PFFT_OK) st = plan_device(*P);
  } catch (const LatticeError& e) {
    st = pfft_status(e.code);
  }
  if (st == PFFT_OK && (flags & (PFFT_FLAG_AUTOTUNE | PFFT_FLAG_TRANSPOSED))) st = plan_route(*P, d, M, flags);
  if (st != PFFT_OK) {
    release(P);
    return st;
  }
  *out = P;
  return PFFT_OK;
}

extern "C" pfft_status pfft_plan_destroy(pfft_plan p) {
  if (!p) return PFFT_ERR_ARG;
  release(p);
  return PFFT_OK;
}

extern "C" pfft_status pfft_plan_route(pfft_plan p, int* fwd, int* inv) {
  if (!p) return PFFT_ERR_ARG;
  if (fwd) *fwd = p->tr && p->tr_fwd ? 1 : 0;
  if (inv) *inv = p->tr && p->tr_inv ? 1 : 0;
  return PFFT_OK;
}

extern "C" pfft_status pfft_plan_info(pfft_plan p, int64_t* m, int* dM, int64_t* eps, int64_t* in_box,
                                      int64_t* out_box) {
  if (!p) return PFFT_ERR_ARG;
  if (m) *m = p->m;
  if (dM) *dM = p->D;
  for (int i = 0; i < p->d; ++i) {
    if (eps) eps[i] = p->eps[i];
    if (in_box) in_box[i] = p->H(i, i);
    if (out_box) out_box[i] = p->G(i, i);
  }
  return PFFT_OK;
}

extern "C" pfft_status pfft_index_map(pfft_plan p, int which, int64_t* coords) {
  if (!p || !coords) return PFFT_ERR_ARG;
  const int d = p->d;
  std::vector<i64> v(d);
  for (i64 s = 0; s < p->m; ++s) {
    switch (which) {
      case PFFT_MAP_INPUT_BOX:
        box_point(p->H, s, coords + s * d);
        break;
      case PFFT_MAP_OUTPUT_BOX:
        box_point(p->G, s, coords + s * d);
        break;
      case PFFT_MAP_INPUT_SNF:
      case PFFT_MAP_OUTPUT_SNF: {
        const bool in = which == PFFT_MAP_INPUT_SNF;
        box_point(in ? p->H : p->G, s, v.data());
        for (int j = 0; j < p->D; ++j) {
          i128 acc = 0;
          for (int c = 0; c < d; ++c) acc += (i128)(in ? p->LAM[j][c] : p->MU[j][c]) * v[c];
          coords[s * p->D + j] = posmod(i64(acc % p->n[j]), p->n[j]);
        }
        break;
      }
      default:
        return PFFT_ERR_ARG;
    }
  }
  return PFFT_OK;
}

extern "C" pfft_status pfft_device_index_map(pfft_plan p, int which, int64_t* slots, void* stream) {
  if (!p || !slots || (which != PFFT_MAP_INPUT_BOX && which != PFFT_MAP_OUTPUT_BOX)) return PFFT_ERR_ARG;
  if (p->D == 0) {
    int64_t zero = 0;
    return cudaMemcpyAsync(slots, &zero, sizeof(zero), cudaMemcpyHostToDevice, (cudaStream_t)stream) ==
                   cudaSuccess
               ? PFFT_OK
               : PFFT_ERR_CUDA;
  }
  PassArgs a = p->rowp;
  return launch_index_probe(a, a, which == PFFT_MAP_INPUT_BOX ? 0 : 1, slots, (cudaStream_t)stream) == 0
             ? PFFT_OK
             : PFFT_ERR_CUDA;
}

// One pass of plan t (kind: row, column or whole tiles), its time recorded under P.
static pfft_status run_pass(pfft_plan_s* P, const pfft_plan_s* t, int kind, int load, int store, int cin, int cout,
                            double scale, const void* in, void* out, cudaStream_t s) {
  const int which = kind == MIX_COL ? 1 : 0;
  if (t->mixed[kind]) {
    MixDesc a = t->mix[kind];
    mix_sides(a, load, store);
    a.conj_in = cin;
    a.conj_out = cout;
    a.scale = scale;
    a.in = in;
    a.out = out;
    P->prof.begin(which, s);
    if ((P->dtype == PFFT_C64 ? launch_mixed_c64(a, s) : launch_mixed_c128(a, s)) != 0) return PFFT_ERR_CUDA;
    P->prof.end(which, s);
    return PFFT_OK;
  }
  PassArgs a = kind == MIX_COL ? t->colp : t->rowp;
  // Bulk copies start on 16 bytes.  The planner checked the rows' offsets inside a
  // signal; a caller's array that starts 8 bytes past such an address (a slice of a
  // tensor) is read and written element by element, by the kernel that rows
  // without whole runs take.  Its exchange, L + L / 32 elements, ends before the
  // stage table of either layout.
  if (a.tma && ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15)) a.tma = a.pipe = 0;
  a.load_mode = load;
  a.store_mode = store;
  a.conj_in = cin;
  a.conj_out = cout;
  a.scale = scale;
  a.in = in;
  a.out = out;
  P->prof.begin(which, s);
  if (launch_pass(a, P->dtype, s) != 0) return PFFT_ERR_CUDA;
  P->prof.end(which, s);
  return PFFT_OK;
}

// The transform of p through the plan t = p->tr of M^T (see pfft_plan_s::tr):
// forward = t's adjoint passes without conjugations, inverse = t's forward
// passes with conjugated input and output.  Kernel time is recorded under p.
static pfft_status transform_transposed(pfft_plan p, const void* in, void* out, cudaStream_t s, bool inverse) {
  pfft_plan_s* t = p->tr;
  const double scale = 1.0 / std::sqrt(double(p->m));
  const int c = inverse ? 1 : 0;
  if (t->pen.empty() || t->mixed[MIX_WHOLE]) {
    return run_pass(p, t, t->mixed[MIX_WHOLE] ? MIX_WHOLE : MIX_ROW, inverse ? MAP_BOX_H : MAP_BOX_G,
                    inverse ? MAP_BOX_G : MAP_BOX_H, c, c, scale, in, out, s);
  }
  if (inverse) {
    pfft_status st = run_pass(p, t, MIX_ROW, MAP_BOX_H, MAP_WS, 1, 0, 1.0, in, t->ws, s);
    if (st != PFFT_OK) return st;
    return run_pass(p, t, MIX_COL, MAP_WS, MAP_BOX_G, 0, 1, scale, t->ws, out, s);
  }
  pfft_status st = run_pass(p, t, MIX_COL, MAP_BOX_G, MAP_WS, 0, 0, 1.0, in, t->ws, s);
  if (st != PFFT_OK) return st;
  return run_pass(p, t, MIX_ROW, MAP_WS, MAP_BOX_H, 0, 0, scale, t->ws, out, s);
}

static pfft_status transform_route(pfft_plan p, const void* in, void* out, cudaStream_t s, bool inverse,
                                   bool via_tr) {
  const double scale = 1.0 / std::sqrt(double(p->m));
  if (p->D == 0) {
    const size_t bytes = size_t(p->batch) * elem_bytes(p->dtype);
    return cudaMemcpyAsync(out, in, bytes, cudaMemcpyDeviceToDevice, s) == cudaSuccess ? PFFT_OK
                                                                                       : PFFT_ERR_CUDA;
  }
  if (via_tr) return transform_transposed(p, in, out, s, inverse);
  const int ci = inverse ? 1 : 0;
  if (p->pen.empty() || p->mixed[MIX_WHOLE]) {
    return run_pass(p, p, p->mixed[MIX_WHOLE] ? MIX_WHOLE : MIX_ROW, inverse ? MAP_BOX_G : MAP_BOX_H,
                    inverse ? MAP_BOX_H : MAP_BOX_G, ci, ci, scale, in, out, s);
  }
  if (!inverse) {
    pfft_status st = run_pass(p, p, MIX_ROW, MAP_BOX_H, MAP_WS, 0, 0, 1.0, in, p->ws, s);
    if (st != PFFT_OK) return st;
    return run_pass(p, p, MIX_COL, MAP_WS, MAP_BOX_G, 0, 0, scale, p->ws, out, s);
  }
  pfft_status st = run_pass(p, p, MIX_COL, MAP_BOX_G, MAP_WS, 1, 0, 1.0, in, p->ws, s);
  if (st != PFFT_OK) return st;
  return run_pass(p, p, MIX_ROW, MAP_WS, MAP_BOX_H, 0, 1, scale, p->ws, out, s);
}

static pfft_status transform(pfft_plan p, const void* in, void* out, void* stream, bool inverse) {
  if (!p || !in || !out || in == out) return PFFT_ERR_ARG;
  const bool via_tr = p->tr && (inverse ? p->tr_inv : p->tr_fwd);
  return transform_route(p, in, out, (cudaStream_t)stream, inverse, via_tr);
}

// Mean time (ms) of one direction by one route over `reps` calls on stream s;
// negative when a call fails.
static float time_route(pfft_plan_s* p, bool inverse, bool via_tr, const void* in, void* out, cudaStream_t s,
                        int reps) {
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    if (e0) cudaEventDestroy(e0);
    cudaGetLastError();
    return -1.0f;
  }
  float ms = -1.0f;
  bool ok = transform_route(p, in, out, s, inverse, via_tr) == PFFT_OK;  // warm-up
  ok = ok && cudaEventRecord(e0, s) == cudaSuccess;
  for (int r = 0; ok && r < reps; ++r) ok = transform_route(p, in, out, s, inverse, via_tr) == PFFT_OK;
  ok = ok && cudaEventRecord(e1, s) == cudaSuccess && cudaEventSynchronize(e1) == cudaSuccess &&
       cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (!ok) {
    cudaStreamSynchronize(s);
    cudaGetLastError();
    return -1.0f;
  }
  return ms / float(reps);
}

// PFFT_FLAG_TRANSPOSED / PFFT_FLAG_AUTOTUNE: plan M^T beside M (same batch and
// precision, this plan's workspace and status word) and route the directions
// through it, always (TRANSPOSED) or where it measures faster (AUTOTUNE: each
// direction timed both ways on zeroed scratch buffers; the transposed route
// must win by 3%).  Plans of the Smith layout or the split-precision form,
// and transposed plans whose row pass is the pipelined kernel (which runs
// only with the conjugations of its own directions), keep the direct route:
// PFFT_ERR_UNSUPPORTED under TRANSPOSED, silently under AUTOTUNE.
static pfft_status plan_route(pfft_plan_s& P, int d, const int64_t* M, unsigned flags) {
  const bool force = (flags & PFFT_FLAG_TRANSPOSED) != 0;
  const pfft_status no = force ? PFFT_ERR_UNSUPPORTED : PFFT_OK;
  if (P.tc || (flags & PFFT_FLAG_LAYOUT_SNF) || P.D == 0) return no;
  std::vector<int64_t> Mt(size_t(d) * d);
  for (int i = 0; i < d; ++i)
    for (int j = 0; j < d; ++j) Mt[size_t(i) * d + j] = M[size_t(j) * d + i];
  pfft_plan_s* T = new (std::nothrow) pfft_plan_s;
  if (!T) return PFFT_ERR_OOM;
  T->batch = P.batch;
  T->dtype = P.dtype;
  T->own_workspace = false;
  pfft_status st;
  try {
    st = plan_host(*T, d, Mt.data());
    if (st == PFFT_OK) st = plan_device(*T);
  } catch (const LatticeError& e) {
    st = pfft_status(e.code);
  }
  if (st == PFFT_OK && (T->rowp.pipe || T->pen.size() != P.pen.size() || T->mixed[MIX_WHOLE] != P.mixed[MIX_WHOLE])) st = PFFT_ERR_UNSUPPORTED;
  if (st != PFFT_OK) {
    plan_release(T);
    return force ? st : PFFT_OK;
  }
  T->ws = P.ws;
  T->rowp.status = T->colp.status = P.status;
  P.tr = T;
  if (force) {
    P.tr_fwd = P.tr_inv = true;
    return PFFT_OK;
  }
  // AUTOTUNE: time both routes of each direction
  const size_t bytes = size_t(P.m) * size_t(P.batch) * elem_bytes(P.dtype);
  void *a = nullptr, *b = nullptr;
  cudaStream_t s = nullptr;
  bool ok = cudaMalloc(&a, bytes) == cudaSuccess && cudaMalloc(&b, bytes) == cudaSuccess &&
            cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) == cudaSuccess &&
            cudaMemsetAsync(a, 0, bytes, s) == cudaSuccess;
  if (ok) {
    const int reps = 3;
    for (int inv = 0; inv < 2; ++inv) {
      const float direct = time_route(&P, inv != 0, false, a, b, s, reps);
      const float via = time_route(&P, inv != 0, true, a, b, s, reps);
      const bool use = direct > 0.0f && via > 0.0f && via < 0.97f * direct;
      (inv ? P.tr_inv : P.tr_fwd) = use;
    }
    cudaStreamSynchronize(s);
  }
  cudaGetLastError();
  if (s) cudaStreamDestroy(s);
  if (a) cudaFree(a);
  if (b) cudaFree(b);
  if (!P.tr_fwd && !P.tr_inv) {
    T->ws = nullptr;
    plan_release(T);
    P.tr = nullptr;
  }
  return PFFT_OK;
}

extern "C" pfft_status pfft_forward(pfft_plan p, const void* in, void* out, void* stream) {
  return transform(p, in, out, stream, false);
}

extern "C" pfft_status pfft_inverse(pfft_plan p, const void* in, void* out, void* stream) {
  return transform(p, in, out, stream, true);
}

static const char* kPassNames[] = {"row_pass", "col_pass"};

extern "C" pfft_status pfft_profile_enable(pfft_plan p, int enable) {
  if (!p) return PFFT_ERR_ARG;
  return p->prof.enable(enable != 0, 2, kPassNames) ? PFFT_OK : PFFT_ERR_CUDA;
}

extern "C" pfft_status pfft_profile_read(pfft_plan p, const char** names, int64_t* launches, double* ms,
                                         int cap, int* n) {
  if (!p) return PFFT_ERR_ARG;
  return p->prof.read(names, launches, ms, cap, n) ? PFFT_OK : PFFT_ERR_CUDA;
}

extern "C" pfft_status pfft_set_wait_limit(pfft_plan p, int64_t spins) {
  if (!p) return PFFT_ERR_ARG;
  if (!p->rowp.tma) return PFFT_ERR_UNSUPPORTED;
  const uint32_t lim = spins < 0 ? kSpinLimit : uint32_t(std::min<int64_t>(spins, int64_t(UINT32_MAX)));
  p->rowp.spin_limit = lim;
  if (p->tr) p->tr->rowp.spin_limit = lim;
  return PFFT_OK;
}

extern "C" pfft_status pfft_last_device_status(pfft_plan p, void* stream) {
  if (!p) return PFFT_ERR_ARG;
  if (!p->status) return PFFT_OK;
  int v = 0;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemcpyAsync(&v, p->status, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return PFFT_ERR_CUDA;
  if (v != 0) cudaMemsetAsync(p->status, 0, sizeof(int), s);
  return pfft_status(v);
}
