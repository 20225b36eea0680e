// Planner of the block contraction (block.cu): turns the products of blocks
// that a contraction sums into output blocks, segments and tiles.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>

#include "../../include/symtensor.h"
#include "plan.h"

namespace sym {

namespace {

void strides_of(const Tensor& T, int64_t s, int64_t* st) {
  int64_t acc = 1;
  for (int l = T.rank - 1; l >= 0; --l) {
    st[l] = acc;
    acc *= T.dim(s, l);
  }
}

// A group of dims of one output block (its row legs, say): sizes, strides in
// the output and, per segment, strides in the operand.  merge() drops unit
// dims and joins neighbours that are contiguous everywhere.
struct Dims {
  std::vector<int64_t> d, o;
  std::vector<std::vector<int64_t>> s;  // [dim][segment]
  void push(int64_t dim, int64_t ostr, std::vector<int64_t> sstr) {
    if (dim == 1) return;
    if (!d.empty() && o.back() == ostr * dim) {
      bool ok = true;
      for (size_t j = 0; j < sstr.size(); ++j) ok = ok && s.back()[j] == sstr[j] * dim;
      if (ok) {
        d.back() *= dim;
        o.back() = ostr;
        s.back() = std::move(sstr);
        return;
      }
    }
    d.push_back(dim);
    o.push_back(ostr);
    s.push_back(std::move(sstr));
  }
};

// The dims right-aligned in kBlkDims slots (the last one fastest); false if there are too many.
bool pack(const Dims& x, int32_t* sizes, uint32_t* mag, int* shf, int32_t* ostr) {
  const int n = (int)x.d.size(), off = kBlkDims - n;
  if (n > kBlkDims) return false;
  for (int i = 0; i < kBlkDims; ++i) ostr[i] = i >= off ? (int32_t)x.o[i - off] : 0;
  *shf = 0;
  for (int i = 1; i < kBlkDims; ++i) {
    sizes[i - 1] = i >= off ? (int32_t)x.d[i - off] : 1;
    int8_t s;
    div_magic(sizes[i - 1], mag[i - 1], s);
    *shf |= (int)(uint8_t)s << (8 * (i - 1));
  }
  return true;
}

// Modelled cost of a tile in SM clocks at full occupancy (throughput) and
// alone (latency), from the kernel's own counts: FP32 128 multiply-adds a
// clock at about half rate for the 8 x 4 microtile and less for the smaller
// ones, FP64 two operations a clock, multiply-adds and the products with the
// coefficients alike, over the live part of the tile; a slab's round trip
// about 700 clocks; 2500 clocks of set-up and stores, shared by the CTAs of an SM.
// FP32 products with coefficients count in the two large shapes, which multiply-adds
// bound; the small one waits for its loads (with a quarter more there too, an SU(2)
// recoupling contraction that takes 150 us on the blocks went to its matrix form, 209).
// kModelScale: measured over modelled time, 1.5 to 1.6 on the contractions of
// the U(1) and SU(2) x U(1) MPS step (D = 2048, 1024) and of the MERA patch;
// FP64 0.9 to 1.2 (those steps, D = 128 to 1500, and SU(2) recoupling contractions).
constexpr double kModelScale = 1.55, kModelScale64 = 1.1;
struct Cost {
  double thr, lat;
};
Cost tile_cost(bool f64, int shape, int64_t m, int64_t n, int64_t k, bool coef) {
  const int TM = blk_rows(f64, shape), TN = blk_cols(f64, shape);
  const double slabs = std::ceil((double)k / blk_slab(f64, shape));
  if (shape == BLK_DOT) {
    const double step = std::max(180.0, 40.0 + 12.0 * (double)(m + n) + (f64 ? 64.0 : 1.0) * (double)(m * n));
    return {step * slabs + 500.0, std::max(step, 900.0) * slabs + 2500.0};
  }
  if (f64) {
    const int64_t gm = shape == BLK_TALL ? 64 : 8, gn = shape == BLK_TALL ? 2 : 16;
    const double lm = (double)(std::min<int64_t>(TM, m + gm - 1) / gm), ln = (double)(std::min<int64_t>(TN, n + gn - 1) / gn);
    const double fma = 64.0 * (lm * ln + (coef ? ln : 0.0)) * (double)k * 1.1;  // four warps' operations, 16 clocks each
    return {fma + 500.0, fma + slabs * 700.0 + 2500.0};
  }
  const double fma = (coef && shape <= BLK_MID ? 1.25 : 1.0) * (double)TM * TN * (double)k / 128.0 /
                     (shape == BLK_BIG ? 0.6 : shape == BLK_MID ? 0.5 : shape == BLK_SMALL ? 0.35 : 0.16);
  return {fma + slabs * 60.0 + 500.0, std::max(fma, slabs * 700.0) + 2500.0};
}

}  // namespace

// The best rates tile_cost knows: 76.8 multiply-adds a clock of an SM in FP32
// (BLK_BIG), below 2 in FP64; whole tiles and latencies only add to that.
double block_floor_us(bool f64, double fma) {
  return (f64 ? kModelScale64 : kModelScale) * fma / (f64 ? 2.0 : 76.8) / 152.0 / 1900.0;
}

double blk_tile_cost(bool f64, const BlkTile& t) {
  const int64_t ks = blk_slab(f64, t.shape);
  return tile_cost(f64, t.shape, t.ob.m - t.r0, t.ob.n - t.c0, std::min<int64_t>(t.ob.ktot, t.s1 * ks) - t.s0 * ks,
                   (t.ob.flags & kBlkCoef) != 0)
      .lat;
}

bool plan_block_phase(Plan& P, int phase, const Tensor& A, const Tensor& B, const Tensor& C,
                      const std::vector<BlkTriple>& triples, const std::vector<int>& freeA,
                      const std::vector<int>& freeB, const std::vector<int>& pairsA, const std::vector<int>& pairsB,
                      double share, double* model_us) {
  const bool f64 = P.f64();
  const int na = (int)freeA.size(), nb = (int)freeB.size(), nc = (int)pairsA.size();
  // tensors and legs of the phase: out legs shared with P (x) and with Q (y),
  // contracted legs z; the result's legs are C = [free A, free B]
  const Tensor &O = phase == 0 ? C : phase == 1 ? A : B, &Pt = phase == 2 ? A : phase == 1 ? C : A,
               &Qt = phase == 2 ? C : B;
  const int p_slot = phase == 1 ? 2 : 0, q_slot = phase == 2 ? 2 : 1;
  const int o_slot = phase == 0 ? DST_OUT : phase == 1 ? DST_DA : DST_DB;
  std::vector<std::pair<int, int>> xo, yo, z;  // (out leg, P leg), (out leg, Q leg), (P leg, Q leg)
  if (phase == 0) {
    for (int i = 0; i < na; ++i) xo.push_back({i, freeA[i]});
    for (int i = 0; i < nb; ++i) yo.push_back({na + i, freeB[i]});
    for (int i = 0; i < nc; ++i) z.push_back({pairsA[i], pairsB[i]});
  } else if (phase == 1) {  // dA = dC B^T
    for (int i = 0; i < na; ++i) xo.push_back({freeA[i], i});
    for (int i = 0; i < nc; ++i) yo.push_back({pairsA[i], pairsB[i]});
    for (int i = 0; i < nb; ++i) z.push_back({na + i, freeB[i]});
  } else {  // dB = A^T dC
    for (int i = 0; i < nc; ++i) xo.push_back({pairsB[i], pairsA[i]});
    for (int i = 0; i < nb; ++i) yo.push_back({freeB[i], na + i});
    for (int i = 0; i < na; ++i) z.push_back({freeA[i], i});
  }
  std::sort(xo.begin(), xo.end());
  std::sort(yo.begin(), yo.end());
  // walk the reduction along whichever operand has its last leg in it
  const bool by_q = !std::any_of(z.begin(), z.end(), [&](auto& l) { return l.first == Pt.rank - 1; });
  std::sort(z.begin(), z.end(), [&](auto& l, auto& r) { return by_q ? l.second < r.second : l.first < r.first; });

  // products grouped by output block
  const int64_t no = O.nsec();
  auto ido = [&](const BlkTriple& t) { return phase == 0 ? t.c : phase == 1 ? t.a : t.b; };
  auto idp = [&](const BlkTriple& t) { return phase == 1 ? t.c : t.a; };
  auto idq = [&](const BlkTriple& t) { return phase == 2 ? t.c : t.b; };
  std::vector<int64_t> first(no + 1, 0);
  for (auto& t : triples) ++first[ido(t) + 1];
  for (int64_t s = 0; s < no; ++s) first[s + 1] += first[s];
  std::vector<const BlkTriple*> by(triples.size());
  {
    std::vector<int64_t> at(first.begin(), first.end() - 1);
    for (auto& t : triples) by[at[ido(t)]++] = &t;
  }
  std::vector<BlkOut> outs;
  std::vector<BlkSeg> segs;
  const int64_t lim = (int64_t)1 << 31;
  if (A.numel() >= lim || B.numel() >= lim || C.numel() >= lim) return false;  // 32-bit offsets in the kernel
  const int seg_base = (int)P.bsegs.size(), out_base = (int)P.bouts.size();
  struct Choice {
    int64_t m, n, k;
    bool coef;
  };
  std::vector<Choice> sizes;
  int64_t so[kMaxDim], sp[kMaxDim], sq[kMaxDim];
  for (int64_t s = 0; s < no; ++s) {
    const int nseg = (int)(first[s + 1] - first[s]);
    strides_of(O, s, so);
    Dims X, Y;
    std::vector<std::vector<int64_t>> xs(xo.size(), std::vector<int64_t>(nseg)), ys(yo.size(), std::vector<int64_t>(nseg));
    std::vector<BlkSeg> ss(nseg);
    int64_t k0 = 0;
    bool pk = false, qk = false;
    for (int j = 0; j < nseg; ++j) {
      const BlkTriple& t = *by[first[s] + j];
      const int64_t ip = idp(t), iq = idq(t);
      strides_of(Pt, ip, sp);
      strides_of(Qt, iq, sq);
      for (size_t i = 0; i < xo.size(); ++i) xs[i][j] = sp[xo[i].second];
      for (size_t i = 0; i < yo.size(); ++i) ys[i][j] = sq[yo[i].second];
      Dims K;
      for (auto& l : z) K.push(Pt.dim(ip, l.first), sp[l.first], {sq[l.second]});
      BlkSeg& g = ss[j];
      g = BlkSeg{};
      int shf;
      int32_t ostr[kBlkDims];
      if (!pack(K, g.kd, g.kmag, &shf, ostr)) return false;
      g.kshf = shf;
      int64_t kn = 1;
      const int off = kBlkDims - (int)K.d.size();
      for (int i = 0; i < kBlkDims; ++i) {
        g.pk[i] = i >= off ? (int32_t)K.o[i - off] : 0;
        g.qk[i] = i >= off ? (int32_t)K.s[i - off][0] : 0;
        if (i >= off) kn *= K.d[i - off];
        if (i >= off && (K.o[i - off] >= lim || K.s[i - off][0] >= lim)) return false;
      }
      if (j == 0 && !K.d.empty()) {
        pk = K.o.back() == 1;
        qk = K.s.back()[0] == 1;
      }
      g.p_off = Pt.offs[ip];
      g.q_off = Qt.offs[iq];
      g.coef = t.coef;
      g.coef_f = (float)t.coef;
      g.k0 = (int)k0;
      g.kn = (int)kn;
      k0 += kn;
      if (k0 >= lim || Pt.block_size(ip) >= lim || Qt.block_size(iq) >= lim) return false;
    }
    int64_t m = 1, n = 1;
    for (size_t i = 0; i < xo.size(); ++i) {
      const int64_t d = O.dim(s, xo[i].first);
      m *= d;
      X.push(d, so[xo[i].first], xs[i]);
    }
    for (size_t i = 0; i < yo.size(); ++i) {
      const int64_t d = O.dim(s, yo[i].first);
      n *= d;
      Y.push(d, so[yo[i].first], ys[i]);
    }
    if (O.block_size(s) >= lim) return false;
    // columns: the narrow side if there is one, else the side with the output's contiguous leg
    const bool x_last = !X.o.empty() && X.o.back() == 1;
    const bool swap = n > 8 && (m <= 8 || x_last);
    BlkOut b{};
    b.off = O.offs[s];
    b.m = (int)(swap ? n : m);
    b.n = (int)(swap ? m : n);
    b.ktot = (int)k0;
    b.seg0 = seg_base + (int)segs.size();
    b.nseg = nseg;
    b.slots = (swap ? q_slot : p_slot) | ((swap ? p_slot : q_slot) << 2) | (o_slot << 4);
    b.flags = ((swap ? qk : pk) ? kBlkPk : 0) | ((swap ? pk : qk) ? kBlkQk : 0);
    int rs, cs;
    if (!pack(swap ? Y : X, b.rd, b.rmag, &rs, b.ro) || !pack(swap ? X : Y, b.cd, b.cmag, &cs, b.co)) return false;
    b.shf = rs | (cs << 16);
    const Dims &R = swap ? Y : X, &Cc = swap ? X : Y;
    for (int j = 0; j < nseg; ++j) {
      BlkSeg& g = ss[j];
      if (g.coef != 1.0) b.flags |= kBlkCoef;
      if (swap) {
        std::swap(g.p_off, g.q_off);
        for (int i = 0; i < kBlkDims; ++i) std::swap(g.pk[i], g.qk[i]);
      }
      const int ro = kBlkDims - (int)R.d.size(), co = kBlkDims - (int)Cc.d.size();
      for (int i = 0; i < kBlkDims; ++i) {
        g.pr[i] = i >= ro ? (int32_t)R.s[i - ro][j] : 0;
        g.qc[i] = i >= co ? (int32_t)Cc.s[i - co][j] : 0;
      }
      segs.push_back(g);
    }
    outs.push_back(b);
    sizes.push_back({b.m, b.n, k0, (b.flags & kBlkCoef) != 0});
  }
  // tile shapes: the cheapest per block, or only the small ones when the
  // launch would otherwise end on a few long tiles
  const double nsm = 152.0;
  double best = 0.0;
  int best_mode = -1;
  double target = 0.0;  // clocks a unit of work may take before it is cut
  auto shape_of = [&](const Choice& c, int mode) {
    int pick = BLK_SMALL;
    double cost = 1e300;
    for (int sh = 0; sh < BLK_SHAPES; ++sh) {
      if (sh < BLK_SMALL && mode == 1) continue;
      if (sh == BLK_TALL && c.n > 8) continue;
      if (sh == BLK_DOT && (c.m > 8 || c.n > 8 || c.k < 512)) continue;
      const int64_t TM = blk_rows(f64, sh), TN = blk_cols(f64, sh);
      // interior tiles, the right and bottom edges, the corner
      const int64_t fm = c.m / TM, fn = c.n / TN, em = c.m % TM, en = c.n % TN;
      double t = 0.0;
      if (fm && fn) t += (double)(fm * fn) * tile_cost(f64, sh, TM, TN, c.k, c.coef).thr;
      if (fm && en) t += (double)fm * tile_cost(f64, sh, TM, en, c.k, c.coef).thr;
      if (em && fn) t += (double)fn * tile_cost(f64, sh, em, TN, c.k, c.coef).thr;
      if (em && en) t += tile_cost(f64, sh, em, en, c.k, c.coef).thr;
      if (t < cost || (t == cost && sh <= BLK_SMALL)) {  // equal for a block within one tile in FP64: the fewer loads
        cost = t;
        pick = sh;
      }
    }
    return pick;
  };
  for (int mode = 0; mode < 2; ++mode) {
    double thr = 0.0, plain = 0.0, lat = 0.0, count = 0.0;
    std::vector<std::pair<double, double>> units;  // (throughput clocks, tiles)
    for (auto& c : sizes) {
      const int sh = shape_of(c, mode);
      const int64_t TM = blk_rows(f64, sh), TN = blk_cols(f64, sh);
      const double full = (double)(c.m / TM) * (double)(c.n / TN);
      const Cost f = tile_cost(f64, sh, TM, TN, c.k, c.coef), e = tile_cost(f64, sh, std::min(c.m, TM), std::min(c.n, TN), c.k, c.coef);
      const double all = (double)((c.m + TM - 1) / TM) * (double)((c.n + TN - 1) / TN);
      thr += f.thr * full + (all - full) * e.thr;
      plain += tile_cost(f64, sh, TM, TN, c.k, false).thr * full +
               (all - full) * tile_cost(f64, sh, std::min(c.m, TM), std::min(c.n, TN), c.k, false).thr;
      lat = std::max(lat, (full > 0 ? f : e).lat);
      units.push_back({f.thr, full});
      units.push_back({e.thr, all - full});
      count += all;
    }
    // an SM's share of this phase; in a batch too, where the largest problem's tiles
    // end the launch (eight two-site problems of 256 <= D <= 1024: 721 us, 747 with the
    // share of eight such problems)
    const double cut = std::max(thr / nsm, 6000.0);
    // the clocks of the busiest SM: tiles go out longest first, one to each SM in
    // turn.  With few tiles -- in FP64, where a few hundred fill the pipe, with
    // more -- that is up to twice the average (an SU(2) recoupling contraction
    // with 172 tiles took 240 us; three sectors of 512 x 512 x 512 in FP32, 192
    // tiles, 65 us a phase where the tensor cores take 25)
    double busy = thr / nsm;
    if (share == 1.0 && (f64 || count < 2.0 * nsm)) {
      for (auto& u : units)
        if (u.first > 2.0 * cut) u = {cut, u.second * u.first / cut};  // cut along its reduction
      std::sort(units.begin(), units.end(), [](auto& a, auto& b) { return a.first > b.first; });
      double next = 0.0, seen = 0.0, first = 0.0;
      for (auto& u : units)
        for (seen += u.second; next < seen; next += nsm) first += u.first;
      if (f64 || first > 24000.0) busy = std::max(busy, first);  // shorter tiles in FP32: the latency covers it
    }
    lat = std::min(lat, 2.0 * cut) * share;  // longer tiles are cut along their reductions
    auto model = [&](double t) {
      return (f64 ? kModelScale64 : kModelScale) * (std::max(t, lat) + 0.3 * std::min(t, lat)) / 1900.0 + 3.0 * share;
    };
    const double us = model(thr / nsm);
    if (best_mode < 0 || us < best) {
      best = us;
      best_mode = mode;
      target = std::max(plain / nsm, 6000.0);
      *model_us = model(busy);
    }
  }
  struct Unit {
    double cost;
    BlkTile t;
    int out;
  };
  std::vector<Unit> tiles;
  // dA's and dB's parts lie side by side (one launch), the forward's in the same place
  const int64_t first_unit = phase == 2 ? P.blk_end : 0;
  const int64_t unit_bytes = kBlkThreads * (f64 ? 8 : 4);
  const int64_t max_units = (int64_t)((double)(kBlkWorkspace / 2) * share) / unit_bytes;
  int64_t units = 0;
  int counters = 0;
  for (size_t i = 0; i < sizes.size(); ++i) {
    const Choice& c = sizes[i];
    const int sh = shape_of(c, best_mode);
    const int TM = blk_rows(f64, sh), TN = blk_cols(f64, sh), KS = blk_slab(f64, sh);
    const int slabs = (int)((c.k + KS - 1) / KS);
    for (int r = 0; r < c.m; r += TM)
      for (int q = 0; q < c.n; q += TN) {
        BlkTile t{};
        t.ob = outs[i];
        t.r0 = r;
        t.c0 = q;
        t.shape = sh;
        // a tile much longer than the launch's share of an SM is cut along its reduction.
        // Both without the coefficients: tiles of one size are cut alike (100 tiles of an
        // FP64 step, 75 of them with signs: 66 us with the 25 others whole, 39 with all cut)
        const double lat = tile_cost(f64, sh, c.m - r, c.n - q, c.k, false).lat;
        int parts = 1;
        if (lat > 2.0 * target) parts = (int)std::min({std::ceil(lat / target), std::max(1.0, slabs / 4.0), 512.0});
        if (units + (int64_t)parts * blk_values(f64, sh) > max_units) parts = 1;
        const int per = parts > 1 ? (slabs + parts - 1) / parts : slabs;
        parts = per > 0 ? (slabs + per - 1) / per : 1;
        for (int p = 0; p < parts; ++p) {
          t.s0 = p * per;
          t.s1 = std::min(slabs, (p + 1) * per);
          t.part = p | (parts << 16);
          t.ws = (int)(first_unit + units);
          t.cnt = P.blk_counters + counters;
          // the segments that meet [s0, s1)
          const BlkSeg* sg = segs.data() + (outs[i].seg0 - seg_base);
          int j0 = 0, j1 = outs[i].nseg;
          while (j0 + 1 < outs[i].nseg && sg[j0 + 1].k0 <= t.s0 * KS) ++j0;
          while (j1 > j0 + 1 && (int64_t)sg[j1 - 1].k0 >= (int64_t)t.s1 * KS) --j1;
          t.ob.seg0 = outs[i].seg0 + j0;
          t.ob.nseg = j1 - j0;
          tiles.push_back({blk_tile_cost(f64, t), t, out_base + (int)i});
        }
        if (parts > 1) {
          units += (int64_t)parts * blk_values(f64, sh);
          ++counters;
        }
      }
    if (tiles.size() > ((size_t)1 << 22)) return false;
  }
  // longest first: the tail of the launch is then made of short tiles
  std::stable_sort(tiles.begin(), tiles.end(), [](auto& a, auto& b) { return a.cost > b.cost; });
  P.bsegs.insert(P.bsegs.end(), segs.begin(), segs.end());
  P.bouts.insert(P.bouts.end(), outs.begin(), outs.end());
  P.blk_range[phase] = {(int)P.btiles.size(), (int)tiles.size()};
  for (auto& t : tiles) {
    P.btiles.push_back(t.t);
    P.btile_out.push_back(t.out);
  }
  P.blk_end = first_unit + units;
  P.blk_units = std::max(P.blk_units, P.blk_end);
  P.blk_counters += counters;
  P.blk_bytes[phase] = (f64 ? 8.0 : 4.0) * ((double)A.numel() + (double)B.numel() + (double)C.numel());
  return true;
}

void drop_blocks(Plan& P) {
  P.bouts.clear();
  P.bsegs.clear();
  P.btiles.clear();
  P.btile_out.clear();
  P.blk_mnk.clear();
  P.blk_units = P.blk_end = 0;
  P.blk_counters = 0;
  P.blocks = false;
  for (int ph = 0; ph < 3; ++ph) {
    P.blk_range[ph] = Range{};
    P.blk_bytes[ph] = P.blk_flops[ph] = 0.0;
  }
}

// Every element that a tile can touch lies inside its tensor: the extreme
// offsets of every block and segment against the tensors' sizes, and every
// reduction's segments end to end.
void validate_blocks(const Plan& P) {
  const int64_t ne[3] = {P.numel_a, P.numel_b, P.numel_c};
  const int64_t lim = (int64_t)1 << 31;
  if (!P.btiles.empty() && std::max({ne[0], ne[1], ne[2]}) >= lim)
    fail(SYM_ERR_UNSUPPORTED, "internal: block contraction of tensors beyond 2^31 elements");
  auto bad = [](const char* what) { fail(SYM_ERR_ARG, std::string("internal: block contraction ") + what); };
  for (int ph = 0; ph < 3; ++ph)
    if (P.blk_range[ph].first < 0 || P.blk_range[ph].count < 0 ||
        (size_t)P.blk_range[ph].first + P.blk_range[ph].count > P.btiles.size())
      bad("tile range");
  auto sides = [&](int ext, const int32_t* d, const uint32_t* mag, int shf, int* size) {
    for (int i = 0; i < kBlkDims - 1; ++i) {
      uint32_t m;
      int8_t s;
      if (d[i] < 1) bad("dim");
      div_magic(d[i], m, s);
      if (m != mag[i] || s != (int8_t)((shf >> (8 * i)) & 0xff)) bad("division constants");
      size[i + 1] = d[i];
    }
    const int64_t inner = (int64_t)d[0] * d[1];
    if (ext < 1 || ext % inner) bad("extent");
    size[0] = (int)(ext / inner);
  };
  auto span = [&](const int* size, const int32_t* st) {
    int64_t r = 0;
    for (int i = 0; i < kBlkDims; ++i) {
      if (st[i] < 0) bad("stride");
      r += (int64_t)(size[i] - 1) * st[i];
    }
    return r;
  };
  auto slot_size = [&](int s) { return s >= 0 && s < 3 ? ne[s] : (int64_t)-1; };
  for (const BlkOut& b : P.bouts) {
    const int ps = b.slots & 3, qs = (b.slots >> 2) & 3, os = (b.slots >> 4) & 7;
    const int64_t no = os == DST_OUT ? ne[2] : os == DST_DA ? ne[0] : os == DST_DB ? ne[1] : -1;
    int rs[kBlkDims], cs[kBlkDims], ks[kBlkDims];
    sides(b.m, b.rd, b.rmag, b.shf, rs);
    sides(b.n, b.cd, b.cmag, b.shf >> 16, cs);
    const int64_t os_ = span(rs, b.ro) + span(cs, b.co);
    if (b.off < 0 || os_ >= lim || b.off + os_ >= no) bad("writes past its tensor");
    if (b.nseg < 0 || b.seg0 < 0 || (size_t)b.seg0 + b.nseg > P.bsegs.size()) bad("segment range");
    int64_t k = 0;
    for (int j = 0; j < b.nseg; ++j) {
      const BlkSeg& g = P.bsegs[b.seg0 + j];
      sides(g.kn, g.kd, g.kmag, g.kshf, ks);
      if (g.k0 != k) bad("segments apart");
      k += g.kn;
      const int64_t pp = span(rs, g.pr) + span(ks, g.pk), qq = span(cs, g.qc) + span(ks, g.qk);
      if (g.p_off < 0 || g.q_off < 0 || pp >= lim || qq >= lim || g.p_off + pp >= slot_size(ps) ||
          g.q_off + qq >= slot_size(qs))
        bad("reads past its tensor");
    }
    if (k != b.ktot || k >= lim) bad("reduction length");
  }
  if (P.btile_out.size() != P.btiles.size()) bad("tile owners");
  for (size_t i = 0; i < P.btiles.size(); ++i) {
    const BlkTile& t = P.btiles[i];
    if (P.btile_out[i] < 0 || (size_t)P.btile_out[i] >= P.bouts.size() || t.shape < 0 || t.shape >= BLK_SHAPES)
      bad("tile");
    const BlkOut& b = P.bouts[P.btile_out[i]];
    BlkOut same = t.ob;
    same.seg0 = b.seg0;
    same.nseg = b.nseg;
    if (std::memcmp(&b, &same, sizeof(b)) != 0) bad("tile's copy of its block");
    if (t.ob.seg0 < b.seg0 || t.ob.nseg < 0 || t.ob.seg0 + t.ob.nseg > b.seg0 + b.nseg) bad("tile's segments");
    if (b.nseg > 0) {
      const BlkSeg &g0 = P.bsegs[t.ob.seg0], &g1 = P.bsegs[t.ob.seg0 + std::max(t.ob.nseg, 1) - 1];
      const int64_t ks = blk_slab(P.f64(), t.shape), k0 = t.s0 * ks, k1 = std::min<int64_t>(b.ktot, t.s1 * ks);
      if (t.ob.nseg < 1 || g0.k0 > k0 || g1.k0 + g1.kn < k1) bad("tile's segments");
    }
    const int part = t.part & 0xffff, nparts = t.part >> 16;
    const int slabs = (b.ktot + blk_slab(P.f64(), t.shape) - 1) / blk_slab(P.f64(), t.shape);
    if (t.r0 < 0 || t.c0 < 0 || t.r0 >= b.m || t.c0 >= b.n || t.r0 % blk_rows(P.f64(), t.shape) ||
        t.c0 % blk_cols(P.f64(), t.shape) || t.s0 < 0 || t.s1 < t.s0 || t.s1 > slabs || part < 0 || part >= nparts)
      bad("tile range");
    if (t.shape == BLK_DOT && (b.m > 8 || b.n > 8)) bad("output too wide for a dot");
    if (nparts == 1 ? (t.s0 != 0 || t.s1 != slabs)
                    : (t.ws < 0 || t.ws + (int64_t)nparts * blk_values(P.f64(), t.shape) > P.blk_units || t.cnt < 0 ||
                       t.cnt >= P.blk_counters))
      bad("tile parts");
  }
}

}  // namespace sym
