// Host tables of the pre-summed de-dispersion (dedisperse_presum.cu).
//
// Channels of each group are taken in units of K = 2^presum adjacent channels
// c0 .. c0 + n - 1 (n = K, fewer at the end of a group).  The unit's reference
// is its last channel e = c0 + n - 1, the highest in frequency and so the
// least delayed (Sec. 1: the delay falls with frequency).  For trial i the
// unit contributes
//   S_rel[t + d(i, e)],   S_rel[u] = sum_j x[c0 + j][u + rel_j],
//   rel_j = d(i, c0 + j) - d(i, e) >= 0   (rel_{n-1} = 0),
// so one series serves every trial with the same tuple rel.  Each series is
// stored twice, copy 1 shifted by one sample, so that a trial whose reference
// delay d is odd reads aligned words of copy 1 at d - 1.  The plan needs:
//   series : every (unit, rel) any trial uses, as rows of the workspace, with
//            the sample range its trials read for outputs t < n_out:
//            [min d', max d' + n_out), d' = the reference delay rounded down
//            to even (copy 1 at d - 1 holds the samples from d on);
//   chunks : per (DM tile, group), its units in order, as many per chunk as fit
//            a shared-memory stage (windows differ in length and number over the
//            band, so a chunk holds more units where they are small); where the
//            wide tile's folds would otherwise be too many, chunks end where its
//            lanes are full;
//   copies : per chunk, the windows of series copies the tile reads -- one per
//            (tuple, parity of d) that occurs, each just long enough for its
//            trials -- packed back to back in the stage: {row, start, (stage
//            byte / 16) | (bytes / 16) << 16, 0}, and last {count, total bytes,
//            units, offset table / 8 entries};
//   offs   : per chunk, at the start of its stage, per (unit, trial) the offset
//            of the trial's first sample inside the stage, in 4-byte words as
//            uint16 (a stage is well below 256 KiB), so that one vector load
//            fetches a warp's offsets for a unit.
// Tiles start at multiples of 64 samples, so nothing depends on the time tile.
#include <algorithm>
#include <array>
#include <vector>

#include "sps_internal.h"

namespace sps {
namespace {

using Rel = std::array<int32_t, 3>;

struct Unit {
  int32_t c0, n;
};

Unit unit_of(int32_t g, int32_t u, int32_t per, int32_t K) {
  return {g * per + K * u, std::min(K, per - K * u)};
}

int32_t ref_delay(const std::vector<int32_t>& d, int32_t C, int32_t i, Unit un) {
  return d[(size_t)i * C + un.c0 + un.n - 1];
}

Rel rel_of(const std::vector<int32_t>& d, int32_t C, int32_t i, Unit un) {
  Rel r{0, 0, 0};
  const int32_t* row = &d[(size_t)i * C];
  for (int32_t j = 0; j + 1 < un.n; j++) r[j] = row[un.c0 + j] - row[un.c0 + un.n - 1];
  return r;
}

// Distinct tuples of one unit over rows [i0, i1], in sorted order.  (Neighbouring
// trials mostly share theirs.)
std::vector<Rel> distinct_rels(const std::vector<int32_t>& d, int32_t C, int32_t i0, int32_t i1, Unit un) {
  std::vector<Rel> v;
  Rel last{-1, -1, -1};
  for (int32_t i = i0; i <= i1; i++) {
    const Rel r = rel_of(d, C, i, un);
    if (r == last && i > i0) continue;
    last = r;
    const auto at = std::lower_bound(v.begin(), v.end(), r);
    if (at == v.end() || *at != r) v.insert(at, r);
  }
  return v;
}

int32_t index_of(const std::vector<Rel>& v, const Rel& r) {
  return (int32_t)(std::lower_bound(v.begin(), v.end(), r) - v.begin());
}

// The copy windows one unit needs in one DM tile of rows [i0, i1]: for tuple
// k of `rels` and parity j, the trials' smallest and largest even-rounded
// reference delay.  Window = [lo rounded down to 8, hi + Tt) samples.
struct TileCopy {
  int32_t k, j, lo, hi;
};

std::vector<TileCopy> tile_copies(const std::vector<int32_t>& d, int32_t C, int32_t i0, int32_t i1, Unit un,
                                  const std::vector<Rel>& rels) {
  std::vector<TileCopy> out;
  for (int32_t i = i0; i <= i1; i++) {
    const int32_t k = rels.size() == 1 ? 0 : index_of(rels, rel_of(d, C, i, un));
    const int32_t de = ref_delay(d, C, i, un), j = de & 1, e = de & ~1;
    size_t q = 0;
    while (q < out.size() && (out[q].k != k || out[q].j != j)) q++;
    if (q == out.size()) {
      out.push_back({k, j, e, e});
    } else {
      out[q].lo = std::min(out[q].lo, e);
      out[q].hi = std::max(out[q].hi, e);
    }
  }
  std::sort(out.begin(), out.end(), [](const TileCopy& a, const TileCopy& b) {
    return a.k != b.k ? a.k < b.k : a.j < b.j;
  });
  return out;
}

int32_t copy_start(const TileCopy& c) { return c.lo & ~7; }

int32_t copy_bytes(const TileCopy& c, int32_t Tt) { return 2 * ((c.hi - copy_start(c) + Tt + 7) / 8 * 8); }

}  // namespace

int64_t count_presum_series(const std::vector<int32_t>& d, int32_t rows, int32_t C, int32_t per, int32_t K) {
  int64_t n = 0;
  const int32_t U = (per + K - 1) / K;
  for (int32_t g = 0; g < C / per; g++)
    for (int32_t u = 0; u < U; u++) n += (int64_t)distinct_rels(d, C, 0, rows - 1, unit_of(g, u, per, K)).size();
  return n;
}

int32_t presum_stage_data(const std::vector<int32_t>& d, int32_t rows, int32_t C, int32_t per, int32_t K,
                          int32_t Di, int32_t cu, int32_t Tt) {
  const int32_t U = (per + K - 1) / K;
  int64_t best = 0;
  for (int32_t i0 = 0; i0 < rows; i0 += Di) {
    const int32_t i1 = std::min(i0 + Di, rows) - 1;
    for (int32_t g = 0; g < C / per; g++)
      for (int32_t u0 = 0; u0 < U; u0 += cu) {
        int64_t bytes = 0;
        for (int32_t u = u0; u < std::min(u0 + cu, U); u++) {
          const Unit un = unit_of(g, u, per, K);
          for (const TileCopy& c : tile_copies(d, C, i0, i1, un, distinct_rels(d, C, i0, i1, un)))
            bytes += copy_bytes(c, Tt);
        }
        best = std::max(best, bytes);
      }
  }
  return (int32_t)std::min<int64_t>(best, INT32_MAX);
}

sps_status build_presum_tables(const std::vector<int32_t>& d, int32_t rows, int32_t C, int32_t per, int32_t n_out,
                               const sps_dedisp_config& cfg, int32_t stage_bytes, PresumTables* out) {
  const int32_t K = 1 << cfg.presum;
  const int32_t G = C / per;
  const int32_t U = (per + K - 1) / K;
  const int32_t Di = cfg.warps_dm * cfg.dms_per_thread;
  const int32_t Tt = cfg.warps_time * 32 * cfg.samples_per_thread;
  const int32_t di_pad = presum_di_pad(cfg);
  const int32_t most = std::min(presum_fold_units(cfg), std::max(kPresumChunkUnits, presum_chunk(cfg)));
  const int32_t n_tiles = (rows + Di - 1) / Di;
  // The wide tile folds at most kWideFolds times.  A fold comes when the next chunk
  // does not fit the lanes and so moves at least fold - most + 1 units; where that
  // leaves too many, chunks are cut so that each moves `fold` units.
  const int32_t fold = presum_fold_units(cfg);
  const bool wide = presum_wide(cfg.dms_per_thread, cfg.samples_per_thread / 2);
  const bool cut = wide && (U - 1) / (fold - most + 1) > kWideFolds;
  if (wide && (U - 1) / fold > kWideFolds)
    return fail(SPS_ERR_UNSUPPORTED, "more folds than the wide tile's counts hold");

  // series: per unit, every tuple over all trials
  std::vector<int32_t> sbase((size_t)G * U);
  std::vector<std::vector<Rel>> all((size_t)G * U);
  out->series.clear();
  out->units.clear();
  out->max_rel = 0;
  for (int32_t g = 0; g < G; g++)
    for (int32_t u = 0; u < U; u++) {
      const Unit un = unit_of(g, u, per, K);
      std::vector<Rel>& v = all[(size_t)g * U + u];
      v = distinct_rels(d, C, 0, rows - 1, un);
      for (const Rel& r : v)
        if (std::min({r[0], r[1], r[2]}) < 0)
          return fail(SPS_ERR_INVALID_ARG, "a lower channel arrives before a higher one");
      std::vector<int32_t> lo(v.size(), INT32_MAX), hi(v.size(), INT32_MIN);
      for (int32_t i = 0; i < rows; i++) {
        const size_t k = (size_t)index_of(v, rel_of(d, C, i, un));
        const int32_t de = ref_delay(d, C, i, un) & ~1;
        lo[k] = std::min(lo[k], de);
        hi[k] = std::max(hi[k], de);
      }
      sbase[(size_t)g * U + u] = (int32_t)out->series.size();
      int32_t ulo = INT32_MAX, uhi = 0;
      for (size_t k = 0; k < v.size(); k++) {
        const int32_t slo = lo[k] & ~7, shi = (hi[k] + n_out + 7) / 8 * 8;
        out->series.push_back({un.c0, un.n, {v[k][0], v[k][1], v[k][2]}, slo, shi, 0});
        ulo = std::min(ulo, slo);
        uhi = std::max(uhi, shi);
      }
      const int32_t max_rel = v.back()[0];  // tuples sorted: the last has the largest first delay
      out->units.push_back({un.c0, un.n, sbase[(size_t)g * U + u], (int32_t)out->series.size(), max_rel, ulo, uhi,
                            0});
      out->max_rel = std::max(out->max_rel, max_rel);
    }

  // chunks per (tile, group): units taken in order while their windows and
  // offsets fit a stage; the offsets of each trial point at its (tuple, parity)
  // copy in the stage, behind the chunk's offset table
  out->chunk_rows.clear();
  out->copies_max = 0;
  std::vector<std::vector<int4>> lists;
  std::vector<int4> heads;
  for (int32_t tile = 0; tile < n_tiles; tile++) {
    const int32_t i0 = tile * Di, i1 = std::min(i0 + Di, rows) - 1;
    for (int32_t g = 0; g < G; g++) {
      const size_t first = lists.size();
      std::vector<std::vector<Rel>> rels(U);
      std::vector<std::vector<TileCopy>> copies(U);
      std::vector<int32_t> bytes(U, 0);
      for (int32_t u = 0; u < U; u++) {
        const Unit un = unit_of(g, u, per, K);
        rels[u] = distinct_rels(d, C, i0, i1, un);
        copies[u] = tile_copies(d, C, i0, i1, un, rels[u]);
        for (const TileCopy& c : copies[u]) bytes[u] += copy_bytes(c, Tt);
      }
      for (int32_t u0 = 0; u0 < U;) {
        int32_t n = 0, need = 0;
        const int32_t end = cut ? std::min(U, (u0 / fold + 1) * fold) : U;
        while (u0 + n < end && n < most && need + bytes[u0 + n] + 2 * di_pad <= stage_bytes) {
          need += bytes[u0 + n] + 2 * di_pad;
          n++;
        }
        if (n == 0) return fail(SPS_ERR_UNSUPPORTED, "a pre-summed unit's windows exceed a stage");
        if (n > 4 && u0 + n < end) n &= ~1;  // units are added two at a time
        int32_t at = n * 2 * di_pad;  // windows follow the offset table
        lists.emplace_back();
        const size_t table = out->offs.size();
        out->offs.resize(table + (size_t)n * di_pad, 0);
        for (int32_t u = u0; u < u0 + n; u++) {
          const Unit un = unit_of(g, u, per, K);
          std::vector<int32_t> dst(copies[u].size());
          for (size_t q = 0; q < copies[u].size(); q++) {
            const TileCopy& c = copies[u][q];
            const int32_t series = sbase[(size_t)g * U + u] + index_of(all[(size_t)g * U + u], rels[u][c.k]);
            dst[q] = at;
            lists.back().push_back({2 * series + c.j, copy_start(c), (at >> 4) | ((copy_bytes(c, Tt) >> 4) << 16), 0});
            at += copy_bytes(c, Tt);
          }
          for (int32_t r = 0; r < di_pad; r++) {
            const int32_t i = std::min(i0 + std::min(r, Di - 1), rows - 1);
            const int32_t k = index_of(rels[u], rel_of(d, C, i, un));
            const int32_t de = ref_delay(d, C, i, un);
            size_t q = 0;
            while (copies[u][q].k != k || copies[u][q].j != (de & 1)) q++;
            const int64_t word = ((int64_t)dst[q] + 2 * ((de & ~1) - copy_start(copies[u][q]))) / 4;
            if (word > 0xFFFF) return fail(SPS_ERR_UNSUPPORTED, "pre-summed staging window beyond 256 KiB");
            out->offs[table + (size_t)(u - u0) * di_pad + r] = (uint16_t)word;
          }
        }
        heads.push_back({(int32_t)lists.back().size(), at - n * 2 * di_pad, n, (int32_t)(table / 8)});
        out->copies_max = std::max<int32_t>(out->copies_max, (int32_t)lists.back().size());
        u0 += n;
      }
      out->chunk_rows.push_back({(int32_t)first, (int32_t)(lists.size() - first), 0, 0});
    }
  }
  if (stage_bytes >= (1 << 18) || out->copies_max >= (1 << 14))
    return fail(SPS_ERR_UNSUPPORTED, "pre-summed stage beyond 256 KiB or 16383 windows");
  out->stage_bytes = stage_bytes;
  out->copies.assign(lists.size() * (size_t)(out->copies_max + 1), int4{-1, 0, 0, 0});
  for (size_t q = 0; q < lists.size(); q++) {
    int4* row = &out->copies[q * (out->copies_max + 1)];
    std::copy(lists[q].begin(), lists[q].end(), row);
    row[out->copies_max] = heads[q];
  }
  return SPS_OK;
}

// Checks, from the delay table alone, what the pass kernel will read through a
// set of tables: for every trial of every (tile, group, unit), its staged
// offset falls inside one window of its chunk's list, that window holds the
// trial's own series (same unit, same relative delays) in the copy of the
// trial's delay parity, the window's first sample plus the offset is the
// trial's even-rounded reference delay d', the window lies inside the stage's
// data, and the series' written range [lo, hi) covers d' .. d' + read_n_out - 1
// (every sample a valid output reads).  The first failure is described in *why.
bool verify_presum_tables(const std::vector<int32_t>& d, int32_t rows, int32_t C, int32_t per, int32_t read_n_out,
                          const sps_dedisp_config& cfg, const PresumTables& t, std::string* why) {
  const int32_t K = 1 << cfg.presum;
  const int32_t G = C / per;
  const int32_t U = (per + K - 1) / K;
  const int32_t Di = cfg.warps_dm * cfg.dms_per_thread;
  const int32_t Tt = cfg.warps_time * 32 * cfg.samples_per_thread;
  const int32_t di_pad = presum_di_pad(cfg);
  const int32_t n_tiles = (rows + Di - 1) / Di;
  auto say = [&](const char* what, int32_t tile, int32_t g, int32_t u, int32_t r) {
    *why = std::string(what) + " (tile " + std::to_string(tile) + ", group " + std::to_string(g) + ", unit " +
           std::to_string(u) + ", trial " + std::to_string(r) + ")";
    return false;
  };
  for (int32_t tile = 0; tile < n_tiles; tile++)
    for (int32_t g = 0; g < G; g++) {
      const int4 chunks = t.chunk_rows[(size_t)tile * G + g];
      // the folds of a block that sums all chunks (one with a share of them makes no more)
      int32_t folds = 0, pending = 0;
      for (int32_t q = 0; q < chunks.y; q++) {
        const int32_t n = t.copies[((size_t)chunks.x + q) * (t.copies_max + 1) + t.copies_max].z;
        if (pending + n > presum_fold_units(cfg)) {
          folds++;
          pending = 0;
        }
        pending += n;
      }
      // a tile's first chunk holds the units its stage is sized for (an even number from six on)
      const bool wide = presum_wide(cfg.dms_per_thread, cfg.samples_per_thread / 2);
      const int32_t sized = std::min(U, presum_chunk(cfg)), held = t.copies[(size_t)chunks.x * (t.copies_max + 1) + t.copies_max].z;
      if (!wide && held < (sized > 4 ? sized & ~1 : sized))
        return say("fewer units in a chunk than its stage is sized for", tile, g, held, 0);
      if (wide && folds > kWideFolds)
        return say("more folds than the wide tile's counts hold", tile, g, folds, 0);
      int32_t chunk = 0, chunk_u0 = 0;  // the unit's chunk and the chunk's first unit
      for (int32_t u = 0; u < U; u++) {
        const int32_t c0 = g * per + K * u, n = std::min(K, per - K * u), e = c0 + n - 1;
        const int4* list = &t.copies[((size_t)chunks.x + chunk) * (t.copies_max + 1)];
        if (u - chunk_u0 == list[t.copies_max].z) {
          chunk_u0 = u;
          chunk++;
          list += t.copies_max + 1;
        }
        if (chunk >= chunks.y) return say("unit in no chunk", tile, g, u, 0);
        const int32_t count = list[t.copies_max].x, table = list[t.copies_max].z * 2 * di_pad;
        const uint16_t* offs = &t.offs[(size_t)list[t.copies_max].w * 8 + (size_t)(u - chunk_u0) * di_pad];
        int32_t sum = 0;
        for (int32_t q = 0; q < count; q++) sum += ((uint32_t)list[q].z >> 16) * 16;
        if (sum != list[t.copies_max].y) return say("window bytes of a chunk", tile, g, u, 0);
        for (int32_t r = 0; r < Di; r++) {
          const int32_t i = tile * Di + r;
          if (i >= rows) break;
          const int32_t* di = &d[(size_t)i * C];
          const int32_t de = di[e], dprime = de & ~1, parity = de & 1;
          const int64_t off = 4 * (int64_t)offs[r];  // stage bytes
          int32_t q = 0;
          for (; q < count; q++) {
            const int32_t dst = (list[q].z & 0xFFFF) * 16, bytes = ((uint32_t)list[q].z >> 16) * 16;
            if (off >= dst && off + 2 * (int64_t)Tt <= (int64_t)dst + bytes) break;
          }
          if (q == count) return say("offset outside every window of the chunk", tile, g, u, r);
          const int32_t dst = (list[q].z & 0xFFFF) * 16, bytes = ((uint32_t)list[q].z >> 16) * 16;
          if (dst < table || dst + bytes > t.stage_bytes) return say("window beyond the stage data", tile, g, u, r);
          const int32_t srow = list[q].x, s = srow / 2;
          if (srow < 0 || s >= (int32_t)t.series.size()) return say("window row outside the series table", tile, g, u, r);
          if (srow % 2 != parity) return say("window of the wrong alignment copy", tile, g, u, r);
          const PresumSeries& ps = t.series[s];
          if (ps.c0 != c0 || ps.n != n) return say("window of another unit's series", tile, g, u, r);
          for (int32_t j = 0; j + 1 < n; j++)
            if (ps.rel[j] != di[c0 + j] - de) return say("window of a series with other relative delays", tile, g, u, r);
          if (list[q].y + (off - dst) / 2 != dprime) return say("offset does not land on the trial's delay", tile, g, u, r);
          if (dprime < ps.lo || (int64_t)dprime + read_n_out > ps.hi)
            return say("a valid output reads outside the series' written range", tile, g, u, r);
        }
      }
      if (chunk + 1 != chunks.y) return say("chunk without units", tile, g, U, 0);
    }
  return true;
}

}  // namespace sps
