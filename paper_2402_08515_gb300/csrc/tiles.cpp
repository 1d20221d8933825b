// Host side of the staged step kernels (kernels_tile.cu): rows are taken in tiles whose columns
// lie in a few contiguous runs of rows, and the runs, the entries' places in them and the order
// of the matrix values are laid out here, once per context.
#include <algorithm>
#include <atomic>
#include <map>
#include <new>

#include "kes_internal.h"

namespace kes {
namespace {

constexpr int kAlign = 4;  // rows: a run of FP32 values starts and ends on 16 bytes
constexpr int kGap = 8;    // runs closer than this many rows are one

struct Run {
  int32_t start, len, dst;
};

// Runs of the ascending, aligned ranges [a, b): merged across small gaps.
void add_range(std::vector<Run>& runs, int32_t a, int32_t b) {
  a = a >= 0 ? a / kAlign * kAlign : -((-a + kAlign - 1) / kAlign * kAlign);
  b = b >= 0 ? (b + kAlign - 1) / kAlign * kAlign : -(-b / kAlign * kAlign);
  if (!runs.empty() && a <= runs.back().start + runs.back().len + kGap) {
    runs.back().len = std::max(runs.back().len, b - runs.back().start);
    return;
  }
  runs.push_back({a, b - a, 0});
}
int32_t place_runs(std::vector<Run>& runs) {
  int32_t at = 0;
  for (Run& r : runs) {
    r.dst = at;
    at += r.len;
  }
  return at;
}
int32_t find_row(const std::vector<Run>& runs, int32_t row) {
  size_t lo = 0, hi = runs.size() - 1;
  while (lo < hi) {
    const size_t mid = (lo + hi + 1) / 2;
    if (runs[mid].start <= row) lo = mid;
    else hi = mid - 1;
  }
  return runs[lo].dst + (row - runs[lo].start);
}

// Ascending union of the column - row differences of a group of slices; empty where the group
// keeps an index instead: a row without its own column (the folded diagonal would land on
// padding), a difference that leads some row out of the mesh, or more than an eighth of zeros.
void group_pattern(const TileInput& in, const TileGroup& g, int64_t lo, int64_t hi, std::vector<int32_t>& pat,
                   std::vector<int32_t>& tmp) {
  pat.clear();
  for (int64_t i = 0; i < g.rows; ++i) {
    const int64_t row = g.row0 + i, s = row / kSliceC, l = row % kSliceC;
    const int32_t n = in.len[row];
    if (n == 0) continue;
    const int32_t* cs = in.col + in.slice_ptr[s] + l;
    size_t at = 0;
    int32_t k = 0;
    bool own = false;
    for (; k < n; ++k) {  // the common case: the row's differences are all in the list
      const int32_t d = static_cast<int32_t>(cs[k * kSliceC] - row);
      own |= d == 0;
      while (at < pat.size() && pat[at] < d) ++at;
      if (at == pat.size() || pat[at] != d) break;
    }
    if (k < n) {
      tmp.clear();
      at = 0;
      own = false;
      for (k = 0; k < n; ++k) {
        const int32_t d = static_cast<int32_t>(cs[k * kSliceC] - row);
        own |= d == 0;
        while (at < pat.size() && pat[at] < d) tmp.push_back(pat[at++]);
        if (at < pat.size() && pat[at] == d) ++at;
        tmp.push_back(d);
      }
      tmp.insert(tmp.end(), pat.begin() + at, pat.end());
      pat.swap(tmp);
    }
    if (!own || static_cast<int64_t>(pat.size()) > g.w + g.w / 8) {
      pat.clear();
      return;
    }
  }
  if (!pat.empty() && (g.row0 + pat.front() < lo || g.row0 + g.rows - 1 + pat.back() >= hi)) pat.clear();
}

}  // namespace

int64_t quad_pos(int64_t w, int64_t k, int64_t lane) {
  const int64_t body = w & ~int64_t(3);
  if (k < body) return (k >> 2) * 4 * kSliceC + 4 * lane + (k & 3);
  if (!(w & 2)) return body * kSliceC + lane;
  return body * kSliceC + (k - body < 2 ? 2 * lane + (k - body) : 2 * kSliceC + lane);
}

bool build_tile_groups(const TileInput& in, TileLayout& out) {
  out.groups.clear();
  for (int j = 0; j < in.n_mesh; ++j)
    for (int64_t r = 0; r < in.mesh_rows[j]; r += kTileGroup) {
      TileGroup g;
      g.row0 = in.mesh_row0[j] + r;
      g.rows = static_cast<int>(std::min<int64_t>(kTileGroup, in.mesh_rows[j] - r));
      g.mesh = j;
      out.groups.push_back(g);
    }
  const int64_t ng = static_cast<int64_t>(out.groups.size());
  std::vector<std::vector<int32_t>> pats(ng);
  int64_t padded = 0, stored = 0;
  // an exception must not leave a thread of a parallel region: it would end the process
  std::atomic<bool> no_memory{false};
#pragma omp parallel
  {
    std::vector<int32_t> tmp;
#pragma omp for schedule(dynamic, 64) reduction(+ : padded, stored)
    for (int64_t i = 0; i < ng; ++i) {
      TileGroup& g = out.groups[i];
      const int64_t s0 = g.row0 / kSliceC, s1 = s0 + g.rows / kSliceC;
      int64_t w = 0;
      for (int64_t s = s0; s < s1; ++s) w = std::max(w, (in.slice_ptr[s + 1] - in.slice_ptr[s]) / kSliceC);
      stored += in.slice_ptr[s1] - in.slice_ptr[s0];
      if (w > kMaxTileWidth) {
        padded += int64_t(1) << 40;
        continue;
      }
      g.w = static_cast<int>(w);
      g.kind = 1;
      if (w > 0) {
        try {
          group_pattern(in, g, in.mesh_row0[g.mesh], in.mesh_row0[g.mesh] + in.mesh_rows[g.mesh], pats[i], tmp);
        } catch (const std::bad_alloc&) {
          no_memory = true;
          pats[i].clear();
        }
      }
      if (!pats[i].empty()) {
        g.kind = 0;
        g.w = static_cast<int>(pats[i].size());
      }
      padded += static_cast<int64_t>(g.w) * g.rows;
    }
  }
  if (no_memory) throw std::bad_alloc();
  // groups of uneven rows would be padded to their longest one: not worth staging
  if (padded > stored + stored / 8) return false;
  std::map<std::vector<int32_t>, int> known;
  int64_t beg = 0;
  for (int64_t i = 0; i < ng; ++i) {
    TileGroup& g = out.groups[i];
    g.beg = beg;
    beg += static_cast<int64_t>(g.w) * (g.rows / kSliceC);
    if (g.kind != 0) continue;
    auto it = known.find(pats[i]);
    if (it == known.end()) {
      it = known.emplace(pats[i], static_cast<int>(out.patterns.size())).first;
      out.patterns.push_back(pats[i]);
    }
    g.pattern = it->second;
    pats[i].clear();
    pats[i].shrink_to_fit();
  }
  if (beg >= (int64_t(1) << 31)) return false;
  out.n_values = beg * kSliceC;
  // per slice, for the kernel that writes the values: place, width, pattern
  out.slice_rec.assign(in.n_slices, int4{0, 0, 0, 0});
  out.pat.clear();
  std::vector<int32_t> at;
  for (const auto& p : out.patterns) {
    at.push_back(static_cast<int32_t>(out.pat.size()));
    out.pat.insert(out.pat.end(), p.begin(), p.end());
  }
  if (out.pat.empty()) out.pat.push_back(0);
  for (const TileGroup& g : out.groups)
    for (int64_t s = g.row0 / kSliceC, q = 0; q < g.rows / kSliceC; ++s, ++q)
      out.slice_rec[s] = int4{static_cast<int>(g.beg + q * g.w), g.w, g.kind, g.kind == 0 ? at[g.pattern] : 0};
  return true;
}

bool build_tiles(const TileInput& in, const TileLayout& lay, int R, TileHost& out) {
  out = TileHost{};
  out.R = R;
  // the runs of a pattern's tile, counted from the tile's first row
  struct PatRuns {
    std::vector<Run> runs;
    std::vector<int32_t> base;
    int xrows = 0, own = 0;
  };
  std::map<std::pair<int, int>, PatRuns> of;  // (pattern, rows)
  struct Tile {
    const TileGroup* g;
    int64_t row0;
    int rows;
  };
  std::vector<Tile> tiles;
  for (const TileGroup& g : lay.groups)
    for (int r = 0; r < g.rows; r += R) tiles.push_back({&g, g.row0 + r, std::min(R, g.rows - r)});
  const int64_t nt = static_cast<int64_t>(tiles.size());
  if (nt >= (int64_t(1) << 31)) return false;
  // index tiles: their runs on their own; where each tile's head goes (16 bytes)
  std::vector<std::vector<Run>> runs_of(nt);
  std::vector<int64_t> head_at(nt + 1, 0);
  for (int64_t t = 0; t < nt; ++t) {
    const TileGroup& g = *tiles[t].g;
    head_at[t + 1] = head_at[t] + 2 + (g.kind == 1 ? int64_t(2) * g.w * tiles[t].rows / 16 : (g.w + 3) / 4);
  }
  if (head_at[nt] >= (int64_t(1) << 31)) return false;
  out.head.assign(head_at[nt], int4{0, 0, 0, 0});
  std::atomic<bool> fits{true}, no_memory{false};
  // the runs and places of an index tile; false: its columns are too scattered
  auto index_tile = [&](int64_t t, std::vector<int32_t>& blocks) {
    const Tile& tl = tiles[t];
    blocks.clear();
    int32_t last = -1;
    for (int i = 0; i < tl.rows; ++i) {
      const int64_t row = tl.row0 + i;
      const int32_t* cs = in.col + in.slice_ptr[row / kSliceC] + row % kSliceC;
      for (int32_t k = 0; k < in.len[row]; ++k) {
        const int32_t b = cs[k * kSliceC] / kAlign;
        if (b != last) blocks.push_back(b);
        last = b;
      }
    }
    for (int i = 0; i < tl.rows; i += kAlign) blocks.push_back(static_cast<int32_t>((tl.row0 + i) / kAlign));
    std::sort(blocks.begin(), blocks.end());
    blocks.erase(std::unique(blocks.begin(), blocks.end()), blocks.end());
    std::vector<Run>& runs = runs_of[t];
    for (int32_t b : blocks) add_range(runs, b * kAlign, (b + 1) * kAlign);
    const int32_t xrows = place_runs(runs);
    if (static_cast<int>(runs.size()) > kMaxRuns || xrows > kMaxStagedRows) return false;
    const int w = tl.g->w;
    for (int i = 0; i < tl.rows; ++i) {
      const int64_t row = tl.row0 + i;
      const int32_t* cs = in.col + in.slice_ptr[row / kSliceC] + row % kSliceC;
      uint16_t* dst =
          reinterpret_cast<uint16_t*>(&out.head[head_at[t] + 2]) + static_cast<int64_t>(i / kSliceC) * w * kSliceC;
      const int32_t own = find_row(runs, static_cast<int32_t>(row));
      for (int k = 0; k < w; ++k)
        dst[quad_pos(w, k, i % kSliceC)] =
            static_cast<uint16_t>(k < in.len[row] ? find_row(runs, cs[k * kSliceC]) : own);
    }
    return true;
  };
#pragma omp parallel
  {
    std::vector<int32_t> blocks;
#pragma omp for schedule(dynamic, 64)
    for (int64_t t = 0; t < nt; ++t) {
      if (tiles[t].g->kind != 1 || !fits || no_memory) continue;  // one tile that does not fit settles it
      try {
        if (!index_tile(t, blocks)) fits = false;
      } catch (const std::bad_alloc&) {
        no_memory = true;
      }
    }
  }
  if (no_memory) throw std::bad_alloc();
  if (!fits) return false;
  std::vector<const PatRuns*> pat_of(nt, nullptr);
  for (int64_t t = 0; t < nt; ++t) {
    const TileGroup& g = *tiles[t].g;
    if (g.kind == 0) {
      const auto key = std::make_pair(g.pattern, tiles[t].rows);
      auto it = of.find(key);
      if (it == of.end()) {
        PatRuns p;
        const auto& pat = lay.patterns[g.pattern];
        for (int32_t d : pat) add_range(p.runs, d, d + tiles[t].rows);
        p.xrows = place_runs(p.runs);
        if (static_cast<int>(p.runs.size()) > kMaxRuns || p.xrows > kMaxStagedRows) return false;
        for (int32_t d : pat) p.base.push_back(find_row(p.runs, d));
        p.own = find_row(p.runs, 0);
        it = of.emplace(key, p).first;
      }
      pat_of[t] = &it->second;
    }
    const auto& runs = g.kind == 0 ? pat_of[t]->runs : runs_of[t];
    out.max_runs = std::max(out.max_runs, static_cast<int>(runs.size()));
  }
  out.seg.assign(static_cast<size_t>(nt) * (out.max_runs + 2), int4{0, 0, 0, 0});
  for (int64_t t = 0; t < nt; ++t) {
    const Tile& tl = tiles[t];
    const TileGroup& g = *tl.g;
    const auto& runs = g.kind == 0 ? pat_of[t]->runs : runs_of[t];
    const int32_t from = g.kind == 0 ? static_cast<int32_t>(tl.row0) : 0;
    int4* slot = &out.seg[static_cast<size_t>(t) * (out.max_runs + 2)];
    for (size_t i = 0; i < runs.size(); ++i) slot[i] = int4{runs[i].start + from, runs[i].len, runs[i].dst, 0};
    slot[out.max_runs] = int4{static_cast<int>(tl.row0), tl.rows, 0, 0};
    const int xrows = runs.back().dst + runs.back().len;
    const int own = g.kind == 0 ? pat_of[t]->own : find_row(runs, static_cast<int32_t>(tl.row0));
    const int64_t beg = g.beg + (tl.row0 - g.row0) / kSliceC * g.w;
    const int64_t units = head_at[t + 1] - head_at[t];
    slot[out.max_runs + 1] = int4{static_cast<int>(beg), tl.rows * g.w, static_cast<int>(head_at[t]), static_cast<int>(16 * units)};
    int4* head = &out.head[head_at[t]];
    head[0] = int4{g.w, g.kind, 0, 0};
    head[1] = int4{static_cast<int>(tl.row0), tl.rows, g.mesh, own};
    if (g.kind == 0) std::copy(pat_of[t]->base.begin(), pat_of[t]->base.end(), reinterpret_cast<int32_t*>(head + 2));
    out.max_xrows = std::max(out.max_xrows, xrows);
    out.max_w = std::max(out.max_w, g.w);
    out.max_head = std::max(out.max_head, static_cast<int>(16 * units));
  }
  return true;
}

}  // namespace kes
