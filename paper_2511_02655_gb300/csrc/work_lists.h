// Layout of the bodies and the work list of the symmetric passes: host code
// without CUDA, so that the lists can be checked for every layout without a GPU.
#pragma once

#include <stdint.h>

#include <algorithm>
#include <vector>

namespace nbody {

// A contiguous run of bodies of one system, the unit of the O(N) kernels and
// of the fixed-order energy reduction.
struct Chunk {
  int32_t sys;
  int32_t begin, end;
  int32_t n_slices;  // partials to combine: slot s of body i is entry row0 + s * stride + i of the partial buffer
  int32_t stride;
  int32_t pad;
  int64_t row0;
};

// Work item of the symmetric force pass (sym_common.cuh): i-bodies [i_begin,
// i_end) of one system (whole i-tiles but for the system's end) against its
// j-bodies [j_begin, j_end), every unordered pair once. Partials of i-bodies go to
// slot slot_i, of j-bodies to slot slot_j (row0 and stride as in Chunk).
struct SymItem {
  int32_t sys;
  int32_t i_begin, i_end;
  int32_t j_begin, j_end;
  int32_t slot_i, slot_j;
  int32_t stride;
  int64_t row0;
};

// The O(N) kernels do their float64 work on GB300's FP64 pipe (about 1/75 of
// the FP32 rate), so that part of their time is the float64 operations per SM: the
// smaller the system, the fewer bodies a chunk has, so that its CTAs cover every
// SM (1024 bodies: 64 CTAs). The rest of the time is the latency of reading each
// body's partials; a combining CTA has several threads per body (slot groups), each
// adding every groups-th slice, so that a body's loads are in flight together.
// Larger systems fill the SMs anyway, and their larger chunks leave fewer chunk
// partials for one CTA to sum into a record.
constexpr int kChunk = 128;  // bodies per chunk at most, and of the staging origin's sums
inline int chunk_bodies(int64_t n_total) {
  return n_total <= 4096 ? 16 : n_total <= 16384 ? 32 : n_total <= 32768 ? 64 : kChunk;
}

struct Tiling {
  int block = 0, ipt = 0, jtile = 0, slice = 0, n_ctas = 0;
  int variant = 0;  // mixed kernels: 0 scalar, 1 packed float32x2, 2 packed with a 4-CTA register cap (force),
                    // 3 symmetric (every unordered pair once)
  int tail = 0;     // slicing of a system's j-range: 0 equal slices, 1 full slices and a halving tail
                    // (symmetric: 0 pieces of one length and a remainder per row of i-tiles, 1 every other
                    // row in pieces a third as long, 2 pieces of a row as equal as whole blocks allow)
};
constexpr int kSymVariant = 3;

constexpr int64_t kMaxSymRows = 64;                      // rows of i-tiles a system is cut into at most

// The systems' bodies and chunks, as the work lists see them.
struct SymLayout {
  int64_t n_total = 0;
  int n_sys = 0;
  std::vector<int64_t> offsets;
  std::vector<Chunk> chunks;  // without slots (Chunk::n_slices, stride, row0: the copies on the device)
  std::vector<int32_t> sys_chunk;
  int j_block = 64;  // j-bodies that a warp of the symmetric pass meets in one block (pieces are whole blocks)
};

// Chunks: runs of <= `bodies` bodies inside one system, and each system's range of them.
inline void cut_chunks(const SymLayout& c, const int64_t bodies, std::vector<Chunk>& chunks,
                       std::vector<int32_t>& sys_chunk) {
  chunks.clear();
  sys_chunk.assign(c.n_sys + 1, 0);
  for (int s = 0; s < c.n_sys; ++s) {
    sys_chunk[s] = (int32_t)chunks.size();
    for (int64_t b = c.offsets[s]; b < c.offsets[s + 1]; b += bodies)
      chunks.push_back(Chunk{s, (int32_t)b, (int32_t)std::min<int64_t>(c.offsets[s + 1], b + bodies), 1, 0, 0, 0});
  }
  sys_chunk[c.n_sys] = (int32_t)chunks.size();
}

inline bool is_sym(const Tiling& t) { return t.variant == kSymVariant; }

// Unordered pairs of all systems.
inline double total_pairs(const SymLayout& c) {
  double p = 0.0;
  for (int s = 0; s < c.n_sys; ++s) {
    const double n = (double)(c.offsets[s + 1] - c.offsets[s]);
    p += 0.5 * n * n;
  }
  return p;
}

// The symmetric pass cuts a system of n bodies into rows of H bodies (whole i-tiles, at most
// kMaxSymRows rows: a body has a slot per row up to its own, so more rows would mean more partials
// to combine than pair work saved) and row r into pieces of about `area` pairs. Rows are whole
// chunks too (both are powers of two): the number of slots is a row's, and the O(N) kernels take
// one number per chunk. It makes a difference to FP64 i-tiles of 64 bodies among chunks of 128.
struct SymRows {
  int64_t n, H, rows, block;  // block: pieces are whole blocks of j-bodies
  SymRows(const SymLayout& c, const Tiling& t, int64_t bodies) : n(bodies), block(c.j_block) {
    const int64_t unit = std::max<int64_t>((int64_t)t.block * t.ipt, chunk_bodies(c.n_total));
    H = unit * std::max<int64_t>(1, (n + unit * kMaxSymRows - 1) / (unit * kMaxSymRows));  // (an empty system has no row)
    rows = (n + H - 1) / H;
  }
  int64_t blocks(int64_t r) const { return (n - r * H + block - 1) / block; }
  // pieces of row r, and for a tail other than 2 the blocks of each (the last may have fewer)
  int64_t pieces(int64_t r, double area, int tail, int64_t* step) const {
    const double ni = (double)std::min(H, n - r * H), pairs = ni * ((double)(n - r * H) - 0.5 * ni);
    const double want = tail == 1 && (r & 1) ? area / 3.0 : area;
    const int64_t nb = blocks(r), p = std::max<int64_t>(1, std::min(nb, (int64_t)(pairs / want + 0.5)));
    *step = std::max<int64_t>(1, (2 * nb + p) / (2 * p));
    return tail == 2 ? p : (nb + *step - 1) / *step;
  }
};

// Work items of a symmetric tiling with the given slice, counted up to `most` and a little beyond.
inline int64_t sym_item_count(const SymLayout& c, const Tiling& t, int64_t slice, int64_t most) {
  const double area = (double)slice * t.block * t.ipt;
  int64_t items = 0, step, last = 0, own = 0;  // own: items of a system of `last` bodies
  for (int s = 0; s < c.n_sys && items <= most; ++s) {
    const int64_t n = c.offsets[s + 1] - c.offsets[s];
    if (n != last) {
      const SymRows R(c, t, n);
      own = 0, last = n;
      for (int64_t r = 0; r < R.rows; ++r) own += R.pieces(r, area, t.tail, &step);
    }
    items += own;
  }
  return items;
}

// Entries of partial sums that a symmetric tiling needs (t.slice as set): a system's bodies times the slots
// of its most used row.
inline int64_t sym_part_rows(const SymLayout& c, const Tiling& t) {
  const double area = (double)t.slice * (double)t.block * t.ipt;
  int64_t rows = 0, step, last = 0, own = 0;  // own: entries of a system of `last` bodies
  for (int s = 0; s < c.n_sys; ++s) {
    const int64_t n = c.offsets[s + 1] - c.offsets[s];
    if (n != last) {
      const SymRows R(c, t, n);
      int64_t most = 0;
      for (int64_t r = 0; r < R.rows; ++r) most = std::max(most, r + 1 + R.pieces(r, area, t.tail, &step));
      own = most * n, last = n;
    }
    rows += own;
  }
  return rows;
}

// Slice of a symmetric tiling (t.tail as set) that makes at most `pieces` work items per CTA of a
// full grid, as many as that allows: one item more than CTAs would cost a whole second round.
constexpr int kSymPieces = 6;
inline int sym_slice(const SymLayout& c, const Tiling& t, int n_ctas, int pieces) {
  const int64_t most = (int64_t)pieces * n_ctas;
  auto fits = [&](int64_t slice) { return sym_item_count(c, t, slice, most) <= most; };
  int64_t lo = 1, hi = 1;  // the least slice that fits lies in (lo, hi], or no slice does (every row one piece)
  while (!fits(hi) && hi < (int64_t)1 << 30) lo = hi, hi *= 2;
  while (hi - lo > std::max<int64_t>(1, lo / 256)) {
    const int64_t mid = (lo + hi) / 2;
    (fits(mid) ? hi : lo) = mid;
  }
  return (int)std::min<int64_t>(hi, 1 << 30);
}

// Work list of the symmetric pass for tiling t (see sym_common.cuh, SymRows), pieces of
// about slice x i-tile pairs. Chunks get their slots; rows is the number of entries the
// partial buffer needs. False if a chunk reaches into a second row: its bodies' slots would differ.
inline bool build_sym_items(const SymLayout& c, const Tiling& t, std::vector<SymItem>& items, std::vector<Chunk>& chunks,
                     int& max_slots, int64_t& rows) {
  items.clear();
  chunks = c.chunks;
  max_slots = 1;
  rows = 0;
  const double area = (double)t.slice * (double)t.block * t.ipt;
  std::vector<int> slots;
  for (int s = 0; s < c.n_sys; ++s) {
    const int64_t b = c.offsets[s], n = c.offsets[s + 1] - b;
    if (n <= 0) continue;
    const SymRows R(c, t, n);
    const int64_t H = R.H;
    slots.assign((size_t)R.rows, 0);
    int most = 0;
    for (int64_t r = 0; r < R.rows; ++r) {
      const int64_t i0 = r * H, ni = std::min(H, n - i0);
      int64_t step;
      const int64_t p = R.pieces(r, area, t.tail, &step);
      auto cut = [&](int64_t k) { return std::min(n, i0 + R.block * (t.tail == 2 ? k * R.blocks(r) / p : k * step)); };
      slots[(size_t)r] = (int)(r + 1 + p);
      most = std::max(most, slots[(size_t)r]);
      for (int64_t k = 0; k < p; ++k) {
        SymItem w{};
        w.sys = s;
        w.i_begin = (int32_t)(b + i0);
        w.i_end = (int32_t)(b + i0 + ni);
        w.j_begin = (int32_t)(b + cut(k));
        w.j_end = (int32_t)(b + cut(k + 1));
        w.slot_j = (int32_t)r;
        w.slot_i = (int32_t)(r + 1 + k);
        w.stride = (int32_t)n;
        w.row0 = rows - b;
        items.push_back(w);
      }
    }
    for (int32_t k = c.sys_chunk[s]; k < c.sys_chunk[s + 1]; ++k) {
      Chunk& ch = chunks[(size_t)k];
      if ((ch.begin - b) / H != (ch.end - 1 - b) / H) return false;
      ch.n_slices = slots[(size_t)((ch.begin - b) / H)];
      ch.stride = (int32_t)n;
      ch.row0 = rows - b;
    }
    max_slots = std::max(max_slots, most);
    rows += (int64_t)most * n;
  }
  // longest first, for the dynamic schedule of the persistent grid
  auto cost = [](const SymItem& w) {
    const int64_t ni = w.i_end - w.i_begin, nj = w.j_end - w.j_begin;
    const int64_t own = std::max<int64_t>(0, std::min(w.i_end, w.j_end) - w.j_begin);  // j-bodies inside the row
    return ni * nj - own * (own - 1) / 2;
  };
  std::stable_sort(items.begin(), items.end(), [&](const SymItem& x, const SymItem& y) { return cost(x) > cost(y); });
  return true;
}

}  // namespace nbody
