"""Work lists of the symmetric passes, checked on the host for every body: the O(N) kernels read each
slot that the pass writes, and no other (csrc/work_lists.h needs no GPU)."""

import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_02655_gb300", "csrc")

DRIVER = r"""
#include "work_lists.h"
using namespace nbody;
// out: bodies that read a slot written not exactly once, slots written and never read, bodies whose
// pairs are not met exactly once, work items
extern "C" int check(const int64_t* sizes, int n_sys, int j_block, int block, int ipt, int slice, int tail,
                     int64_t* out) {
  SymLayout c;
  c.n_sys = n_sys, c.j_block = j_block;
  c.offsets.push_back(0);
  for (int s = 0; s < n_sys; ++s) c.offsets.push_back(c.offsets.back() + sizes[s]);
  c.n_total = c.offsets.back();
  cut_chunks(c, chunk_bodies(c.n_total), c.chunks, c.sys_chunk);
  Tiling t;
  t.block = block, t.ipt = ipt, t.slice = slice, t.tail = tail, t.variant = kSymVariant;
  std::vector<SymItem> items;
  std::vector<Chunk> chunks;
  int max_slots;
  int64_t rows;
  if (!build_sym_items(c, t, items, chunks, max_slots, rows)) return 1;
  if (sym_item_count(c, t, slice, 1 << 30) != (int64_t)items.size()) return 3;  // (empty systems included)
  if (rows != sym_part_rows(c, t)) return 2;
  std::vector<int> written((size_t)rows);
  std::vector<int64_t> met((size_t)c.n_total);
  for (const SymItem& w : items) {
    for (int64_t i = w.i_begin; i < w.i_end; ++i) written[(size_t)(w.row0 + (int64_t)w.slot_i * w.stride + i)]++;
    for (int64_t j = w.j_begin; j < w.j_end; ++j) written[(size_t)(w.row0 + (int64_t)w.slot_j * w.stride + j)]++;
    // partners met as an i-body: the piece's later bodies; as a j-body: the row's earlier bodies
    for (int64_t i = w.i_begin; i < w.i_end; ++i)
      met[(size_t)i] += std::max<int64_t>(0, w.j_end - std::max<int64_t>(w.j_begin, i + 1));
    for (int64_t j = w.j_begin; j < w.j_end; ++j)
      met[(size_t)j] += std::max<int64_t>(0, std::min<int64_t>(w.i_end, j) - w.i_begin);
  }
  for (int k = 0; k < 4; ++k) out[k] = 0;
  for (const Chunk& k : chunks)
    for (int64_t i = k.begin; i < k.end; ++i) {
      bool bad = false;
      for (int s = 0; s < k.n_slices; ++s) {
        int& w = written[(size_t)(k.row0 + (int64_t)s * k.stride + i)];
        bad |= w != 1;
        w = 0;
      }
      out[0] += bad;
      out[2] += met[(size_t)i] != sizes[k.sys] - 1;
    }
  for (int w : written) out[1] += w != 0;
  out[3] = (int64_t)items.size();
  return 0;
}
"""


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    d = tmp_path_factory.mktemp("work_lists")
    src, lib = d / "driver.cpp", d / "libdriver.so"
    src.write_text(DRIVER)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    f = ctypes.CDLL(str(lib)).check

    def run(sizes, j_block, block, ipt, slice_, tail):
        out = (ctypes.c_int64 * 4)()
        assert f((ctypes.c_int64 * len(sizes))(*sizes), len(sizes), j_block, block, ipt, slice_, tail, out) == 0
        return list(out)
    return run


LAYOUTS = {"65": [65], "1400": [1400], "17000": [17000], "33000": [33000], "36000": [36000], "45001": [45001],
           "512x256": [256] * 512, "200x200": [200] * 200, "300x200": [200] * 300, "80x500": [500] * 80,
           "60x512": [512] * 60, "40x4500": [4500] * 40, "mixed": [0, 1, 300, 40001, 2, 700, 0, 4097, 63]}


@pytest.mark.parametrize("tail", [0, 1, 2])
@pytest.mark.parametrize("layout", LAYOUTS)
@pytest.mark.parametrize("j_block,block,ipt", [(32, 64, 1), (32, 128, 1), (32, 256, 1), (32, 128, 2), (64, 128, 1),
                                               (64, 128, 2), (64, 256, 2), (64, 256, 4)])
def test_slots_read_are_slots_written(check, j_block, block, ipt, layout, tail):
    for slice_ in (160, 1 << 30):
        wrong, unread, pairs, items = check(LAYOUTS[layout], j_block, block, ipt, slice_, tail)
        assert (wrong, unread, pairs) == (0, 0, 0) and items > 0, (slice_, wrong, unread, pairs)
