"""The host side of the log-prob kernels' plan (csrc/vocab_plan.cuh), compiled with a plain C++ compiler."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_24840_b200", "csrc")


def _run(tmp_path, body):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "plan.cpp"
    src.write_text('#include <cstdio>\n#include <cstdlib>\n#include <initializer_list>\n#include "vocab_plan.cuh"\n'
                   '#define CHECK(c) do { if (!(c)) { std::printf("%s: sm %d chunks %d splits %d\\n", #c, sm, chunks, splits); std::exit(1); } } while (0)\n'
                   "int main() {\n" + body + "\n  return 0;\n}\n")
    subprocess.check_call([gxx, "-std=c++17", "-O2", "-Wall", "-I", CSRC, str(src), "-o", str(tmp_path / "plan")])
    out = subprocess.run([str(tmp_path / "plan")], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout


def test_segments_blocks_and_groups_cover_the_vocabulary_on_any_number_of_sms(tmp_path):
    """Every chunk belongs to one segment, every segment to one block and every block to one group, in order; every segment is dealt
    once; the tables are not written past their ends.  Up to 600 SMs: more than a segment's number has bits for."""
    _run(tmp_path, r"""
  const int sms[] = {1, 2, 3, 15, 16, 17, 132, 147, 148, 160, 254, 255, 256, 257, 300, 511, 600};
  const int counts[] = {1, 2, 3, 16, 17, 64, 100, 147, 148, 149, 255, 256, 257, 300, 591, 594, 601, 1000, 4097, 8388607};
  const int cuts[] = {1, 2, 3, 4, 7, 8, 16, 33, 63, 64};
  for (int sm : sms) for (int chunks : counts) for (int cut : cuts) {
    const int splits = cut < chunks ? cut : chunks;
    const VocabPlan v = make_vocab_plan(sm, chunks, splits);
    CHECK(v.splits >= 1 && v.splits <= v.n_mid && v.n_mid <= v.n_sub && v.n_mid <= MAX_SPLITS && v.n_sub <= sm && v.n_sub <= chunks);
    CHECK(v.chunk_of_sub(0) == 0 && v.chunk_of_sub(v.n_sub) == chunks);
    CHECK(v.mid_begin[0] == 0 && v.mid_begin[v.n_mid] == v.n_sub && v.group_begin[0] == 0 && v.group_begin[v.splits] == v.n_mid);
    for (int i = 0; i < v.n_sub; ++i) CHECK(v.chunk_of_sub(i) == (int)((long long)i * chunks / v.n_sub) && v.chunk_of_sub(i) < v.chunk_of_sub(i + 1));
    for (int i = 0; i < v.n_mid; ++i) CHECK(v.mid_begin[i] < v.mid_begin[i + 1]);
    for (int g = 0; g < v.splits; ++g) CHECK(v.group_begin[g] < v.group_begin[g + 1]);
    bool dealt[600] = {};
    for (int j = 0; j < v.n_sub; ++j) {
      const int s = v.nth_sub(j);
      CHECK(s >= 0 && s < v.n_sub && !dealt[s]);
      CHECK(v.chunk_of_sub(s + 1) - v.chunk_of_sub(s) == v.per_sub + (j < v.n_long ? 1 : 0));
      dealt[s] = true;
    }
  }""")


def test_the_combining_kernel_fits_beside_the_log_prob_kernel(tmp_path):
    """Whatever the vocabulary and the tail: where all blocks of the combining kernel fit at once, four an SM, one of them and one of the
    log-prob kernel (its 195 KB) are within the shared memory of an SM; and no block takes fewer tokens than that, 32 KB, 32 tokens or an
    SM's share of the tail allow."""
    _run(tmp_path, r"""
  const size_t beside = 4 * 48 * 1024 + 1024 + 256 + 64 * 28, sm_bytes = 228 * 1024, reserved = 1024;
  const int sm = 148;
  int most = 0, beyond = 0;
  for (int chunks = 1; chunks <= 600; ++chunks) for (int splits = 1; splits <= 64 && splits <= chunks; splits += splits < 8 ? 1 : 7) for (int halves = 1; halves <= 2; ++halves) {
    const VocabPlan v = make_vocab_plan(sm, chunks, splits);
    for (long rows : {1L, 100L, 148L, 149L, 888L, 1000L, 2800L, 3552L, 3553L, 3996L, 4200L, 9472L}) {
      const int group = combine_group(v, halves, rows, sm, beside);
      CHECK(group >= 1 && group <= 32 && group <= (rows + sm - 1) / sm);
      const size_t token = combine_bytes(v, halves), bytes = group * token;
      const bool fits = beside + bytes + 2 * reserved <= sm_bytes, at_once = (rows + group - 1) / group <= 4 * sm;
      CHECK(bytes <= 32 * 1024);
      CHECK(group == 32 || group == (rows + sm - 1) / sm || bytes + token > (fits ? sm_bytes - beside - 2 * reserved : 32 * 1024));
      // past the line only where the smaller blocks would not fit at once
      if (!fits) { ++beyond; CHECK(rows > (long)((sm_bytes - beside - 2 * reserved) / token) * 4 * sm); }
      CHECK(fits || !at_once || rows > (long)((sm_bytes - beside - 2 * reserved) / token) * 4 * sm);
      most = group > most ? group : most;
    }
  }
  const int chunks = 0, splits = 0;
  CHECK(most == 32 && beyond > 0);""")
