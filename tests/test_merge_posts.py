"""The tile walker's posts of merges: every interleaving of one poster, which reuses a place for
posts of growing size, and two helpers, walked through on the CPU with the functions that the
kernel uses (csrc/gwcp_post.cuh). Every merge is done once, and the poster leaves its wait only
when all are done. The same walk finds the fault of the two-word form (the number of merges read
after the draw), so it does look where that one went wrong."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <set>
#include <string>
#include <vector>
#include "gwcp_post.cuh"
using namespace gwcp;

static const int kSizes[] = {SIZES};
static const int kPosts = sizeof(kSizes) / sizeof(int), kHelpers = 2, kTries = 2;

struct Walker {
  int pc, tries, j;  // j: the merge drawn
  uint32_t w;
};
struct State {
  uint32_t word, total, open, done;  // (total: the two-word form only)
  int post;                          // which post the place holds
  int begun[8], ended;               // its merges
  Walker t[1 + kHelpers];            // t[0]: the poster
};
enum { ANNOUNCE, OPEN, LOOK, SEEN, DRAW, LIMIT, BEGIN, END, WAIT, CLOSE, STOP };

static bool wrong = false;

// one step of walker i; false: it cannot go on now
static bool step(State& s, int i) {
  Walker& t = s.t[i];
  const int none = i == 0 ? WAIT : LOOK;  // where a walker goes that draws nothing
  switch (t.pc) {
    case ANNOUNCE: s.done = 0; s.open = 1; t.pc = OPEN; return true;
    case OPEN:
      std::memset(s.begun, 0, sizeof(s.begun));
      s.ended = 0;
      s.total = uint32_t(kSizes[s.post]);
      s.word = SPLIT ? 0u : post_open(uint32_t(kSizes[s.post]));
      t.pc = SEEN;
      return true;
    case LOOK:  // a helper: is there an open post?
      if (t.tries == 0) { t.pc = STOP; return true; }
      if (!s.open) return false;
      --t.tries;
      t.pc = SEEN;
      return true;
    case SEEN: t.pc = SPLIT || post_left(s.word) ? DRAW : none; return true;
    case DRAW:
      t.w = s.word++;
      t.pc = SPLIT ? LIMIT : post_left(t.w) ? BEGIN : none;
      t.j = SPLIT ? int(t.w) : int(post_merge(t.w));
      if (!SPLIT && t.pc == BEGIN && t.j + 1 == int(post_merges(t.w))) s.open = 0;
      return true;
    case LIMIT:
      t.pc = t.w < (1u << 30) && t.w < s.total ? BEGIN : none;
      if (t.pc == BEGIN && t.w + 1 == s.total) s.open = 0;
      return true;
    case BEGIN:
      if (t.j >= kSizes[s.post] || s.begun[t.j]++) wrong = true;  // not a merge of this post, or a second time
      t.pc = END;
      return true;
    case END: ++s.ended; ++s.done; t.pc = i == 0 ? SEEN : LOOK; return true;
    case WAIT:
      if (s.done < uint32_t(kSizes[s.post])) return false;
      for (int j = 0; j < kSizes[s.post]; ++j) wrong |= s.begun[j] != 1;
      wrong |= s.ended != kSizes[s.post];
      t.pc = CLOSE;
      return true;
    case CLOSE:
      s.word = SPLIT ? 1u << 30 : kPostClosed;
      if (s.post + 1 < kPosts) { ++s.post; t.pc = ANNOUNCE; } else { t.pc = STOP; }
      return true;
    default: return false;
  }
}

int main() {
  State s;
  std::memset(&s, 0, sizeof(s));
  s.word = SPLIT ? 1u << 30 : kPostClosed;
  s.t[0].pc = ANNOUNCE;
  for (int i = 1; i <= kHelpers; ++i) { s.t[i].pc = LOOK; s.t[i].tries = kTries; }
  std::set<std::string> seen;
  std::vector<State> todo{s};
  size_t finished = 0;
  while (!todo.empty() && !wrong) {
    State a = todo.back();
    todo.pop_back();
    bool moved = false;
    for (int i = 0; i <= kHelpers; ++i) {
      State b = a;
      if (!step(b, i)) continue;
      moved = true;
      if (seen.insert(std::string(reinterpret_cast<char*>(&b), sizeof(b))).second) todo.push_back(b);
    }
    if (!moved) {
      if (a.t[0].pc != STOP) { std::printf("stuck\n"); return 1; }
      ++finished;
    }
  }
  std::printf("%s %zu %zu\n", wrong ? "wrong" : "right", seen.size(), finished);
  return 0;
}
"""


def explore(tmp_path, split, sizes):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "posts.cpp", tmp_path / "posts"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", f"-DSPLIT={int(split)}", f"-DSIZES={sizes}", "-I",
                           os.path.join(ROOT, "paper_2111_12478_gb300", "csrc"), str(src), "-o", str(exe)])
    word, states, ends = subprocess.check_output([str(exe)], text=True).split()
    assert int(states) > 100
    return word, int(ends)


@pytest.mark.parametrize("sizes", ["2,3", "2,4", "3,2", "2,3,4"])
def test_every_merge_once(tmp_path, sizes):
    word, ends = explore(tmp_path, False, sizes)
    assert word == "right" and ends > 0


def test_the_walk_finds_a_limit_read_after_the_draw(tmp_path):
    assert explore(tmp_path, True, "2,3")[0] == "wrong"
