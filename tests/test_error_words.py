"""The layer entry points' error words (csrc/errword.h, host code): a word that a failed
call left set fails no later call, and none is handed out while a launch of an earlier
call may still write it.  The waits and the kernels' writes are faked."""
import pathlib
import re
import shutil
import subprocess

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_1610_03918_gb300" / "csrc"

MAIN = r"""
#include <cstdio>
#include "errword.h"
using namespace picgb;

static ErrWords pool;
static volatile int words[64];

struct Wait {   // what the wait returns, and what a kernel writes before it ends
  Drain d;
  int written, *word_seen;
  int *calls;
  Drain operator()() const {
    ++*calls;
    if (written) *const_cast<int *>(words + *word_seen) = written;
    return d;
  }
};

#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)

int main() {
  int calls = 0, k = 0;
  {   // a wait that gave up is reported by its own call ...
    ErrLease<Wait> a(pool, words, Wait{Drain::kEnded, 2, &k, &calls});
    k = a.index();
    CHECK(k == 0 && a.end() == 2 && a.index() == -1);
  }
  CHECK(calls == 1);
  {   // ... and by no later one, though it left the word set
    CHECK(words[0] == 2);
    ErrLease<Wait> a(pool, words, Wait{Drain::kEnded, 0, &k, &calls});
    CHECK(a.index() == 0 && words[0] == 0 && a.end() == 0);
  }
  {   // a call that is left without an end still waits for its launches
    calls = 0;
    { ErrLease<Wait> a(pool, words, Wait{Drain::kEnded, 3, &k, &calls}); k = a.index(); }
    CHECK(calls == 1 && words[0] == 3);
    ErrLease<Wait> b(pool, words, Wait{Drain::kEnded, 0, &k, &calls});
    CHECK(b.index() == 0 && b.end() == 0);
  }
  {   // launches that never run give the word back
    for (int q = 0; q < 200; ++q) {
      ErrLease<Wait> a(pool, words, Wait{Drain::kNotRun, 0, &k, &calls});
      CHECK(a.index() == 0 && a.end() == -1);
    }
  }
  {   // calls in progress have different words
    ErrLease<Wait> a(pool, words, Wait{Drain::kEnded, 0, &k, &calls}), b(pool, words, Wait{Drain::kEnded, 0, &k, &calls});
    CHECK(a.index() == 0 && b.index() == 1);
  }
  // a wait that fails: its word is not handed out again, and with all of them gone a
  // call is refused, not kept waiting
  for (int q = 0; q < 64; ++q) {
    ErrLease<Wait> a(pool, words, Wait{Drain::kUnknown, 0, &k, &calls});
    CHECK(a.index() == q && a.end() == -1);
  }
  ErrLease<Wait> a(pool, words, Wait{Drain::kEnded, 0, &k, &calls});
  CHECK(a.index() == -1 && a.end() == -1);
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_error_words(tmp_path):
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = tmp_path / "main"
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-pthread", "-I", str(CSRC),
                    str(tmp_path / "main.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_entry_points_end_every_call_that_launched():
    # between the word's drawing and the end of the call no status is returned past it
    text = (CSRC / "unet.cu").read_text()
    parts = text.split("ErrWord word(s);")[1:]
    assert len(parts) == 5
    for part in parts:
        body = part[part.index("return PIC_ECUDA;") + 1:part.index("\n}\n")]   # behind the refusal without a word
        body = body[:body.rindex("word.end(") + 9]
        assert not re.search(r"\breturn (?!word\.end\()", body)
