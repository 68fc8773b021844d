"""The context's workspace against an allocator with a limit (host code, compiled
here): what it asks for and gives up, in order, for each call."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1605_05773_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include "d8_workspace.h"
struct Mem {
  size_t room;
  std::map<void*, size_t> held;
  void* alloc(size_t n) {
    size_t sum = n;
    for (auto& h : held) sum += h.second;
    std::printf(" %s%zu", sum > room ? "no" : "+", n);
    if (sum > room) return nullptr;
    void* p = std::malloc(1);
    held[p] = n;
    return p;
  }
  void release(void* p) {
    std::printf(" -%zu", held[p]);
    held.erase(p);
    std::free(p);
  }
};
int main(int argc, char** argv) {
  Mem mem{(size_t)std::atoi(argv[1]), {}};
  d8::Workspace ws;
  for (int k = 2; k + 1 < argc; k += 2) {
    if (argv[k][0] == 'r') {  // room changes
      mem.room = (size_t)std::atoi(argv[k + 1]);
      continue;
    }
    const bool ok = ws.ensure(mem, (size_t)std::atoi(argv[k]), (size_t)std::atoi(argv[k + 1]));
    std::printf(" %s%zu;", ok ? "=" : "fail", ws.bytes);
    if ((ws.p != nullptr) != (ws.bytes > 0)) return 1;
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    d = tmp_path_factory.mktemp("ws")
    (d / "m.cpp").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-I", CSRC, str(d / "m.cpp"), "-o", str(d / "m")], check=True)
    return str(d / "m")


@pytest.mark.parametrize("args, want", [
    # one size: the old block goes first, so that old and new need not fit together
    ("100 60 60 80 80 50 50", "+60 =60; -60 +80 =80; =80;"),
    ("100 60 60 200 200 60 60", "+60 =60; -60 no200 fail0; +60 =60;"),
    # room for both sizes
    ("100 50 10 50 10", "+50 =50; =50;"),
    # no room for the larger one: the smaller, and later calls ask no more
    ("30 50 10 50 10 50 10", "no50 +10 =10; =10; =10;"),
    # a block that holds the smaller size is kept when the larger finds no room, once
    ("60 20 20 50 10 50 10 40 10 45 10", "+20 =20; no50 =20; =20; +40 -20 =40; no45 =40;"),
    ("100 20 20 50 10 r 20 60 10", "+20 =20; +50 -20 =50; no60 =50;"),
    # neither fits
    ("5 50 10 4 4", "no50 no10 fail0; +4 =4;"),
    # a new block: the refusal is forgotten
    ("30 50 10 r 100 50 10 60 60 200 70", "no50 +10 =10; =10; -10 +60 =60; -60 no200 +70 =70;"),
])
def test_what_is_asked_for(exe, args, want):
    r = subprocess.run([exe, *args.split()], capture_output=True, text=True)
    assert r.returncode == 0
    print(r.stdout)
    assert " ".join(r.stdout.split()) == want
