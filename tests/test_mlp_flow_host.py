"""The MMA threads' order of waits and issues (pnp_mlpflow.cuh), run on the host: the
parities of a run in which every wait succeeds, and, with each wait in turn running
out, that nothing issued is still under way when the kernel goes on to free its
tensor memory; and how the weight gradients' CTAs are shared out over fewer SMs."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1701_02005_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "pnp_mlpflow.cuh"

#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); std::exit(1); } } while (0)

// waits: the one numbered `fail` runs out; a barrier's k-th use has parity k & 1
struct Base {
  int fail, waits = 0, under_way = 0, issued = 0, commits = 0, drains = 0;
  bool gave_up = false;
  explicit Base(int f) : fail(f) {}
  bool wait(int (&uses), unsigned phase) {
    CHECK(!gave_up && drains == 0 && phase == (unsigned)(uses & 1));
    ++uses;
    gave_up = waits++ == fail;
    return !gave_up;
  }
  void issue() { CHECK(!gave_up); ++issued; ++under_way; }
  bool drain() { ++drains; under_way = 0; return true; }
};

struct Net : Base {
  using Base::Base;
  int uses[2] = {0, 0}, mmas[2][5] = {};
  bool ready(int h, unsigned phase) { return wait(uses[h], phase); }
  void forward(int l, int h) {   // half h needs the halves up to h of this layer's hand-over
    CHECK(uses[0] == commits + 1 && uses[1] == commits + (l == 0 || h ? 1 : 0));
    ++mmas[0][l];
    issue();
  }
  void backward(int l) {
    CHECK(uses[0] == commits + 1 && uses[1] == commits + 1);
    ++mmas[1][l];
    issue();
  }
  void commit() { ++commits; }
};

struct Wg : Base {
  using Base::Base;
  int fulls[3] = {}, frees[2] = {}, sums[2] = {}, slots = 0;
  bool freed(int b, unsigned phase) { return wait(frees[b], phase); }
  bool full(int q, unsigned phase) { return wait(fulls[q], phase); }
  void product(int q, int b, bool acc) {
    CHECK(q == issued % 3 && b == issued / 2 % 2 && acc == (issued % 2 != 0));
    CHECK(acc || sums[b] == frees[b]);   // the block's last sum has been read
    issue();
  }
  void commit_slot(int q) { CHECK(q == slots % 3); ++slots; }
  void commit_sum(int b) { ++sums[b]; }
};

template <typename Ops, typename F>
void each_wait(F run) {
  Ops all(-1);
  CHECK(run(all) && all.drains == 1 && all.under_way == 0);
  for (int f = 0; f < all.waits; ++f) {
    Ops o(f);
    CHECK(!run(o) && o.drains == 1 && o.under_way == 0 && o.waits == f + 1);
  }
}

int main() {
  for (int tiles = 1; tiles <= 5; ++tiles) {
    Net inf(-1), trn(-1);
    CHECK((pnp::flow_network<5, false>(inf, 0, tiles, 2)) && (pnp::flow_network<5, true>(trn, 0, tiles, 2)));
    const int mine = (tiles + 1) / 2;
    CHECK(inf.commits == 5 * mine && trn.commits == 9 * mine);
    for (int l = 0; l < 5; ++l) {
      CHECK(inf.mmas[0][l] == mine * (l ? 2 : 1) && inf.mmas[1][l] == 0);
      CHECK(trn.mmas[0][l] == mine * (l ? 2 : 1) && trn.mmas[1][l] == (l ? mine : 0));
    }
    each_wait<Net>([&](Net& o) { return pnp::flow_network<5, false>(o, 0, tiles, 2); });
    each_wait<Net>([&](Net& o) { return pnp::flow_network<5, true>(o, 0, tiles, 2); });
  }
  for (int tiles = 0; tiles <= 13; ++tiles) {
    Wg w(-1);
    CHECK((pnp::flow_wgrad<3, 2>(w, tiles)) && w.issued == tiles && w.slots == tiles);
    CHECK(w.sums[0] + w.sums[1] == (tiles + 1) / 2);
    each_wait<Wg>([&](Wg& o) { return pnp::flow_wgrad<3, 2>(o, tiles); });
  }
  std::puts("ok");
}
"""


SHARES = r"""
#include <cstdio>
#include "pnp_mlpflow.cuh"

int main() {
  const int full[5] = {24, 36, 36, 36, 20};
  for (int sms = 0; sms <= 200; ++sms) {
    int s[5], sum = 0, most = sms < 152 ? sms : 152;
    pnp::share_ctas(full, 152, sms, s);
    for (int l = 0; l < 5; ++l) {
      sum += s[l];
      const double part = full[l] * most / 152.0;
      if (s[l] < 1 || s[l] > full[l] || (most >= 5 && (s[l] < part - 2 || s[l] > part + 2)) ||
          (sms >= 152 && s[l] != full[l]))
        return std::printf("%d SMs: layer %d gets %d\n", sms, l, s[l]), 1;
    }
    // one wave, and no SM without a CTA; below eight SMs the layers' ones alone can exceed it
    if (most >= 8 ? sum != most : sum > 8) return std::printf("%d SMs: %d CTAs\n", sms, sum), 1;
  }
  std::puts("ok");
}
"""


@pytest.mark.parametrize("program", [PROGRAM, SHARES], ids=["order", "shares"])
def test_host_side_of_the_network_kernels(program, tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "flow.cpp", tmp_path / "flow"
    src.write_text(program)
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
