"""What the copying and multiplying warps leave behind when a bounded wait gives
up: the roles of csrc/ring_roles.cuh compiled for the host, with waits that
fail at every possible place.  Whatever was issued must have been waited for
when a role returns (a copy that lands, or a matrix instruction that completes,
after the CTA has given its memory back is a fault).  No GPU."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_05034_gb300", "csrc")

TC = r"""
#include <cstdio>
#include <set>
#include <vector>
#include "ring_roles.cuh"

// Stages 0 .. nst-1 of the stencil.  The wait numbered `fail` of a role (and
// every later one before the drain) gives up.
template <int S>
int copy_role(int nst, int fail, bool* raised) {
  std::vector<int> issued;
  std::set<int> landed;  // stages known to have landed
  int waits = 0;
  bool gave_up = false;
  dwfk::tc_copy_role<S>(
      nst,
      [&](int b, unsigned par) {
        const int h = (int)issued.size() - S;  // done: the MMAs of the slot's last use, so its copies too
        if (b != h % S || (int)par != ((h / S) & 1)) { std::printf("done(%d) of stage %d\n", b, h); return false; }
        if (waits++ >= fail) { gave_up = true; return false; }
        landed.insert(h);
        return true;
      },
      [&](int b, unsigned par) {
        for (int h = (int)issued.size() - 1; h >= 0; h--)
          if (h % S == b) {
            if ((int)par == ((h / S) & 1)) landed.insert(h);
            break;
          }
        return true;
      },
      [&](int g, int b) {
        if (b != g % S || gave_up) std::printf("issue after giving up\n");
        issued.push_back(g);
      },
      [&]() { *raised = true; });
  for (int g : issued)
    if (!landed.count(g)) { std::printf("S %d nst %d fail %d: copy of stage %d in flight\n", S, nst, fail, g); return 1; }
  return *raised != gave_up;
}

template <int S, int NBUF>
int mma_role(int nst, int fail, bool* raised) {
  std::vector<int> issued;
  int waits = 0, complete = 0;  // stages known to be complete
  bool gave_up = false;
  auto w = [&]() { if (waits++ >= fail) gave_up = true; return !gave_up; };
  dwfk::tc_mma_role<S, NBUF>(
      nst, [&](int, unsigned) { return w(); }, [&](int, unsigned) { return w(); },
      [&](int b, unsigned par) {
        const int h = (int)issued.size() - 1;
        if (b == h % S && (int)par == ((h / S) & 1)) complete = h + 1;
        return true;
      },
      [&](int h, int d, int t, int b) {
        if (gave_up || h != (int)issued.size() || d != h % 9 || t != h / 9 % NBUF || b != h % S) std::printf("order\n");
        issued.push_back(h);
      },
      [&]() { *raised = true; });
  if (complete != (int)issued.size()) { std::printf("S %d nst %d fail %d: MMAs in flight\n", S, nst, fail); return 1; }
  return *raised != gave_up;
}

int main() {
  int bad = 0;
  for (int nst = 0; nst <= 45; nst += 9)
    for (int fail = 0; fail <= 2 * nst + 8; fail++) {
      bool r[5] = {false, false, false, false, false};
      bad += copy_role<2>(nst, fail, r) + copy_role<3>(nst, fail, r + 1) + copy_role<4>(nst, fail, r + 2);
      bad += mma_role<3, 1>(nst, fail, r + 3) + mma_role<4, 2>(nst, fail, r + 4);
    }
  std::printf("bad %d\n", bad);
  return bad != 0;
}
"""


def _run(tmp_path, source):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "roles.cpp"
    src.write_text(source)
    exe = tmp_path / "roles"
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", CSRC, "-x", "c++", str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "bad 0", r.stdout


def test_coarse_stencil_roles_leave_nothing_in_flight(tmp_path):
    _run(tmp_path, TC)


STREAM = r"""
#include <cstdio>
#include <set>
#include <utility>
#include <vector>
#include "ring_roles.cuh"

static int produce(const std::vector<int>& runs, int fail) {
  const unsigned slots[4] = {3, 3, 2, 2};
  unsigned issued[4] = {0, 0, 0, 0};
  std::set<std::pair<int, unsigned>> landed;  // (ring, use)
  int waits = 0, bad = 0;
  bool gave_up = false, raised = false;
  const auto issue = [&](int ring, int slot) {
    if (gave_up || (unsigned)slot != issued[ring] % slots[ring]) bad++;
    issued[ring]++;
  };
  dwfk::StreamProducer p;
  for (int nt : runs) {
    if (!p.ok) break;
    p.run(
        nt,
        [&](int ring, int slot, unsigned par) {  // the use before the next one of the slot was read, so it had landed
          const unsigned k = issued[ring] - slots[ring];
          if ((unsigned)slot != k % slots[ring] || par != ((k / slots[ring]) & 1)) bad++;
          if (waits++ >= fail) { gave_up = true; return false; }
          landed.insert({ring, k});
          return true;
        },
        [&](int, int slot) { issue(dwfk::RING_C, slot); }, [&](int, int slot) { issue(dwfk::RING_L, slot); },
        [&](int, int part, int slot) { issue(dwfk::RING_Y + part, slot); });
  }
  p.finish(
      [&](int ring, int slot, unsigned par) {
        for (unsigned k = issued[ring]; k-- > 0;)
          if (k % slots[ring] == (unsigned)slot) {
            if (par == ((k / slots[ring]) & 1)) landed.insert({ring, k});
            break;
          }
        return true;
      },
      [&]() { raised = true; });
  for (int r = 0; r < 4; r++)
    for (unsigned k = 0; k < issued[r]; k++)
      if (!landed.count({r, k})) { std::printf("fail %d: ring %d use %u in flight\n", fail, r, k); bad++; }
  return bad + (raised != gave_up);
}

int main() {
  int bad = 0;
  const std::vector<std::vector<int>> all = {{1}, {2}, {3}, {7}, {1, 1, 1}, {4, 2, 5}, {32, 5}};
  for (const auto& runs : all) {
    int n = 8;
    for (int nt : runs) n += 4 * nt + 2;
    for (int fail = 0; fail <= n; fail++) bad += produce(runs, fail);
  }
  std::printf("bad %d\n", bad);
  return bad != 0;
}
"""


def test_streaming_hop_producer_leaves_nothing_in_flight(tmp_path):
    """Also where it is a consumer that gave up (no wait of the producer fails)
    and where the z half of a halo step failed after its y half was issued."""
    _run(tmp_path, STREAM)
