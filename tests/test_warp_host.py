"""The arithmetic of the kernels' warp operations (csrc/warp.cuh), compiled for the host and checked there."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), 'paper_1809_05608_gb300', 'csrc')


def _run(tmp_path, body):
    nvcc = shutil.which('nvcc') or '/usr/local/cuda/bin/nvcc'
    if not os.path.exists(nvcc):
        pytest.skip('no nvcc')
    src = tmp_path / 't.cu'
    src.write_text('#include <cstdio>\n#include <cstdlib>\n#include "warp.cuh"\nusing namespace mgfld;\n'
                   '#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\\n", __LINE__, #x); std::exit(1); } } '
                   'while (0)\n' + body)
    exe = tmp_path / 't'
    r = subprocess.run([nvcc, '-std=c++17', '-gencode', 'arch=compute_103a,code=sm_103a', '-I', CSRC, str(src), '-o',
                        str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


def test_reduction_members(tmp_path):
    """A reduction over a group's part of a warp: every lane of that part names all of it and nobody else, in blocks
    of whole groups of every size, the last warp of the block in part."""
    _run(tmp_path, '''
int main() {
  for (int n = 1; n <= 32; ++n)
    for (int threads = n; threads <= 256; threads += n)
      for (int t = 0; t < threads; ++t) {
        const int warp = t / 32 * 32, live = threads - warp < 32 ? threads - warp : 32;
        unsigned expect = 0;
        for (int l = 0; l < live; ++l)
          if ((warp + l) / n == t / n) expect |= 1u << l;
        CHECK(group_lanes(t - warp, t % n, n, live) == expect);
      }
}
''')


def test_no_members_left_to_convergence():
    """No kernel takes the lanes that happen to be converged for the members of an operation."""
    for name in os.listdir(CSRC):
        if name.endswith(('.cu', '.cuh')):
            assert '__activemask' not in open(os.path.join(CSRC, name)).read(), name


def test_wait_keeps_the_warp_together(tmp_path):
    """The wait of a warp whose lanes see the copy complete at different looks: every lane takes part in the same
    votes and comes out with the same answer."""
    _run(tmp_path, '''
int main() {
  // what each of 4 lanes sees at the first look and after the bounded wait
  for (int first = 0; first < 16; ++first)
    for (int last = 0; last < 16; ++last) {
      const bool vote[2] = {first == 15, last == 15};
      int votes0 = -1;
      for (int l = 0; l < 4; ++l) {
        int votes = 0;
        const bool got = warp_wait([&]() { return (first >> l & 1) != 0; }, [&]() { return (last >> l & 1) != 0; },
                                   [&](bool) { CHECK(votes < 2); return vote[votes++]; });
        if (l == 0) votes0 = votes;
        CHECK(votes == votes0 && got == (vote[0] || vote[1]));
      }
    }
}
''')


def test_copies_in_flight_when_a_wait_gives_up(tmp_path):
    """The ring uses a warp has to drain when the wait for use u gives up: the one waited for up to the last one issued,
    in the order in which the substitution issues and waits (the top-down half with its middle zone, the
    bottom-up half without)."""
    _run(tmp_path, '''
int main() {
  for (int S = 2; S <= 4; S *= 2)
    for (int NG = 0; NG <= 9; ++NG)
      for (int mid = 0; mid < 2; ++mid) {
        const int NU = 2 * NG + mid;
        int last = -1;
        auto issue = [&](int u) { if (u < NU) { CHECK(u == last + 1); last = u; } };
        auto wait = [&](int u) { CHECK(ring_last_issued(u, S, NU) == last && last >= u); };
        for (int u = 0; u < S; ++u) issue(u);
        if (NG > 0) wait(0);
        for (int v = 0; v < NG; ++v) {                       // inward
          if (v > 0) issue(v - 1 + S);
          if (v + 1 < NG) wait(v + 1);
        }
        int u = NG;
        if (mid) {
          wait(u);
          if (u > 0) issue(u - 1 + S);
          ++u;
        }
        if (NG > 0) wait(u);
        for (int w = 0; w < NG; ++w, ++u) {                  // outward
          if (u > 0) issue(u - 1 + S);
          if (w + 1 < NG) wait(u + 1);
        }
        CHECK(last == NU - 1 || NU == 0);
      }
}
''')
