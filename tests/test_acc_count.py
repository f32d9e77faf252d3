"""The rule that keeps the accumulator's words from overflowing (csrc/acc_count.h), run on the host over random orders
of launches, captured graphs that are replayed or dropped, and resets."""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_26691_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "acc_count.h"
using namespace st;

struct Op { bool clear; double base, add; bool far; };

// what a word can hold: digits since its carries were last propagated, and far commits among them
struct Word {
  double digits = 0; bool far = false;
  void check(unsigned seed) const {
    // 2^31 digits, 2^30 beside far commits (2^20 to spare)
    const double limit = far ? 1073741824.0 + 1048576.0 : 2147483648.0;
    if (digits > limit) { std::printf("seed %u: %.0f digits, far %d\n", seed, digits, (int)far); std::exit(1); }
  }
};

int main() {
  for (unsigned seed = 0; seed < 3000; ++seed) {
    std::mt19937 rng(seed);
    auto below = [&](double n) { return std::uniform_real_distribution<double>(0, n)(rng); };
    AccCount host; AccDeviceCount dev{0, 0, 0}; Word w;
    std::vector<std::vector<Op>> graphs;
    const double most = seed % 3 ? 1073741824.0 : 3e8;  // digits of a launch
    auto execute = [&](const Op& o) {  // on the device, in device mode
      if (o.clear) { acc_cleared(dev); w = Word(); return; }
      if (acc_decide(dev, o.base, o.add)) w = Word{1, false};
      w.digits += o.add; w.far = w.far || o.far; w.check(seed);
    };
    auto op = [&](bool capturing) -> Op {
      Op o{below(1) < 0.05, 0, (double)(long long)below(most), below(1) < 0.3};
      if (o.clear) {
        if (!host.cleared(capturing)) w = Word();
        return o;
      }
      const AccCount::Action act = host.launch(o.add, o.far, capturing);
      if (act == AccCount::kAskDevice) { o.base = host.adds; return o; }
      if (act == AccCount::kPropagate) w = Word{1, false};
      w.digits += o.add; w.far = w.far || o.far; w.check(seed);
      return o;
    };
    for (int i = 0; i < 60; ++i) {
      const double r = below(1);
      if (i > 10 && r < 0.1) {  // captured, not run
        graphs.emplace_back();
        for (int k = 1 + (int)below(3); k > 0; --k) graphs.back().push_back(op(true));
      } else if (!graphs.empty() && r < 0.4) {
        for (const Op& o : graphs[(size_t)below(graphs.size())]) execute(o);
      } else {
        const bool on_device = host.on_device;
        const Op o = op(false);
        if (on_device) execute(o);
      }
    }
  }
  return 0;
}
"""


def test_no_word_can_overflow(tmp_path):
    src = tmp_path / "acc.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "acc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("prec,grid,sort", [("fp64", 16, False), ("mixed_f32", 16, True), ("mixed_f32", 12, False),
                                            ("mixed_bf16", 16, True)])
@pytest.mark.parametrize("replays", [0, 1, 3])
def test_captured_steps_replay_as_steps(prec, grid, sort, replays):
    """Steps captured into a graph, replayed some times (or dropped) between steps that are not: the state and the
    sources, bit for bit, of the same steps one after the other; after a reset too."""
    import torch

    from paper_2603_26691_gb300 import inputs
    from paper_2603_26691_gb300.sim import Sim

    n, dt = 5000, 1e-3
    pos, vel, d, _ = inputs.particles(1, 0, n, vmax=1.0)
    out = []
    for captured in (False, True):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            sim = Sim(grid, precision=prec, stream=stream)
            sim.set_params(reorder_every=0)
            sim.set_fluid(inputs.taylor_green(grid))
            sim.add_particles(pos, d, vel)
            if sort:
                sim.reorder()
            sim.step(2, dt)
            got = []
            if captured:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream):
                    sim.step(3, dt)
            for _ in range(2):
                for _ in range(replays):
                    if captured:
                        graph.replay()
                    else:
                        sim.step(3, dt)
                    sim.step(1, dt)
                got.append(sim.sources(host=True, reset=True))
            stream.synchronize()
            got += sim.particles()
            sim.close()
        out.append(got)
    for a, b in zip(*out):
        assert np.array_equal(a, b)
