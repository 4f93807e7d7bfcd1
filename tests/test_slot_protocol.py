"""The INT4 GEMM's TMEM slots: who waits for which phase of which mbarrier, over every interleaving of its warp roles.

An mbarrier's parity tells a phase from its neighbours only.  A role that watches a use of a slot which others issue can come so late
that they are two phases further, and then waits for good; one that skips a use can take an older phase for the one it waits for.  The
walk of the two code-MMA warps is plain C++, compiled here; the roles around it are restated as lists of waits and arrivals, and every
state that the five of them can reach together is visited.
"""
import ctypes
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_27003_b200", "csrc")
MODEL = r"""
#include <algorithm>
#include <unordered_set>
#include <vector>
#include "tmem_slots.h"
using w4a4::CodeSlotWalk;

struct Op { bool wait; int bar; uint32_t parity; int done; };   // wait: `done` phases must have completed when it is let through
using Program = std::vector<Op>;
enum { EMPTY = 0, FULL = 2, OP_FULL = 4, OP_EMPTY = OP_FULL + 8, BARS = OP_EMPTY + 8 };

// 0: every state ends in completion; 1: a wait let through before its phase; 2: a state from which nobody can go on; 3: a use in the wrong slot
static int explore(const std::vector<Program>& roles, const int* counts) {
  std::vector<std::vector<std::vector<int>>> arrivals(roles.size());   // [role][position][barrier]
  for (size_t a = 0; a < roles.size(); ++a) {
    std::vector<int> n(BARS, 0);
    arrivals[a].push_back(n);
    for (const Op& op : roles[a]) {
      if (!op.wait) ++n[op.bar];
      arrivals[a].push_back(n);
    }
  }
  std::vector<std::vector<int>> stack = {std::vector<int>(roles.size(), 0)};
  std::unordered_set<uint64_t> seen;
  auto key = [&](const std::vector<int>& s) { uint64_t k = 0; for (int pc : s) k = k * 256 + pc; return k; };
  seen.insert(key(stack[0]));
  while (!stack.empty()) {
    const std::vector<int> s = stack.back();
    stack.pop_back();
    bool moved = false, finished = true;
    for (size_t a = 0; a < roles.size(); ++a) {
      if (s[a] == static_cast<int>(roles[a].size())) continue;
      finished = false;
      const Op& op = roles[a][s[a]];
      if (op.wait) {
        int n = 0;
        for (size_t b = 0; b < roles.size(); ++b) n += arrivals[b][s[b]][op.bar];
        const int phases = n / counts[op.bar];
        if ((phases & 1u) == op.parity) continue;   // the phase of that parity is the running one
        if (phases < op.done) return 1;
      }
      moved = true;
      std::vector<int> t = s;
      ++t[a];
      if (seen.insert(key(t)).second) stack.push_back(t);
    }
    if (!moved && !finished) return 2;
  }
  return 0;
}

// `observer`: the two code warps share the groups of a stage instead of the slots, the second one watches a tile's first use; and
// without that wait (2).
extern "C" int slots(int tiles, int lr_stages, int groups, int ring, int observer) {
  const int stages = (groups + 1) / 2;
  std::vector<Program> roles(6);   // producer, code warps, scale warp, two epilogue warps
  int counts[BARS];
  for (int i = 0; i < BARS; ++i) counts[i] = i < FULL ? 2 : (i < OP_FULL ? 2 : (i < OP_EMPTY ? 1 : 3));
  bool wrong = false;
  auto wait = [&](int role, int bar, uint32_t parity, int done) { roles[role].push_back({true, bar, parity, done}); };
  auto arrive = [&](int role, int bar) { roles[role].push_back({false, bar, 0, 0}); };
  auto stage_full = [&](int role, int n) { wait(role, OP_FULL + n % ring, (n / ring) & 1, n / ring + 1); };
  auto stage_done = [&](int role, int n) { arrive(role, OP_EMPTY + n % ring); };
  // the release of the slot's previous use: use u is the (u / 2)th of slot u % 2
  auto slot_free = [&](int role, int u) { wait(role, EMPTY + u % 2, ((u / 2) & 1) ^ 1, u / 2); };
  for (int w = 0; w < 2; ++w) {
    CodeSlotWalk walk(w);
    int use = 0, stage = 0;
    auto issue = [&](int u) {   // by the walk's own account of slot and parity
      wrong = wrong || walk.own != static_cast<uint32_t>(u % 2);
      arrive(1 + w, FULL + walk.own);
      walk.issued();
    };
    auto own_free = [&](int u) { wait(1 + w, EMPTY + walk.own, walk.free_parity(), u / 2); };
    for (int tile = 0; tile < tiles; ++tile) {
      if (observer == 1) slot_free(1 + w, use);
      if (lr_stages > 0) {
        const bool mine = observer ? w == 0 : walk.owns_next();
        if (mine && !observer) own_free(use);
        if (mine && observer == 2) slot_free(1 + w, use);
        for (int l = 0; l < lr_stages; ++l) stage_full(1 + w, stage), stage_done(1 + w, stage++);
        if (mine) observer ? arrive(1 + w, FULL + use % 2) : issue(use);
        walk.pass(1), ++use;
      }
      const int v = observer ? w : static_cast<int>(walk.group());
      for (int st = 0; st < stages; ++st) {
        stage_full(1 + w, stage);
        const int in_stage = std::min(2, groups - 2 * st);
        if (v < in_stage) {
          const int u = use + 2 * st + v;
          if (observer) slot_free(1 + w, u), arrive(1 + w, FULL + u % 2);
          else own_free(u), issue(u);
        }
        stage_done(1 + w, stage++);
      }
      walk.pass(groups), use += groups;
    }
  }
  const int uses = (lr_stages > 0) + groups, n_stages = lr_stages + stages;
  for (int n = 0; n < tiles * n_stages; ++n) {
    wait(0, OP_EMPTY + n % ring, ((n / ring) & 1) ^ 1, n / ring);
    arrive(0, OP_FULL + n % ring);
  }
  int use = 0, stage = 0;
  for (int tile = 0; tile < tiles; ++tile) {
    if (lr_stages > 0) {
      slot_free(3, use), arrive(3, FULL + use % 2), ++use;
      for (int l = 0; l < lr_stages; ++l) stage_full(3, stage), stage_done(3, stage++);
    }
    for (int st = 0; st < stages; ++st) {
      stage_full(3, stage);
      for (int v = 0; v < std::min(2, groups - 2 * st); ++v) slot_free(3, use), arrive(3, FULL + use % 2), ++use;
      stage_done(3, stage++);
    }
  }
  for (int e = 4; e < 6; ++e)
    for (int u = 0; u < tiles * uses; ++u) wait(e, FULL + u % 2, (u / 2) & 1, u / 2 + 1), arrive(e, EMPTY + u % 2);
  for (const Program& p : roles) if (p.size() > 255) return -1;
  return wrong ? 3 : explore(roles, counts);
}
"""


@pytest.fixture(scope="module")
def slots(tmp_path_factory):
    d = tmp_path_factory.mktemp("slots")
    src, lib = d / "slots.cpp", d / "slots.so"
    src.write_text(MODEL)
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, "-o", str(lib), str(src)], check=True)
    return ctypes.CDLL(str(lib)).slots


@pytest.mark.parametrize("lr_stages", [0, 1, 3])
@pytest.mark.parametrize("groups", [1, 2, 3, 4, 5])
def test_no_interleaving_stalls_or_runs_early(slots, lr_stages, groups):
    for ring in (2, 5):
        assert slots(4, lr_stages, groups, ring, 0) == 0


@pytest.mark.parametrize("lr_stages,groups", [(0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (3, 4)])
def test_the_model_finds_a_warp_that_only_watches(slots, lr_stages, groups):
    # The second code warp does not issue a tile's first use: a poll after its release and the next use's of that slot stalls.
    assert slots(4, lr_stages, groups, 5, 1) == 2


@pytest.mark.parametrize("lr_stages,groups", [(0, 3), (1, 2)])
def test_the_model_finds_a_wait_for_an_older_phase(slots, lr_stages, groups):
    # Without that wait an odd number of uses per tile moves a warp to the other slot, one phase of which it has not seen.
    assert slots(4, lr_stages, groups, 5, 2) in (1, 2)


def test_no_warp_wide_instruction_hangs_on_a_lanes_own_answer():
    # PTX: a .sync.aligned instruction under a predicate that the lanes of a warp see differently is undefined.  So in each inline
    # assembly block the predicate's last writer in front of such an instruction is a vote.
    guarded = 0
    for name in sorted(n for n in os.listdir(CSRC) if n.endswith((".cu", ".cuh", ".h"))):
        for block in re.findall(r"asm\s*(?:volatile)?\s*\((.*?)\);", open(os.path.join(CSRC, name)).read(), flags=re.S):
            code = re.sub(r"//[^\n]*", "", "".join(re.findall(r'"((?:[^"\\]|\\.)*)"', block))).replace("\\n", "\n")
            lines = [line.strip() for line in re.split(r"[;\n]", code) if line.strip()]
            for i, line in enumerate(lines):
                m = re.match(r"@!?(\w+)\s+\S*\.sync\.aligned", line)
                if m is None:
                    continue
                guarded += 1
                writers = [w for w in lines[:i] if re.match(rf"(?!@|\.reg)\S+\s+{m.group(1)}\b", w)]
                assert writers and writers[-1].startswith("vote.sync.all.pred"), (name, line)
    assert guarded > 0


@pytest.mark.gpu
@pytest.mark.parametrize("K,r", [(64, 0), (64, 16), (128, 32), (192, 0), (192, 96), (704, 64)])
def test_a_late_issuing_warp_changes_nothing(K, r):
    import torch
    import paper_2605_27003_b200 as w4
    from test_gpu_parity import guarded, guards_intact
    from workloads import generator as gen
    # Three tiles per CTA and more, every parity of slot uses per tile; 20 us are some twenty of these tiles.
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N, dev = 2560, "cuda:0"
    M = 128 * (-(-3 * sms // (N // 128))) + 33
    x = gen.make_activations(M, K, seed=3)
    layer = gen.make_layer_svd(K, N, r, x[:1024], seed=4, bias_std=0.01)
    ctx = w4.Context(0, M, K, r)
    lay = w4.Layer(ctx, [layer.to(dev)], num_bins=1)
    xd, clip = x.to(dev), torch.full((1, 1, 1), 0.9, dtype=torch.float32, device=dev)
    y = torch.empty(M, N, dtype=torch.bfloat16, device=dev)
    w4.w4a4_linear_forward(lay.ptr, xd, M, 0, 0, clip, y)
    for warp in (1, 2, 3):
        buf, late = guarded((M, N), torch.bfloat16, 1234.0)
        w4.w4a4_debug_late_gemm(lay.ptr, M, 0, late, warp, 20000)
        torch.cuda.synchronize()
        ctx.check()
        assert torch.equal(y, late) and guards_intact(buf, 1234.0)
    lay.close()
    ctx.close()
