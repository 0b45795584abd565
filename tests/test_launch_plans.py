"""The launch plans of pf16_plan.h, compiled for the host on their own: the split-K
reduction's groups of splits for every split count the weight gradients take, the
buffer ring of the pipelined stem pooling under every order of its events, and the load
modes that the GEMM is launched with."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_1911_07384_gb300.build import CSRC

SHIM = """
#include "pf16_plan.h"
extern "C" void splitk(int splits, long long total, int* out) {
  const pf16::SplitkPlan p = pf16::splitk_plan(splits, total);
  out[0] = p.tree_groups_log2, out[1] = p.leaves_log2, out[2] = p.groups_log2, out[3] = p.leaf_step;
}
extern "C" int modes_ok(int a, int b, int transform) { return pf16::gemm_modes_ok(a, b, transform != 0); }
// stage, full barrier and parity of tiles start, start + by, ...
extern "C" void ring(int start, int by, int stages, int groups, int n, int* out) {
  pf16::RingPos r = pf16::ring_start(start);
  for (int i = 0; i < n; ++i, r.advance(by, stages, pf16::ring_bars(stages, groups)))
    out[3 * i] = r.stage, out[3 * i + 1] = r.bar, out[3 * i + 2] = (int)r.phase;
}
"""


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    d = tmp_path_factory.mktemp("plans")
    (d / "shim.cpp").write_text(SHIM)
    cxx = shutil.which("g++") or shutil.which("c++")
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "shim.so"),
                    str(d / "shim.cpp")], check=True)
    return ctypes.CDLL(os.path.join(str(d), "shim.so"))


@pytest.mark.parametrize("total", [64, 96, 128, 256, 303, 304, 305, 512, 1152, 4096, 20000, 77823, 77824, 131072])
def test_splitk_groups(plans, total):
    """A CTA's 256 threads hold every group of a chunk, a thread at most 16 splits, and
    groups and splits per thread multiply to the padded split count."""
    out = (ctypes.c_int * 4)()
    for splits in list(range(1, 1025)) + [2048, 4096]:
        plans.splitk(splits, ctypes.c_longlong(total), out)
        tree, leaves, groups, step = out
        assert 0 <= groups <= 8 and 0 <= leaves <= 4, (splits, tuple(out))
        assert groups + leaves == (splits - 1).bit_length(), (splits, tuple(out))
        assert 0 <= tree <= 8 and tree <= groups + leaves, (splits, tuple(out))
        # a group lies inside a run of the tree, or is two single splits half of them apart
        if groups >= tree:
            assert step == 1
        else:
            assert leaves == 1 and groups + 1 == tree and step == 1 << groups


def _positions(plans, start, by, stages, groups, n):
    out = (ctypes.c_int * (3 * n))()
    plans.ring(start, by, stages, groups, n, out)
    return [tuple(out[3 * i:3 * i + 3]) for i in range(n)]


@pytest.mark.parametrize("stages,groups", [(2, 2), (3, 2), (4, 2), (3, 1), (3, 3), (4, 3), (5, 3)])
def test_ring_waits(plans, stages, groups):
    """Every reachable order of copies issued and landed (in any order) and of groups passing
    their waits and releasing their buffers: a wait by parity (true while the barrier's
    present phase has the other parity) never passes before its own tile's copy has landed,
    every tile is taken, and the schedule cannot stop."""
    tiles = 3 * stages * groups + 2
    prod = _positions(plans, 0, 1, stages, groups, tiles)
    cons = {g + groups * i: p for g in range(groups)
            for i, p in enumerate(_positions(plans, g, groups, stages, groups, (tiles - g + groups - 1) // groups))}
    bars = 1 + max(p[1] for p in prod)
    # state: tiles issued, those of them in flight, and each group's steps (even: waiting for
    # its next tile, odd: holding it)
    todo, seen = [(0, frozenset(), (0,) * groups)], set()
    while todo:
        state = todo.pop()
        if state in seen:
            continue
        seen.add(state)
        issued, flight, steps = state
        landed = [u for u in range(issued) if u not in flight]
        phase = [sum(prod[u][1] == b for u in landed) for b in range(bars)]
        freed = [sum(prod[g + groups * i][0] == s for g in range(groups) for i in range(steps[g] // 2))
                 for s in range(stages)]
        nxt = [(issued, flight - {u}, steps) for u in flight]
        if issued < tiles and freed[prod[issued][0]] == issued // stages:
            nxt.append((issued + 1, flight | {issued}, steps))
        for g in range(groups):
            u = g + groups * (steps[g] // 2)
            if u >= tiles:
                continue
            if steps[g] % 2 == 0:
                stage, bar, parity = cons[u]
                if phase[bar] % 2 == parity:
                    continue
                assert u in landed, f"group {g} passes the wait for tile {u} before its copy has landed: {state}"
                assert stage == prod[u][0]
            nxt.append((issued, flight, steps[:g] + (steps[g] + 1,) + steps[g + 1:]))
        assert nxt or all(g + groups * (steps[g] // 2) >= tiles for g in range(groups)), f"stopped in {state}"
        todo += nxt


def test_gemm_load_modes(plans):
    """Six pairs, two of them with an operand transform; every other is refused."""
    tiled_k, tiled_mn, im2col_k, im2col_mn, tap3d_mn = range(5)
    pairs = {(tiled_k, tiled_k), (im2col_k, tiled_k), (tiled_k, tiled_mn), (im2col_k, tap3d_mn),
             (tiled_mn, tiled_mn), (tiled_mn, im2col_mn)}
    for a in range(-1, 7):
        for b in range(-1, 7):
            assert bool(plans.modes_ok(a, b, 0)) == ((a, b) in pairs)
            assert bool(plans.modes_ok(a, b, 1)) == ((a, b) in {(tiled_k, tiled_k), (tiled_mn, tiled_mn)})
