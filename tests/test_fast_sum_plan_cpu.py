"""Host side of the near image sum by expansions (csrc/fmm.cu), without a GPU: where
fmm_plan and fmm_fit put the boxes, run by a small program (tests/native) whose device
allocations and copies land in host memory."""
import math
import os
import subprocess

import numpy as np
import pytest

from paper_1912_04501_gb300 import _build, workloads

HERE = os.path.dirname(os.path.abspath(__file__))
ORDERS = {0: 24, 1: 48, 2: 48}  # series per precision: single, double, double-float


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("plan") / "fast_sum_plan")
    objs = [os.path.join(_build.BUILD, os.path.splitext(s)[0] + ".o") for s in _build.SOURCES]
    _build.build(force=not all(map(os.path.exists, objs)))
    wrap = [a for f in ("Malloc", "Free", "MemcpyAsync", "MemsetAsync", "StreamSynchronize", "GetLastError")
            for a in ("-Xlinker", "--wrap=cuda" + f)]
    subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "-O1", "-o", exe,
                    os.path.join(HERE, "native", "fast_sum_plan.cu"), *objs, *wrap], check=True)
    return exe


def _run(exe, cell, *commands, doubled=0):
    """Per command (status, {precision: (on, walls, held, boxes or None)}); boxes:
    (ox, oy, h, gx, gy, levels, wall level, first centre)."""
    text = [f"{doubled} 24 1", *(f"{v!r}" for v in [*map(float, cell["e1"]), *map(float, cell["e2"]),
                                                    *map(float, cell["centre"])]), str(len(cell["bodies"]))]
    for b in cell["bodies"]:
        text.append(f"{b['n']} {b['a']!r} {b['b']!r} {float(b['xc'][0])!r} {float(b['xc'][1])!r}")
    for c in commands:
        if c[0] == "plan":
            text.append(f"plan {c[1]}")
        else:
            text.append("set " + " ".join(repr(float(v)) for v in [*c[1], *np.ravel(c[2])]))
    r = subprocess.run([exe], input=" ".join(text), capture_output=True, text=True, check=True, timeout=60)
    out = []
    for line in r.stdout.splitlines():
        w = line.split()
        if w[0] in ("plan", "set", "freed"):
            out.append((dict(zip(w[1::2], map(int, w[2::2]))), {}))
        elif w[0] == "prec":
            prec = int(w[1])
            out[-1][1][prec] = (int(w[3]), int(w[5]), int(w[7]), None)
        else:
            out[-1][1][prec] = (*out[-1][1][prec][:3], [float(v) for v in w[1:]])
    return out


def _nodes(cell, xc):
    xs, ws = [], []
    for b, x in zip(cell["bodies"], xc):
        t = 2 * np.pi * np.arange(b["n"]) / b["n"]
        c, s = math.cos(b["theta"]), math.sin(b["theta"])
        p = np.stack([b["a"] * np.cos(t), b["b"] * np.sin(t)], 1)
        d = np.stack([-b["a"] * np.sin(t), b["b"] * np.cos(t)], 1)
        xs.append(p @ np.array([[c, s], [-s, c]]) + np.asarray(x))
        ws.append(2 * np.pi / b["n"] * np.linalg.norm(d, axis=1))
    return np.concatenate(xs) - np.asarray(cell["centre"]), np.concatenate(ws)


def _tail(cell, e2, xc, box, order):
    """Largest first term left out of the walls' series, sum_j w_j (|eta_j| / |W|)^P over
    sum_j w_j, over the collocation points and far images."""
    ox, oy, h, _, _, _, wall = box[:7]
    if wall < 0:
        return 0.0
    X, w = _nodes(cell, xc)
    H = h * 2 ** wall
    centre = np.array([ox, oy]) + (np.floor((X - [ox, oy]) / H) + 0.5) * H
    eta = np.linalg.norm(X - centre, axis=1)
    s = 0.5 * np.polynomial.legendre.leggauss(24)[0]
    e1, e2 = np.asarray(cell["e1"], float), np.asarray(e2, float)
    worst = 0.0
    for a, b in ((e1, e2), (e2, e1)):
        for k in (-1, 0, 1):
            for shift in (-2 * a + k * b, a + k * b):
                p = (-0.5 * a + s[:, None] * b - shift)[:, None]
                r = eta / np.linalg.norm(p - centre[None], axis=2)
                worst = max(worst, float((w * np.minimum(r, 10.0) ** order).sum(1).max() / w.sum()))
    return worst


def relisted(cell, past):
    """The same suspension with bodies listed by another lattice image, their centres up to
    `past` beyond the cell (in lattice coordinates) yet inside the rectangle around it."""
    e1, e2, c = (np.asarray(cell[k], float) for k in ("e1", "e2", "centre"))
    E = np.column_stack([e1, e2])
    half = 0.5 * (abs(e1[0]) + max(abs(e2[0]), 0.5 * abs(e1[0])))
    xc, moved = [], 0
    for b in cell["bodies"]:
        x = np.asarray(b["xc"], float) - c
        s = np.linalg.solve(E, x)
        for m in (-1, 1):
            if 0.5 < abs(s[0] + m) <= 0.5 + past and abs(x[0] + m * e1[0]) < half:
                x = x + m * e1
                moved += 1
                break
        xc.append(x + c)
    return np.array(xc), moved


@pytest.mark.parametrize("skew", [0.0, -0.3, -0.45, 0.45])
@pytest.mark.parametrize("bodies,nodes", [(25, 256), (60, 130)])
def test_boxes_follow_a_configuration(program, skew, bodies, nodes):
    """Whatever configuration is set, the boxes hold every node and the walls' series
    leave out less than single precision's or double's rounding (sizes that
    bie_apply_static takes: the boxes' counts never change)."""
    cell = workloads.random_cell(bodies, 0.3, (1.0, 3.0), 5e-3, nodes, 1001, e2=(skew, 1.0))
    home = np.array([b["xc"] for b in cell["bodies"]])
    rng = np.random.default_rng(3)
    states = [(cell["e2"], home), *[(cell["e2"], relisted(cell, p)[0]) for p in (0.1, 0.3, 0.45)],
              (cell["e2"], home + rng.integers(-1, 2, (len(home), 1)) * np.asarray(cell["e1"])),
              ((0.9 * skew, 0.6), home), ((skew, 1.7), home), (cell["e2"], home + [3.0, 0.0]), (cell["e2"], home)]
    assert skew == 0 or relisted(cell, 0.45)[1] > 0
    res = _run(program, cell, ("plan", 0), *[("set", e2, xc) for e2, xc in states])
    for (e2, xc), (status, precs) in zip([(cell["e2"], home), *states], res):
        assert status["rc"] == 0
        X = _nodes(cell, xc)[0]
        for prec, (on, walls, _, box) in precs.items():
            assert on and walls
            ox, oy, h, gx, gy = box[:5]
            assert (X >= [ox, oy]).all() and (X <= [ox + gx * h, oy + gy * h]).all()
            assert box[7] == np.float32(ox + 0.5 * h) and box[8] == np.float32(oy + 0.5 * h)
            assert _tail(cell, e2, xc, box, ORDERS[prec]) < (6e-8 if prec == 0 else 1e-12), (prec, e2)
    # back where it began: the boxes as planned
    assert res[len(states)][1] == res[0][1]


@pytest.mark.parametrize("seed", [1, 2, 3])
@pytest.mark.parametrize("bodies,nodes", [(3, 1024), (25, 256), (100, 160)])
def test_walls_series_of_sheared_cells(program, bodies, nodes, seed):
    """The double series leave out less than a rounding for every source, whatever the
    shear, where a box's corner nearest to an image holds the source farthest from the
    box's centre."""
    for skew in (0.3, 0.45, 0.5):
        cell = workloads.random_cell(bodies, 0.3, (1.0, 3.0), 1e-2 if bodies < 60 else 2e-3, nodes, 1000 + seed,
                                     e2=(skew, 1.0), equal_area=seed != 2, max_tries=2000000)
        precs = _run(program, cell, ("plan", 0))[0][1]
        home = np.array([b["xc"] for b in cell["bodies"]])
        for prec in (1, 2):
            on, walls, _, box = precs[prec]
            assert on and walls
            assert _tail(cell, cell["e2"], home, box, ORDERS[prec]) < 1e-16, (prec, skew)


@pytest.mark.parametrize("doubled", [0, 1])
def test_short_memory_leaves_the_direct_sum(program, doubled):
    """An allocation that fails costs its precision the boxes (the moments', all three),
    never the context: no error is left, nothing half made stays, and a configuration can
    be set all the same."""
    cell = workloads.random_cell(40, 0.25, (1.0, 2.0), 5e-3, 200, 2, e2=(0.2, 1.0))
    home = np.array([b["xc"] for b in cell["bodies"]])
    for fail in range(0, 5):
        plan, state, end = _run(program, cell, ("plan", fail), ("set", cell["e2"], home + [0.4, 0.0]), doubled=doubled)
        off = {0: (), 1: (0,), 2: (1,), 3: (2,), 4: (0, 1, 2)}[fail]
        for status, precs in (plan, state):
            assert status["rc"] == 0 and status["error"] == 0
            assert status["calls"] == 4
            assert status["live"] == (0 if fail == 4 else 4 - len(off)) and status["work"] == (fail != 4)
            for prec, (on, _, held, _) in precs.items():
                assert (on, held) == ((0, 0) if prec in off else (1, 1))
        assert end[0]["live"] == 0


def test_large_cells_are_planned_anew(program):
    """Beyond the sizes that bie_apply_static takes, a configuration that leaves the grid
    gets another one (the leaves stay as small as they were), memory permitting."""
    cell = workloads.random_cell(60, 0.25, (1.0, 2.0), 5e-3, 200, 2, e2=(0.2, 1.0))
    home = np.array([b["xc"] for b in cell["bodies"]])
    away = home + np.array([[4.0 * (k == 5), 0.0] for k in range(len(home))])
    for fail in (0, 6, 8):
        plan, inside, out, back, end = _run(program, cell, ("plan", fail), ("set", cell["e2"], home),
                                            ("set", cell["e2"], away), ("set", cell["e2"], home))
        assert inside[1] == plan[1] and (inside[0]["calls"], out[0]["calls"], back[0]["calls"]) == (4, 8, 8)
        off = {0: (), 6: (1,), 8: (0, 1, 2)}[fail]
        X = _nodes(cell, away)[0]
        for status, precs in (out, back):
            assert status["rc"] == 0 and status["error"] == 0
            assert status["live"] == (0 if fail == 8 else 4 - len(off)) and status["work"] == (fail != 8)
            for prec, (on, _, held, box) in precs.items():
                assert (on, held) == ((0, 0) if prec in off else (1, 1))
                if on:
                    ox, oy, h, gx, gy = box[:5]
                    assert h < 1.5 * plan[1][prec][3][2]
                    assert (X >= [ox, oy]).all() and (X <= [ox + gx * h, oy + gy * h]).all()
        assert end[0]["live"] == 0
