"""The FP32 QL sweep on a tridiagonal T (csrc/lanczos.cu, ql_fp32) under any order in which a warp's lanes may run: every
lane computes the rotations from shared d and e while lane 0 writes their new values, so each rotation needs a warp
barrier between a lane's reads and lane 0's stores.  The lanes run here as Python generators that give way at every
shared access, with the barriers that the source has."""
import os
import random
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = open(os.path.join(ROOT, "paper_2205_02491_gb300", "csrc", "lanczos.cu")).read()
F = np.float32


def rotation_loop():
    body = SRC[SRC.index("bool ql_fp32("):]
    body = body[:body.index("\n}\n")]
    loop = body[body.index("for (; i >= l; --i) {"):]
    return loop[:re.search(r"\n      }\n", loop).start()]


def barrier_in_loop():
    """A warp barrier after the rotation's reads and before lane 0's stores."""
    loop = re.sub(r"//[^\n]*", "", rotation_loop())
    store = loop.index("if (lane == 0)")
    return "__syncwarp()" in loop[loop.index("d[i]"):store]


def lane_sweeps(lane, sh, Z, barrier):
    """One lane of ql_fp32 on sh = {"d", "e"} and its row Z of the eigenvectors; yields "sync" at a barrier."""
    d, e = sh["d"], sh["e"]
    k = len(d)
    for l in range(k):
        for _ in range(60):
            yield "sync"
            small = [i >= k - 1 or abs(e[i]) <= F(5.9604645e-8) * (abs(d[i]) + abs(d[i + 1]) + F(1e-3)) for i in range(l, k)]
            mm = l + small.index(True)
            yield "sync"  # the ballots
            if mm == l:
                break
            el, dl, dl1 = e[l], d[l], d[l + 1]
            yield
            g = (dl1 - dl) / (F(2) * el)
            h = np.sqrt(g * g + F(1))
            g = d[mm] - dl + el / (g + (h if g >= 0 else -h))
            yield
            sn, cs, p, di1 = F(1), F(1), F(0), d[mm]
            z0 = Z[mm]
            for i in range(mm - 1, l - 1, -1):
                yield
                f, b, di = sn * e[i], cs * e[i], d[i]
                q = f * f + g * g
                if not q > F(1e-36):
                    sh["failed"].add(lane)
                    return
                if barrier:
                    yield "sync"
                ri = F(1) / np.sqrt(q)
                c0 = Z[i]
                sn, cs = f * ri, g * ri
                g = di1 - p
                t = (di - g) * sn + F(2) * cs * b
                p = sn * t
                yield
                if lane == 0:
                    e[i + 1] = q * ri
                    d[i + 1] = g + p
                g = cs * t - b
                Z[i + 1] = sn * c0 + cs * z0
                z0 = cs * c0 - sn * z0
                di1 = di
            Z[l] = z0
            yield "sync"
            if lane == 0:
                d[l] -= p
                e[l] = g
                e[mm] = F(0)
            yield "sync"


def run_warp(d, e, seed, barrier):
    """seed None: the lanes in lockstep."""
    k = len(d)
    sh = {"d": d.copy(), "e": e.copy(), "failed": set()}
    Z = [np.eye(k, dtype=F)[r] for r in range(k)]
    lanes = {r: lane_sweeps(r, sh, Z[r], barrier) for r in range(k)}
    rnd = random.Random(seed)
    at_barrier = set()
    while lanes:
        free = [r for r in lanes if r not in at_barrier]
        if not free:
            at_barrier.clear()
            continue
        for r in (free if seed is None else [rnd.choice(free)]):
            try:
                if next(lanes[r]) == "sync":
                    at_barrier.add(r)
            except StopIteration:
                del lanes[r]
    return sh, np.stack(Z)


@pytest.mark.parametrize("k", [2, 3, 6])
def test_lanes_may_run_in_any_order(k):
    g = np.random.default_rng(k)
    d, e = g.standard_normal(k).astype(F), np.append(g.uniform(0.3, 1.0, k - 1), 0.0).astype(F)
    with np.errstate(all="ignore"):
        ref, Zr = run_warp(d, e, None, True)
        assert not ref["failed"]
        T = np.diag(d.astype(float)) + np.diag(e[:-1].astype(float), 1) + np.diag(e[:-1].astype(float), -1)
        assert np.max(np.abs(np.sort(ref["d"]) - np.linalg.eigvalsh(T))) <= 32 * k * 2.0 ** -24 * np.linalg.norm(T, 2)
        for seed in range(60):
            sh, Z = run_warp(d, e, seed, barrier_in_loop())
            assert not sh["failed"] and np.array_equal(sh["d"], ref["d"]) and np.array_equal(Z, Zr), seed
