"""The lanes per restart of a plain launch, asked of the host function itself:
its one pass over the library chooses what the estimate summed ligand by
ligand in FP64 chooses, and does not take longer than a few reads of the
offsets."""
import ctypes as C
import math
import time

import numpy as np
import pytest

from paper_2303_06150_gb300 import build

SMS = 152
# lanes, and slots of the shapes with few and with many increments in flight
SLOTS = {8: (2, 5), 16: (1, 3), 32: (1, 2)}
# chain (us, us per cost) and throughput (cost per us) of 8, 16 and 32 lanes
MODELS = [(8, 60.0, 0.0085, 1.294e6), (16, 42.0, 0.0030, 0.908e6), (32, 42.0, 0.0023, 0.498e6)]


@pytest.fixture(scope="module")
def pick():
    f = C.CDLL(build.build())._ZN5ligen15dock_pick_lanesEPKiS1_iiiiiii
    f.argtypes = [C.c_void_p] * 2 + [C.c_int] * 7

    def bind(atoms, rot, R, n_rigid, n_theta, passes, fmt=0):
        a, r = (np.concatenate([[0], np.cumsum(v)]).astype(np.int32) for v in (atoms, rot))
        args = (a.ctypes.data, r.ctypes.data, len(atoms), R, n_rigid, n_theta, passes, fmt, SMS)
        return lambda keep=(a, r): f(*args)
    return bind


def _sweep(G, n_theta):
    """Increments in flight of the shape with the fewest slots that hold them all, and its chunks."""
    slots = next((s for s in SLOTS[G] if G * s >= n_theta), SLOTS[G][-1])
    return slots, -(-n_theta // (G * slots))


def _estimate(atoms, rot, R, n_rigid, n_theta, passes):
    if len(atoms) * R > 400 * SMS:
        return {8: 0.0}
    N, n = np.asarray(atoms, float), np.asarray(rot, float)
    rigid, moving = n_rigid * N, passes * n * (N + 4) / 4
    out = {}
    for G, us, per_cost, rate in MODELS:
        slots, chunks = _sweep(G, n_theta)
        s36, c36 = _sweep(G, 36)
        work = (rigid + 36 * G * slots * chunks / (G * s36 * c36) * moving + 2000).sum()
        longer = chunks * slots ** 0.5 / (c36 * s36 ** 0.5) - 1
        chain = (rigid + 36 * moving).max() + 36 * longer * moving.max()
        out[G] = math.hypot(us + per_cost * chain, work * R / rate)
    return out


def test_one_pass_chooses_what_the_sums_choose(pick):
    rng = np.random.default_rng(1)
    seen = set()
    for _ in range(4000):
        L = int(np.exp(rng.uniform(0, np.log(1500))))
        atoms = rng.integers(1, int(rng.integers(2, 257)), L)
        rot = rng.integers(0, int(rng.integers(1, 34)), L)
        args = (int(np.exp(rng.uniform(0, np.log(300)))), int(rng.integers(1, 25)),
                int(rng.choice([1, 2, 4, 12, 24, 36, 72, 180])), int(rng.choice([0, 1, 2, 3, 10, 1000])))
        est = _estimate(atoms, rot, *args)
        got = pick(atoms, rot, *args, fmt=int(rng.integers(0, 3)))()
        assert est[got] <= min(est.values()) * (1 + 1e-9)
        seen.add(got)
    assert seen == {8, 16, 32}


# measured launches (256 restarts, 24 rotations, 3 passes) whose fastest lanes are well ahead of the others
@pytest.mark.parametrize("ligands,atoms,rot,n_theta,fastest", [
    (40, (24, 52), (2, 10), 180, (16, 32)), (20, (24, 52), (2, 10), 180, (16, 32)), (80, (24, 52), (2, 10), 120, (16, 32)),
    (20, (100, 120), (20, 30), 180, (16, 32)), (5, (100, 120), (20, 30), 180, (32,)), (40, (100, 120), (20, 30), 120, (16, 32)),
    (160, (100, 120), (20, 30), 12, (8,)), (160, (24, 52), (2, 10), 12, (8,)), (80, (12, 24), (1, 3), 180, (16,))])
def test_other_increments(pick, ligands, atoms, rot, n_theta, fastest):
    rng = np.random.default_rng(0)
    assert pick(rng.integers(atoms[0], atoms[1] + 1, ligands), rng.integers(rot[0], rot[1] + 1, ligands), 256, 24,
                n_theta, 3)() in fastest


def test_host_time_of_a_large_library(pick):
    def best(f):
        t = []
        for _ in range(100):
            t0 = time.perf_counter()
            f()
            t.append(time.perf_counter() - t0)
        return min(t)

    off = np.arange(60001, dtype=np.int64)
    # three of numpy's passes over 60,000 numbers: 48 us where this takes 54 and three scalar FP64 passes took 287
    yard = best(lambda: (np.diff(off).max(), (off * off).sum(), off.max()))
    assert best(pick(np.full(60000, 20), np.full(60000, 3), 1, 24, 36, 3)) <= 3 * yard
