"""Host model of the order of the mixed paths' U cubes and of the epilogue's lanes (no GPU).

Every group tensor is stored as its term of W (C0[a][b][c] = U0, C1[b][a][c] =
U1, C2[b][c][a] = U2) in 8^3 cubes, the three group terms of a cube side by side
and U^g[a][b][c] at ucube_off(a & 7, b & 7, c & 7) of its cube, a innermost
(tcorr_internal.cuh, store_u_cubes).  The epilogue's lane 8 j + i of warp w takes
b = i, c = i ^ j ^ 4 (w & 1) and a = i ^ n(j) ^ (w >> 1), then a ^ 4, of an orbit's
cubes (epilogue.cu).
"""
import itertools

import numpy as np
import pytest

N = (0, 2, 3, 1)
PERMS = list(itertools.permutations(range(3)))


def ucube_off(la, lb, lc):
    return (lb << 6) | (lc << 3) | la


def lanes(w, h):
    for lane in range(32):
        i, j = lane & 7, lane >> 3
        yield i ^ N[j] ^ (w >> 1) ^ (4 * h), i, i ^ j ^ ((w & 1) << 2)


def test_n_is_the_kernels_expression():
    assert [((j & 1) << 1) ^ ((j >> 1) * 3) for j in range(4)] == list(N)


def test_lanes_cover_every_element_orbit_once():
    got = sorted(t for w in range(8) for h in range(2) for t in lanes(w, h))
    assert got == sorted(itertools.product(range(8), repeat=3))


@pytest.mark.parametrize("perm", PERMS)
def test_every_read_touches_32_banks(perm):
    for w, h in itertools.product(range(8), range(2)):
        ts = [tuple(t[p] for p in perm) for t in lanes(w, h)]
        assert len({(x * 64 + y * 8 + z) % 32 for x, y, z in ts}) == 32  # a cube term
        assert len({(x * 8 + y) % 32 for x, y, _ in ts}) == 32           # an 8 x 8 ovov block


@pytest.mark.parametrize("pb", [4, 8, 16])
def test_a_warps_store_is_whole_sectors_in_runs(pb):
    pc = 128 // pb
    for wq in range(4):  # 32 rows of the tile, 8 values of a: (cube, 32-byte sector) of each lane
        rows = [divmod(r, pc) for r in range(32 * wq, 32 * wq + 32)]
        cells = {((b >> 3, c >> 3), ucube_off(0, b & 7, c & 7) // 8) for b, c in rows}
        assert len(cells) == 32
        for cube in {c for c, _ in cells}:
            s = sorted(x for c, x in cells if c == cube)
            assert s == list(range(s[0], s[0] + len(s)))  # one run per cube


@pytest.mark.parametrize("v", [8, 13, 21])
def test_stores_and_epilogue_reads_agree(v):
    rng = np.random.default_rng(v)
    nb = (v + 7) // 8
    U = [rng.standard_normal((v, v, v)) for _ in range(3)]
    task = np.full(3 * nb ** 3 * 512, np.nan)
    for b, c, a in itertools.product(range(v), repeat=3):
        A, B, C = a >> 3, b >> 3, c >> 3
        cubes = ((A * nb + B) * nb + C) * 3, ((B * nb + A) * nb + C) * 3 + 1, ((B * nb + C) * nb + A) * 3 + 2
        for g in range(3):
            task[cubes[g] * 512 + ucube_off(a & 7, b & 7, c & 7)] = U[g][a, b, c]
    for x, y, z in itertools.product(range(v), repeat=3):
        base = (((x >> 3) * nb + (y >> 3)) * nb + (z >> 3)) * 3 * 512
        lx, ly, lz = x & 7, y & 7, z & 7
        # the reads of slot (x, y, z): (middle, fast, slow), (slow, fast, middle), (slow, middle, fast)
        w = (task[base + ly * 64 + lz * 8 + lx] + task[base + 512 + lx * 64 + lz * 8 + ly]
             + task[base + 1024 + lx * 64 + ly * 8 + lz])
        assert w == pytest.approx(U[0][x, y, z] + U[1][y, x, z] + U[2][z, x, y], rel=1e-14, abs=1e-14)


SLOTS = [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]  # abc, acb, bac, bca, cab, cba


@pytest.mark.parametrize("kind,orbit", [(2, (0, 0, 1)), (3, (0, 1, 1)), (4, (1, 1, 1))])
def test_repeated_blocks_meet_every_element_once(kind, orbit):
    """The element orbits and slot masks of the epilogue's repeated-block form."""
    trip = [(x, y, z) for x in range(8) for y in range(x, 8) for z in range(y, 8)]
    pair = [(x, y) for x in range(8) for y in range(x, 8)]
    if kind == 4:
        els = trip
    elif kind == 2:
        els = [(x, y, z) for x, y in pair for z in range(8)]
    else:
        els = [(x, y, z) for y, z in pair for x in range(8)]
    met = []
    for la, lb, lc in els:
        ab, bc = kind != 3 and la == lb, kind != 2 and lb == lc
        count = (1 if bc else 0x13) if ab else (0xd if bc else 0x3f)
        e = [(orbit[0], la), (orbit[1], lb), (orbit[2], lc)]
        met += [tuple(e[d] for d in SLOTS[q]) for q in range(6) if count >> q & 1]
    want = {tuple((p[d], l[d]) for d in range(3)) for p in {tuple(orbit[d] for d in s) for s in SLOTS}
            for l in itertools.product(range(8), repeat=3)}
    assert len(met) == len(set(met)) and set(met) == want


def test_slot_composition():
    """P[q]: the slots of acb, bac, cba, bca, cab of the element at slot q."""
    P = [(1, 2, 5, 3, 4), (0, 4, 3, 5, 2), (3, 0, 4, 1, 5), (2, 5, 1, 4, 0), (5, 1, 2, 0, 3), (4, 3, 0, 2, 1)]
    for q, s in enumerate(SLOTS):
        want = [tuple(s[d] for d in SLOTS[k]) for k in (1, 2, 5, 3, 4)]
        assert [SLOTS[k] for k in P[q]] == want
