"""CPU model of the block schedule of the cluster eigensolver (hj_eig_kernel): the columns lie in two blocks of b per CTA;
a sweep rotates the pairs inside the blocks, then in every round all pairs of the CTA's two blocks, after which the blocks
move by the circle method.  The model checks what the kernel relies on: every pair of columns meets exactly once a
sweep, the pairs of a step are disjoint, no two blocks land in one place, and 2 Ce - 1 moves bring every block home, which
the final look-up of the eigenvalues uses.  The shapes are read from the kernel's source."""
import os
import re

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2306_00632_gb300", "csrc", "eig_hj.cu")


def _shapes():
    """(C, RPL, BT) of the launches."""
    with open(SRC) as f:
        found = re.findall(r"HjShape<\w+, (\d+), (\d+), (\d+)>;", f.read())
    return [tuple(map(int, s)) for s in found]


def _deal(C, BT, rc):
    """CTAs that take part and columns of a block."""
    Ce = max(1, min(C, (rc + 2 * BT - 1) // (2 * BT)))
    return Ce, max(1, ((rc + Ce - 1) // Ce + 1) // 2)


def _home(Ce, b):
    """blocks[cta][block]: the columns of each; position g of block blk of CTA c holds column (2 g + blk) Ce + c."""
    return [[[(2 * g + blk) * Ce + c for g in range(b)] for blk in range(2)] for c in range(Ce)]


def _steps(Ce, b, blocks):
    """The pairs of every step of a sweep; blocks is moved along."""
    even = (b + 1) & ~1
    for step in range(even - 1):
        pairs = []
        for c in range(Ce):
            for blk in range(2):
                for k in range(even // 2):
                    i, j = (even - 1, step) if k == 0 else ((step + k) % (even - 1), (step - k) % (even - 1))
                    i, j = min(i, j), max(i, j)
                    if j < b:
                        pairs.append((blocks[c][blk][i], blocks[c][blk][j]))
        yield pairs
    for _ in range(2 * Ce - 1):
        for k in range(b):
            yield [(blocks[c][0][g], blocks[c][1][(g + k) % b]) for c in range(Ce) for g in range(b)]
        if Ce == 1:
            continue
        landed = {}
        for c in range(Ce):   # top blocks move right (the first stays), bottom blocks left
            top = (0, 0) if c == 0 else ((Ce - 1, 1) if c == Ce - 1 else (c + 1, 0))
            bottom = (1, 0) if c == 0 else (c - 1, 1)
            for place, block in ((top, blocks[c][0]), (bottom, blocks[c][1])):
                assert place not in landed
                landed[place] = block
        assert len(landed) == 2 * Ce
        for (c, blk), block in landed.items():
            blocks[c][blk] = block


@pytest.mark.parametrize("Ce", range(1, 17))
@pytest.mark.parametrize("b", [1, 2, 3, 4, 5, 8, 9])
def test_every_pair_once_and_blocks_home(Ce, b):
    blocks = _home(Ce, b)
    met = set()
    for pairs in _steps(Ce, b, blocks):
        cols = [x for p in pairs for x in p]
        assert len(cols) == len(set(cols))
        for p in pairs:
            p = tuple(sorted(p))
            assert p not in met
            met.add(p)
    n = 2 * Ce * b
    assert len(met) == n * (n - 1) // 2
    assert blocks == _home(Ce, b)


def test_shapes_hold_their_columns():
    shapes = _shapes()
    assert len(shapes) >= 5
    for C, RPL, BT in shapes:
        rows = 32 * RPL
        bmax = (rows // C + 1) // 2
        assert 2 * bmax <= 32   # one lane per column in the search for the pivot
        assert (rows - 1) // C < 2 * bmax   # the Cholesky's columns of one CTA
        for rc in range(1, rows + 1):
            Ce, b = _deal(C, BT, rc)
            assert b <= bmax and 2 * b * Ce >= rc
            # idle CTAs and columns past rc: player k is where the last look-up expects it
            home = _home(Ce, b)
            assert sorted(x for c in home for blk in c for x in blk) == list(range(2 * b * Ce))


@pytest.mark.parametrize("rc,C,BT", [(5, 4, 4), (17, 8, 4), (40, 16, 4), (33, 4, 12)])
def test_rotations_in_this_order_converge(rc, C, BT):
    g = np.random.default_rng(rc)
    A = g.standard_normal((rc + 3, rc))
    sv = np.linalg.svd(A, compute_uv=False)
    Ce, b = _deal(C, BT, rc)
    for _ in range(12):
        rotated = False
        for pairs in _steps(Ce, b, _home(Ce, b)):
            for p, q in pairs:
                if p >= rc or q >= rc:
                    continue
                x, y = A[:, p].copy(), A[:, q].copy()
                prod = x @ y
                if abs(prod) <= 1e-14 * np.linalg.norm(x) * np.linalg.norm(y):
                    continue
                rotated = True
                d = y @ y - x @ x
                t = 2 * prod / (d + np.copysign(np.hypot(d, 2 * prod), d))
                u = t / (1 + np.sqrt(1 + t * t))
                s = 2 * u / (1 + u * u)
                x -= u * y   # the kernel's shears
                y += s * x
                x -= u * y
                A[:, p], A[:, q] = x, y
        if not rotated:
            break
    assert not rotated
    assert np.allclose(np.sort(np.linalg.norm(A, axis=0))[::-1], sv, rtol=1e-12)
