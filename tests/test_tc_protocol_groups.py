"""CPU model of conv2's in-place schedule in gf_flow_tc.cu for any number of
epilogue groups (issuing thread r and group r take every NG-th tile through a
ring of nb accumulators; a group writes h2 of tile t over h1 once tiles
.. t + r have completed): no deadlock exactly when r <= NG nb + (r mod NG), no
accumulator refilled before it is read, no write under a queued read; and the
rings that the launches use."""
import ctypes as C
import random

import pytest

from test_tc_protocol import geometry


def fits(r, nb, ng):
    return r <= ng * nb + r % ng


def conv2_phase(nt, r, nb, ng, p_first, rng):
    """One conv2 phase under a random schedule; False if it deadlocks."""
    queue = {g: [] for g in range(ng)}          # issued, not completed (in order per thread)
    issued, drained, waiting = [0] * ng, [0] * ng, [False] * ng
    done, filled = set(), [set() for _ in range(ng)]
    tiles = [list(range(g, nt, ng)) for g in range(ng)]
    wrote = [0] * ng
    while any(wrote[g] < len(tiles[g]) for g in range(ng)):
        moves = []
        for g in range(ng):
            if issued[g] < len(tiles[g]) and issued[g] - drained[g] < nb:
                moves.append(("issue", g))
            if queue[g]:
                moves.append(("mma", g))
            if not waiting[g] and drained[g] < len(tiles[g]) and tiles[g][drained[g]] in done:
                moves.append(("drain", g))
            if waiting[g] and all(t in done for t in range(min(tiles[g][wrote[g]] + r, nt - 1) + 1)):
                moves.append(("write", g))
        if not moves:
            return False
        kind, g = rng.choice(moves)
        if kind == "issue":
            slot = issued[g] % nb
            assert slot not in filled[g], "accumulator refilled before it was read"
            filled[g].add(slot)
            queue[g].append(tiles[g][issued[g]])
            issued[g] += 1
        elif kind == "mma":
            done.add(queue[g].pop(0))
        elif kind == "drain":
            filled[g].discard(drained[g] % nb)
            drained[g] += 1
            waiting[g] = True
        else:
            t = tiles[g][wrote[g]]
            lo, hi = p_first + 96 * t, p_first + 96 * t + 95
            for u in set(range(nt)) - done:     # queued now or issued later
                assert 96 * u + 96 + 2 * p_first - 1 < lo or 96 * u > hi, "h2 written over positions still to be read"
            wrote[g] += 1
            waiting[g] = False
    return True


@pytest.mark.parametrize("ng", [2, 4])
@pytest.mark.parametrize("nd,L", [(2, 8), (2, 64), (3, 8), (3, 12), (3, 16)])
@pytest.mark.parametrize("nb", [1, 2, 3, 4, 8])
def test_deadlocks_exactly_when_the_rings_are_short(nd, L, nb, ng):
    p_first, nt, r = geometry(nd, L)
    for seed in range(4):
        ok = conv2_phase(nt, r, nb, ng, p_first, random.Random(seed))
        assert ok == (fits(min(r, nt - 1), nb, ng) or fits(r, nb, ng)), (nt, r)


def test_rings_of_four_groups_fit_every_shape():
    from paper_2208_08903_gb300 import _abi
    lib = _abi.load()
    n = 0
    for nd, Ls in ((2, range(4, 66, 2)), (3, range(4, 18, 2))):
        for L in Ls:
            for c, n2 in ((8, 32), (16, 48)):
                hid = (C.c_int32 * _abi.GF_MAX_HIDDEN)(*([c, c] + [0] * (_abi.GF_MAX_HIDDEN - 2)))
                if lib.gf_flow_tensor_core_supported(C.byref(_abi.FlowShapeExC(nd, L, 4, 2, hid, 3, 1, 0.01))):
                    assert fits(geometry(nd, L)[2], min(4, 512 // (4 * n2)), 4), (nd, L, c)
                    n += 1
    assert n >= 10
