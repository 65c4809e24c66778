"""The 2D pruning pass's closed forms (cp_prune.cu works them out for 32
vertices at a time), compared with the lookup table on all 256 masks: the H0
link, where each top cell held by a vertex dies, and which vertices have
survivors or a root."""
import pytest

import prune_restatement as pr


@pytest.fixture(scope="module")
def lib():
    from paper_2606_04801_gb300 import _lib, build

    build.build()
    return _lib.load()


def test_closed_forms(lib):
    for raw in range(512):
        if raw & 16:
            continue
        e = pr.entry(lib, 2, raw)
        n = [(raw >> k) & 1 for k in range(9)]
        up, left, right, down = n[1], n[3], n[5], n[7]
        co = [n[0] & up & left, n[2] & up & right, n[6] & down & left, n[8] & down & right]
        # the first face in L(v) in the order up, left, right, down
        faces = [up, left, right, down]
        assert (e & 7) == (faces.index(1) if any(faces) else 7)
        # quadrants 0, 1 die across +y, 2 across +x, 3 towards the highest one not held
        for t in range(4):
            code = (e >> (9 + 4 * t)) & 15
            if not co[t]:
                assert code == 15, (raw, t)
            elif t < 2:
                assert code == t + 2
            elif t == 2:
                assert code == 3
            else:
                rest = [k for k in (2, 1, 0) if not co[k]]
                assert code == (rest[0] if rest else 8)
        # the faces not followed, around the vertex, by a quadrant: exactly one unless there is an event
        s = [up & ~co[1], right & ~co[3], down & ~co[2], left & ~co[0]]
        h0, dual = (e >> 3) & 0x3F, (e >> 41) & 0xFFF
        event = bool(h0 or dual or (e & 7) == 7 or all(co))
        assert event == (sum(v & 1 for v in s) != 1), raw
        assert h0 < 16 and dual < 16
