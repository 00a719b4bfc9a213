"""The hand-overs of the kernel that runs a depthwise 3x3 layer and the pointwise layer behind it in one launch, walked through on
the host for every way the library cuts such a pair: no role may wait for something that only its own later steps bring about."""
from collections import defaultdict

import pytest

SIZES = [(7, 7), (14, 14), (28, 28), (37, 37), (56, 56), (112, 112), (13, 17), (1, 126), (3, 130)]


def _roles(lay, tiles, res):
    """Every role of a CTA with `tiles` tiles as a generator: ("wait", barrier, phases that have to be complete) or ("done", barrier)."""
    S, parts, slots, bufs = lay["slabs"], lay["parts"], lay["slots"], lay["out_bufs"]

    def accumulator(e):      # of GEMM 2: index, uses before this one
        return (e & 1, e >> 1) if lay["accs2"] == 2 else (0, e)

    def activations():
        for u in range(tiles * S * lay["loads"]):
            i, use = u % lay["a_stages"], u // lay["a_stages"]
            yield "wait", ("empty", i), use
            yield "done", ("full", i)

    def diagonals():
        for v in range(tiles * S):
            yield "wait", ("dempty", v & 1), v >> 1
            yield "done", ("dfull", v & 1)

    def depthwise():
        u = 0
        for v in range(tiles * S):
            yield "wait", ("tempty1", v & 1), v >> 1
            yield "wait", ("dfull", v & 1), (v >> 1) + 1
            for _ in range(lay["loads"]):
                i, use = u % lay["a_stages"], u // lay["a_stages"]
                yield "wait", ("full", i), use + 1
                yield "done", ("empty", i)
                u += 1
            yield "done", ("dempty", v & 1)
            yield "done", ("tfull1", v & 1)

    def weights():
        for u in range(parts * S if lay["w_res"] else tiles * parts * S):
            i, use = u % lay["w_stages"], u // lay["w_stages"]
            yield "wait", ("wempty", i), use
            yield "done", ("wfull", i)

    def pointwise():
        u = 0
        for l in range(tiles):
            for q in range(parts):
                d, use2 = accumulator(l * parts + q)
                yield "wait", ("tempty2", d), use2
                for s in range(S):
                    g = l * S + s
                    if q == 0:
                        yield "wait", ("slot_full", g % slots), g // slots + 1
                    w = (q * S + s, 0) if lay["w_res"] else (u % lay["w_stages"], u // lay["w_stages"])
                    yield "wait", ("wfull", w[0]), w[1] + 1
                    if not lay["w_res"]:
                        yield "done", ("wempty", w[0])
                    if q == parts - 1:
                        yield "done", ("slot_free", g % slots)
                    u += 1
                yield "done", ("tfull2", d)

    def epilogue():
        o = 0
        for l in range(tiles + lay["defer"]):
            if l < tiles:
                for s in range(S):
                    g = l * S + s
                    yield "wait", ("slot_free", g % slots), g // slots
                    yield "wait", ("tfull1", g & 1), (g >> 1) + 1
                    yield "done", ("tempty1", g & 1)
                    yield "done", ("slot_full", g % slots)
            if l == 0 if lay["defer"] else l == tiles:
                continue
            for _ in range(parts):
                d, use2 = accumulator(o)
                yield "wait", ("res_full" if res else "out_free", o % bufs), o // bufs + (1 if res else 0)
                yield "wait", ("tfull2", d), use2 + 1
                yield "done", ("tempty2", d)
                yield "done", ("out_full", o % bufs)
                o += 1

    def mover():
        for o in range(tiles * parts):
            yield "wait", ("out_full", o % bufs), o // bufs + 1
            yield "done", ("out_free", o % bufs)

    def fetcher():
        for o in range(tiles * parts if res else 0):
            yield "wait", ("out_free", o % bufs), o // bufs
            yield "done", ("res_full", o % bufs)

    return [f() for f in (activations, diagonals, depthwise, weights, pointwise, epilogue, mover, fetcher)]


def _stuck(lay, tiles, res):
    """What the roles still wait for when none of them can go on ([]: all of them have finished)."""
    phases = defaultdict(int)
    pending = [[r, next(r, None)] for r in _roles(lay, tiles, res)]
    moved = True
    while moved:
        moved = False
        for p in pending:
            while p[1] is not None and (p[1][0] == "done" or phases[p[1][1]] >= p[1][2]):
                if p[1][0] == "done":
                    phases[p[1][1]] += 1
                p[1] = next(p[0], None)
                moved = True
    return [p[1] for p in pending if p[1] is not None]


def _layout(h, w, c, c_out, stride, n, res):
    from paper_2202_05239_b200 import api
    return api.f8_debug_dwpw_layout(api.ConvDesc(n, h, w, c, c, 3, 3, stride, 1, 0, 0, 0, 4, 7, 4, 0), c_out, res)


@pytest.mark.parametrize("res", [False, True])
def test_no_layout_waits_in_a_circle(res):
    seen = {}
    for h, w in SIZES:
        for stride in (1, 2):
            for c in range(16, 1281, 16):
                for c_out in list(range(16, 321, 16)) + [384, 512, 768, 1024]:
                    lay = _layout(h, w, c, c_out, stride, 2, res)
                    if lay is not None:
                        seen.setdefault(tuple(v for k, v in lay.items() if k not in ("wanted", "tiles")), (lay, (h, w, c, c_out, stride)))
    assert any(l["accs2"] == 1 and l["slabs"] > l["slots"] for l, _ in seen.values())      # one wide part: the narrowest of them all
    assert any(l["parts"] > 1 and l["defer"] for l, _ in seen.values())
    for lay, shape in seen.values():
        for tiles in (1, 2, 5):
            assert not _stuck(lay, tiles, res), (shape, lay, tiles, _stuck(lay, tiles, res))


def test_the_walk_finds_a_circle():
    """The walk itself: a wide part with a deferred second epilogue and more slabs than slots."""
    lay = dict(slabs=4, slots=2, parts=1, accs2=1, defer=1, loads=1, a_stages=3, w_stages=4, w_res=1, out_bufs=1)
    assert not _stuck(lay, 1, False) and _stuck(lay, 2, False)
    assert not _stuck(dict(lay, defer=0), 5, False) and not _stuck(dict(lay, accs2=2), 5, False)
