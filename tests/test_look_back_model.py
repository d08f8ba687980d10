"""The order the fold kernels' look-back has to give: a slot is stored by the tile of its last access, after
every tile its accesses run through has read its initial value.

The model is the happens-before relation of the memory model, over one chain of tiles: program order within a
thread, a release and the acquire that reads it, and barriers (of the block or of the warp) among the threads
that meet at them.  Shuffles are left out: they move values and order nothing."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_10158_gb300", "csrc")


def chain(warp_barrier, tiles=4, lanes=3, seen_lane=2):
    """Edges between events (tile, thread, step).  In each tile but the first, lane `seen_lane` acquires the
    descriptor of the tile before and lane 0 releases the tile's own."""
    edges = set()

    def program(tile, thread, steps):
        for a, b in zip(steps, steps[1:]):
            edges.add(((tile, thread, a), (tile, thread, b)))

    def barrier(tile, before, after):
        for i in range(lanes):
            for j in range(lanes):
                edges.add(((tile, i, before), (tile, j, after)))

    for t in range(tiles):
        for i in range(lanes):
            program(t, i, ["load", "loaded", "look", "acquired", "release", "published", "carried", "store"])
        barrier(t, "load", "loaded")                     # the values read come before the block's barrier
        if warp_barrier:
            barrier(t, "acquired", "release")            # the look-back's end
        barrier(t, "published", "carried")               # the carry handed to the block
        if t:
            edges.add(((t - 1, 0, "release"), (t, seen_lane, "acquired")))
    return edges


def reaches(edges, a, b):
    follow = {}
    for x, y in edges:
        follow.setdefault(x, []).append(y)
    todo, seen = [a], {a}
    while todo:
        for y in follow.get(todo.pop(), ()):
            if y not in seen:
                seen.add(y)
                todo.append(y)
    return b in seen


def ordered(edges, tiles=4, lanes=3):
    return all(reaches(edges, (t, i, "load"), (tiles - 1, j, "store"))
               for t in range(tiles - 1) for i in range(lanes) for j in range(lanes))


def test_every_load_comes_before_the_store():
    assert ordered(chain(warp_barrier=True))


def test_without_the_warp_barrier_the_chain_breaks():
    """A tile's WHOLE stands for all tiles before it, but the acquire of those was another lane's."""
    assert not ordered(chain(warp_barrier=False))
    assert ordered(chain(warp_barrier=False, seen_lane=0))        # the lane that publishes


def test_the_source_has_the_barrier():
    text = open(os.path.join(CSRC, "det_common.cuh")).read()
    at = text.index("S look_back(")
    body = re.sub(r"//[^\n]*", "", text[at:text.index("\n}\n", at)])
    assert "ld128_acquire" in body and "return" in body
    assert re.search(r"__syncwarp\(\);\s*return sum;\s*$", body.rstrip())
    assert body.count("return") == 1                              # on every way out
    for name in ("det_fold.cu", "det_oe.cu"):                     # and nobody looks back without it
        code = open(os.path.join(CSRC, name)).read()
        assert "ld128_acquire" not in code and re.search(r"look_back<\w+>\(desc", code), name
