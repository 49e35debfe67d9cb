"""The multi-step kernel's hand-out, checked in its source: the orders of memory that a run on one GPU
cannot show."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2608_23786_gb300", "csrc", "stepper_march.cuh")


def _body(name):
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    start = text.index("{", re.search(rf"\b(?:void|bool) {name}\(", text).start())
    depth = 0
    for k in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return text[start:k]


def test_the_counters_of_all_lanes_are_ordered_before_the_tile_is_handed_out():
    """Several lanes acquire a counter each and one lane publishes the tile; __all_sync and
    __any_sync order no memory, __syncwarp does: it stands between the looks and the publication."""
    body = _body("march_hand_out")
    looks = body.rindex("__any_sync")
    publish = body.index("if (lane == 0) {", looks)
    assert body.index("ld_acquire_gpu") < looks < publish < body.index("st_release_cta(out", publish)
    assert "__syncwarp()" in body[looks:publish]


def test_every_warp_of_a_tile_orders_its_lanes_before_it_arrives():
    body = re.sub(r"//[^\n]*", "", open(SRC).read())
    arrive = body.rindex("mbar_arrive(")
    assert "__syncwarp()" in body[body.rindex("scatter_all", 0, arrive):arrive]


def test_a_wait_gives_up_by_time_and_by_looks():
    """Time alone would take a launch that was switched out for a second for one without progress."""
    body = _body("march_give_up").replace("\n", " ")
    assert re.search(r"looks < kMarchLimitLooks \|\| global_ns\(\) - t0 <= kMarchLimitNs\) return false", body)
    calls = re.findall(r"march_give_up\(([^)]*)\)", re.sub(r"//[^\n]*", "", open(SRC).read()))
    assert len(calls) == 4 and calls.count("t0, it, a.err") == 3
