"""Kernels launched while their predecessor drains (programmatic dependent launch), read as source: they wait before
they touch memory, and promise nothing about buffers that the predecessor still writes."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_01076_gb300", "csrc")

# uploaded by copies in front of the first launch of a chain; no kernel writes them
COPIED = ("BatchSweep", "int2", "int")


def kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__ void\s*(?:__launch_bounds__\([^{;]*?\)\s*)?(\w+)\(([^{;]*?)\)\s*\{", text):
            depth, at = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[at], 0)
                at += 1
            yield m.group(1), m.group(2), text[m.end():at]


def test_dependent_kernels_promise_nothing_about_the_state():
    seen = []
    for name, params, body in kernels():
        if "follow_predecessor()" not in body:
            continue
        seen.append(name)
        for p in params.split(","):
            if "__restrict__" in p:
                assert re.match(r"\s*const (%s) \*__restrict__" % "|".join(COPIED), p), (name, p)
        # pointer parameters are read behind the wait only
        before = body[:body.index("follow_predecessor()")]
        for p in re.findall(r"\*(?:__restrict__ )?\s*(\w+)", params):
            assert not re.search(r"\b%s\b" % p, before), (name, p)
    assert sorted(seen) == ["batch_sweep_kernel", "step_kernel", "sweep_kernel", "tile_kernel"]


def test_every_dependent_launch_is_of_a_waiting_kernel():
    waiting = {name for name, _, body in kernels() if "follow_predecessor()" in body}
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = open(path).read()
        for m in re.finditer(r"launch_following\((\w+)", text):
            if m.group(1) == "void":            # the definition
                continue
            names = {m.group(1)} if m.group(1) != "kernel" else set(re.findall(r"kernel = (?:seam \? )?(\w+_kernel)", text))
            assert names and names <= waiting, (path, names)
