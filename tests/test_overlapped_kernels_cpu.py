"""Kernels that may become resident before the launch ahead of them has ended: each begins with
start_after_previous(), and uses what it returns (a read-only load is held back by nothing else)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2101_07163_gb300", "csrc")


def sources():
    return {f: open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC))
            if f.endswith((".cu", ".cuh"))}


def kernel_bodies(text):
    """name -> body of every __global__ function (up to the brace that closes it)."""
    out = {}
    for m in re.finditer(r"__global__", text):
        head = re.compile(r"(\w+_kernel)\s*\(").search(text, m.end())
        i = text.index("{", head.end())
        depth, j = 1, i + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        out[head.group(1)] = text[i:j]
    return out


def test_every_overlapped_kernel_depends_on_its_wait():
    src = sources()
    bodies = {}
    for text in src.values():
        bodies.update(kernel_bodies(text))
    plain = {m for text in src.values() for m in re.findall(r"(\w+_kernel)(?:<[^;]*?>)?<<<", text)}
    overlapped = sorted(set(bodies) - plain)
    assert {"march_kernel", "row_kernel", "two_kernel", "two_tile_kernel", "adj_collide_kernel",
            "batch_two_kernel"} <= set(overlapped)
    for name in overlapped:
        uses = re.findall(r"(.*)start_after_previous\(\)", bodies[name])
        assert len(uses) == 1, name
        assert re.search(r"[+(]\s*$", uses[0]), name + " drops the result"
    for name in plain:
        assert "start_after_previous" not in bodies[name], name
