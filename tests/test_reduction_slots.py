"""The interior point's reductions over the grid share a few slots of partial
results: a block that writes a slot must know that every block has read it.

The parts of an iteration are followed in the order in which the kernels call
them, with the slots that each reduction writes and reads and the grid barriers
between them as the source has them.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1908_05834_gb300", "csrc")
EVENT = re.compile(r"ip_partials<(\w+), (\d+)>\(|ip_totals\(S, A\.part, (\d+), (\d+)\)|(bar\.sync)\(\)|(ip_check)<")


def _events(source, name):
    """("write" | "read", slots) and ("barrier", ()) of a part, in order."""
    body = re.search(r"\bbool %s\(.*?\n}\n" % name, source, re.S).group(0)
    out = []
    for m in EVENT.finditer(body):
        if m.group(1):
            out.append(("write", [0] * (m.group(1) != "false") + list(range(1, int(m.group(2)) + 1))))
        elif m.group(3):
            out.append(("read", list(range(int(m.group(3)), int(m.group(4))))))
        elif m.group(5):
            out.append(("barrier", []))
        elif name != "ip_check":
            out += _events(source, "ip_check")
    return out


def test_no_slot_is_written_before_all_blocks_have_read_it():
    with open(os.path.join(CSRC, "ip.cuh")) as f:
        source = f.read()
    for parts in (["ip_check"], ["ip_steps", "ip_corrector"], ["ip_steps", "ip_step"],
                  ["ip_steps", "ip_corrector", "ip_steps", "ip_step"]):
        unread, written = set(), set()  # read, or written, since the last barrier
        seen = 0
        for part in parts:
            for what, slots in _events(source, part):
                seen += what != "barrier"
                if what == "barrier":
                    unread, written = set(), set()
                elif what == "write":
                    assert not unread & set(slots), f"{parts}: {part} writes slots that other blocks may still read"
                    written |= set(slots)
                else:
                    assert not written & set(slots), f"{parts}: {part} reads slots that other blocks may not have written"
                    unread |= set(slots)
        assert seen >= 2 * len(parts)
