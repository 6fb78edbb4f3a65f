"""The exchange of row maxima between the warps of the persistent row quantizers, on the CPU.

Per row group each warp writes its maximum to shared memory, passes one CTA barrier and reads the
maxima of all warps. Every interleaving of a few warps over a few groups is walked here: with one
buffer a fast warp's write for the next group can overtake a slow warp's read, with the buffers
taken in turn it cannot. The kernels' number of buffers is read from their source."""

import os
import re

import pytest

from paper_2606_07116_gb300 import build as B


def violations(warps, groups, bufs):
    """Whether some interleaving lets a read see another group's maximum. A warp's program per group
    is write, barrier, then one read per warp; a state is every warp's (group, step) and the buffers."""
    reads = warps
    steps = 2 + reads  # write, barrier, reads

    def at_barrier(pos, k):
        return pos[k] % steps == 1

    start = ((0,) * warps, tuple(((-1,) * warps) for _ in range(bufs)))
    seen, stack = {start}, [start]
    while stack:
        pos, mem = stack.pop()
        moves = []
        for k in range(warps):
            g, s = divmod(pos[k], steps)
            if g == groups or s == 1:
                continue
            new_mem = mem
            if s == 0:
                row = list(mem[g % bufs])
                row[k] = g
                new_mem = tuple(tuple(row) if b == g % bufs else mem[b] for b in range(bufs))
            elif mem[g % bufs][s - 2] != g:
                return True
            moves.append((tuple(p + 1 if i == k else p for i, p in enumerate(pos)), new_mem))
        # The barrier lets everyone through once every warp has arrived at the same group's.
        if all(at_barrier(pos, k) for k in range(warps)) and len({p // steps for p in pos}) == 1:
            moves.append((tuple(p + 1 for p in pos), mem))
        for m in moves:
            if m not in seen:
                seen.add(m)
                stack.append(m)
    return False


def _kernel_source(name):
    with open(os.path.join(B.CSRC, "quant.cu")) as f:
        text = f.read()
    start = text.index(f"{name}(const QuantArgs a) {{")
    bufs = re.search(r"constexpr int kRowMaxBufs = (\d+);", text)
    return text[start:text.index("\n}\n", start)], int(bufs.group(1)) if bufs else 1


def test_one_buffer_is_overtaken():
    assert violations(2, 2, 1)
    assert violations(3, 2, 1)


@pytest.mark.parametrize("kernel,array", [("quantize_rows_1k_kernel", "wmax"),
                                          ("quantize_mx_1k_kernel", "wmaxx")])
def test_kernels_take_enough_buffers_in_turn(kernel, array):
    body, bufs = _kernel_source(kernel)
    assert not violations(2, 4, bufs)
    assert not violations(3, 3, bufs)
    # The array has that many buffers, and every access names the group's.
    uses = re.findall(rf"\b{array}(\[[^\]]*\])", body)
    assert uses[0] == "[kRowMaxBufs]" and len(uses) == 3 and all(u == "[turn]" for u in uses[1:])
    assert bufs == 2 and body.count("const uint32_t turn = ring.turn();") == 1


@pytest.mark.parametrize("S", [1, 2, 3])
def test_ring_turn_is_the_parity_of_the_group(S):
    """RowRing::turn() from the slot and its phase."""
    s = phase = 0
    for i in range(6 * S):
        assert (s + (S & phase)) & 1 == i & 1
        s += 1
        if s == S:
            s, phase = 0, phase ^ 1
