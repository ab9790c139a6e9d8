"""The shared-memory rings of the tensor-core kernels that two warps issue from, as a
model on the host: every order in which the loader, the two issuing warps, the
copies and the MMAs' completions can interleave, with the mbarriers' parity
waits.  No order may end with a wait that nothing satisfies, or let a warp use
a slot that does not hold its slice.  Arrival counts and who arrives are read
from the kernels' sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2102_11576_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def explore(slots, slices, release, counts, acts):
    """First fault over all interleavings, or None.

    slices: loads in order, slice q into slot q % slots; release(q): the
    (barrier, phase) the loader waits for before it loads q, or None.  counts: arrivals
    per phase of every releasing barrier.  acts[w][q]: what warp w does once it has
    seen slice q land: (barrier, "mma"), (barrier, "arrive") or None."""
    names = sorted(counts)
    at = {b: k for k, b in enumerate(names)}
    warps = len(acts)

    def arrive(bars, b):  # bars: (phase, arrivals so far) of every releasing barrier
        k = at[b]
        ph, n = bars[k]
        n += 1
        return bars[:k] + (((ph + 1, 0) if n == counts[b] else (ph, n)),) + bars[k + 1:]

    # (next load, loads in flight, full phases, slice each slot holds, issuers' positions, commits in flight, bars)
    start = (0, frozenset(), (0,) * slots, (-1,) * slots, (0,) * warps, ((),) * warps, ((0, 0),) * len(names))
    seen, todo = {start}, [start]
    while todo:
        q, flying, full, holds, pos, commits, bars = todo.pop()
        nxt = []
        if q < slices:
            r = release(q)
            if r is None or (bars[at[r[0]]][0] & 1) != (r[1] & 1):
                nxt.append((q + 1, flying | {q}, full, holds, pos, commits, bars))
        for f in flying:
            s = f % slots
            nxt.append((q, flying - {f}, full[:s] + (full[s] + 1,) + full[s + 1:], holds[:s] + (f,) + holds[s + 1:],
                        pos, commits, bars))
        for w in range(warps):
            p = pos[w]
            if p < slices and (full[p % slots] & 1) != ((p // slots) & 1):
                act = acts[w][p]
                c, b = commits, bars
                if act and act[1] == "mma":
                    if holds[p % slots] != p:
                        return f"warp {w} multiplies slice {holds[p % slots]} for {p}"
                    c = c[:w] + (c[w] + (act[0],),) + c[w + 1:]
                elif act:
                    b = arrive(b, act[0])
                nxt.append((q, flying, full, holds, pos[:w] + (p + 1,) + pos[w + 1:], c, b))
            if commits[w]:
                nxt.append((q, flying, full, holds, pos, commits[:w] + (commits[w][1:],) + commits[w + 1:],
                            arrive(bars, commits[w][0])))
        if not nxt and not (q == slices and all(p == slices for p in pos)):
            return f"stuck: next load {q}, issuers at {pos}"
        for n in nxt:
            if n not in seen:
                seen.add(n)
                todo.append(n)
    return None


def alternating(stages, slices, arrivals, bystander):
    """dst_gemm_tile.inc, two issuing warps: warp w multiplies the slices of its parity."""
    empty = [f"empty{s}" for s in range(stages)]
    acts = [[(empty[q % stages], "mma") if (q & 1) == w else ((empty[q % stages], "arrive") if bystander else None)
             for q in range(slices)] for w in range(2)]
    return explore(stages, slices, lambda q: (empty[q % stages], q // stages - 1) if q >= stages else None,
                   {b: arrivals for b in empty}, acts)


def digits(slices, arrivals, bystander):
    """digit.cuh: eight digit tiles a slice in a ring of six; the top warp multiplies the first four."""
    step = [f"step{i}" for i in range(8)]
    tiles = 8 * slices
    top = [(step[q % 8], "mma") if q % 8 < 4 else ((step[q % 8], "arrive") if bystander else None)
           for q in range(tiles)]
    bottom = [(step[q % 8], "mma") for q in range(tiles)]
    return explore(6, tiles, lambda q: (step[(q - 6) % 8], (q - 6) // 8) if q >= 6 else None,
                   {b: arrivals(i) for i, b in enumerate(step)}, [top, bottom])


@pytest.mark.parametrize("stages,slices", [(2, 8), (3, 8), (4, 10)])
def test_alternating_issuers(stages, slices):
    src = source("dst_gemm_tile.inc")
    arrivals = {"1": 1, "kIssuers": 2}[re.search(r"mbar_init\(&empty\[s\], (\w+)\);", src).group(1)]
    assert alternating(stages, slices, arrivals, "mbar_arrive(&empty[s])" in src) is None
    assert alternating(stages, slices, 1, False) is not None  # the owner's release alone does not do


@pytest.mark.parametrize("slices", [2, 3])
def test_digit_issuers(slices):
    src = source("digit.cuh")
    n = re.search(r"mbar_init\(&step\[s\], (.+?)\);", src).group(1)
    arrivals = {"2": lambda i: 2, "s < 4 ? 2 : 1": lambda i: 2 if i < 4 else 1}[n]
    assert digits(slices, arrivals, "mbar_arrive(&step[i])" in src) is None
    assert digits(slices, lambda i: 2 if i < 4 else 1, False) is not None
