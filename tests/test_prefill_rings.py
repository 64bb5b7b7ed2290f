"""Host model of the prefill kernel's rings: no wait may pass on the phase of another turn.

An mbarrier wait names a phase by its parity only, so a wait for turn t of a ring's slot also passes while turn t - 1 is
still incomplete.  A group of dequantization warps takes every fourth unit of 128 k and does not wait for the loads of the
others, and bulk copies complete in any order.  The model walks the kernel's agents as far as they get with one load that never
arrives (or the MMAs stopped at one unit) and looks for a wait that passes although its slot's turn before is the one withheld."""
import os
import re

import pytest

GROUPS = 4
ORDER = ("packed", "buffer", "x")                             # a group's waits for a unit: packed words, weight buffer, activations
SRC = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_11248_b200", "csrc", "mpgemm.cu")).read()


def load_barriers(ring, stages, int8):
    """Over how many stages the kernel's "loaded" barriers of a ring take turns (P packed words, X activations)."""
    own = re.search(r"constexpr int [^;]*\b%s_LOAD_BARS = (\d+)" % ring, SRC)
    if own is None or (ring == "X" and not int8):
        return stages                                         # a barrier for every slot of the ring
    if ring == "P":
        assert SRC.count("ploaded0 + 8 * (pc % P_LOAD_BARS)") == 2 and "(pc / P_LOAD_BARS) & 1u" in SRC
    else:
        assert SRC.count("xloaded0 + 8 * (INT8 ? xc % X_LOAD_BARS :") == 2 and "(INT8 ? xc / X_LOAD_BARS :" in SRC
    return int(own.group(1))


def wrong_turn(segments, p_stages, wbufs, xu, x_stages, withheld, int8):
    """segments: units of each.  withheld: ("packed" | "x", stage) that never arrives, ("mma", unit) that is never issued
    or ("group", unit) that is never begun.
    Returns the wait (kind, unit) that passes on the wrong turn, or None."""
    p_of, x_of, x_last, parts = [], [], [], []                # unit -> stage; stage -> last unit (x) and units (packed)
    for n in segments:
        u0 = len(p_of)
        for i in range(n):
            if i % 2 == 0:
                parts.append([])
            if i % xu == 0:
                x_last.append(0)
            p_of.append(len(parts) - 1)
            x_of.append(len(x_last) - 1)
            parts[-1].append(u0 + i)
            x_last[-1] = u0 + i
    units = len(p_of)
    read, ready, done = [False] * units, [False] * units, 0   # words in registers; weights and activations handed on; MMAs committed
    loads = {"packed": [0, len(parts)], "x": [0, len(x_last)]}
    bars = {"packed": load_barriers("P", p_stages, int8), "x": load_barriers("X", x_stages, int8)}
    at = [[g, 0] for g in range(GROUPS)]                      # a group's unit, the wait it stands at

    def loaded(kind, stage):
        return stage < loads[kind][0] and withheld != (kind, stage)

    moved = True
    while moved:
        moved = False
        while loads["packed"][0] < len(parts) and (loads["packed"][0] < p_stages or all(read[u] for u in parts[loads["packed"][0] - p_stages])):
            loads["packed"][0] += 1
            moved = True
        while loads["x"][0] < len(x_last) and (loads["x"][0] < x_stages or x_last[loads["x"][0] - x_stages] < done):
            loads["x"][0] += 1
            moved = True
        while done < units and ready[done] and withheld != ("mma", done):
            done += 1
            moved = True
        for a in at:
            while a[0] < units:
                u, kind = a[0], ORDER[a[1]]
                if withheld == ("group", u):
                    break
                if kind == "buffer":
                    passes = u < wbufs or u - wbufs < done
                    wrong = u >= 2 * wbufs and u - 2 * wbufs >= done
                else:
                    stage, turns = (p_of if kind == "packed" else x_of)[u], bars[kind]
                    passes = loaded(kind, stage)
                    wrong = stage >= turns and not loaded(kind, stage - turns)
                if wrong:
                    return kind, u
                if not passes:
                    break
                moved = True
                a[1] += 1
                if a[1] == 2:
                    read[u] = True                            # the words are freed after the wait for the weight buffer
                if a[1] == len(ORDER):
                    ready[u] = True
                    a[0], a[1] = u + GROUPS, 0
    return None


def walks(nu):
    """Walks of a worker: whole tiles; the end of one tile, whole tiles, the beginning of another; a piece alone."""
    whole = 3 + 24 // nu
    yield [nu] * whole
    for first in {1, 2, 3, nu // 2, nu - 1}:
        if 0 < first < nu:
            for last in {1, 3, nu - 1}:
                if 0 < last < nu:
                    yield [first] + [nu] * (1 + 16 // nu) + [last]
                    yield [first, last]


def check(segments, p_stages, wbufs, xu, x_stages, int8=False):
    for kind in ("packed", "x", "mma", "group"):
        for i in range(sum(segments)):
            got = wrong_turn(segments, p_stages, wbufs, xu, x_stages, (kind, i), int8)
            assert got is None, (segments, p_stages, wbufs, xu, x_stages, (kind, i), got)


# (weight buffers, units and stages of activations, admitted unit counts of a tile): what launch_mpgemm_variant chooses,
# and launch_mpgemm_ternary_i8 (whole tiles only, 2-bit weights)
RINGS = {
    "fp16, up to 64 tokens": (6, 2, 8, lambda nu: nu >= 4),
    "fp16, up to 128 tokens": (6, 2, 4, lambda nu: nu >= 4),
    "fp16, up to 64 tokens, short K": (4, 2, 8, lambda nu: nu < 4),
    "fp16, up to 128 tokens, short K": (4, 2, 4, lambda nu: nu < 4),
    "fp16, up to 256 tokens": (4, 1, 4, lambda nu: True),
}
RINGS_INT8 = {
    "up to 128 tokens": (8, 2, 8, lambda nu: nu >= 8),
    "up to 128 tokens, short K": (4, 2, 8, lambda nu: nu < 8),
    "up to 192 tokens": (4, 2, 4, lambda nu: True),
    "up to 256 tokens": (8, 2, 4, lambda nu: nu >= 8),
    "up to 256 tokens, short K": (4, 2, 4, lambda nu: nu < 8),
}


@pytest.mark.parametrize("name", list(RINGS))
def test_no_wait_for_packed_words_passes_on_the_turn_before(name):
    wbufs, xu, x_stages, admits = RINGS[name]
    for p_stages in (8, 4):                                   # 2-bit weights; 3 and 4
        for nu in (n for n in (1, 2, 3, 4, 5, 6, 7, 9, 12) if admits(n)):
            for segments in walks(nu):
                check(segments, p_stages, wbufs, xu, x_stages)


@pytest.mark.parametrize("name", list(RINGS_INT8))
def test_no_wait_for_activations_of_the_integer_path_passes_on_the_turn_before(name):
    wbufs, xu, x_stages, admits = RINGS_INT8[name]
    for nu in (n for n in (1, 2, 3, 4, 5, 7, 8, 9, 11, 13, 20) if admits(n)):
        check([nu] * (3 + 24 // nu), 8, wbufs, xu, x_stages, int8=True)


def test_tensor_memory_is_taken_after_the_wait_and_before_the_signal():
    # A predecessor that signals early and allocates tensor memory on the same SM afterwards would wait for this kernel's columns,
    # and this kernel for its end; the same between this kernel and a successor of that kind.
    kernel = SRC[SRC.index("mpgemm_kernel(const __grid_constant__"):SRC.index("// ---- stage 1")]
    wait, signal = (kernel.index("griddepcontrol." + w) for w in ("wait;", "launch_dependents;"))
    allocs = [m.start() for m in re.finditer(r"tcgen05_alloc2?\(", kernel)]
    assert len(allocs) == 2 and wait < min(allocs) and max(allocs) < signal
    assert kernel.count("griddepcontrol.") == 2
