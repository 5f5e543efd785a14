"""The hand-over between the threads of k_mlp_forward (csrc/lbm_mlp.cu), every interleaving, on the CPU.

An mbarrier wait names one parity bit, so it tells a phase apart from the next one only: a thread that has not looked
while two phases completed waits for a phase that depends on itself.  The model has the kernel's agents -- the epilogue
warps, the thread that issues the first layer's products, the one that issues the others', and the tensor core that
completes each in order -- and its barriers: accumulator full (one per agent that issues), first accumulator read,
epilogue done.  ``last`` says whether the last layer's epilogue arrives at epilogue done too.
"""

import pytest


def _stuck(tiles, layers, warps, last):
    """A reachable state in which nothing can happen and not all is done, or None."""
    per = layers if last else layers - 1  # epilogue-done phases of a tile

    def passed(done, phase):  # try_wait.parity: the phase of that parity is not the one running
        return (done & 1) != (phase & 1)

    # state: per warp (tile, layer); first issuer's tile; second issuer's (tile, layer, epilogue phases seen);
    # completed products of either; arrivals at the first-accumulator-read and epilogue-done barriers
    start = ((0, 0),) * warps, 0, (0, 1, 0), (0, 0), 0, 0
    seen, todo = {start}, [start]
    while todo:
        state = todo.pop()
        epi, first, second, full, read, done = state
        after = []
        for w, (j, l) in enumerate(epi):
            if j == tiles:
                continue
            hidden = j * (layers - 1) + l - 1
            if passed(full[0], j) if l == 0 else passed(full[1], hidden):
                at = (j, l + 1) if l + 1 < layers else (j + 1, 0)
                after.append((epi[:w] + (at,) + epi[w + 1:], first, second, full, read + (l == 0),
                              done + (last or l + 1 < layers)))
        if first < tiles and (first == 0 or passed(read // warps, first - 1)):
            after.append((epi, first + 1, second, full, read, done))
        j, l, saw = second
        if j < tiles:
            if saw < j * per + l:
                if passed(done // warps, saw):
                    after.append((epi, first, (j, l, saw + 1), full, read, done))
            else:
                at = (j, l + 1, saw) if l + 1 < layers else (j + 1, 1, saw)
                after.append((epi, first, at, full, read, done))
        issued = first, j * (layers - 1) + l - 1
        for r in range(2):
            if full[r] < issued[r]:
                after.append((epi, first, second, (full[0] + (r == 0), full[1] + (r == 1)), read, done))
        if not after and not (first == tiles and j == tiles and all(e == (tiles, 0) for e in epi)):
            return state
        for s in after:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return None


@pytest.mark.parametrize("layers", [2, 3, 4, 6])
@pytest.mark.parametrize("warps", [1, 2])
def test_no_interleaving_stops(layers, warps):
    assert _stuck(3, layers, warps, last=False) is None


@pytest.mark.parametrize("layers", [2, 3, 4])
def test_an_arrival_of_the_last_layer_can_lap_the_waiting_thread(layers):
    assert _stuck(3, layers, 1, last=True) is not None
