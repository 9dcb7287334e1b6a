"""The end of the network's CTA pairs (csrc/vrm_mlp.cu, k_mlp_fused): a model of
the commits that the leading CTA sends to both, each landing after a delay of
its own, and of the parity waits before a CTA may end.  With the waits on the
drain barrier and on the last commit of every ring stage and slot, no arrival
lands in a CTA that has ended; with the leading CTA's wait on its own drain
barrier alone, some do."""
import random

import pytest

RING = 5
SLABS = (2, 4, 4, 4)  # per layer of a tile


class Barrier:
    """Arrivals that each complete one phase."""

    def __init__(self):
        self.at = []

    def wait(self, t, parity):
        """First moment from t on at which the phase under way is not of `parity`."""
        times = sorted(self.at)
        done = sum(a <= t for a in times)
        while done & 1 == parity:
            t = times[done]
            done += 1
        return t


def run(my_tiles, rng, waits):
    total = sum(SLABS) * my_tiles
    cta = [dict(wempty=[Barrier() for _ in range(RING)], hfree=[Barrier() for _ in range(2)], drain=Barrier(),
                load=0.0, tile=0.0) for _ in range(2)]

    def commit(t, name, k=None):
        for c in cta:
            b = c[name] if k is None else c[name][k]
            b.at.append(t + rng.expovariate(1.0) ** 3)  # (long tails: late arrivals)

    t, g = 0.0, 0
    for p in range((my_tiles + 1) // 2):
        for layer, nk in enumerate(SLABS):
            for s in range(2 if 2 * p + 1 < my_tiles else 1):
                i = 2 * p + s
                if layer == 0:  # the slot's input follows the last layer of its tile before
                    for c in cta:
                        if i >= 2:
                            c["tile"] = c["hfree"][s].wait(c["tile"], (i // 2 - 1) & 1)
                    t = max(t, *(c["tile"] for c in cta))
                for _ in range(nk):
                    for c in cta:  # the CTA's half of the slab
                        if g >= RING:
                            c["load"] = c["wempty"][g % RING].wait(c["load"], (g // RING - 1) & 1)
                    t = max(t, *(c["load"] for c in cta)) + 0.1
                    commit(t, "wempty", g % RING)
                    g += 1
                if layer == 3:
                    commit(t, "hfree", s)
    assert g == total
    commit(t, "drain")
    ends = []
    for rank, c in enumerate(cta):
        end = t
        if waits == "all":
            # the weights' thread, and beside it the inputs'
            end = c["load"]
            for k in range(max(total - RING, 0), total):
                end = c["wempty"][k % RING].wait(end, (k // RING) & 1)
            end = c["drain"].wait(end, 0)
            tile = c["tile"]
            for i in range(max(my_tiles - 2, 0), my_tiles):
                tile = c["hfree"][i % 2].wait(tile, (i // 2) & 1)
            end = max(end, tile)
        elif rank == 0:
            end = c["drain"].wait(end, 0)
        ends.append(end)
    end = max(ends)  # the cluster barrier
    return all(a <= end for c in cta for b in [c["drain"]] + c["wempty"] + c["hfree"] for a in b.at)


@pytest.mark.parametrize("my_tiles", [1, 2, 3, 4, 5, 8, 13])
def test_no_arrival_lands_in_a_cta_that_has_ended(my_tiles):
    rng = random.Random(my_tiles)
    assert all(run(my_tiles, rng, "all") for _ in range(300))
    assert not all(run(my_tiles, rng, "leader's drain") for _ in range(300))
