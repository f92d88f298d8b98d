"""Host logic of the work split of launches of more than 256 tokens (no GPU).
What the kernel rests on: every chunk of every unit belongs to one cluster; a
cluster has at most two segments of cut units, one that begins its unit and one
that does not (a partial slot each); units that share a ticket index do not
exist; and, since no cluster waits for another, the units are finished once
each whatever the order in which the clusters run -- one after the other
included, as when another program's launches hold the SMs."""
import ctypes
import random

import pytest

from paper_2403_00835_gb300.cllm import load

FIELDS = ("row_units", "ntiles", "bn", "kchunks", "cpc", "clusters")


def plan(gate_up, M, K, T, clusters, split=1):
    f = load().cllm_test_plan_wide
    f.argtypes = [ctypes.c_int] * 6 + [ctypes.POINTER(ctypes.c_int)]
    out = (ctypes.c_int * 6)()
    assert f(gate_up, M, K, T, clusters, split, out) == 0
    return dict(zip(FIELDS, list(out)))


def segments(p, cluster):
    """(unit, k0, k1, first, last contributor) of a cluster, as the kernel walks them."""
    units = p["row_units"] * p["ntiles"]
    n, kc, cpc = p["clusters"], p["kchunks"], p["cpc"]
    whole = units // n * n
    for u in range(cluster, whole, n):
        yield u, 0, kc, cluster, cluster
    rest = (units - whole) * kc
    c, c1 = min(rest, cluster * cpc), min(rest, (cluster + 1) * cpc)
    while c < c1:
        u, k0 = divmod(c, kc)
        k1 = min(kc, k0 + c1 - c)
        yield u + whole, k0, k1, u * kc // cpc, ((u + 1) * kc - 1) // cpc
        c += k1 - k0


CASES = [(0, 12288, 4096, 500), (0, 4096, 4096, 500), (1, 11008, 4096, 500), (0, 4096, 11008, 500),
         (0, 4096, 11008, 2048), (0, 768, 256, 300), (1, 688, 256, 300), (0, 256, 688, 1025),
         (0, 2048, 256, 257), (0, 128, 8192, 2048), (0, 128, 64, 257), (0, 640, 72, 300)]


@pytest.mark.parametrize("clusters", [76, 36, 3, 1])
@pytest.mark.parametrize("gate_up,M,K,T", CASES)
def test_wide_split(gate_up, M, K, T, clusters):
    p = plan(gate_up, M, K, T, clusters)
    units, kc = p["row_units"] * p["ntiles"], p["kchunks"]
    assert p["row_units"] * (256 if gate_up else 512) >= M and kc * 64 >= K
    assert p["bn"] % 16 == 0 and p["bn"] <= 128 and p["ntiles"] * p["bn"] >= T > (p["ntiles"] - 1) * p["bn"]
    assert 1 <= p["clusters"] <= clusters and 1 <= p["cpc"] <= kc
    covered, tickets, shared = {}, {}, {}
    for c in range(p["clusters"]):
        slots = set()
        for u, k0, k1, first, last in segments(p, c):
            assert 0 <= u < units and first <= c <= last < p["clusters"]
            for k in range(k0, k1):
                assert (u, k) not in covered
                covered[u, k] = c
            if last > first:
                assert (k0 == 0) == (c == first)
                assert c == first or c not in slots  # at most one segment that continues a unit
                slot = (c, c == first)
                assert slot not in slots
                slots.add(slot)
                assert tickets.setdefault(first, u) == u
                shared.setdefault(u, set()).add(c)
                assert len(set(range(first, last + 1))) == last - first + 1
    assert len(covered) == units * kc
    # the arrival protocol, clusters run one at a time in any order: each unit
    # is finished once, by its last contributor, with every other sum stored
    for seed in range(3):
        order = list(range(p["clusters"]))
        random.Random(seed).shuffle(order)
        count, stored, finished = {}, set(), []
        for c in order:
            for u, k0, k1, first, last in segments(p, c):
                if last > first:
                    if count.get(first, 0) != last - first:
                        stored.add((c, c == first))
                        count[first] = count.get(first, 0) + 1
                        continue
                    assert all((o, o == first) in stored for o in range(first, last + 1) if o != c)
                finished.append(u)
        assert sorted(finished) == list(range(units))


def test_whole_units_without_split():
    for gate_up, M, K, T in CASES:
        p = plan(gate_up, M, K, T, 76, split=0)
        for c in range(p["clusters"]):
            assert all(k0 == 0 and k1 == p["kchunks"] and first == last == c
                       for u, k0, k1, first, last in segments(p, c))


def test_bad_arguments_are_rejected():
    f = load().cllm_test_plan_wide
    f.argtypes = [ctypes.c_int] * 6 + [ctypes.POINTER(ctypes.c_int)]
    out = (ctypes.c_int * 6)()
    assert f(0, 0, 64, 300, 76, 1, out) == -1 and f(0, 128, 64, 300, 0, 1, out) == -1
    assert f(0, 128, 64, 300, 76, 1, None) == -1
