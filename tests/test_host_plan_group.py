"""Host logic of the engine's weight-GEMM work split up to 256 tokens (no GPU).
Tiles form groups of 4; the CTAs of one residue mod 4 share a (group, chunk)
space cut into equal contiguous ranges.  What the kernels rest on: the split
does not depend on the token count (a row's bits do not depend on the launch's
width); every chunk of every tile belongs to one CTA; the four CTAs of a range
run over the same K range (a pair shares activations); the first contributor
of a shared tile ends its range in it and the others begin theirs in it."""
import ctypes

import pytest

from paper_2403_00835_gb300.cllm import load

FIELDS = ("mtiles", "size", "kchunks", "cpc", "bn", "bn_max", "maxc", "grid")
# (weight tiles, K): the 7B launches (QKV, O, gate/up, down, LM head), the small
# decoders' and some with groups that are not full
SHAPES = [(96, 4096), (32, 4096), (172, 4096), (32, 11008), (250, 4096), (252, 4096),
          (6, 256), (2, 256), (11, 256), (2, 688), (16, 256), (1, 8), (5, 72), (7, 1000)]


def plan(mtiles, K, T, sms=152):
    f = load().cllm_test_plan_group
    f.argtypes = [ctypes.c_int] * 4 + [ctypes.POINTER(ctypes.c_int)]
    f.restype = ctypes.c_int
    out = (ctypes.c_int * 8)()
    assert f(mtiles, K, T, sms, out) == 0
    return dict(zip(FIELDS, list(out)))


@pytest.mark.parametrize("mtiles,K", SHAPES)
def test_group_split_covers_every_tile_once(mtiles, K):
    p = plan(mtiles, K, 16)
    for T in (1, 17, 64, 65, 128, 129, 256):
        q = plan(mtiles, K, T)
        assert all(q[k] == p[k] for k in ("kchunks", "cpc", "maxc", "grid"))
        assert q["bn"] == -(-T // 16) * 16 and q["bn_max"] == min(b for b in (32, 64, 128, 256) if b >= q["bn"])
    size, kc, cpc, grid = p["size"], p["kchunks"], p["cpc"], p["grid"]
    assert size == 4 and kc % 2 == 0 and kc * 64 >= K and cpc % 2 == 0 and cpc >= 4
    assert grid % size == 0 and grid <= 152
    owner = {}
    maxc = 1
    for cta in range(grid):
        j, q = cta % size, cta // size
        total = (mtiles - j + size - 1) // size * kc  # as cta_range
        for c in range(min(total, q * cpc), min(total, (q + 1) * cpc)):
            tile = c // kc * size + j
            assert tile < mtiles and (tile, c % kc) not in owner
            owner[tile, c % kc] = q
    assert len(owner) == mtiles * kc
    for tile in range(mtiles):
        g = tile // size
        qs = [owner[tile, k] for k in range(kc)]
        first, last = g * kc // cpc, ((g + 1) * kc - 1) // cpc
        assert sorted(set(qs)) == list(range(first, last + 1)) and qs == sorted(qs)
        maxc = max(maxc, last - first + 1)
        if last > first:
            assert g * kc < (first + 1) * cpc < (g + 1) * kc  # the owner's range ends in the tile
            assert all(g * kc < q * cpc for q in range(first + 1, last + 1))
        # neighbours of the group run over the same ranges
        mate = tile ^ 1
        if mate < mtiles:
            assert qs == [owner[mate, k] for k in range(kc)]
    assert maxc == p["maxc"]


@pytest.mark.parametrize("mtiles,K,share", [(96, 4096, 42), (32, 4096, 14), (172, 4096, 74), (32, 11008, 38)])
def test_group_split_keeps_the_7b_shares(mtiles, K, share):
    assert plan(mtiles, K, 16)["cpc"] == share


@pytest.mark.parametrize("sms", [152, 151, 150, 148, 7, 4])
def test_group_split_launches_no_more_ctas_than_it_is_given(sms):
    for mtiles, K in SHAPES:
        assert plan(mtiles, K, 16, sms)["grid"] <= sms


def test_bad_arguments_are_rejected():
    f = load().cllm_test_plan_group
    f.argtypes = [ctypes.c_int] * 4 + [ctypes.POINTER(ctypes.c_int)]
    out = (ctypes.c_int * 8)()
    assert f(0, 64, 16, 152, out) == -1 and f(4, 64, 257, 152, out) == -1
    assert f(4, 64, 16, 0, out) == -1 and f(4, 64, 16, 152, None) == -1
