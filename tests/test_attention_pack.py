"""The schedule scoring contexts use (kvprm_plan_attention with KVPRM_PLAN_PACK; no GPU): shared
partial pages and packed short runs.  Against the block tables, recomputed here: every cached token
of every candidate scored exactly once per kv head, every partial slot owned by one (candidate, kv
head), lanes of a pack within the bounds the kernel relies on, and the pages of the plan without
packing the same as before."""
import collections

import numpy as np
import pytest

import paper_2607_09153_gb300.kvprm as kp


def coverage(p, group, tc):
    """(b, g, page, valid) counts and the slots of every (b, g)."""
    got, used = collections.Counter(), collections.defaultdict(list)

    def score(b, g, pages, last):
        for i, pg in enumerate(pages):
            got[(int(b), int(g), int(pg), last if i == len(pages) - 1 else 16)] += 1

    for s in p["segs"]:
        kind, g, c, nc, off, npg, last, slot = (int(x) for x in s)
        assert npg >= 1 and 1 <= last <= 16
        if kind == 3:
            lanes = p["cands"][c:c + 6 * nc].reshape(nc, 6)
            assert 1 <= nc <= 8 and lanes[:, 3].max() == npg and lanes[:, 3].min() >= 1 and group <= 8
            for b, lg, lo, ln, lv, ls in lanes:
                score(b, lg, p["pages"][lo:lo + ln], int(lv))
                used[(int(b), int(lg))].append(int(ls))
            continue
        pages = p["pages"][off:off + npg]
        cands = [c] if kind == 0 else p["cands"][c:c + nc]
        reps = {0: 1 if group <= 8 else min(8, npg), 1: 8 // max(nc, 1), 2: 1}[kind]
        assert kind != 2 or tc
        for k, b in enumerate(cands):
            score(b, g, pages, last)
            used[(int(b), g)] += ([slot + i for i in range(reps)] if kind == 0 else
                                  [int(p["slots"][slot + w]) for w in range(reps * nc) if w % nc == k])
    return got, used


def check(bt, sl, n_kv, group, n_ctas, share):
    bt, sl = np.asarray(bt, np.int32), np.asarray(sl, np.int32)
    p = kp.kvprm_plan_attention(bt, sl, n_kv, group, n_ctas, share | kp.KVPRM_PLAN_PACK)
    want = collections.Counter()
    for b in range(len(sl)):
        npg = (int(sl[b]) + 15) // 16
        for g in range(n_kv):
            for j in range(npg):
                want[(b, g, int(bt[b, j]), 16 if j < npg - 1 else int(sl[b]) - 16 * (npg - 1))] += 1
    got, used = coverage(p, group, share >= 2)
    assert got == want
    for b in range(len(sl)):
        for g in range(n_kv):
            base, cnt = int(p["slot_base"][b * n_kv + g]), int(p["nslots"][b * n_kv + g])
            assert sorted(used[(b, g)]) == list(range(base, base + cnt))
    assert p["n_ctas"] <= n_ctas and p["cta_seg"][0] == 0 and np.all(np.diff(p["cta_seg"]) >= 0)
    return p


def own_pages(lens, start=0):
    bt = np.zeros((len(lens), max(1, max((L + 15) // 16 for L in lens))), np.int32)
    nxt = start
    for b, L in enumerate(lens):
        n = (L + 15) // 16
        bt[b, :n] = nxt + np.arange(n)
        nxt += n
    return bt


@pytest.mark.parametrize("n, top, kind", [(1, 5, 3), (40, 16, 3), (64, 17, 3), (201, 333, 3), (9, 9000, 0),
                                          (37, 4000, 0)])
@pytest.mark.parametrize("group", [7, 12])
def test_short_private_runs(n, top, kind, group):
    rng = np.random.default_rng(n + top)
    lens = rng.integers(0, top + 1, n).tolist()
    p = check(own_pages(lens), lens, 4, group, 152, 3)
    kinds = set(p["segs"][:, 0].tolist())
    assert kinds == {kind if group <= 8 else 0}, "long runs and groups of more than eight heads keep the other form"


@pytest.mark.parametrize("depth, group", [(2, 6), (4, 6), (5, 2), (6, 7), (8, 1)])
@pytest.mark.parametrize("share", [1, 3])
def test_shared_partial_pages(depth, group, share):
    # a depth-k readout: rows b k .. b k + k - 1 list the same pages, the last of them partial
    lens = [1, 15, 16, 17, 100, 0, 333, 640]
    bt, sl = np.repeat(own_pages(lens), depth, axis=0), np.repeat(lens, depth)
    p = check(bt, sl, 2, group, 152, share)
    assert not (p["segs"][:, 0] == 0).any(), "no one-page private run is left"


def test_a_page_full_for_some_and_partial_for_others():
    # candidates 0, 1 end inside page 3 (same length), 2 ends there earlier, 3 and 4 go on past it
    bt = np.array([[0, 1, 3, 0], [0, 1, 3, 0], [0, 1, 3, 0], [0, 1, 3, 5], [0, 1, 3, 6]], np.int32)
    for share in (1, 3):
        p = check(bt, [41, 41, 37, 64, 50], 2, 7, 16, share)
        tail = [s for s in p["segs"] if int(s[6]) == 9]   # 41 = 2 x 16 + 9: one run of candidates 0 and 1
        assert tail and all(int(s[0]) == 1 and int(s[3]) == 2 for s in tail)


def test_random_sharing():
    rng = np.random.default_rng(5)
    for _ in range(60):
        n, mb = int(rng.integers(1, 30)), int(rng.integers(1, 12))
        bt = rng.integers(0, int(rng.integers(mb, 40 * mb)), (n, mb))
        sl = rng.integers(0, 16 * mb + 1, n)
        if rng.random() < 0.5:   # copies of whole rows share every page, the partial one included
            src = rng.integers(0, n, n)
            bt, sl = bt[src], sl[src]
        check(bt, sl, int(rng.integers(1, 5)), int(rng.integers(1, 9)), int(rng.integers(1, 153)),
              int(rng.integers(0, 4)))
