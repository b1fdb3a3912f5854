"""Packed short runs and shared partial pages on the GPU, at the edges of both: lanes of one page, of
a partial page, of different lengths in one pack, more lanes than warps; a candidate without a cache
among them; and a depth-k readout whose verify tokens share pages that end anywhere.  Against the
oracle, with the scoring tolerances."""
import pytest

import kvsynth as ks
from tests.gpu_util import compare, require_gpu, run_gpu

pytestmark = pytest.mark.gpu


def arch(hd, group, n_kv):
    return ks.Arch(1, 256, group * n_kv, n_kv, hd, 256)


@pytest.mark.parametrize("hd, group, n_kv, lens", [
    (128, 7, 2, [(13 * b) % 330 for b in range(60)]),     # one pack per CTA, lanes cut to the common length
    (128, 8, 4, [1] * 200 + [0, 16, 17]),                 # partial single pages
    (64, 1, 2, [16 * (b % 5) for b in range(90)]),        # full pages only, empty caches
    (64, 8, 1, [90 + b for b in range(256)]),             # every candidate of the largest call
])
def test_packed_runs(hd, group, n_kv, lens):
    require_gpu()
    w = ks.distinct("pack", arch(hd, group, n_kv), 800 + len(lens), lens, gain_std=0.2)
    t = ks.Tables.make(0.2)
    r, attn, _, sc = run_gpu(w, t)
    compare(w, t, gpu_rewards=r, gpu_attn=attn, label=f"packed hd {hd} G {group} n {len(lens)}")
    sc.close()


@pytest.mark.parametrize("hd, group, depth", [(128, 6, 4), (64, 2, 3), (128, 7, 7), (128, 1, 8), (128, 4, 2)])
def test_shared_partial_pages(hd, group, depth):
    require_gpu()
    lens = [1, 15, 16, 17, 64, 65, 0, 200, 333]
    w = ks.distinct("tails", arch(hd, group, 2), 830 + depth, lens, gain_std=0.2)
    t = ks.Tables.make(0.2)
    r, attn, _, sc = run_gpu(w, t, depth=depth)
    compare(w, t, gpu_rewards=r, gpu_attn=attn, label=f"tails hd {hd} G {group} depth {depth}", depth=depth)
    sc.close()
