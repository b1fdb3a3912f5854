"""The call's tables on their way to the device (one kernel reading pinned host memory) and the
rewards on their way out: odd table sizes (parts that end inside a 16-byte quad, empty parts, more
than one launch round of quads), two calls in flight that share the staging buffer, and the
caller's device buffer written by the head kernel instead of a copy; and the caller's vectors (embedding,
gains, head rows), which may start at any element, on every image that reads them."""
import numpy as np
import pytest

import kvsynth as ks
from tests.gpu_util import P_PLUS_ATOL, make_scorer, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens", [[0], [1], [16, 17, 0], [5, 300, 31, 64, 129], [40] * 33,
                                  list(range(1, 4097, 97))])
def test_tables_and_rewards(lens):
    torch = require_gpu()
    import paper_2607_09153_gb300 as kp
    w = ks.distinct("setup", ks.ARCH_TINY, 60 + len(lens), lens)
    dev = ks.DeviceInputs(w, ks.Tables.make())
    n = len(lens)
    sc = make_scorer(dev, n + 3, w.max_blocks)
    bt, sl = np.asarray(w.block_table), np.asarray(w.seq_lens)
    want = [sc.score(dev.pool, bt, sl), sc.score(dev.pool, bt[::-1], sl[::-1])]
    # both orders in flight at once, each into its own buffer (at an address that is no multiple of 16)
    out = [torch.full((n + 1,), -1.0, dtype=torch.float32, device="cuda")[1:] for _ in range(2)]
    for _ in range(3):
        sc.score_async(dev.pool, bt, sl, out[0])
        sc.score_async(dev.pool, np.ascontiguousarray(bt[::-1]), np.ascontiguousarray(sl[::-1]), out[1])
    torch.cuda.synchronize()
    for o, r in zip(out, want):
        assert np.array_equal(o.cpu().numpy(), r)
    # the two orders are scheduled differently: the same up to fp32 rounding order
    assert np.abs(want[0] - want[1][::-1]).max() <= P_PLUS_ATOL
    for i in range(n):   # the last call's tables on the device: reversed order
        b = n - 1 - i
        j = np.arange(sl[b])
        assert np.array_equal(kp.kvprm_resolve(sc.ctx, i, int(sl[b])), bt[b, j // 16].astype(np.int64) * 16 + j % 16)
    sc.close()


@pytest.mark.parametrize("shift", [1, 2, 3, 4])
def test_vectors_at_any_address(shift):
    # embedding, gains and head rows that start anywhere (2-byte aligned views) score as aligned ones do
    torch = require_gpu()
    w = ks.distinct("shift", ks.ARCH_TINY, 90, [33, 128, 5])
    t = ks.Tables.make(0.2)
    dev = ks.DeviceInputs(w, t)
    sc = make_scorer(dev, 3, w.max_blocks)
    want = sc.score(dev.pool, w.block_table, w.seq_lens)
    sc.close()

    def moved(v):
        buf = torch.zeros(v.numel() + 8, dtype=v.dtype, device="cuda")
        buf[shift:shift + v.numel()] = v.reshape(-1)
        return buf[shift:shift + v.numel()]

    for k in (ks.EMBED, ks.FINAL_NORM, ks.W_PLUS, ks.W_MINUS):
        dev.top[k] = moved(dev.top[k])
    for layer in dev.layers:
        for k in (ks.ATTN_NORM, ks.MLP_NORM):
            layer[k] = moved(layer[k])
    sc = make_scorer(dev, 3, w.max_blocks)
    assert np.array_equal(sc.score(dev.pool, w.block_table, w.seq_lens), want)
    sc.close()


# a residual epilogue of each image: 32 padded columns (small), 48 (the fewest of the large one, also as 12
# candidates of four verify tokens), 64, 80 (CTA pairs), 144 (pairs of half of the columns)
@pytest.mark.parametrize("n, depth", [(32, 1), (33, 1), (12, 4), (49, 1), (80, 1), (129, 1)])
@pytest.mark.parametrize("shift", [1, 2])
def test_gains_at_any_address(n, depth, shift):
    require_gpu()
    w = ks.distinct("gains", ks.Arch(2, 256, 4, 2, 64, 704), 95 + n, [(11 * b) % 50 for b in range(n)], gain_std=0.2)
    dev = ks.DeviceInputs(w, ks.Tables.make(0.2))

    def rewards():
        sc = make_scorer(dev, n * depth, w.max_blocks)
        sc.set_depth(depth)
        r = sc.score(dev.pool, w.block_table, w.seq_lens)
        sc.close()
        return r

    want = rewards()
    for layer in dev.layers:
        for k in (ks.ATTN_NORM, ks.MLP_NORM):
            buf = layer[k].new_zeros(layer[k].numel() + 8)
            buf[shift:shift + layer[k].numel()] = layer[k].reshape(-1)
            layer[k] = buf[shift:shift + layer[k].numel()]
    assert np.array_equal(rewards(), want)
