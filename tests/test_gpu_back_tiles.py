"""The tensor-core attention backward at the edges of its tiles (8 pages of 16 tokens, 4 candidates a
step, 8 rows a candidate): shared runs one page short of a tile, one over and several tiles long;
candidates that fill a step, leave one over or are split over tiles because the pages alone would
leave the GPU idle; both head widths; the narrowest and widest groups; row counts whose workspace
arrays do not end on 16 bytes.  Against the fp64 oracle with the gradient's tolerance
(tests/test_gpu_steering.py), and eagerly against the captured graph.  And a candidate that is not finite, whose
rows must not reach the gradient of pages that it does not read."""
import numpy as np
import pytest

import kvsynth as ks
from tests.gpu_util import make_scorer, require_gpu
from tests.test_gpu_steering import _compare, _gpu_grad, _oracle

pytestmark = pytest.mark.gpu


def arch(hd, group, n_kv=2):
    return ks.Arch(1, 256, group * n_kv, n_kv, hd, 256)


@pytest.mark.parametrize("hd, group, cands, pages, own", [
    (128, 7, 2, 1, [1, 16]),
    (128, 7, 3, 7, [0, 5, 33]),
    (128, 8, 4, 8, [16, 17, 0, 140]),
    (128, 1, 5, 9, [3] * 5),
    (128, 6, 9, 17, [0] * 9),
    (64, 8, 8, 16, [20, 1] * 4),
    (64, 2, 13, 25, [130] * 13),
    (64, 7, 5, 8, [15] * 5),
])
def test_shared_runs(hd, group, cands, pages, own):
    require_gpu()
    t = ks.Tables.make(0.2)
    segs = [[(1, 16 * pages)] + ([(10 + b, own[b])] if own[b] else []) for b in range(cands)]
    w = ks.workload_from_segments("back_tiles", arch(hd, group), 700 + pages, segs, gain_std=0.2)
    p, grad, dev, sc = _gpu_grad(w, t)
    p_ref, ref, _, _ = _oracle(w, t)
    _compare(f"hd {hd} G {group}: {cands} candidates, {pages} shared pages", w, p, grad, p_ref, ref)
    sc.close()


@pytest.mark.parametrize("n, group, n_kv", [(65, 7, 1), (27, 7, 2), (3, 5, 1), (66, 3, 1)])
def test_odd_rows(n, group, n_kv):
    # n x n_q that is no multiple of four (n >= 64 takes the large-batch projections)
    require_gpu()
    t = ks.Tables.make(0.2)
    w = ks.distinct("back_rows", arch(64, group, n_kv), 720 + n, [(37 * b) % 90 for b in range(n)], gain_std=0.2)
    p, grad, dev, sc = _gpu_grad(w, t)
    p_ref, ref, _, _ = _oracle(w, t)
    _compare(f"{n} candidates of {group * n_kv} heads", w, p, grad, p_ref, ref)
    sc.close()


# The bad candidate's rows stay in shared memory, in its place of a step of four; three row stages on, the same CTA
# takes a step that leaves this place empty beside a candidate: a private page's (places 0, 1), or a step of three.
@pytest.mark.parametrize("groups, bad, own", [([(4, 128)], 1, 9728), ([(8, 608 * 16), (3, 1216 * 16)], 3, 16)])
@pytest.mark.parametrize("which, value", [(0, "inf"), (1, "nan")])
def test_a_candidate_that_is_not_finite(groups, bad, own, which, value):
    torch = require_gpu()
    t = ks.Tables.make(0.2)
    segs = [[(1 + i, shared), (10 + 10 * i + b, own)] for i, (cands, shared) in enumerate(groups) for b in range(cands)]
    w = ks.workload_from_segments("back_nan", arch(64, 2), 750, segs, gain_std=0.2)
    p, grad, dev, sc = _gpu_grad(w, t)
    sc.close()
    pages = [set(w.block_table[b, :int(w.seq_lens[b]) // 16].tolist()) for b in range(len(segs))]
    dev.pool[0, int(w.block_table[bad, int(w.seq_lens[bad]) // 16 - 1]), which, :, 3, :] = float(value)
    p2, grad2, _, sc = _gpu_grad(w, t, dev)
    sc.close()
    others = [b for b in range(len(segs)) if b != bad]
    assert not np.isfinite(p2[bad]) and np.array_equal(p2[others], p[others])
    clean = sorted(set().union(*pages) - pages[bad])
    assert torch.equal(grad2[0][clean], grad[0][clean])


def _split(x):
    """x as the sum of its bf16 high and low parts, fp32 in, fp64 out."""
    hi = ks.bf16_bits_to_f64(ks.f64_to_bf16_bits(x))
    return hi + ks.bf16_bits_to_f64(ks.f64_to_bf16_bits(x - hi))


def test_softmax_weights_far_below_the_maximum():
    """Keys with one element, so that a score is one product and its rounding is known: each row of dV is then
    w dO, and w = exp(score - lse) can be read off it.  The backward rounds score - lse once (up to 2^-19 at 46 to
    62) and takes expf; the rounding and the weight's split into two bf16 are followed here, for every fp32 lse near
    the fp64 one.  What is left is expf's error (up to two ulp, 2.4e-7), which moves a few splits by 2^-17 = 7.6e-6,
    the fp32 sums and the dropped product of the low parts: 4.9e-7 in the mean.  An exponent that is rounded twice,
    as by exp2 of the product with log2(e), adds up to 2.6e-6 and many such moves: 1.75e-6."""
    torch = require_gpu()
    import paper_2607_09153_gb300 as kp
    heads, hd, lens = 8, 64, list(range(60, 68))
    a = ks.Arch(1, 256, heads, heads, hd, 256)
    w = ks.distinct("back_exp", a, 760, lens, gain_std=0.2)
    t = ks.Tables.make(0.2)
    dev = ks.DeviceInputs(w, t)
    sc = make_scorer(dev, len(lens), w.max_blocks)
    kp.kvprm_set_debug(sc.ctx, 2)
    sc.score(dev.pool, w.block_table, w.seq_lens)
    q, k_self = torch.empty((2, len(lens), heads, hd), dtype=torch.float32, device="cuda")
    kp.kvprm_debug_layers(sc.ctx, 1, q.data_ptr())
    kp.kvprm_debug_layers(sc.ctx, 2, k_self.data_ptr())
    torch.cuda.synchronize()
    q, k_self = q.cpu().numpy(), k_self.cpu().numpy()
    sc.close()
    rng = np.random.default_rng(4)
    dev.pool[:, :, 0] = 0
    keys = {}
    for b, L in enumerate(lens):
        for h in range(heads):
            e = int(np.abs(q[b, h]).argmax())
            k = ks.bf16_bits_to_f64(ks.f64_to_bf16_bits(8 * rng.uniform(-62, -46, L) / q[b, h, e]))
            k[0] = 0   # the largest score, and with the verify token's own the whole of lse
            keys[b, h] = k * _split(q[b, h, e].astype(np.float64)) / 8
            j = np.arange(L)
            dev.pool[0, torch.as_tensor(w.block_table[b, j // 16].astype(np.int64)), 0, h, torch.as_tensor(j % 16), e] = \
                torch.as_tensor(k, dtype=dev.pool.dtype, device="cuda")
    _, grad, _, sc = _gpu_grad(w, t, dev)
    sc.close()
    off = []
    for (b, h), s in keys.items():
        j = np.arange(1, len(s))
        dv = grad[0, torch.as_tensor(w.block_table[b, j // 16].astype(np.int64)), 1, h, torch.as_tensor(j % 16)]
        dv = dv.cpu().numpy().astype(np.float64)
        lw = np.log(dv @ (dv / np.linalg.norm(dv, axis=1, keepdims=True)).mean(0))   # ln w and a constant
        lse = np.float32(np.logaddexp(0, (q[b, h].astype(np.float64) * k_self[b, h]).sum() / 8))
        fits = []
        for i in range(-64, 65):
            x = (s[1:] - (np.float64(lse) + i * np.spacing(lse))).astype(np.float32)
            r = lw - np.log(_split(np.exp(x.astype(np.float64)).astype(np.float32).astype(np.float64)))
            fits.append(np.abs(r - np.median(r)))
        off.append(min(fits, key=np.mean))
    assert np.concatenate(off).mean() <= 1e-6
