"""One context, one call after another of a different kind: plans with a fused combine, packed short runs, long ragged
runs, shared pages, the tensor-core launch, the attention entry point, another readout depth and the gradient.  Nothing
of a call's plan may reach the next: every result is, bit for bit, that of a context made for this call alone (the
gradient: within the order of its sums)."""
import itertools

import numpy as np
import pytest

import kvsynth as ks
from tests.gpu_util import make_scorer, require_gpu

pytestmark = pytest.mark.gpu

# (cache segments of every candidate)
BATCHES = {
    "equal": [[(b, 160)] for b in range(8)],                      # fused combine
    "short": [[(20 + b, 1 + 7 * b)] for b in range(9)],           # packed
    "long": [[(40 + b, 300 + 171 * b)] for b in range(7)],        # persistent, private runs
    "prefix": [[(60, 96), (61 + b, 21)] for b in range(10)],      # shared pages (head_dim 128: on the tensor cores)
    "one": [[(80, 47)]],
}


@pytest.mark.parametrize("arch", [ks.Arch(2, 256, 14, 2, 128, 512), ks.Arch(2, 256, 4, 2, 64, 512)])
def test_calls_of_every_kind_after_one_another(arch):
    torch = require_gpu()
    import paper_2607_09153_gb300 as kp
    names = list(BATCHES)
    w = ks.workload_from_segments("reuse", arch, 960, [s for k in names for s in BATCHES[k]], gain_std=0.2)
    dev = ks.DeviceInputs(w, ks.Tables.make(0.2))
    first = dict(zip(names, np.cumsum([0] + [len(BATCHES[k]) for k in names])))
    rows = {k: slice(first[k], first[k] + len(BATCHES[k])) for k in names}
    tables = {k: (np.ascontiguousarray(w.block_table[rows[k]]), np.ascontiguousarray(w.seq_lens[rows[k]])) for k in names}
    gen = torch.Generator(device="cuda").manual_seed(3)
    qkv = [torch.randn((10, h, arch.head_dim), generator=gen, device="cuda")
           for h in (arch.n_q_heads, arch.n_kv_heads, arch.n_kv_heads)]
    st = torch.cuda.current_stream().cuda_stream

    def call(sc, kind, batch):
        bt, sl = tables[batch]
        n = len(sl)
        if kind == "attention":
            out = torch.zeros_like(qkv[0])
            kp.kvprm_attention(sc.ctx, dev.pool[0].data_ptr(), dev.n_pages, bt, sl, n, *(x.data_ptr() for x in qkv),
                               out.data_ptr(), st)
        elif kind == "grad":
            out = torch.zeros(dev.pool.shape, dtype=torch.float32, device="cuda")
            kp.kvprm_score_grad(sc.ctx, dev.pool.data_ptr(), dev.n_pages, bt, sl, n, out.data_ptr(), st)
        else:
            sc.set_depth(kind)
            out = torch.from_numpy(sc.score(dev.pool, bt, sl))
            sc.set_depth(1)
        kp.kvprm_check_device(sc.ctx)
        return out.cpu()

    def scorer():
        return make_scorer(dev, 48, w.max_blocks)

    calls = [(kind, batch) for kind in (1, 4, "attention", "grad") for batch in names]
    want = {}
    for c in calls:
        sc = scorer()
        want[c] = call(sc, *c)
        sc.close()
    sc = scorer()
    order = [c for pair in itertools.permutations(calls, 2) for c in pair]   # each kind after each other one
    for c in order:
        got = call(sc, *c)
        if c[0] == "grad":
            assert ((got - want[c]).norm() / want[c].norm()).item() < 1e-4, c
        else:
            assert torch.equal(got, want[c]), c
    sc.close()
