"""Buffers that a context makes after its creation (the first gradient call's, the debug captures', an adapter's)
are zeroed before the caller's work on them, whatever its stream: the calls run on a stream that does not wait for
the legacy default stream, which is kept busy meanwhile.  Against the same calls on the default stream."""
import dataclasses

import pytest

import kvsynth as ks
from tests.gpu_util import make_scorer, require_gpu

pytestmark = pytest.mark.gpu

ARCH = ks.Arch(2, 512, 8, 2, 64, 2048)


def _grads(sc, dev, w, stream, calls):
    torch = require_gpu()
    import paper_2607_09153_gb300 as kp
    out = [torch.zeros(dev.pool.shape, dtype=torch.float32, device="cuda") for _ in range(calls)]
    torch.cuda.synchronize()
    if stream.cuda_stream:
        torch.cuda._sleep(100_000_000)   # about 50 ms on the default stream
    for g in out:   # the first while the default stream is busy, the rest once it has caught up
        kp.kvprm_score_grad(sc.ctx, dev.pool.data_ptr(), dev.n_pages, w.block_table, w.seq_lens, w.n_candidates,
                            g.data_ptr(), stream.cuda_stream)
        torch.cuda.synchronize()
    kp.kvprm_check_device(sc.ctx)
    return out


@pytest.mark.parametrize("group_of", [ARCH, ks.Arch(2, 512, 16, 1, 64, 512)])   # tcgen05, CUDA cores
def test_first_gradient_calls(group_of):
    torch = require_gpu()
    w = ks.shared_prefix("streams", group_of, 940, 5, 70, 45, gain_std=0.2)
    dev = ks.DeviceInputs(w, ks.Tables.make(0.2))
    sc = make_scorer(dev, 5, w.max_blocks)
    want = _grads(sc, dev, w, torch.cuda.default_stream(), 1)[0]
    sc.close()
    sc = make_scorer(dev, 5, w.max_blocks)
    for g in _grads(sc, dev, w, torch.cuda.Stream(), 2):
        assert ((g - want).norm() / want.norm()).item() < 1e-4   # sums in another order
    sc.close()


def test_first_gradient_call_on_a_captured_stream():
    # refused before anything is made, so that the call after it makes its buffers
    torch = require_gpu()
    import paper_2607_09153_gb300 as kp
    w = ks.shared_prefix("streams_c", ARCH, 942, 5, 70, 45, gain_std=0.2)
    dev = ks.DeviceInputs(w, ks.Tables.make(0.2))
    sc = make_scorer(dev, 5, w.max_blocks)
    want = _grads(sc, dev, w, torch.cuda.default_stream(), 1)[0]
    sc.close()
    sc = make_scorer(dev, 5, w.max_blocks)
    s, g = torch.cuda.Stream(), torch.zeros(dev.pool.shape, dtype=torch.float32, device="cuda")
    x = torch.ones(4, device="cuda")
    with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=s, capture_error_mode="relaxed"):
        x += 1
        with pytest.raises(kp.KvprmError) as e:
            kp.kvprm_score_grad(sc.ctx, dev.pool.data_ptr(), dev.n_pages, w.block_table, w.seq_lens, w.n_candidates,
                                g.data_ptr(), s.cuda_stream)
    assert e.value.code == kp.KVPRM_EUNSUPPORTED
    got = _grads(sc, dev, w, torch.cuda.default_stream(), 1)[0]
    assert ((got - want).norm() / want.norm()).item() < 1e-4
    sc.close()


def test_debug_capture_and_adapter():
    torch = require_gpu()
    import paper_2607_09153_gb300 as kp
    n = 5
    w = ks.distinct("streams_l", dataclasses.replace(ARCH, lora_rank=64), 941, [40, 0, 17, 100, 64], gain_std=0.2)
    dev = ks.DeviceInputs(w, ks.Tables.make(0.2))

    a = dev.arch
    names = dict(zip(ks.LORA_KINDS, ("a_qkv", "b_qkv", "a_o", "b_o", "a_gate_up", "b_gate_up", "a_down", "b_down")))
    factors = [{names[k]: L[k] for k in ks.LORA_KINDS} for L in dev.layers]

    def run(stream):
        sc = make_scorer(dev, n, w.max_blocks)
        r = torch.zeros(n, device="cuda")
        attn = torch.empty((a.n_layers, n, a.n_q_heads * a.head_dim), device="cuda")
        torch.cuda.synchronize()
        if stream.cuda_stream:
            torch.cuda._sleep(100_000_000)
        sc.set_lora(0)
        sc.set_lora(a.lora_rank, a.lora_alpha, factors)   # its buffers are there: zeroed again
        kp.kvprm_set_debug(sc.ctx, 1)
        sc.score_async(dev.pool, w.block_table, w.seq_lens, r, stream=stream)
        kp.kvprm_debug_attn_out(sc.ctx, attn.data_ptr())
        torch.cuda.synchronize()
        sc.close()
        return r.cpu(), attn.cpu()

    want, got = run(torch.cuda.default_stream()), run(torch.cuda.Stream())
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
