"""The projections where the choice of kernel image and ring depth changes: 32, 33, 48, 49 and 64, 65, 80, 81
candidates (the padded columns step by 16), a gate/up that only fits one wave with a stage less, a down
projection whose K loop gets twice the CTAs, the adapter's A x on either image, and an adapter with more K
tiles than the weights.  One kernel alone
against an fp64 product (fp32 accumulation over K = 18,944: below 1e-5 of the largest output), and whole
layers against the oracle with the scoring tolerances.  And an adapter's launches beside one another against the
same launches one after the other."""
import dataclasses

import numpy as np
import pytest

import kvsynth as ks
from tests.gpu_util import compare, make_scorer, require_gpu, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    require_gpu()
    w = ks.distinct("proj_img", ks.Arch(1, 3584, 28, 4, 128, 18944), 1, [16])
    sc = make_scorer(ks.DeviceInputs(w, ks.Tables.make()), 96, 4)
    yield sc
    sc.close()


@pytest.mark.parametrize("M, K, n", [(3584, 18944, 33), (3584, 18944, 48), (3584, 18944, 49), (3584, 18944, 65),
                                     (3584, 18944, 80), (37888, 3584, 33), (37888, 3584, 48), (1000, 192, 40)])
def test_projection(ctx, M, K, n):
    torch = require_gpu()
    import paper_2607_09153_gb300 as kp
    rng = np.random.default_rng(M + K + n)
    Wb, Xb = ks.f64_to_bf16_bits(rng.normal(0, 0.02, (M, K))), ks.f64_to_bf16_bits(rng.normal(0, 1, (n, K)))
    W, X = (torch.from_numpy(b.view(np.int16)).cuda() for b in (Wb, Xb))
    Y = torch.full((n, M), float("nan"), dtype=torch.float32, device="cuda")
    kp.kvprm_projection(ctx.ctx, W.data_ptr(), M, K, X.data_ptr(), n, Y.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    ref = ks.bf16_bits_to_f64(Xb) @ ks.bf16_bits_to_f64(Wb).T
    assert np.abs(Y.cpu().numpy().astype(np.float64) - ref).max() / np.abs(ref).max() < 1e-5


@pytest.mark.parametrize("n, rank", [(5, 512), (32, 64), (33, 0), (48, 128), (49, 0), (65, 64), (80, 0), (81, 64)])
def test_layers(n, rank):
    require_gpu()
    arch = dataclasses.replace(ks.Arch(2, 320, 5, 5, 64, 9792), lora_rank=rank)
    w = ks.distinct("images", arch, 900 + n, [(7 * b) % 50 for b in range(n)], gain_std=0.2)
    t = ks.Tables.make(0.2)
    r, attn, _, sc = run_gpu(w, t)
    compare(w, t, gpu_rewards=r, gpu_attn=attn, label=f"n {n} rank {rank}")
    sc.close()


@pytest.mark.parametrize("arch, n", [(ks.Arch(3, 1536, 12, 2, 128, 8960), 16), (ks.Arch(3, 1536, 12, 2, 128, 8960), 48),
                                     (ks.Arch(2, 256, 4, 2, 64, 704), 201)])
@pytest.mark.parametrize("rank", [64, 256])
def test_adapter_beside_the_weights(monkeypatch, arch, n, rank):
    """A projection with an adapter starts while its A x still runs and reads x after the mark that A x leaves: calls
    of two different batches in turn, queued behind one another, against launches that wait for their predecessor's
    end.  The same kernels in the same order of sums, so bit for bit."""
    torch = require_gpu()
    w = ks.distinct("beside", dataclasses.replace(arch, lora_rank=rank), 950 + n, [(7 * b) % 90 for b in range(n)],
                    gain_std=0.2)
    dev = ks.DeviceInputs(w, ks.Tables.make(0.2))
    bt, sl = np.asarray(w.block_table), np.asarray(w.seq_lens)
    batches = [(bt, sl), (np.ascontiguousarray(np.roll(bt, 1, 0)), np.ascontiguousarray(np.roll(sl, 1)))]
    sc = make_scorer(dev, n, w.max_blocks)
    out = torch.zeros((40, n), dtype=torch.float32, device="cuda")
    for i in range(40):
        sc.score_async(dev.pool, *batches[i % 2], out[i])
    torch.cuda.synchronize()
    sc.close()
    monkeypatch.setenv("KVPRM_NO_PDL", "1")
    sc = make_scorer(dev, n, w.max_blocks)
    for k, b in enumerate(batches):
        want = torch.from_numpy(sc.score(dev.pool, *b))
        assert all(torch.equal(o, want) for o in out[k::2].cpu())
    sc.close()
