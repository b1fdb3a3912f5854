"""Projections on CTA pairs (two CTAs, an M = 256 MMA, half of the activation tile read from each): plain pairs
and pairs that hold half of the columns, with and without a cluster reduction, every epilogue, an adapter's extra
K tiles and K tiles that do not divide among the ranks, at padded columns around the choice of the form and up to
the largest.  Against the oracle with the scoring tolerances.  And, on the host, that a plan's clusters are placed
in one wave."""
import dataclasses

import pytest

import kvsynth as ks
import paper_2607_09153_gb300 as kp
from tests.gpu_util import compare, make_scorer, require_gpu, run_gpu
from tests.test_gpu_steering import _compare, _gpu_grad, _oracle

# QKV and O: pairs at 80 to 128 padded columns, halves beyond; down (11 K tiles over 4 ranks): pairs
SMALL = ks.Arch(2, 256, 4, 2, 64, 704)
# QKV (36 m-tiles, 18 clusters of 8 do not fit): halves from 96, two ranks
WIDE = ks.Arch(1, 512, 28, 4, 128, 1024)
# gate/up has more tiles than the chip has SMs: pairs, of an even and of an odd number of 128-row units
GATE_UP = ks.Arch(1, 128, 2, 2, 64, 9984)
GATE_UP_ODD = ks.Arch(1, 128, 2, 2, 64, 9856)
PLACED = {1: 152, 2: 76, 4: 36, 8: 15, 16: 7}   # clusters of CTAs that fill an SM, on 152 SMs


@pytest.mark.parametrize("arch", [ks.ARCH_1P5B, ks.ARCH_7B, ks.ARCH_8B, SMALL, WIDE])
@pytest.mark.parametrize("rank", [0, 256])
def test_clusters_are_placed(arch, rank):
    for n_pad in range(16, 257, 16):
        for M, K in [(arch.qkv_rows, arch.d_model), (arch.d_model, arch.n_q_heads * arch.head_dim), (arch.d_model, arch.d_ff)]:
            p = kp.kvprm_plan_projection(M, K + rank, n_pad, 152, True, False)
            clusters = (p["m_tiles"] + p["tiles_per_cta"] - 1) // p["tiles_per_cta"]
            if p["smem_bytes"] + 1024 > 228 * 1024 // 2 and p["cluster"] > 1:
                assert clusters <= PLACED[p["cluster"]], (M, K, n_pad)


@pytest.mark.gpu
@pytest.mark.parametrize("arch", [ks.ARCH_1P5B, ks.ARCH_7B, ks.ARCH_8B, SMALL, WIDE, GATE_UP])
def test_clusters_are_placed_by_the_device(arch):
    """The same of the launches themselves: where a CTA fills an SM, no more clusters than the device holds at once
    with the shared memory and cluster size that the launch has (not the plan's table of what GPCs place)."""
    require_gpu()
    w = ks.distinct("placed", ks.Arch(1, 128, 2, 2, 64, 128), 810, [16])
    sc = make_scorer(ks.DeviceInputs(w, ks.Tables.make(0.2)), 256, w.max_blocks)
    checked = 0
    for n_pad in range(16, 257, 16):
        for M, K, gu in [(arch.qkv_rows, arch.d_model, False), (arch.d_model, arch.n_q_heads * arch.head_dim, False),
                         (arch.d_model, arch.d_ff, False), (arch.d_ff, arch.d_model, True)]:
            for rank in (0, 64, 256):
                p = kp.kvprm_plan_projection(M, K + rank, n_pad, 152, True, gu)
                if p["smem_bytes"] + 1024 > 228 * 1024 // 2 and p["cluster"] * (1 + p["pair"]) > 1:
                    clusters, placed = kp.kvprm_debug_projection_placement(sc.ctx, M, K + rank, n_pad, gu)
                    assert 0 < clusters <= placed, (M, K, n_pad, gu, rank, p)
                    checked += 1
    assert checked
    sc.close()


@pytest.mark.gpu
@pytest.mark.parametrize("arch, n, rank", [(SMALL, 48, 0), (SMALL, 64, 64), (SMALL, 65, 0), (SMALL, 128, 64),
                                           (SMALL, 129, 0), (SMALL, 145, 256),
                                           (SMALL, 208, 64), (SMALL, 256, 0), (WIDE, 88, 0), (WIDE, 129, 64), (WIDE, 176, 0),
                                           (WIDE, 250, 0), (GATE_UP, 48, 0), (GATE_UP, 128, 64), (GATE_UP, 161, 0),
                                           (GATE_UP_ODD, 49, 0), (GATE_UP_ODD, 80, 64),
                                           (GATE_UP_ODD, 256, 0)])
def test_layers(arch, n, rank):
    require_gpu()
    w = ks.distinct("pairs", dataclasses.replace(arch, lora_rank=rank), 700 + n, [(5 * b) % 40 for b in range(n)],
                    gain_std=0.2)
    t = ks.Tables.make(0.2)
    r, attn, _, sc = run_gpu(w, t)
    compare(w, t, gpu_rewards=r, gpu_attn=attn, label=f"d {arch.d_model} n {n} rank {rank}")
    sc.close()


@pytest.mark.gpu
def test_gradient():
    """The backward's products and the gate and up values that the forward keeps for it."""
    require_gpu()
    w = ks.distinct("pairs_grad", GATE_UP, 790, [(7 * b) % 20 for b in range(166)], gain_std=0.2)
    t = ks.Tables.make(0.2)
    p, grad, dev, sc = _gpu_grad(w, t)
    p_ref, ref, _, _ = _oracle(w, t)
    _compare("166 candidates", w, p, grad, p_ref, ref)
    sc.close()


@pytest.mark.gpu
def test_two_streams():
    """Two contexts' pairs on two streams at once: the rewards of either alone, bit for bit."""
    torch = require_gpu()
    t = ks.Tables.make(0.2)
    runs = []
    for arch, n in [(GATE_UP, 96), (WIDE, 130)]:
        w = ks.distinct("pairs_streams", arch, 800 + n, [(5 * b) % 40 for b in range(n)], gain_std=0.2)
        dev = ks.DeviceInputs(w, t)
        sc = make_scorer(dev, n, w.max_blocks)
        alone = torch.tensor(sc.score(dev.pool, w.block_table, w.seq_lens))
        runs.append((w, dev, sc, alone, torch.zeros(n, device="cuda"), torch.cuda.Stream()))
    torch.cuda.synchronize()
    for _ in range(8):
        for w, dev, sc, _, out, st in runs:
            sc.score_async(dev.pool, w.block_table, w.seq_lens, out, stream=st)
    torch.cuda.synchronize()
    for _, _, sc, alone, out, _ in runs:
        assert torch.equal(out.cpu(), alone)
        sc.close()
