"""The sequentially decoded block as one launch, at the edges of its split of the work.

bf16 engine: the cooperative kernel runs groups of at most 16 or 32 samples side by side and cuts the cache into 16-key tiles
and units of 64 or 128 keys; 132 tokens cross both, the batches leave groups and ranks short or without samples.  fp32 engine:
1, 2 or 4 samples per cluster.
"""
import threading

import numpy as np
import pytest
import torch

from oracle import tarflow_oracle as O
from paper_2505_24791_b200 import binding, synth
from tests.gpu_util import Model, rel_l2

pytestmark = pytest.mark.gpu

REL_L2, MAX_ABS = 2e-2, 5e-2  # bf16 engine against the fp64 oracle: the tolerances of every other bf16 test
PATHS = 5e-3                  # two orders of summation of the same bf16 products: the bound used for the other step kernels
FP32_MAX = 1e-4               # fp32 engine against the fp64 oracle


@pytest.mark.parametrize("width,batch,classes", [(128, 1, 0), (128, 40, 0), (256, 15, 10), (256, 130, 0), (512, 3, 0), (512, 65, 10),
                                                 (1024, 1, 0), (1024, 18, 10), (1024, 33, 0)])
def test_bf16_block_in_one_launch(monkeypatch, width, batch, classes):
    cfg = synth.config("cfg2", H=24, W=22, n_blocks=1, n_layers=2, width=width, n_heads=width // 64, n_classes=classes)
    z = synth.make_latents(cfg, 7, B=batch)
    lab = synth.make_labels(cfg, B=batch) if classes else None
    out = {}
    for path in ("0", "1"):
        monkeypatch.setenv("TARFLOW_SEQ_PERSIST", path)
        with Model(cfg, max_batch=batch) as m:
            out[path] = m.inverse_sequential(z, lab)
            pick = sorted({0, batch // 2, batch - 1})
            if path == "1":  # a sample's arithmetic depends neither on the batch nor on its place in it
                for p in pick:
                    alone = m.inverse_sequential(z[p:p + 1], None if lab is None else lab[p:p + 1])
                    assert np.array_equal(alone[0], out[path][p])
            xo = O.model_inverse_sequential(m.blocks, z[pick], None if lab is None else lab[pick], cfg)
        x = out[path][pick]
        assert np.isfinite(out[path]).all() and rel_l2(x, xo) <= REL_L2 and np.abs(x - xo).max() <= MAX_ABS
    assert rel_l2(out["1"], out["0"]) <= PATHS


@pytest.mark.parametrize("batch", [1, 17, 37])
def test_fp32_block_in_one_launch(batch):
    cfg = synth.config("cfg1", H=14, W=10, n_blocks=1)
    z = synth.make_latents(cfg, 8, B=batch)
    with Model(cfg, max_batch=batch) as m:
        x = m.inverse_sequential(z, None)
        assert np.abs(x - O.model_inverse_sequential(m.blocks, z, None, cfg)).max() <= FP32_MAX


def test_bf16_block_whose_launch_is_refused_runs_as_a_chain(monkeypatch):
    cfg = synth.config("cfg2", H=12, W=12, n_blocks=2, n_layers=1, width=128, n_heads=2)
    z = synth.make_latents(cfg, 9, B=5)
    monkeypatch.setenv("TARFLOW_SEQ_PERSIST", "0")
    with Model(cfg, max_batch=5) as m:
        chain = m.inverse_sequential(z, None)
    monkeypatch.delenv("TARFLOW_SEQ_PERSIST")
    with Model(cfg, max_batch=5) as m:
        at_once = m.inverse_sequential(z, None)
        binding.tf_debug_set(m.m, binding.TF_DEBUG_REFUSE_BLOCK_LAUNCH, 1)
        for profile in (0, 2):
            binding.tf_profile_enable(m.m, profile)
            assert np.array_equal(m.inverse_sequential(z, None), chain)
        binding.tf_profile_enable(m.m, 0)
        x, _, _, rc = m.inverse(z, None, [0, 1], 1e-3, m.L + 1)    # nothing of the refusal is left for later launches to report
        assert rc == 0 and np.isfinite(x).all()
        binding.tf_debug_set(m.m, binding.TF_DEBUG_REFUSE_BLOCK_LAUNCH, 0)
        assert np.array_equal(m.inverse_sequential(z, None), at_once)


def test_bf16_blocks_of_two_models_on_two_streams():
    """Launches whose CTAs wait on one another take turns: two handles, two threads, two streams, as many blocks as each decodes."""
    cfg = synth.config("cfg2", H=12, W=12, n_blocks=4, n_layers=2, width=256, n_heads=4)
    B = 70   # more than half of the GPU's SMs each
    z = torch.from_numpy(synth.make_latents(cfg, 10, B=B)).cuda()
    with Model(cfg, max_batch=B) as a, Model(cfg, max_batch=B) as b:
        want = a.inverse_sequential(z.cpu().numpy(), None)
        got, failed = {}, []

        def decode(m, name):
            try:
                stream = torch.cuda.Stream()
                with torch.cuda.stream(stream):
                    x = torch.empty_like(z)
                    for _ in range(8):
                        x.fill_(float("nan"))
                        binding.tf_inverse_sequential(m.m, z, None, B, x)
                        got.setdefault(name, []).append(x.cpu().numpy())
            except Exception as e:  # noqa: BLE001 -- reported below, by the test's own thread
                failed.append(e)

        torch.cuda.synchronize()
        threads = [threading.Thread(target=decode, args=(m, n)) for n, m in (("a", a), ("b", b))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not failed, failed
        for name in ("a", "b"):
            assert len(got[name]) == 8 and all(np.array_equal(x, want) for x in got[name])


@pytest.mark.parametrize("width,batch", [(128, 9), (512, 5), (1024, 6)])
def test_bf16_block_of_one_layer_reads_the_rows_it_has_just_written(width, batch):
    """With one layer a step's new keys and values are read by bulk copies of the very next layer walked; 150 tokens fill several
    units of the ring."""
    cfg = synth.config("cfg2", H=30, W=20, n_blocks=1, n_layers=1, width=width, n_heads=width // 64)
    z = synth.make_latents(cfg, 12, B=batch)
    with Model(cfg, max_batch=batch) as m:
        x = m.inverse_sequential(z, None)
        xo = O.model_inverse_sequential(m.blocks, z, None, cfg)
        assert rel_l2(x, xo) <= REL_L2 and np.abs(x - xo).max() <= MAX_ABS
        assert all(np.array_equal(m.inverse_sequential(z, None), x) for _ in range(5))


@pytest.mark.parametrize("before_the_end", [1, 0, -1])
def test_bf16_block_when_the_exchange_numbers_start_over(before_the_end):
    """A batch of 40 leaves words in rows that a batch of 1 does not touch.  Started over at the end of the 32-bit range, the
    numbers of the batch of 1 end where those words' numbers begin: the second batch of 40 must not take them for its own."""
    cfg = synth.config("cfg2", H=12, W=12, n_blocks=1, n_layers=2, width=128, n_heads=2)
    numbers = (2 * cfg["n_layers"] + 1) * (synth.seq_len(cfg) - 1) + 1   # of one block
    z = synth.make_latents(cfg, 11, B=40)
    with Model(cfg, max_batch=40) as m:
        want = m.inverse_sequential(z, None)
        alone = m.inverse_sequential(z[:1], None)
        last = 2 ** 32 - 1
        # the whole block still fits, one number is missing, or nearly all of them are
        start = {1: last - numbers, 0: last - numbers + 1, -1: last - 1}[before_the_end]
        binding.tf_debug_set(m.m, binding.TF_DEBUG_EXCHANGE_NUMBER, start)
        assert np.array_equal(m.inverse_sequential(z[:1], None), alone)
        for _ in range(2):
            assert np.array_equal(m.inverse_sequential(z, None), want)
        with pytest.raises(binding.TarflowError):
            binding.tf_debug_set(m.m, binding.TF_DEBUG_EXCHANGE_NUMBER, 1)


def test_fp32_sample_that_diverges_leaves_its_cluster_mates_alone():
    """Four samples share a cluster here and a CTA has five heads, 20 (sample, head) pairs for 16 warps: a warp goes on to the
    pair of another sample with the first one's rows still in its registers."""
    cfg = synth.config("cfg1", H=16, W=12, n_blocks=1, n_layers=1, width=160, n_heads=40, mlp_ratio=1)
    z = synth.make_latents(cfg, 13, B=80)
    with Model(cfg, max_batch=80) as m:
        want = m.inverse_sequential(z, None)
        assert np.isfinite(want).all()
        z[4] = 3e38
        x = m.inverse_sequential(z, None)
        others = np.arange(80) != 4
        assert not np.isfinite(x[4]).all() and np.array_equal(x[others], want[others])


@pytest.mark.parametrize("over", [{}, dict(width=96, n_heads=3, n_blocks=1), dict(H=14, W=10, width=160, n_heads=40, mlp_ratio=1, n_layers=1)])
def test_fp32_sample_does_not_depend_on_the_batch(over):
    """Every direction of the fp32 engine, one sample alone, a few, and as part of a batch that fills clusters with two or four
    samples and the products' widest tiles: the same bits."""
    cfg = synth.config("cfg1", **over)
    K, B = cfg["n_blocks"], 90
    z = synth.make_latents(cfg, 14, B=B)
    with Model(cfg, max_batch=B) as m:
        calls = {"sequential": lambda x: (m.inverse_sequential(x, None),),
                 "jacobi": lambda x: m.inverse(x, None, [1] * K, 1e-5, m.L + 1)[::2],
                 "forward": lambda x: m.forward(x, None)}
        for name, call in calls.items():
            whole = call(z)
            for pick in (slice(0, 1), slice(57, 60), slice(B - 30, B)):
                part = call(z[pick])
                assert np.array_equal(part[0], whole[0][pick]), (name, pick)
                if name != "sequential":   # sweep counts [blocks, samples], log-determinants
                    assert np.array_equal(part[1], whole[1][..., pick]), (name, pick)
