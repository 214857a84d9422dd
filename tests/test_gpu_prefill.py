"""Prefill of several prompts at once: a chunk's rows may belong to several streams, and prompts are cut
at chunk borders.  A row's sums are taken in the same order whatever its chunk holds, so the cache must
hold bit for bit what each prompt leaves when it is prefilled alone, and the verify step from there must
agree with the oracle.
"""
import numpy as np
import pytest
import torch

from paper_2505_15380_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hd,hq,hkv,d,f,lens", [
    (64, 4, 2, 128, 256, [300, 18, 65, 2000, 130, 66]),      # more rows than a chunk: a prompt is cut in two
    (128, 4, 1, 256, 640, [64, 129, 1, 20]),                 # tile and chunk edges; a prompt without cached rows
    (32, 16, 1, 136, 264, [33, 80]),                         # 16 query heads per kv head: 4 rows per attention tile
])
def test_prompts_together_equal_prompts_alone(hd, hq, hkv, d, f, lens):
    from paper_2505_15380_b200 import binding
    shape = synth.ModelShape(3, d, hq, hkv, hd, f, 301, 8, 1e4, weight_dtype=synth.BF16)
    wl = synth.Workload("prefill", shape, shape, len(lens), 3, 1.0, 0, tuple(lens), 2, d, d + 1)
    model = binding.Model(shape, synth.weights_blob(shape, synth.make_weights(shape, d)))
    prefixes = [synth.make_prefix(wl, b) for b in range(len(lens))]
    none = np.zeros(0, np.int32)
    together, alone = (binding.Streams(model, len(lens), max(lens) + 8, 3) for _ in range(2))
    together.kv.zero_()
    alone.kv.zero_()
    together.prefill(prefixes)
    for b in range(len(lens)):
        alone.prefill([p if i == b else none for i, p in enumerate(prefixes)])
    for gs in (together, alone):
        assert gs.last_status() == 0
        n, pend = gs.get_state()
        assert list(n) == [x - 1 for x in lens] and list(pend) == [int(p[-1]) for p in prefixes]
    assert torch.equal(together.kv, alone.kv)
    pages = sum(-(-n // 64) for n in lens) + len(lens)
    paged = binding.PagedStreams(model, len(lens), pages, -(-max(lens) // 64) + 1, 3)
    paged.kv.zero_()
    paged.prefill(prefixes)
    assert paged.last_status() == 0
    _, _, table = paged.paged_state()
    for b, n in enumerate(lens):
        for pg in range(-(-(n - 1) // 64)):
            a, z = pg * 64, min(pg * 64 + 64, n - 1)
            assert torch.equal(paged.kv[:, table[b, pg], :, :, : z - a], together.kv[:, b, :, :, a:z])


def test_verify_after_a_prefill_of_several_chunks():
    from tests.gpu_case import run_case
    shape = synth.ModelShape(2, 128, 4, 2, 64, 256, 300, 8, 1e4, weight_dtype=synth.BF16)
    wl = synth.Workload("prefill", shape, shape, 4, 4, 0.8, 25, (1300, 17, 900, 260), 2, 5, 6)
    run_case(wl, beta=0.4, sigma=1.0, logit_tol=2e-3)


def test_short_prompts_beside_others_equal_prompts_alone():
    """Prompts of at most 16 rows take the persistent kernel, whoever joins beside them."""
    from paper_2505_15380_b200 import binding
    lens = [300, 17, 2, 40, 9]
    shape = synth.ModelShape(3, 128, 4, 2, 64, 256, 301, 8, 1e4, weight_dtype=synth.BF16)
    wl = synth.Workload("prefill", shape, shape, len(lens), 3, 1.0, 0, tuple(lens), 2, 5, 6)
    model = binding.Model(shape, synth.weights_blob(shape, synth.make_weights(shape, 5)))
    prefixes = [synth.make_prefix(wl, b) for b in range(len(lens))]
    together, alone = (binding.Streams(model, len(lens), max(lens) + 8, 3) for _ in range(2))
    together.kv.zero_()
    alone.kv.zero_()
    together.prefill(prefixes)
    for b in range(len(lens)):
        alone.prefill([p if i == b else np.zeros(0, np.int32) for i, p in enumerate(prefixes)])
    for gs in (together, alone):
        assert gs.last_status() == 0
        n, pend = gs.get_state()
        assert list(n) == [x - 1 for x in lens] and list(pend) == [int(p[-1]) for p in prefixes]
    assert torch.equal(together.kv, alone.kv)
