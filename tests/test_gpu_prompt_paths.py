"""The prompt pass at the edges of its paths, teacher-forced against the oracle: chunks of up to 256 tokens (projections split
along K, finished by kernels of their own) and above (pairs of CTAs, finished in the epilogue), and prompts around the
attention's 128 x 128 tiles.  The decode steps behind it read the cache that each path filled."""
import numpy as np
import pytest

from paper_2305_13144_b200 import synth
from parity_util import HIDDEN_TOL, LOGIT_TOL, engine, teacher_forced

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,head_dim,ffn,lens", [
    (2, 128, 264, [1]),
    (2, 128, 264, [16, 1, 15]),                  # 32 tokens: the token tile is full
    (3, 64, 520, [127, 2]),                      # 129 tokens
    (2, 128, 256, [128, 127]),
    (4, 64, 1000, [256]),                        # the longest chunk of the split path, two query tiles
    (2, 128, 264, [257]),                        # the shortest of the paired path, a query tile with one row
    (3, 64, 520, [129, 128, 1, 255]),            # 513 tokens: a third token tile with one
    (1, 128, 8, [300, 385, 64]),
])
def test_prompt_lengths_and_paths(heads, head_dim, ffn, lens):
    shape = synth.ModelShape(n_layers=2, d_model=heads * head_dim, n_heads=heads, head_dim=head_dim, d_ffn=ffn, vocab=300)
    w = synth.make_weights(shape, seed=31)
    rng = np.random.default_rng(6)
    prompts = [rng.integers(3, shape.vocab, size=n).tolist() for n in lens]
    el, eh, _ = teacher_forced(shape, w, prompts, [3] * len(lens), cap=3, max_ctx=max(lens) + 4, max_prefill=max(256, sum(lens)),
                               kv_tokens=sum(lens) + 64 * len(lens))
    assert el <= LOGIT_TOL and eh <= HIDDEN_TOL, (el, eh)


@pytest.mark.parametrize("heads,ffn,lens", [
    (4, 1000, [257]),                            # two token tiles of 160 (the second with 97), nothing cut
    (16, 264, [200, 100]),                       # q,k,v: 48 units for 74 pairs, not cut either
    (16, 5000, [256, 256]),                      # two full tiles of 256; down: 16 units in four to six parts each
    (24, 264, [200, 100]),                       # o: 24 units in three or four parts each, over two tiles of 160
    (32, 2000, [130, 127]),                      # q,k,v: a full round of pairs, then 22 units in parts; o and gate/up too
    (8, 16384, [300]),                           # down: 8 units of 256 k-blocks in nine or ten parts each
    (2, 16384, [425, 425, 424, 426]),            # seven token tiles, the down projection's in groups of four and three
])
def test_cut_and_grouped_projections_of_the_paired_path(heads, ffn, lens):
    shape = synth.ModelShape(n_layers=1, d_model=heads * 128, n_heads=heads, head_dim=128, d_ffn=ffn, vocab=300)
    w = synth.make_weights(shape, seed=35)
    rng = np.random.default_rng(12)
    prompts = [rng.integers(3, shape.vocab, size=n).tolist() for n in lens]
    el, eh, _ = teacher_forced(shape, w, prompts, [2] * len(lens), cap=2, max_ctx=max(lens) + 4, max_prefill=max(256, sum(lens)),
                               kv_tokens=sum(lens) + 64 * len(lens))
    assert el <= LOGIT_TOL and eh <= HIDDEN_TOL, (el, eh)


@pytest.mark.parametrize("lens", [[280, 100, 120, 30], [100, 120, 30, 300], [300, 299, 1]])
def test_chunks_of_both_paths_in_one_batch(lens):
    """Chunks of at most 300 tokens: some run on pairs of CTAs, some with their projections split along K."""
    shape = synth.ModelShape(n_layers=2, d_model=256, n_heads=2, head_dim=128, d_ffn=264, vocab=300)
    w = synth.make_weights(shape, seed=32)
    rng = np.random.default_rng(10)
    prompts = [rng.integers(3, shape.vocab, size=n).tolist() for n in lens]
    el, eh, _ = teacher_forced(shape, w, prompts, [3] * len(lens), cap=3, max_ctx=max(lens) + 4, max_prefill=300,
                               kv_tokens=sum(lens) + 64 * len(lens))
    assert el <= LOGIT_TOL and eh <= HIDDEN_TOL, (el, eh)


def test_hidden_states_are_there_when_the_call_returns():
    """dump_hidden read on another stream right behind ss_prefill, without waiting for the engine's."""
    import torch
    from paper_2305_13144_b200 import api
    shape = synth.ModelShape(n_layers=8, d_model=2048, n_heads=16, head_dim=128, d_ffn=4096, vocab=300)
    eng = engine(shape, synth.make_weights(shape, seed=33), max_ctx=1100, max_prefill=2048, kv_tokens=9000)
    cu = np.arange(9, dtype=np.int32) * 1000               # four chunks
    ids = np.random.default_rng(11).integers(3, shape.vocab, size=8000).astype(np.int32)
    for _ in range(3):
        dh = torch.zeros(8, shape.d_model, device="cuda")
        torch.cuda.synchronize()
        api.ss_prefill(eng, ids, cu, None, 2, dump_hidden=dh)
        at_return = dh.cpu()                               # torch's stream, not the engine's
        torch.cuda.synchronize()
        api.ss_release_batch(eng)
        assert torch.equal(at_return, dh.cpu()) and (at_return.abs().amax(dim=1) > 0).all()
