"""ss_logits_noalloc(): the entry point for callers that may not allocate device memory (code
inside someone else's graph capture or allocator callback, or a process whose memory belongs to
another pool).  Its scratch is a fixed array inside the library that all calls share, so the
check is made on two calls in a row with different inputs: each must reproduce the logits that
the engine's own entry points (ss_prefill / ss_decode_step with dump_logits) computed from the
same hidden states, and the logits the CPU oracle's final norm + LM head give for them, within
the tolerance of the other GPU tests (2e-2 of the largest logit).
This file sorts last on purpose: a failure here cannot hide the other tests in a -x run."""
import numpy as np
import pytest

from oracle import decoder as od
from paper_2305_13144_b200 import synth

pytestmark = pytest.mark.gpu


def test_noalloc_logits_match_engine_on_two_calls_in_a_row():
    import torch
    from paper_2305_13144_b200 import api
    shape = synth.TINY
    w = synth.make_weights(shape, seed=1234)
    bits = {k: synth.to_bf16_bits(v) for k, v in w.items()}
    eng = api.make_engine(shape, api.runtime_cfg(16, 128, 512, 16, 2048), bits)
    oracle = od.Decoder(w, n_layers=shape.n_layers, n_heads=shape.n_heads, head_dim=shape.head_dim,
                        rms_eps=shape.rms_eps, rope_theta=shape.rope_theta, eos_id=shape.eos_id)
    gain = torch.from_numpy(bits["final_norm"].view(np.int16)).cuda().view(torch.bfloat16)
    head = torch.from_numpy(bits["lm_head"].view(np.int16)).cuda().view(torch.bfloat16)
    g = synth.group_tiny(seed=3)
    B = 5
    toks = np.concatenate([g.prompt(i) for i in range(B)]).astype(np.int32)
    cu = np.zeros(B + 1, dtype=np.int32)
    cu[1:] = np.cumsum(g.prompt_len[:B])
    dl = torch.zeros(B, shape.vocab, dtype=torch.float32, device="cuda")
    dh = torch.zeros(B, shape.d_model, dtype=torch.float32, device="cuda")
    mine = torch.full((B, shape.vocab), float("nan"), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    api.ss_prefill(eng, toks, cu, None, 8, dump_logits=dl, dump_hidden=dh)
    for call in range(2):
        torch.cuda.synchronize()
        api.ss_logits_noalloc(dh, gain, head, shape.rms_eps, mine)
        torch.cuda.synchronize()
        ref, got = dl.cpu().numpy(), mine.cpu().numpy()
        assert np.isfinite(got).all()
        err = np.max(np.abs(got - ref)) / np.max(np.abs(ref))
        assert err <= 2e-2, (call, err)
        exp = oracle.logits_of(dh.cpu().numpy().astype(np.float64))        # the oracle on the same hidden states
        err_o = np.max(np.abs(got - exp)) / np.max(np.abs(exp))
        assert err_o <= 2e-2, (call, err_o)
        mine.fill_(float("nan"))
        api.ss_decode_step(eng, dump_logits=dl, dump_hidden=dh)      # new hidden states for the second call
    api.ss_release_batch(eng)


def test_noalloc_rejects_sizes_beyond_its_array():
    import torch
    from paper_2305_13144_b200 import api
    d, V = 64, 256
    gain = torch.ones(d, dtype=torch.bfloat16, device="cuda")
    head = torch.zeros(V, d, dtype=torch.bfloat16, device="cuda")
    h = torch.zeros(17, d, dtype=torch.float32, device="cuda")
    out = torch.zeros(17, V, dtype=torch.float32, device="cuda")
    with pytest.raises(api.SSError) as e:
        api.ss_logits_noalloc(h, gain, head, 1e-6, out)              # 17 rows > 16
    assert e.value.code == api.SS_ERR_CAPACITY


@pytest.mark.parametrize("rows,d,vocab,offset", [(1, 64, 130, 0), (5, 192, 1000, 1), (16, 4096, 4097, 0), (3, 8192, 129, 3)])
def test_noalloc_sizes_and_alignments(rows, d, vocab, offset):
    """Rows that do not fill the summing kernel's groups, vocabularies that end inside a tile, inputs that begin `offset`
    elements behind a 16-byte boundary, against fp64.  The normalised input is rounded once (2^-9 at most, relative), so
    the result is off by no more than that in the 2-norm but for the fp32 sums: 3e-3."""
    import torch
    from paper_2305_13144_b200 import api
    gen = torch.Generator(device="cuda")
    gen.manual_seed(rows + d)
    h = torch.empty(rows * d + offset, device="cuda").normal_(0.0, 2.0, generator=gen)[offset:].view(rows, d)
    gain = torch.empty(d + offset, device="cuda").uniform_(0.5, 1.5, generator=gen).to(torch.bfloat16)[offset:]
    head = torch.empty(vocab, d, device="cuda").normal_(0.0, 0.02, generator=gen).to(torch.bfloat16)
    out = torch.full((rows, vocab), float("nan"), device="cuda")
    torch.cuda.synchronize()
    for _ in range(2):
        api.ss_logits_noalloc(h, gain, head, 1e-6, out)
    torch.cuda.synchronize()
    x = h.double() * torch.rsqrt(h.double().square().mean(1, keepdim=True) + 1e-6) * gain.double()
    ref = x @ head.double().T
    assert float((out.double() - ref).norm() / ref.norm()) <= 3e-3


def test_noalloc_inside_a_graph_capture():
    """What the call exists for: captured beside other work, replayed with other inputs, the results of a plain call.  The
    captured launches depend on one another in the plain way, so that a framework can read the graph's edges with the calls
    that know no other (cudaGraphGetEdges fails on edges that carry data of their own)."""
    import ctypes
    import torch
    from paper_2305_13144_b200 import api
    n, d, V = 7, 512, 1000
    gen = torch.Generator(device="cuda")
    gen.manual_seed(9)
    head = torch.empty(V, d, device="cuda").normal_(0.0, 0.02, generator=gen).to(torch.bfloat16)
    gain = torch.ones(d, device="cuda", dtype=torch.bfloat16)
    src, h, out, after = (torch.zeros(n, k, device="cuda") for k in (d, d, V, V))
    api.ss_logits_noalloc(h, gain, head, 1e-6, out)                      # the first call on a device, outside of a capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        h.copy_(src)
        api.ss_logits_noalloc(h, gain, head, 1e-6, out)
        after.copy_(out)
        api.ss_logits_noalloc(h, gain, head, 1e-6, out)
    rt = ctypes.CDLL("libcudart.so.12")
    nodes, edges = ctypes.c_size_t(0), ctypes.c_size_t(0)
    raw = ctypes.c_void_p(graph.raw_cuda_graph())
    assert rt.cudaGraphGetNodes(raw, None, ctypes.byref(nodes)) == 0 and nodes.value >= 8
    frm, to = ((ctypes.c_void_p * 64)() for _ in range(2))
    edges.value = 64
    assert rt.cudaGraphGetEdges(raw, frm, to, ctypes.byref(edges)) == 0
    assert edges.value == nodes.value - 1                                 # a chain
    graph.instantiate()
    for seed in range(3):
        src.normal_(0.0, 2.0, generator=gen)
        want = torch.zeros(n, V, device="cuda")
        api.ss_logits_noalloc(src, gain, head, 1e-6, want)
        out.zero_(), after.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert want.abs().max() > 0 and torch.equal(out, want) and torch.equal(after, want)
