"""The kernels of a call overlap (programmatic dependent launch): a kernel sets up, and starts to load its weights, while the one before it is finishing.  Whatever the caller enqueued
before the call, on the same stream, has to be finished before any of that: here weights, activations, states and the workspace are rewritten by kernels right before the call, with
nothing in between, and the results have to be those of a call with the stream idle, bit for bit -- eagerly, two calls in a row, and replayed from a captured graph.  The workspace is
filled with NaN each time: a kernel that reads another one's output too early finds those."""
import numpy as np
import pytest
import torch

from paper_2511_15927_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2511_15927_b200 import build
    build.build()
    import tests.gpu_util as g
    return g


def _tensors(o):
    if isinstance(o, torch.Tensor):
        return [o]
    if isinstance(o, dict):
        o = list(o.values())
    return [t for v in o for t in _tensors(v)] if isinstance(o, (list, tuple)) else []


def _mixer(G, dtype, shape, state=False, flags=None, chunk=0):
    from paper_2511_15927_b200 import binding as dm
    cfg = G.cfg_of(shape, dtype, dm.DM_FLAGS_DEFAULT if flags is None else flags, chunk=chunk)
    wf, wr = I.make_mixer_weights(shape, 5, dtype, perturb=True)
    dw = [G.dev_dir_weights(wf, dtype), G.dev_dir_weights(wr, dtype)]
    x = G.dev(I.make_activations(shape, 5, dtype), dtype)
    y = torch.empty_like(x)
    ws = G.workspace(dm.dm_bimamba_workspace_bytes(cfg))
    cw = tuple(dm.make_dir_weights(w) for w in dw)
    if not state:
        return (lambda st: dm.dm_bimamba_forward(cfg, cw, x.data_ptr(), y.data_ptr(), ws.data_ptr(), ws.numel(), st)), _tensors([dw, x]), [y], ws
    s, c = I.make_states(shape, 5, dtype)
    s, c = G.dev(s.astype(np.float32)), G.dev(c, dtype)
    so, co = torch.empty_like(s), torch.empty_like(c)
    return (lambda st: dm.dm_bimamba_block_step(cfg, cw, x.data_ptr(), s.data_ptr(), c.data_ptr(), so.data_ptr(), co.data_ptr(), y.data_ptr(), ws.data_ptr(), ws.numel(), st)), \
        _tensors([dw, x, s, c]), [y, so, co], ws


def _stack(G, kind, shape, layers=3, V=304):
    from paper_2511_15927_b200 import binding as dm
    dtype, B, L, d = I.BF16, shape.batch, shape.seqlen, shape.d_model
    sw = I.make_stack_weights(shape, layers, V, seed=6, dtype=dtype, perturb=True)
    keep = [G.dev_stack_weights(sw, dtype)]
    csw, arr = dm.make_stack_weights(keep[0])
    scfg = dm.dm_stack_cfg(G.cfg_of(shape, dtype), layers, V, 1e-5)
    tok = G.dev(I.make_tokens(B, L, V - 8, V - 8, seed=6).astype(np.int32))
    logits, out = torch.empty(B, L, V, device="cuda", dtype=torch.bfloat16), torch.empty_like(tok)
    if kind == "cond":
        I.add_block_weights(sw, shape, 2 * d, 32, seed=6, dtype=dtype)
        keep += [G.dev_block_weights(sw, dtype), G.dev(np.asarray(I.make_timestep_embedding(B, 32, seed=6), np.float32))]
        cbw, blk = dm.make_block_weights(keep[1]), dm.dm_block_cfg(2 * d, 32, 1e-5)
        ws = G.workspace(dm.dm_denoise_cond_workspace_bytes(scfg, blk))
        call = lambda st: dm.dm_denoise_step_cond(scfg, blk, csw, cbw, tok.data_ptr(), keep[2].data_ptr(), logits.data_ptr(), out.data_ptr(), None, ws.data_ptr(), ws.numel(), st)
    elif kind == "sample":
        r = np.random.default_rng(6)
        keep += [G.dev(r.random((B, L), dtype=np.float32)), G.dev(r.random((B, L), dtype=np.float32))]
        ws = G.workspace(dm.dm_denoise_sample_workspace_bytes(scfg))
        smp = dm.dm_sample_cfg(V - 8, V - 7, 0.5)
        call = lambda st: dm.dm_denoise_sample_step(scfg, None, csw, None, tok.data_ptr(), 0, smp, keep[1].data_ptr(), keep[2].data_ptr(), out.data_ptr(), None, ws.data_ptr(), ws.numel(), st)
        return (lambda st: (arr, call(st))), _tensors([keep, tok]), [out], ws
    elif kind == "hybrid_block":
        prefix, heads = 100, d // 64
        keep += [[{"w_qkv": torch.randn(3 * d, d, device="cuda").mul_(d ** -0.5).bfloat16(), "w_o": torch.randn(d, d, device="cuda").mul_(d ** -0.5).bfloat16()} if i % 2 == 0 else None
                  for i in range(layers)],
                 [torch.randn(layers, B, prefix + L, d, device="cuda").bfloat16() for _ in range(2)],
                 [torch.randn(layers, B, shape.n_heads, shape.headdim, shape.d_state, device="cuda").mul_(0.5), torch.randn(layers, B, shape.d_conv - 1, shape.conv_ch, device="cuda").bfloat16()]]
        caw = dm.make_attn_weights(keep[1])
        (kc, vc), (s, c) = keep[2], keep[3]
        so, co = torch.empty_like(s), torch.empty_like(c)
        states, ast = (dm.dm_layer_state * layers)(), (dm.dm_attn_state * layers)()
        for i in range(layers):
            states[i] = dm.dm_layer_state(s[i].data_ptr(), c[i].data_ptr(), so[i].data_ptr(), co[i].data_ptr())
            ast[i] = dm.dm_attn_state(kc[i].data_ptr(), vc[i].data_ptr(), prefix, prefix + L)
        ws = G.workspace(dm.dm_denoise_hybrid_workspace_bytes(scfg))
        call = lambda st: dm.dm_denoise_step_hybrid_block(scfg, None, dm.dm_hybrid_cfg(2, heads), csw, None, caw, tok.data_ptr(), 0, logits.data_ptr(), out.data_ptr(), states, ast,
                                                          ws.data_ptr(), ws.numel(), st)
        return (lambda st: (arr, call(st))), _tensors([keep, tok]), [logits, out, so[1], co[1]], ws
    else:
        ws = G.workspace(dm.dm_denoise_workspace_bytes(scfg))
        call = lambda st: dm.dm_denoise_step(scfg, csw, tok.data_ptr(), logits.data_ptr(), out.data_ptr(), None, ws.data_ptr(), ws.numel(), st)
    return (lambda st: (arr, call(st))), _tensors([keep, tok]), [logits, out], ws


CASES = {
    "mixer_long": lambda G: _mixer(G, I.BF16, I.MixerShape(1, 4100, 128, 2, 128, 4, 4)),               # prep partly inside the scan launch
    "mixer_1k_pairs": lambda G: _mixer(G, I.BF16, I.MixerShape(2, 700, 512, 2, 128, 4, 32)),
    "mixer_chunk32": lambda G: _mixer(G, I.BF16, I.MixerShape(1, 2100, 128, 2, 16, 4, 4), chunk=32),
    "mixer_narrow": lambda G: _mixer(G, I.BF16, I.MixerShape(2, 300, 256, 2, 16, 4, 8), state=True),       # d_state 16: chains of half heads, whole ones, two to an SM
    "mixer_narrow_whole": lambda G: _mixer(G, I.BF16, I.MixerShape(5, 300, 256, 2, 16, 4, 8), state=True),
    "mixer_narrow_two": lambda G: _mixer(G, I.BF16, I.MixerShape(10, 300, 256, 2, 16, 4, 8)),
    "mixer_tied": lambda G: _mixer(G, I.BF16, I.MixerShape(2, 200, 256, 2, 64, 4, 8), flags=15),
    "mixer_f32": lambda G: _mixer(G, I.F32, I.MixerShape(2, 300, 128, 2, 16, 4, 8), state=True),
    "block_32": lambda G: _mixer(G, I.BF16, I.MixerShape(4, 32, 512, 2, 128, 4, 16), state=True),
    "block_48": lambda G: _mixer(G, I.BF16, I.MixerShape(4, 48, 256, 2, 128, 4, 16), state=True),
    "stack": lambda G: _stack(G, "plain", I.MixerShape(2, 150, 256, 2, 32, 4, 8)),
    "stack_narrow": lambda G: _stack(G, "plain", I.MixerShape(2, 150, 256, 2, 16, 4, 8)),
    "stack_few_rows": lambda G: _stack(G, "plain", I.MixerShape(1, 100, 256, 2, 32, 4, 8), V=38016),     # the vocabulary's tiles taken in turn
    "stack_cond": lambda G: _stack(G, "cond", I.MixerShape(2, 150, 256, 2, 32, 4, 8)),
    "hybrid_block": lambda G: _stack(G, "hybrid_block", I.MixerShape(3, 32, 256, 2, 64, 4, 8)),
    "sample": lambda G: _stack(G, "sample", I.MixerShape(2, 100, 256, 2, 32, 4, 8)),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_calls_follow_what_the_stream_holds(G, name):
    from paper_2511_15927_b200 import binding as dm
    torch.manual_seed(7)
    call, inputs, outputs, ws = CASES[name](G)
    kept = [t.clone() for t in inputs]
    current = lambda: torch.cuda.current_stream().cuda_stream

    def spoil():
        for t in inputs:
            t.fill_(float("nan") if t.is_floating_point() else 0)
        for t in outputs:
            t.fill_(float("nan") if t.is_floating_point() else -7)
        ws.fill_(0xFF)                                          # every float in it is NaN

    def restore():
        for t, k in zip(inputs, kept):
            t.copy_(k)

    def take():
        torch.cuda.synchronize()
        dm.dm_check(current())
        return [t.clone() for t in outputs]

    ws.fill_(0xFF)
    torch.cuda.synchronize()
    call(current())
    want = take()
    assert all(not torch.isnan(t).any() for t in want if t.is_floating_point())
    same = lambda got: all(torch.equal(a, b) for a, b in zip(got, want))
    for _ in range(3):                                          # everything is written right before the call
        spoil()
        torch.cuda.synchronize()
        torch.cuda._sleep(200000)                               # the copies and the call wait in the stream together
        restore()
        call(current())
        assert same(take())
    # spoiled right behind the first call, restored right before the second: neither sees the other's inputs
    spoil()
    restore()
    call(current())
    first = [t.clone() for t in outputs]
    spoil()
    restore()
    call(current())
    assert same(take()) and same(first)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(current())
    for _ in range(2):
        spoil()
        torch.cuda._sleep(200000)
        restore()
        graph.replay()
        assert same(take())
