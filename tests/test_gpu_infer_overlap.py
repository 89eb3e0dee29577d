"""Inference calls and training steps launched back to back, each kernel set up
under the one before it, give the bits of the same calls with the device idle
between them: several chunks a call, inputs and outputs used again by the next
call, the low-confidence tests on, weights that change between the calls; and
the same inference calls replayed from a graph."""
import pytest

pytestmark = pytest.mark.gpu


def _model(ctx, x, y, width, layers):
    from paper_2312_04830_gb300 import binding
    sg = binding.Surrogate(ctx, width=width, hidden_layers=layers, max_batch=1024, infer_chunk=1024, seed=11)
    sg.fit_normalization(x, y)
    sg.set_confidence(0.2)
    sg.set_transport_confidence(0.2)
    return sg


@pytest.mark.parametrize("kind", ["resident", False])
@pytest.mark.parametrize("width,layers", [(256, 3), (512, 2)])
def test_back_to_back_equals_one_by_one(prlib, cuda, species, width, layers, kind):
    import torch
    from paper_2312_04830_gb300 import binding, workloads as W
    ctx = binding.PropertyContext(species)
    T, p, Y = W.training_states(4096, seed=2)
    d = lambda a: torch.as_tensor(a, device=cuda).float().contiguous()
    x = torch.cat([d(T)[None], d(p)[None], d(Y)])
    y = ctx.props(x[0].contiguous(), x[1].contiguous(), x[2:].contiguous(), "fp32")[0]
    n = 3000   # three chunks, the last one ragged
    parts = [(x[0, k:k + n].contiguous(), x[1, k:k + n].contiguous(), x[2:, k:k + n].contiguous()) for k in (0, 500, 1096)]

    def run(idle):
        sg = _model(ctx, x, y, width, layers)
        sg.set_fused_infer(kind)
        loss = torch.zeros(8, device=cuda)
        out, fb = torch.empty((6, n), device=cuda), torch.empty(n, dtype=torch.uint8, device=cuda)
        a, got = [t.clone() for t in parts[0]], []
        for k in range(8):
            for dst, src in zip(a, parts[k % 3]):
                dst.copy_(src)
            if idle:
                torch.cuda.synchronize()
            sg.infer(*a, out=out, used_fallback=fb)
            if idle:
                torch.cuda.synchronize()
            got += [out.clone(), fb.clone()]
            sg.train_step(x, y, 1024, 1e-3, sample_seed=k + 1, loss_out=loss[k:])
            if idle:
                torch.cuda.synchronize()
        sg.sync_status()
        w = torch.as_tensor(sg.get_params())
        return sg, got + [loss], w
    sg, busy, w1 = run(False)
    s2, idle, w2 = run(True)
    assert torch.equal(w1, w2)
    for k, (u, v) in enumerate(zip(busy, idle)):
        assert torch.equal(u.view(torch.int32) if u.dtype == torch.float32 else u,
                           v.view(torch.int32) if v.dtype == torch.float32 else v), k
    # a graph of two calls
    st = torch.cuda.Stream()
    outs = [torch.empty((6, n), device=cuda) for _ in range(2)]
    fbs = [torch.empty(n, dtype=torch.uint8, device=cuda) for _ in range(2)]
    with torch.cuda.stream(st):
        sg.infer(*parts[1], out=outs[0], used_fallback=fbs[0], stream=st)
        st.synchronize()
        ref = [(o.clone(), f.clone()) for o, f in [sg.infer(*parts[k], stream=st) for k in (1, 2)]]
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            for k in (0, 1):
                sg.infer(*parts[k + 1], out=outs[k], used_fallback=fbs[k], stream=st)
        for o in outs:
            o.zero_()
        for _ in range(3):
            graph.replay()
    torch.cuda.synchronize()
    for (o, f), u, v in zip(ref, outs, fbs):
        assert torch.equal(o.view(torch.int32), u.view(torch.int32)) and torch.equal(f, v)
    sg.sync_status()
    sg.close()
    s2.close()
    ctx.close()
