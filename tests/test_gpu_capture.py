"""Calls captured by a caller into a CUDA graph of their own, where the kernels'
programmatic launches become programmatic edges between graph nodes: with
copies, a fill and a second stream among them, replayed on changing inputs,
the graph gives what the same calls give one by one."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DEV = "cuda"


@pytest.fixture(scope="module")
def acid():
    import __graft_entry__ as g

    g.build()
    from paper_2607_12358_gb300 import acid as a

    return a


@pytest.mark.parametrize("dtype,rows,d,heads", [(torch.bfloat16, 1500, 1920, 15), (torch.bfloat16, 700, 1920, 30),
                                                (torch.float32, 200, 576, 9)])
def test_captured_calls_equal_eager_calls(acid, dtype, rows, d, heads):
    g = torch.Generator(device=DEV).manual_seed(7)
    rand = lambda *s, dt=dtype: torch.randn(*s, device=DEV, generator=g).to(dt)  # noqa: E731
    x, prev, w, wo = rand(rows, d), rand(rows, d), 0.05 * rand(3 * d, d), 0.05 * rand(d, d)
    sh, sc, gate, b = (rand(d, dt=torch.float32) for _ in range(4))
    ws = torch.empty(acid.attention_workspace_size(d // heads), dtype=torch.uint8, device=DEV)
    dws = torch.empty(acid.drift_workspace_size(rows * d), dtype=torch.uint8, device=DEV)
    y, qkv, att, out = (torch.empty(rows, n, device=DEV, dtype=dtype) for n in (d, 3 * d, d, d))
    side = torch.empty(rows, d, device=DEV, dtype=dtype)
    rel = torch.empty(2, dtype=torch.float64, device=DEV)
    other = torch.cuda.Stream()

    def calls():
        acid.acid_layernorm_mod(x, sh, sc, out=y, out_dtype=dtype)
        fork = torch.cuda.Event()
        fork.record()
        other.wait_event(fork)
        with torch.cuda.stream(other):
            acid.acid_cache_apply(y, prev, out=side)
        acid.acid_linear_forward(y, w, None, out=qkv)
        acid.acid_attention_forward(qkv[:, :d], qkv[:, d:2 * d], qkv[:, 2 * d:], heads, out=att, workspace=ws)
        out.copy_(x)
        acid.acid_linear_forward(att, wo, b, "gated_res", gate=gate, residual=out, out=out)
        join = torch.cuda.Event()
        join.record(other)
        torch.cuda.current_stream().wait_event(join)
        rel.zero_()
        acid.acid_drift_signal(side, out, out_rel=rel[:1], workspace=dws)

    calls()  # sets the kernels up
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls()
    for seed in (1, 2, 3):
        x.copy_(torch.randn(rows, d, device=DEV, generator=g))
        calls()
        torch.cuda.synchronize()
        want = [t.clone() for t in (y, side, qkv, att, out, rel)]
        for t in (y, side, qkv, att, out, rel):
            t.fill_(float("nan"))
        graph.replay()
        graph.replay()  # a replay right behind another
        torch.cuda.synchronize()
        acid.check_device_error()
        for got, ref in zip((y, side, qkv, att, out, rel), want):
            assert torch.isfinite(ref.double()).all() and torch.equal(got, ref)
