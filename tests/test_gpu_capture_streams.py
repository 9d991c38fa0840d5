"""While a stream capture that one call of a context takes part in is open, other batch calls of
the same context on another stream, with workspaces of their own, run as always: the context's
second stream, which the captured call took into the capture, is left out."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["forward", "emission", "gradient", "jacobian"])
def test_a_call_beside_an_open_capture(call):
    import torch
    from paper_1912_07759_gb300 import synthetic as S
    from paper_1912_07759_gb300 import transit as T
    ctx = T.TransitContext(0)
    tables = T.XsecTables(ctx, S.make_tables(1, 2, 4, 5, 3000, with_cia=False))
    bins = T.Bins(ctx, tables, *S.bins_logspaced(10))
    spec_h = S.batch_spec(2)
    spec = T.BatchSpec(spec_h, max_layers=40)
    B = 5
    th = torch.tensor(S.draw_theta(3, B, spec_h), device="cuda")
    gbin = torch.ones(B, bins.n_bin, dtype=torch.float64, device="cuda")

    def space():
        n = T.batch_workspace_size(ctx, tables, spec, bins, B, with_adjoint=True)
        return torch.empty(n, dtype=torch.uint8, device="cuda")
    ws_a, ws_b = space(), space()

    def beside():
        if call == "forward":
            out = T.forward_transit_batch(ctx, tables, spec, th, None, bins, workspace=ws_b)[0]
        elif call == "emission":
            out = T.forward_emission_batch(ctx, tables, spec, th, None, bins, workspace=ws_b)[0]
        elif call == "gradient":
            out = T.adjoint_transit(ctx, tables, spec, th, None, bins, gbin=gbin, workspace=ws_b)[1]
        else:
            out = T.adjoint_transit(ctx, tables, spec, th, None, bins, want_grad=False,
                                    want_jac=True, workspace=ws_b)[4]
        return out.clone()
    want = beside()
    binned, _ = T.forward_transit_batch(ctx, tables, spec, th, None, bins, workspace=ws_a)
    torch.cuda.synchronize()
    captured = torch.zeros_like(binned)
    status = torch.zeros(B, dtype=torch.int32, device="cuda")
    other = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="relaxed"):
        T.forward_transit_batch(ctx, tables, spec, th, None, bins, workspace=ws_a,
                                out_binned=captured, out_status=status)
        with torch.cuda.stream(other):
            got = beside()
        T.forward_transit_batch(ctx, tables, spec, th, None, bins, workspace=ws_a,
                                out_binned=captured, out_status=status)   # in the capture again
    other.synchronize()
    assert torch.equal(got, want)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(captured, binned)
    assert torch.equal(beside(), want)                       # and with the second stream again
    ctx.sync_status()
