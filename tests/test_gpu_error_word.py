"""The error word that operator calls read from pinned host memory: a bounded wait that runs out
is reported by the allocating and the allocation-free entry point alike, by each for its own
call only, and the next call on the context succeeds."""
import pytest

from paper_1101_0423_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", ["dev", "static"])
@pytest.mark.parametrize("opname", ["DEO", "C", "CCDAG"])
def test_timeout_is_reported_by_the_call_that_met_it(gpu_lib, first, opname):
    import torch
    dwf, dims, ns = gpu_lib, (4, 2, 4, 4), 6
    om, sg = inputs.weights("cosine", ns)
    x = torch.from_numpy(inputs.gaussian_source(dims, ns, seed=71)).cuda()
    op = getattr(dwf, "OP_" + opname)
    with dwf.Context(dims, ns, 1.8, 0.05, om, sg, inputs.gauge_field(dims, 0.5, seed=70)) as ctx:
        def call(which):
            out = torch.full_like(x, float("nan"))
            f = dwf.dwf_apply_eo_dev if which == "dev" else dwf.dwf_apply_eo_dev_static
            f(ctx.h, op, dwf.PREC_F32, 1, x, out, stream=torch.cuda.current_stream())
            return out
        want = call("dev")
        dwf.dwf_debug_set_wait(ctx.h, 1024, skip_copies=True)
        try:
            with pytest.raises(dwf.DwfError) as e:
                call(first)
            assert e.value.status == dwf.DWF_ETIMEOUT
        finally:
            dwf.dwf_debug_set_wait(ctx.h, 0, skip_copies=False)
        for which in ("static", "dev"):
            assert torch.equal(call(which), want)
