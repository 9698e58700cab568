"""The time-out path of the decode kernel, exercised without hanging or faulting anything: the workspace is
told to treat the intermediate vector that the CTAs exchange between the two phases as never complete,
and that no device-side wait may last longer than about a millisecond.  The kernel has to return by itself,
report SLICEMOE_STATUS_WAIT_TIMEOUT, and the same workspace has to work again once it is re-initialised."""
import time

import numpy as np
import pytest

from oracle import moe
from paper_2512_12990_b200 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


def test_wait_timeout_is_reported_and_the_workspace_recovers():
    import torch
    from paper_2512_12990_b200 import binding as B
    sh = synth.SHAPES["tiny"]
    layer = H.Layer(sh, range(sh.n_experts))
    logits = synth.router_logits_normal(sh.seed, ("timeout-logits",), 1, sh.n_experts)
    ids, w, _ = moe.route_topk(logits, sh.top_k)
    prec = (ids >= 4).astype(np.uint8)
    xbits, x64 = H.x_inputs(sh, 1, "timeout-x")
    x = H.to_dev_bf16(xbits)
    args = (torch.from_numpy(ids.astype(np.int32)).cuda(), torch.from_numpy(prec).cuda(),
            torch.from_numpy(w.astype(np.float32)).cuda())
    y_ref = moe.expert_ffn(x64, layer.oracle_list(), ids, prec, w)

    # a normal call first
    y = B.slicemoe_expert_ffn(layer.cshape, layer.experts_tbl, x, *args, layer.ws)
    torch.cuda.synchronize()
    assert B.slicemoe_get_status(layer.ws) == 0
    H.assert_close(y.cpu().numpy(), y_ref, "before the time-out")

    # one arrival that never comes, and a limit of 2 million cycles (about a millisecond)
    B.slicemoe_workspace_set_wait(layer.ws, 2_000_000, extra_arrivals=1)
    y_bad = torch.full((1, sh.hidden), 7.0, dtype=torch.float32, device="cuda")
    t0 = time.time()
    B.slicemoe_expert_ffn(layer.cshape, layer.experts_tbl, x, *args, layer.ws, y=y_bad)
    torch.cuda.synchronize()
    assert time.time() - t0 < 5.0, "the kernel must return by itself"
    status = B.slicemoe_get_status(layer.ws)
    assert status & B.STATUS_WAIT_TIMEOUT
    assert torch.all(y_bad == 7.0), "the output is not written when h was never complete"

    # re-initialised, the workspace works again (and the limit is back to its default)
    B.lib().slicemoe_workspace_init(layer.ws.data_ptr(), layer.ws.numel(), None)
    y2 = B.slicemoe_expert_ffn(layer.cshape, layer.experts_tbl, x, *args, layer.ws)
    torch.cuda.synchronize()
    assert B.slicemoe_get_status(layer.ws) == 0
    assert torch.equal(y2, y), "same bits as before the time-out"


@pytest.mark.parametrize("T,limit", [(4, 2_000_000), (17, 200_000)])
def test_wait_timeout_of_several_tokens(T, limit):
    """The same for the kernels that take several tokens at once, in one pass and in two: their waits for the weights run
    out, y stays as it was, and the workspace works again.  (200,000 cycles: less than what the producers give copies on
    their way, which is a floor of their own.)"""
    import torch
    from paper_2512_12990_b200 import binding as B
    sh = synth.Shape("batch-timeout", 512, 384, 12, 3, 64, n_shared=1, shared_inter=256, n_layers=1, seed=7300)
    layer = H.Layer(sh, range(sh.n_experts))
    rng = np.random.default_rng(T)
    ids = np.stack([rng.permutation(sh.n_experts)[:sh.top_k] for _ in range(T)]).astype(np.int32)
    lists = [torch.from_numpy(a).cuda() for a in (ids, rng.integers(0, 2, ids.shape).astype(np.uint8), rng.random(ids.shape).astype(np.float32))]
    x = H.to_dev_bf16(H.x_inputs(sh, T, "batch-timeout-x")[0])

    def call(y=None):
        y = B.slicemoe_layer(layer.cshape, layer.experts_tbl, layer.shared_tbl, None, x, *lists, layer.ws, y=y)
        torch.cuda.synchronize()
        return y

    y = call()
    assert B.slicemoe_get_status(layer.ws) == 0
    B.slicemoe_workspace_set_wait(layer.ws, limit, extra_arrivals=1)
    y_bad = torch.full((T, sh.hidden), 7.0, device="cuda")
    t0 = time.time()
    call(y_bad)
    assert time.time() - t0 < 5.0, "the kernels must return by themselves"
    assert B.slicemoe_get_status(layer.ws) == B.STATUS_WAIT_TIMEOUT
    assert torch.all(y_bad == 7.0)
    B.lib().slicemoe_workspace_init(layer.ws.data_ptr(), layer.ws.numel(), None)
    assert torch.equal(call(), y) and B.slicemoe_get_status(layer.ws) == 0


def test_a_short_limit_is_not_spent_on_the_launch_before():
    """The down projection of several tokens starts while gate/up still runs.  Its waits are counted from the end of that
    launch: a limit of 40,000 cycles, 20 us, lets a pass through whose gate/up alone takes longer."""
    import torch
    from paper_2512_12990_b200 import binding as B
    E, k, T, h, inter = 16, 4, 16, 4096, 1408
    g = torch.Generator(device="cuda").manual_seed(5)
    pack = lambda n, c: B.slicemoe_pack(torch.randn((n, c), generator=g, device="cuda").mul_(0.02), 32)
    experts = [dict(gate=pack(inter, h), up=pack(inter, h), down=pack(h, inter)) for _ in range(E)]
    table, shape = B.expert_table(experts), B.make_shape(h, inter, E, k, 32)
    ws = B.new_workspace(shape)
    ids = torch.stack([torch.randperm(E, generator=g, device="cuda")[:k] for _ in range(T)]).to(torch.int32)
    prec = torch.randint(0, 2, (T, k), generator=g, device="cuda").to(torch.uint8)
    w, x = torch.rand((T, k), generator=g, device="cuda"), torch.randn((T, h), generator=g, device="cuda").bfloat16()
    want = B.slicemoe_layer(shape, table, None, None, x, ids, prec, w, ws)
    B.slicemoe_workspace_set_wait(ws, 40_000)
    for _ in range(20):
        assert torch.equal(B.slicemoe_layer(shape, table, None, None, x, ids, prec, w, ws), want)
    assert B.slicemoe_get_status(ws) == 0
