"""How the batch-1 decode kernel deals its gate/up tasks (16 rows of a slot) to the CTAs: both-slice tasks one by one, then two
MSB-only ones to each CTA that got one less, then the rest.  Shapes at the edges of that rule on a device of 148 SMs, against
the float64 oracle; and down projections whose chunks go several times round the ring."""
import numpy as np
import pytest

from oracle import moe
from paper_2512_12990_b200 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu

CASES = [
    # hidden, inter, top_k, both-slice entries, group, shared inter
    (256, 4736, 2, 1, 128, 0),      # 296 both-slice tasks: every CTA has two, nobody is short; 296 MSB-only ones
    (256, 4736, 2, 1, 128, 128),    # 304: 140 CTAs are short of one; more MSB-only tasks than their two each
    (128, 1280, 2, 1, 64, 0),       # 80 and 80: 68 CTAs are short, and get one or two
    (128, 128, 2, 1, 32, 0),        # 8 and 8: most CTAs have nothing to do
    (128, 128, 1, 0, 128, 0),       # MSB-only tasks alone
    (256, 1280, 8, 2, 128, 0),      # one or two both-slice tasks and many MSB-only ones: an odd number of the former
    (256, 1280, 8, 8, 64, 128),     # both-slice tasks alone
    (4096, 1152, 8, 5, 32, 2176),   # 17 units of down tiles a row block, 34 for the CTAs with two, in a ring of 8
    (2304, 2176, 4, 2, 128, 2176),  # two chunks to a slot, the second one block wide
]


@pytest.mark.parametrize("hidden,inter,k,n_both,group,shared_inter", CASES)
def test_task_dealing_and_ring_laps(hidden, inter, k, n_both, group, shared_inter):
    import torch
    from paper_2512_12990_b200 import binding as B
    sh = synth.Shape("deal", hidden, inter, k + 1, k, group, n_shared=1 if shared_inter else 0, shared_inter=shared_inter, seed=9100 + inter + k)
    layer = H.Layer(sh, range(sh.n_experts))
    ids = np.array([np.random.default_rng(k).permutation(sh.n_experts)[:k]], dtype=np.int32)
    prec = (np.arange(k) < n_both).astype(np.uint8)[None, ::-1].copy()
    w = np.linspace(0.4, 0.1, k)[None]
    xbits, x64 = H.x_inputs(sh, 1)
    want = moe.layer(x64, layer.oracle_list(), ids, prec, w, shared=layer.oracle_shared)
    args = (H.to_dev_bf16(xbits), torch.from_numpy(ids).cuda(), torch.from_numpy(prec).cuda(), torch.from_numpy(w.astype(np.float32)).cuda(), layer.ws)
    y = [B.slicemoe_layer(layer.cshape, layer.experts_tbl, layer.shared_tbl, None, *args) for _ in range(4)]
    torch.cuda.synchronize()
    assert B.slicemoe_get_status(layer.ws) == 0
    H.assert_close(y[0].cpu().numpy(), want, f"{hidden} x {inter}, {n_both} of {k} from both slices")
    assert all(torch.equal(y[0], v) for v in y[1:])


@pytest.mark.parametrize("hidden,inter,k,n_both,group,shared_inter", [
    (2048, 2048, 3, 1, 128, 0),     # 68 CTAs with a group that has a gate/up task and no chunk of the first output rows
    (2560, 2048, 1, 0, 128, 4096),  # 40
    (2048, 1024, 2, 1, 64, 0),
])
def test_rows_between_the_phases(hidden, inter, k, n_both, group, shared_inter):
    """A group's rows of partial sums belong to gate/up until the epilogue has taken them: also where the group has nothing to wait
    for in the down projection.  Many launches back to back and with another kernel between them, all of one result."""
    import torch
    from paper_2512_12990_b200 import binding as B
    sh = synth.Shape("rows", hidden, inter, k + 1, k, group, n_shared=1 if shared_inter else 0, shared_inter=shared_inter, seed=9300 + inter + k)
    layer = H.Layer(sh, range(sh.n_experts))
    ids = np.arange(k, dtype=np.int32)[None]
    prec = (np.arange(k) < n_both).astype(np.uint8)[None]
    w = np.linspace(0.4, 0.1, k)[None]
    xbits, x64 = H.x_inputs(sh, 1)
    want = moe.layer(x64, layer.oracle_list(), ids, prec, w, shared=layer.oracle_shared)
    args = (H.to_dev_bf16(xbits), torch.from_numpy(ids).cuda(), torch.from_numpy(prec).cuda(), torch.from_numpy(w.astype(np.float32)).cuda(), layer.ws)
    y = torch.empty((400, 1, hidden), device="cuda")
    other = torch.zeros(1 << 20, device="cuda")
    for i in range(400):
        B.slicemoe_layer(layer.cshape, layer.experts_tbl, layer.shared_tbl, None, *args, y=y[i])
        if i % 3 == 2:
            other.add_(1.0)
    torch.cuda.synchronize()
    assert B.slicemoe_get_status(layer.ws) == 0
    H.assert_close(y[0].cpu().numpy(), want, f"{hidden} x {inter}")
    assert torch.equal(y, y[:1].expand_as(y))


@pytest.mark.parametrize("hidden,inter,k,n_both,group,shared_inter", [
    (2048, 2048, 3, 1, 128, 0),
    (2560, 2048, 1, 0, 128, 4096),
    (4096, 1152, 8, 5, 32, 2176),
    (256, 1280, 8, 2, 64, 128),
])
def test_the_same_tasks_by_every_way_to_the_list(hidden, inter, k, n_both, group, shared_inter):
    """The list read behind the wait, ahead of it (resident), or worked out in the kernel: one plan, the same bits.  And lists of
    which some or all entries name no expert, for which the plan and the ring of the down projection are cut anew."""
    import torch
    from paper_2512_12990_b200 import binding as B
    n_shared = 1 if shared_inter else 0
    sh = synth.Shape("ways", hidden, inter, k + 2, k, group, n_shared=n_shared, shared_inter=shared_inter, seed=9500 + inter + k)
    layer = H.Layer(sh, range(sh.n_experts))
    xbits, x64 = H.x_inputs(sh, 1)
    x = H.to_dev_bf16(xbits)
    logits = torch.from_numpy(np.random.default_rng(k).standard_normal((1, k + 2)).astype(np.float32)).cuda()
    tables = (layer.cshape, layer.experts_tbl, layer.shared_tbl, None, x)
    for _ in range(20):
        routed, ids, prec, w = B.slicemoe_layer_routed(*tables, logits, layer.ws, rank_high=n_both)
        assert prec.sum() == n_both
        plain = B.slicemoe_layer(*tables, ids, prec, w, layer.ws)
        torch.cuda.synchronize()  # the lists are complete before what precedes the next call begins
        resident = [B.slicemoe_layer(*tables, ids, prec, w, layer.ws, flags=B.LISTS_RESIDENT) for _ in range(4)]
        assert torch.equal(plain, routed) and all(torch.equal(plain, r) for r in resident)
    assert B.slicemoe_get_status(layer.ws) == 0
    n_ids, n_prec, n_w = ids.cpu().numpy(), prec.cpu().numpy(), w.cpu().numpy().astype(np.float64)
    for dropped in {(0,), (k - 1,), tuple(range(k))}:
        kept = [j for j in range(k) if j not in dropped]
        some = ids.clone()
        some[:, list(dropped)] = torch.tensor([-1, k + 2] * k, dtype=torch.int32, device="cuda")[:len(dropped)]
        torch.cuda.synchronize()
        y = [B.slicemoe_layer(*tables, some, prec, w, layer.ws, flags=f) for f in (0, B.LISTS_RESIDENT) for _ in range(3)]
        assert B.slicemoe_get_status(layer.ws) == 1
        if kept:
            want = moe.layer(x64, layer.oracle_list(), n_ids[:, kept], n_prec[:, kept], n_w[:, kept], shared=layer.oracle_shared)
        else:
            want = sum((moe.expert_ffn_one(x64[0], e, 1) for e in layer.oracle_shared), np.zeros(hidden))[None]
        if np.any(want):
            H.assert_close(y[0].cpu().numpy(), want, f"without entries {dropped}")
        else:
            assert not y[0].any()
        assert all(torch.equal(y[0], v) for v in y[1:])
