"""Several tokens through slicemoe_layer and slicemoe_layer_routed in one pass of the batch kernels, against the float64 oracle,
at the sizes where their split can go wrong: the fewest tokens that take them, runs of exactly, less and more than eight
pairs of an expert, one token more than a pass holds, each group size, several chunks of the down projection.  Tolerance
as for one token."""
import numpy as np
import pytest

from oracle import moe
from paper_2512_12990_b200 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,hidden,inter,group,n_shared,shared_inter,gated,bits", [
    (4, 128, 128, 32, 0, 0, False, (8, 4)),       # the smallest layer, the fewest tokens
    (8, 384, 640, 64, 2, 128, False, (8, 4)),     # runs of exactly eight for the shared experts
    (9, 256, 2176, 128, 1, 256, True, (8, 4)),    # one more than a run holds; two chunks of the down projection
    (16, 2176, 128, 128, 1, 2304, True, (6, 3)),  # a whole pass; the shared expert wider than the routed ones
    (17, 256, 256, 32, 0, 0, False, (4, 2)),      # a pass and one token
])
def test_batches_against_the_oracle(T, hidden, inter, group, n_shared, shared_inter, gated, bits):
    import torch
    from paper_2512_12990_b200 import binding as B
    E, k = 6, 3
    sh = synth.Shape("batch", hidden, inter, E, k, group, n_shared=n_shared, shared_inter=shared_inter,
                     shared_sigmoid_gate=gated, n_layers=1, seed=7000 + T)
    L = H.Layer(sh, range(E), b_high=bits[0], b_low=bits[1])
    rng = np.random.default_rng(T)
    ids = np.stack([rng.permutation(E)[:k] for _ in range(T)]).astype(np.int32)
    ids[:, 0] = np.where(ids[:, 1:].min(axis=1) > 0, 0, ids[:, 0])  # expert 0 has many pairs
    ids[1] = [4, 4, 2]                                              # an expert twice in a token
    prec = rng.integers(0, 2, (T, k)).astype(np.uint8)
    w = rng.random((T, k)).astype(np.float32)
    xbits, x64 = H.x_inputs(sh, T, "batch-x")
    x = H.to_dev_bf16(xbits)

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()

    def layer(ids_, ws):
        y = B.slicemoe_layer(L.cshape, L.experts_tbl, L.shared_tbl, L.gate_vec_dev, x, dev(ids_), dev(prec), dev(w), ws)
        torch.cuda.synchronize()
        return y.cpu().numpy(), B.slicemoe_get_status(ws)

    def oracle(ids_, prec_, w_):
        return moe.layer(x64, L.oracle_list(), ids_, prec_, w_.astype(np.float64), shared=L.oracle_shared, shared_gate_vec=L.gate_vec)

    y_ref = oracle(ids, prec, w)
    y, status = layer(ids, L.ws)
    assert status == 0
    for t in range(T):
        H.assert_close(y[t], y_ref[t], f"token {t}")
    # a workspace without the batch part: token after token
    y, status = layer(ids, B.new_workspace(L.cshape)[:L.ws.numel() - 256])
    assert status == 0
    for t in range(T):
        H.assert_close(y[t], y_ref[t], f"token {t} alone")
    # an id out of range is skipped and reported; the workspace is fit for the next call
    bad, w_ref = ids.copy(), w.copy()
    bad[T - 1, 1], w_ref[T - 1, 1] = E, 0.0
    y, status = layer(bad, L.ws)
    assert status & B.STATUS_BAD_EXPERT_ID
    H.assert_close(y, oracle(ids, prec, w_ref), "bad id skipped")
    # routed in the same call
    logits = synth.router_logits_normal(sh.seed, ("batch-logits",), T, E)
    y, ids_r, prec_r, w_r = B.slicemoe_layer_routed(L.cshape, L.experts_tbl, L.shared_tbl, L.gate_vec_dev, x,
                                                    dev(logits.astype(np.float32)), L.ws, rank_high=1)
    torch.cuda.synchronize()
    assert B.slicemoe_get_status(L.ws) == 0
    ids_ref, _, _ = moe.route_topk(logits, k)
    assert np.array_equal(ids_r.cpu().numpy(), ids_ref)
    H.assert_close(y.cpu().numpy(), oracle(ids_ref, prec_r.cpu().numpy(), w_r.cpu().numpy()), "routed")


def _random_lists(rng, T, E, k):
    ids = np.stack([rng.permutation(E)[:k] for _ in range(T)]).astype(np.int32)
    return ids, rng.integers(0, 2, (T, k)).astype(np.uint8), rng.random((T, k)).astype(np.float32)


def test_a_result_buffer_may_start_on_any_float():
    """As for one token, nothing is asked of y's alignment: a view one float into a buffer gets the same bits."""
    import torch
    from paper_2512_12990_b200 import binding as B
    T, E, k = 4, 6, 3
    sh = synth.Shape("batch", 256, 128, E, k, 64, n_shared=0, shared_inter=0, shared_sigmoid_gate=False, n_layers=1, seed=7100)
    L = H.Layer(sh, range(E))
    ids, prec, w = (torch.from_numpy(a).cuda() for a in _random_lists(np.random.default_rng(1), T, E, k))
    x = H.to_dev_bf16(H.x_inputs(sh, T, "batch-y")[0])
    want = B.slicemoe_layer(L.cshape, L.experts_tbl, None, None, x, ids, prec, w, L.ws)
    buf = torch.full((T * sh.hidden + 2,), 7.0, device="cuda")
    y = buf[1:-1].view(T, sh.hidden)
    assert y.data_ptr() % 8 == 4
    B.slicemoe_layer(L.cshape, L.experts_tbl, None, None, x, ids, prec, w, L.ws, y=y)
    torch.cuda.synchronize()
    assert torch.equal(y, want) and buf[0] == 7.0 and buf[-1] == 7.0


@pytest.mark.parametrize("group,bits", [(128, (8, 4)), (64, (6, 3)), (32, (8, 4)), (32, (4, 2))])
def test_a_token_does_not_depend_on_the_others_of_its_batch(group, bits):
    """The form of the arithmetic follows from the run that a token's pair falls into: alone or with one other pair, among
    up to eight, at one precision or both.  None of that shows in the token's result, bit for bit."""
    import torch
    from paper_2512_12990_b200 import binding as B
    E, k, hidden = 12, 3, 640
    sh = synth.Shape("batch", hidden, 384, E, k, group, n_shared=1, shared_inter=256, shared_sigmoid_gate=True, n_layers=1, seed=7200 + group)
    L = H.Layer(sh, range(E), b_high=bits[0], b_low=bits[1])
    x_all = H.to_dev_bf16(H.x_inputs(sh, 16, "batch-alone")[0])
    mine, mine_w = np.array([3, 7, 5], np.int32), np.array([0.5, 0.3, 0.2], np.float32)

    def call(others, others_prec, my_prec):
        """Token 0 keeps its list; the others' lists [T - 1, k] vary."""
        T = len(others) + 1
        ids = np.concatenate([mine[None], others]).astype(np.int32)
        prec = np.concatenate([my_prec[None], others_prec]).astype(np.uint8)
        w = np.concatenate([mine_w[None], np.full((T - 1, k), 0.25, np.float32)])
        y = B.slicemoe_layer(L.cshape, L.experts_tbl, L.shared_tbl, L.gate_vec_dev, x_all[:T].contiguous(),
                             *(torch.from_numpy(a).cuda() for a in (ids, prec, w)), L.ws)
        torch.cuda.synchronize()
        assert B.slicemoe_get_status(L.ws) == 0
        return y[0].cpu()

    for my_prec in (np.array([1, 0, 1], np.uint8), np.array([0, 1, 0], np.uint8)):
        elsewhere = np.array([0, 1, 2])                                   # none of the token's experts: it is alone with each
        want = call(np.tile(elsewhere, (3, 1)), np.zeros((3, k)), my_prec)
        assert want.abs().max() > 0
        for T in (4, 5, 9, 16):
            for shared_with in (1, T - 1):                                # one other pair, or all of them
                for p in (0, 1):
                    others = np.tile(elsewhere, (T - 1, 1))
                    others[:shared_with] = mine[None]
                    got = call(others, np.full((T - 1, k), p), my_prec)
                    assert torch.equal(got, want), f"T {T}, {shared_with} others at precision {p}"
        got = call(np.tile(mine, (7, 1)), np.arange(7)[:, None] % 2 * np.ones((1, k)), my_prec)
        assert torch.equal(got, want), "others at either precision"


@pytest.mark.parametrize("T", [4, 16])
def test_the_widest_hidden_with_the_smallest_groups(T):
    """Hidden 4096 at group 32: the digits of eight tokens leave the gate/up kernel one ring stage per group."""
    import torch
    from paper_2512_12990_b200 import binding as B
    E, k = 6, 3
    sh = synth.Shape("batch", 4096, 128, E, k, 32, n_shared=1, shared_inter=256, shared_sigmoid_gate=True, n_layers=1, seed=7400 + T)
    L = H.Layer(sh, range(E))
    ids, prec, w = _random_lists(np.random.default_rng(T), T, E, k)
    xbits, x64 = H.x_inputs(sh, T, "batch-wide")
    y = B.slicemoe_layer(L.cshape, L.experts_tbl, L.shared_tbl, L.gate_vec_dev, H.to_dev_bf16(xbits),
                         *(torch.from_numpy(a).cuda() for a in (ids, prec, w)), L.ws)
    torch.cuda.synchronize()
    assert B.slicemoe_get_status(L.ws) == 0
    y_ref = moe.layer(x64, L.oracle_list(), ids, prec, w.astype(np.float64), shared=L.oracle_shared, shared_gate_vec=L.gate_vec)
    for t in range(T):
        H.assert_close(y[t].cpu().numpy(), y_ref[t], f"token {t}")
