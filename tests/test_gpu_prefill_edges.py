"""slicemoe_prefill_layer at the edges of its token tiles, in the narrow form (tiles of up to 96 tokens) and the wide one (192),
with the pairs counted by one block and by several, and with x on 4 bytes only.  Per token against the float64 oracle, tolerance
as for the decode path."""
import numpy as np
import pytest

from oracle import moe
from paper_2512_12990_b200 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,E,k,group,n_shared", [
    (1, 8, 2, 64, 0), (16, 8, 2, 32, 1), (17, 8, 2, 128, 0), (33, 8, 2, 64, 2),  # narrow: one tile an expert
    (96, 8, 2, 128, 1),      # its widest tile
    (97, 8, 2, 128, 1),      # the wide form's narrowest use of a second warpgroup's columns
    (97, 16, 2, 64, 0),      # narrow, expert 0's tokens cut into two tiles
    (192, 4, 1, 32, 1), (193, 4, 1, 64, 1),  # wide: one tile, two
    (1025, 4, 4, 64, 0),     # 4,100 pairs: more than one block counts
])
def test_tile_edges(T, E, k, group, n_shared):
    import torch
    from paper_2512_12990_b200 import binding as B
    sh = synth.Shape("pf_edges", 384, 256, E, k, group, n_shared=n_shared, shared_inter=128 if n_shared else 0,
                     shared_sigmoid_gate=n_shared == 1, n_layers=1, seed=7100 + T)
    L = H.Layer(sh, range(E))
    rng = np.random.default_rng(T + E)
    # every token goes to expert 0 and to k - 1 others
    ids = np.stack([np.concatenate(([0], 1 + rng.permutation(E - 1)[:k - 1])) for _ in range(T)]).astype(np.int32)
    w = rng.random((T, k)).astype(np.float32)
    ep = (np.arange(E) % 2).astype(np.uint8)
    xbits, x64 = H.x_inputs(sh, T, "edges-x")
    x = H.to_dev_bf16(xbits)
    ws = B.new_prefill_workspace(L.cshape, T)

    def layer(x_, ep_):
        y, status = B.slicemoe_prefill_layer(L.cshape, L.experts_tbl, L.shared_tbl, L.gate_vec_dev, x_, torch.from_numpy(ids).cuda(),
                                             torch.from_numpy(w).cuda(), torch.from_numpy(ep_).cuda(), ws)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        return y.cpu().numpy()

    y = layer(x, ep)
    some = sorted(set(range(T)) & {0, 1, 15, 16, 31, 47, 48, 63, 64, 79, 95, 96, 97, 111, 112, 191, 192, T - 2, T - 1})
    y_ref = moe.layer(x64[some], L.oracle_list(), ids[some], ep[ids[some]], w[some].astype(np.float64), shared=L.oracle_shared,
                      shared_gate_vec=L.gate_vec)
    for i, t in enumerate(some):
        H.assert_close(y[t], y_ref[i], f"token {t}")
    # the same rows two elements further on: x on 4 bytes takes the other copy of the gather kernel, with the same result but for
    # the shared expert's gate, whose 384 fp32 products it adds in another order: by at most 384 x 2^-24 of the sum of
    # their sizes (about 5), 1.1e-4, a quarter of that in the sigmoid, below 1e-4 of the shared expert's part
    shifted = torch.empty(x.numel() + 2, dtype=x.dtype, device=x.device)[2:].view_as(x)
    shifted.copy_(x)
    assert shifted.data_ptr() % 16 == 4
    y2 = layer(shifted, ep)
    if sh.shared_sigmoid_gate:
        assert H.errors(y2, y)[0] <= 1e-4
    else:
        assert np.array_equal(y2, y)


def test_calls_in_a_row_through_the_same_buffers():
    """Kernels of a call start before the one ahead has ended and read the plan, x and the tables then: prompts that take
    turns in one workspace, with nothing in between, each give what they give alone."""
    import torch
    from paper_2512_12990_b200 import binding as B
    E, k, hidden = 12, 3, 512
    sh = synth.Shape("edges", hidden, 256, E, k, 128, n_shared=1, shared_inter=256, shared_sigmoid_gate=True, n_layers=1, seed=8900)
    L = H.Layer(sh, range(E))
    rng = np.random.default_rng(9)
    prompts = []
    for T in (5, 300, 40):
        ids = np.stack([rng.permutation(E)[:k] for _ in range(T)]).astype(np.int32)
        if T == 40:
            ids[:] = [1, 2, 3]
        prompts.append((H.to_dev_bf16(H.x_inputs(sh, T, f"row-{T}")[0]), torch.from_numpy(ids).cuda(), torch.rand((T, k), device="cuda"),
                        torch.from_numpy(rng.integers(0, 2, E).astype(np.uint8)).cuda()))
    ws = B.new_prefill_workspace(L.cshape, 300)

    def call(p):
        return B.slicemoe_prefill_layer(L.cshape, L.experts_tbl, L.shared_tbl, L.gate_vec_dev, *p, ws)

    alone = []
    for p in prompts:
        ws.fill_(0)
        alone.append(call(p)[0])
        torch.cuda.synchronize()
    out = [call(p) for _ in range(20) for p in prompts]
    torch.cuda.synchronize()
    for i, (y, status) in enumerate(out):
        assert int(status) == 0 and torch.equal(y, alone[i % 3]), f"call {i}"
