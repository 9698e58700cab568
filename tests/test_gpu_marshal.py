"""The native argument marshalling behind binding.py: outputs given or allocated, streams, optional arguments, errors."""
import numpy as np
import pytest

from paper_2512_12990_b200 import binding as B
from paper_2512_12990_b200 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tokens", [1, 3])
def test_given_and_allocated_outputs_are_the_same_bits(tokens):
    import torch
    sh = synth.SHAPES["tiny"]
    layer = H.Layer(sh, range(sh.n_experts))
    xbits, _ = H.x_inputs(sh, tokens, "marshal-x")
    x = H.to_dev_bf16(xbits)
    logits = torch.from_numpy(synth.router_logits_normal(sh.seed, ("marshal",), tokens, sh.n_experts)).cuda()
    ids, w, prec = B.slicemoe_route_topk(logits, sh.top_k, rank_high=1)
    assert B.slicemoe_route_topk(logits, sh.top_k, want_prec=False)[2] is None
    assert ids.shape == (tokens, sh.top_k) and ids.dtype == torch.int32 and prec.dtype == torch.uint8
    ref = B.slicemoe_layer(layer.cshape, layer.experts_tbl, None, None, x, ids, prec, w, layer.ws)
    y = torch.full((tokens, sh.hidden), float("nan"), device="cuda")
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    assert B.slicemoe_layer(layer.cshape, layer.experts_tbl, None, None, x, ids, prec, w, layer.ws, y=y, stream=side) is y
    side.synchronize()
    assert torch.equal(y, ref)
    assert torch.equal(B.slicemoe_expert_ffn(layer.cshape, layer.experts_tbl, x, ids, prec, w, layer.ws), ref)
    out = B.slicemoe_layer_routed(layer.cshape, layer.experts_tbl, None, None, x, logits, layer.ws, rank_high=1)
    assert all(torch.equal(a, b) for a, b in zip(out, (ref, ids, prec, w)))
    out = B.slicemoe_layer_routed(layer.cshape, layer.experts_tbl, None, None, x, logits, layer.ws, rank_high=1, y=y, want_lists=False)
    assert out[0] is y and out[1:] == (None, None, None)
    pws = B.new_prefill_workspace(layer.cshape, tokens)
    eprec = torch.ones(sh.n_experts, dtype=torch.uint8, device="cuda")
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    a = B.slicemoe_prefill_layer(layer.cshape, layer.experts_tbl, None, None, x, ids, w, eprec, pws)
    b = B.slicemoe_prefill_layer(layer.cshape, layer.experts_tbl, None, None, x, ids, w, eprec, pws, y=y, status=status)
    assert b[0] is y and b[1] is status and torch.equal(a[0], y) and int(a[1]) == int(status) == 0


def test_errors_are_exceptions():
    import torch
    logits = torch.zeros((1, 8), device="cuda")
    with pytest.raises(B.SliceMoEError) as e:
        B.slicemoe_route_topk(logits, 9)
    assert e.value.code == B.E_INVALID_ARG and "slicemoe_route_topk" in str(e.value)
    with pytest.raises(AssertionError):
        B.slicemoe_route_topk(logits.double(), 2)
    with pytest.raises(AssertionError):
        B.slicemoe_pack(torch.zeros((16, 256), device="cuda").t(), 64)
    with pytest.raises(B.SliceMoEError) as e:
        B.slicemoe_pack(torch.zeros((16, 128), device="cuda"), 48)
    assert e.value.code == B.E_UNSUPPORTED
    shape = B.make_shape(256, 128, 8, 2, 64)
    ws = B.new_workspace(shape)
    x = torch.zeros((1, 256), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(B.SliceMoEError) as e:
        B.slicemoe_layer(shape, None, None, None, x, logits, logits, logits, ws)
    assert e.value.code == B.E_INVALID_ARG
    with pytest.raises((TypeError, BufferError)):
        B.slicemoe_layer(None, None, None, None, x, logits, logits, logits, ws)
    assert np.isfinite(x.float().cpu().numpy()).all()


def test_outputs_have_storages_of_their_own():
    """A packed matrix and a routing list can be saved and loaded, and an output that is kept keeps nothing else."""
    import io
    import torch
    m = B.slicemoe_pack(torch.randn((32, 256), device="cuda"), 64)
    routed = B.slicemoe_route_topk(torch.randn((3, 8), device="cuda"), 2)
    shape = B.make_shape(256, 128, 8, 2, 64)
    layer = H.Layer(synth.SHAPES["tiny"], range(8))
    x = torch.zeros((1, 256), dtype=torch.bfloat16, device="cuda")
    out = B.slicemoe_layer_routed(shape, layer.experts_tbl, None, None, x, torch.randn((1, 8), device="cuda"), B.new_workspace(shape))
    for group in ([m.msb, m.lsb, m.scale, m.zp], routed, out):
        assert len({t.untyped_storage().data_ptr() for t in group}) == len(group)
        assert all(t.storage_offset() == 0 and t.untyped_storage().nbytes() == t.numel() * t.element_size() for t in group)
        f = io.BytesIO()
        torch.save(list(group), f)
        f.seek(0)
        assert all(torch.equal(a, b) for a, b in zip(torch.load(f), group))


def test_running_out_of_memory_is_torchs_own_error():
    import torch
    W = torch.zeros((16384, 4096), device="cuda")          # 256 MB; its planes take 32 MB each
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + (8 << 20)) / total)
    try:
        with pytest.raises(torch.OutOfMemoryError):
            B.slicemoe_pack(W, 128)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert B.slicemoe_pack(W, 128).N == 16384
