"""The calls' host side in native code (kvq_call) against the binding's general way: the same bytes for what it takes, and the same
exceptions for what it leaves."""
import pytest
import torch

from paper_2605_05699_b200 import binding as kb
from paper_2605_05699_b200 import workloads as wl


def calls(plan, x, lam, packed, scales, out, pos, stream=None):
    """Every call that has a native form, on caches [S, T, .] (the flat calls see them as S T rows)."""
    flat = packed.view(-1, packed.shape[-1]), scales.view(-1, scales.shape[-1])
    n = flat[0].shape[0]
    kb.kvq_encode(plan, x.view(-1, x.shape[-1])[:n], lam, *flat, n, stream=stream)
    kb.kvq_append(plan, x[:, 0].contiguous(), lam, packed, scales, 1, 2, stream=stream)
    kb.kvq_append_at(plan, x[:, 1].contiguous(), lam, packed, scales, pos, 2, stream=stream)
    kb.kvq_flush_block(plan, x[:, :2].contiguous(), lam, packed, scales, out, 0, 2, stream=stream)
    kb.kvq_decode(plan, *flat, lam, out.view(-1, out.shape[-1]), n, stream=stream)


def test_the_native_module_has_been_built():
    kb.lib()
    assert kb._native is not None


@pytest.mark.parametrize("native", [True, False])
def test_what_is_refused_stays_refused(native, monkeypatch):
    """No device needed: every one of these stops before the library is called."""
    kb.lib()
    if not native:
        monkeypatch.setattr(kb, "_native", None)
    plan = kb.Plan(64)
    h = plan.handle
    x, lam = torch.zeros(4, 64, dtype=torch.float16), torch.ones(64)
    p, s = torch.zeros(4, 8, 32, dtype=torch.uint8), torch.zeros(4, 8, 2, dtype=torch.float16)
    with pytest.raises(ValueError, match="x must live on a CUDA device"):
        kb.kvq_encode(h, x, lam, p, s)
    with pytest.raises(ValueError, match="packed must live"):
        kb.kvq_decode(h, p, s, lam, x)
    with pytest.raises(ValueError, match="x_new must live"):
        kb.kvq_append(h, x, lam, p, s, 0)
    with pytest.raises(ValueError, match="x_new must live"):
        kb.kvq_append_at(h, x, lam, p, s, torch.zeros(1, dtype=torch.int64))
    with pytest.raises(ValueError, match="x_block must live"):
        kb.kvq_flush_block(h, x.view(4, 1, 64), lam, p, s, x, 0)
    with pytest.raises(ValueError):
        kb.kvq_flush_block(h, x, lam, p, s, x, 0)          # not [S, rows, D]
    with pytest.raises(AttributeError):
        kb.kvq_encode(h, [1.0], lam, p, s)
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("D,dtype", [(64, "f16"), (256, "bf16")])
def test_native_and_general_calls_give_the_same_bytes(D, dtype, monkeypatch):
    S, T = 3, 5
    plan = kb.Plan(D, 32, 3)
    x = wl.make_vectors(S * T, D, dtype, "gaussian", 1, device="cuda").view(S, T, D)
    lam = wl.make_lambda(2, D, 2).cuda()
    pos = torch.tensor([3], dtype=torch.int64, device="cuda")
    side = torch.cuda.Stream()
    got = []
    for native, stream in ((True, None), (False, None), (True, torch.cuda.current_stream()), (True, side)):
        with monkeypatch.context() as m:
            if not native:
                m.setattr(kb, "_native", None)
            b = [torch.zeros(S, T, D // 2, dtype=torch.uint8, device="cuda"), torch.zeros(S, T, D // 32, dtype=torch.float16, device="cuda"),
                 torch.zeros(S, T, D, dtype=x.dtype, device="cuda")]
            torch.cuda.synchronize()
            if stream is side:   # on a side stream as the current one
                with torch.cuda.stream(side):
                    calls(plan.handle, x, lam, *b, pos)
            else:
                calls(plan.handle, x, lam, *b, pos, stream)
            torch.cuda.synchronize()
            got.append(b)
    for b in got[1:]:
        assert all(bool((u == v).all()) for u, v in zip(got[0], b))
    assert bool(got[0][0].any()) and bool(got[0][2].any())
    # what needs a device to be refused: the same exceptions both ways
    p, s, o = got[0]
    for native in (True, False):
        with monkeypatch.context() as m:
            if not native:
                m.setattr(kb, "_native", None)
            with pytest.raises(ValueError, match="x must be contiguous"):
                kb.kvq_encode(plan.handle, x[:, ::2], lam, p, s)
            with pytest.raises(TypeError, match="float16 or bfloat16"):
                kb.kvq_encode(plan.handle, x.float(), lam, p, s)
            with pytest.raises(kb.KvqError) as e:
                kb.kvq_append(plan.handle, x[:, 0].contiguous(), lam, p, s, T, 2)   # past the end of the cache
            assert e.value.status == kb.KVQ_ERR_INVALID_ARG
    plan.close()
