"""Decode steps at the sizes where one form of the attention gives way to another, against fp64 softmax attention."""
import pytest
import torch

from paper_2512_07090_b200 import binding as tfb
from launched import launched, ran
from test_gpu_parity import ATTN_TOL, DEV, _qkv, attn_rel_err, to_np
from test_gpu_parity import test_decode_attention_uneven_positions_and_skips as _uneven_positions_and_skips

pytestmark = pytest.mark.gpu


def _form(call, items):
    """How the visible keys of a work item are divided: by the kernels launched and their CTAs."""
    names = launched(call)
    assert "decode_decide_kernel" in names[0][0]
    if "decode_attention_stream_kernel" in names[1][0]:
        return "pieces" if "decode_combine_kernel" in names[-1][0] else "stream"
    assert "decode_attention_split_kernel" in names[1][0]
    return "scratch" if len(names) == 3 else "whole" if names[1][1] == items else "cluster"


@pytest.mark.parametrize("workspace", [True, False])
@pytest.mark.parametrize("B,S,Hkv,G,window,forms", [      # with a workspace, without
    (8, 420, 8, 4, 0, "cluster cluster"), (4, 777, 8, 4, 0, "cluster cluster"), (1, 300, 40, 1, 0, "cluster cluster"), (3, 129, 10, 2, 0, "cluster cluster"),
    (2, 512, 8, 4, 100, "whole whole"),                                                      # a window too short to be split
    (8, 1000, 8, 4, 0, "cluster cluster"), (4, 1800, 8, 2, 0, "cluster cluster"), (3, 1100, 12, 1, 0, "cluster cluster"),   # they learn of a skip with keys in flight
    (1, 3800, 4, 2, 0, "cluster cluster"), (1, 6000, 4, 2, 0, "scratch cluster"),            # a long one as a cluster, a short one through scratch
    (18, 600, 8, 4, 0, "scratch whole"), (70, 300, 8, 4, 0, "whole whole"), (80, 300, 8, 4, 0, "whole whole"),   # one wave (the attention starts early), two, three
    (20, 300, 8, 8, 0, "whole whole"),                                                       # eight heads a group
    (6, 30000, 4, 1, 0, "pieces cluster"), (300, 200, 8, 1, 0, "pieces stream"),             # last tiles of 1 to 64 keys
    (3, 3000, 32, 1, 0, "scratch stream"), (7, 1200, 40, 1, 0, "pieces stream"),
    (18, 130, 40, 1, 0, "whole stream"), (18, 130, 8, 1, 0, "whole whole")])                # three waves of short items, one
def test_decode_attention_forms(B, S, Hkv, G, window, forms, workspace):
    ctx, shape, params, qn, k, v, st, O, skip = _step(B, S, Hkv, G, seed=S, window=window)
    if workspace:
        ctx.ensure_workspace(shape, params)
    pos = torch.zeros(B, dtype=torch.int32, device=DEV)
    step = lambda: ctx.tf_decode_step(shape, params, 0.0, qn, k, v, pos, st, O, None, skip)
    step()
    assert _form(step, B * Hkv) == forms.split()[0 if workspace else 1]
    ctx.close()
    _uneven_positions_and_skips(B, S, Hkv, G, window, workspace)


def _step(B, S, Hkv, G, seed, window=0):
    q, k, v = _qkv(B, S, Hkv * G, Hkv, torch.bfloat16, seed=seed)
    qn = q[:, -1].contiguous()
    shape = tfb.make_shape(None, k, v, window=window, n_q_heads=Hkv * G)
    shape.q_stride[:] = [qn.stride(0), 0, qn.stride(1)]
    shape.o_stride[:] = list(shape.q_stride)
    params = tfb.default_params(prune_ratio=0.5, warmup_tokens=0)
    ctx = tfb.Context(0)
    st = tfb.DecodeState(B, Hkv, DEV)
    st.tau.fill_(9.0)
    return ctx, shape, params, qn, k, v, st, torch.empty_like(qn), torch.empty(B, dtype=torch.uint8, device=DEV)


def _exact(qn, k, v, b, n):
    Hkv = k.shape[2]
    s = torch.einsum("hgd,nhd->hgn", qn[b].double().view(Hkv, -1, 128), k[b, :n].double()) / 128 ** 0.5
    return torch.einsum("hgn,nhd->hgd", s.softmax(-1), v[b, :n].double()).reshape(-1, 128)


@pytest.mark.parametrize("B,S,Hkv,G,kernel,ctas", [
    (1, 8192, 8, 4, "split", 64), (4, 4096, 8, 4, "split", 128), (1, 30000, 8, 1, "split", 64), (1, 4000, 40, 1, "split", 120),   # clusters at any length
    (20, 1000, 8, 4, "split", 160), (1, 8192, 2, 8, "split", 2),      # no room for clusters, none for eight heads a group
    (1, 200, 100, 1, "split", 100), (4, 1000, 40, 1, "split", 160),   # whole items: short ones, several an SM
    (1, 3000, 100, 1, "stream", 148), (1, 384, 90, 1, "stream", 148)])
def test_steps_without_a_workspace_are_split_as_far_as_clusters_go(B, S, Hkv, G, kernel, ctas):
    ctx, shape, params, qn, k, v, st, O, skip = _step(B, S, Hkv, G, seed=S)
    pos = torch.full((B,), S - 1, dtype=torch.int32, device=DEV)
    step = lambda: ctx.tf_decode_step(shape, params, 0.0, qn, k, v, pos, st, O, None, skip)
    step()
    assert ctx.tf_get_status()[0] == tfb.TF_OK
    for b in range(B):
        assert attn_rel_err(to_np(O[b]), _exact(qn, k, v, b, S).cpu().numpy()) < ATTN_TOL[torch.bfloat16], b
    assert ran(step, f"decode_attention_{kernel}_kernel") == ctas
    ctx.close()


@pytest.mark.parametrize("B,S,Hkv,kernel,ctas", [
    (12, 250, 32, "split", 384), (24, 250, 32, "stream", 148),            # 18 tiles per SM
    (7, 1000, 40, "split", 280), (7, 1200, 40, "stream", 148),            # 34: a full wave
    (16, 832, 32, "split", 512), (16, 896, 32, "stream", 148)])           # 48: two of them
def test_ungrouped_steps_either_side_of_the_streaming_kernel(B, S, Hkv, kernel, ctas):
    ctx, shape, params, qn, k, v, st, O, skip = _step(B, S, Hkv, 1, seed=S)
    ctx.ensure_workspace(shape, params)
    pos = torch.full((B,), S - 1, dtype=torch.int32, device=DEV)
    step = lambda: ctx.tf_decode_step(shape, params, 0.0, qn, k, v, pos, st, O, None, skip)
    step()
    assert ctx.tf_get_status()[0] == tfb.TF_OK
    for b in (0, B - 1):
        assert attn_rel_err(to_np(O[b]), _exact(qn, k, v, b, S).cpu().numpy()) < ATTN_TOL[torch.bfloat16], b
    assert ran(step, f"decode_attention_{kernel}_kernel") == ctas
    ctx.close()


@pytest.mark.parametrize("B,S,Hkv,G,launches", [(1, 1000, 8, 4, 2), (1, 600, 40, 1, 2), (3, 500, 6, 2, 2), (1, 4000, 40, 1, 3), (16, 500, 32, 1, 2)])
def test_split_decode_loses_nothing_before_the_result_is_rounded(B, S, Hkv, G, launches):
    """The error against 64 bits is that of rounding the exact result to bf16 (to 2 %): clusters of every group size, ungrouped
    heads through scratch and unsplit."""
    ctx, shape, params, qn, k, v, st, O, skip = _step(B, S, Hkv, G, seed=S)
    ctx.ensure_workspace(shape, params)
    n0 = ctx.launches
    ctx.tf_decode_step(shape, params, 0.0, qn, k, v, torch.full((B,), S - 1, dtype=torch.int32, device=DEV), st, O, None, skip)
    assert ctx.launches - n0 == launches
    assert ctx.tf_get_status()[0] == tfb.TF_OK
    err = rounding = 0.0
    for b in range(B):
        ref = _exact(qn, k, v, b, S)
        err += float((O[b].double() - ref).square().sum())
        rounding += float((ref.bfloat16().double() - ref).square().sum())
    assert err < 1.02 ** 2 * rounding, (err ** 0.5, rounding ** 0.5)
    ctx.close()
