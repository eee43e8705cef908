"""Selections at the sizes where one form gives way to another: exchanges of the cluster form, waits that give up, short sequences."""
import numpy as np
import pytest
import torch

from paper_2512_07090_b200 import binding as tfb

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _select(ctx, score, ratio, theta=None):
    B, S = score.shape
    shape = tfb.tf_shape()
    shape.batch, shape.seq, shape.n_q_heads, shape.n_kv_heads, shape.head_dim, shape.dtype = B, S, 32, 32, 128, tfb.TF_BF16
    params = tfb.default_params(prune_ratio=ratio, warmup_tokens=4)
    keep = torch.full((B, S), 7, dtype=torch.uint8, device=DEV)
    idx = torch.full((B, S), -7, dtype=torch.int32, device=DEV)
    nk = torch.full((B,), -7, dtype=torch.int32, device=DEV)
    ctx.tf_select(shape, params, score, keep, idx, nk, theta)
    return keep, idx, nk


def _expect(score, ratio):
    S = len(score)
    order = sorted(range(4, S), key=lambda t: (-score[t], -t))          # equal scores go from the highest index down
    pruned = set(order[:min(S - 4, int(np.floor(ratio * S)))])
    return [t for t in range(S) if t not in pruned]


# spread scores (two passes), all of them in one binade and close together (three and four passes), many equal ones
@pytest.mark.parametrize("kind", ["spread", "close", "closer", "ties"])
@pytest.mark.parametrize("S", [1025, 2048, 2049, 9000, 32768])           # clusters of 4 and 8, every register count
def test_cluster_selection_passes(S, kind):
    rng = np.random.default_rng(S)
    x = rng.standard_normal((2, S)) * 0.05
    if kind != "spread":
        x = 0.5 + rng.random((2, S)) * {"close": 1e-3, "closer": 2e-6, "ties": 1e-3}[kind]
    if kind == "ties":
        x = np.round(x, 5)
    score = x.astype(np.float32)
    ctx = tfb.Context(0)
    ctx.tf_set_select_path(2)
    keep, idx, nk = _select(ctx, torch.from_numpy(score).to(DEV), 0.4)
    assert ctx.tf_get_status()[0] == tfb.TF_OK
    for b in range(2):
        want = _expect(score[b], 0.4)
        assert int(nk[b]) == len(want)
        got = idx[b].cpu().numpy()
        assert np.array_equal(got[:len(want)], want) and np.all(got[len(want):] == -1)
        assert np.array_equal(np.flatnonzero(keep[b].cpu().numpy()), want)
    ctx.close()


def test_a_selection_whose_waits_give_up_keeps_nothing_or_the_right_tokens():
    """On a limit of no cycles an exchange that is not there at the first look counts as missing: the status says so, and all outputs
    of that sequence say that nothing is kept, so that neither the list nor the mask leads on to numbers that were never exchanged."""
    score = (np.random.default_rng(3).standard_normal((8, 20000)) * 0.05).astype(np.float32)
    dev = torch.from_numpy(score).to(DEV)
    want = [_expect(s, 0.5) for s in score]
    ctx = tfb.Context(0)
    ctx.tf_set_select_path(2)
    codes = []
    for limit in (0, 0, 0, -1):
        ctx.tf_set_wait_limits(wait_cycles=limit)
        theta = torch.full((8,), 7.0, device=DEV)
        keep, idx, nk = _select(ctx, dev, 0.5, theta)
        codes.append(ctx.tf_get_status()[0])
        for b in range(8):
            got, n, mask = idx[b].cpu().numpy(), int(nk[b]), keep[b].cpu().numpy()
            if codes[-1] == tfb.TF_OK or n > 0:
                assert n == len(want[b]) and np.array_equal(got[:n], want[b]) and np.all(got[n:] == -1)
                assert np.array_equal(np.flatnonzero(mask), want[b])
                assert float(theta[b]) == np.delete(score[b], want[b]).min()
            else:
                assert np.all(got == -1) and not mask.any() and float(theta[b]) == np.inf
        ctx.tf_clear_status()
    assert tfb.TF_ERR_TIMEOUT in codes[:3] and set(codes[:3]) <= {tfb.TF_OK, tfb.TF_ERR_TIMEOUT} and codes[3] == tfb.TF_OK
    ctx.close()


@pytest.mark.parametrize("S,H", [(1, 1), (33, 8), (33, 9), (240, 32), (240, 64),       # 8, 16, 32 lanes a token, one or two heads a lane
                                 (240, 65), (241, 8), (241, 32)])                    # too many heads; too long
@pytest.mark.parametrize("case", ["plain", "ties", "nan", "eligible", "threshold", "none"])
def test_short_sequences_in_one_launch_give_the_bits_of_the_two_steps(S, H, case):
    rng = np.random.default_rng(100 * S + H)
    B = 3
    sim = [torch.from_numpy((rng.standard_normal((B, S, H)) * 0.1).astype(np.float32)).to(DEV) for _ in range(2)]
    if case == "ties":
        for s in sim:
            s[:, 1::2] = s[:, :1]
    if case == "nan":
        sim[0][1, S // 2, H // 2] = float("nan")
    kw = dict(prune_ratio=0.0 if case == "none" else 0.4, warmup_tokens=2)
    if case == "eligible":
        kw["eligible"] = el = torch.from_numpy((rng.random((B, S)) < 0.3).astype(np.uint8)).to(DEV)
    if case == "threshold":
        kw["threshold"] = tau = torch.tensor([-0.02, 0.0, 0.5], device=DEV)
        kw["select_mode"] = tfb.TF_SELECT_THRESHOLD
    params = tfb.default_params(**kw)
    shape = tfb.tf_shape()
    shape.batch, shape.seq, shape.n_q_heads, shape.n_kv_heads, shape.head_dim, shape.dtype = B, S, H, H, 128, tfb.TF_F32
    got = []
    ctx = tfb.Context(0)
    for path in (1, 0):
        ctx.tf_set_select_path(path)
        out = [torch.full((B, S), -3.0, device=DEV), torch.full((B, S), 9, dtype=torch.uint8, device=DEV),
               torch.full((B, S), -9, dtype=torch.int32, device=DEV), torch.full((B,), -9, dtype=torch.int32, device=DEV), torch.full((B,), -9.0, device=DEV)]
        n0 = ctx.launches
        ctx.tf_score_select(shape, params, sim[0], sim[1], *out)
        assert ctx.launches - n0 == (1 if path == 0 and S <= 240 and H <= 64 else 2)
        got.append(out)
        alone = [torch.empty_like(o) for o in out[1:]]                       # step a4 alone on these scores
        ctx.tf_select(shape, params, out[0], *alone)
        for a, o in zip(alone, out[1:]):
            assert torch.equal(a, o)
    for a, o in zip(*got):
        assert torch.equal(a.view(torch.int32) if a.dtype == torch.float32 else a, o.view(torch.int32) if o.dtype == torch.float32 else o)
    ctx.close()
