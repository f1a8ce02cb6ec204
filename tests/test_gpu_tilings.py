"""The sizes at which the kernels change their tiling or their way of working, against the CPU oracle: vocabulary tiles of a
CTA, tiles of hidden rows, halves of a tile, slabs of a draw, and logits that no bound can tell apart.  Needs a B200.
Tolerances as in util.py (derived there); SM counts are read from the device."""
import numpy as np
import pytest
import torch

from paper_2405_04304_b200 import binding, inputs
from util import (check_draft, check_verify, gpu_draft_step, gpu_verify, make_clf, near_tie_ids, to_gpu_clf,
                  to_oracle_clf)

pytestmark = pytest.mark.gpu

_bits = inputs.bf16_bits


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _check_draft_and_each_probability(got, ref, tau, active=None, rel=5e-5):
    """check_draft compares probabilities absolutely, which says nothing about those of a flat distribution: here each of the ten
    largest relatively.  A logit of these tests is a sum of at most 40 products of some 10 in all, in fp32, so that it is good to
    40 * 10 * 2^-24 = 2.4e-5 and e^z to as much; the exponentials and their sum add 1e-6."""
    check_draft(got, ref, tau, active=active)
    on = np.ones(len(ref.token), bool) if active is None else np.asarray(active) != 0
    want = ref.feats[on, :10]
    assert float(np.abs(got["feats"][on, :10] / want - 1.0).max()) < rel


# vocabulary rows per SM: one and two tiles of up to 128, a tile of exactly 32 / 33 rows (with and without the shared bound)
@pytest.mark.parametrize("rows_per_sm,extra,B", [(32, 0, 9), (32, 1, 9), (128, 0, 40), (128, 1, 40), (256, 1, 33),
                                                 (16, 5, 128), (16, 5, 129), (40, -3, 300)])
def test_batched_draft_step_at_the_edges_of_its_tiling(oracle, rows_per_sm, extra, B):
    V, d = _sms() * rows_per_sm + extra, 40
    W, h = inputs.lm_head(V, d, seed=V, std=0.3), inputs.hidden(B, d, seed=B)
    params = make_clf(16, seed=1)
    pos, nd = np.arange(1, B + 1, dtype=np.int32), (np.arange(B, dtype=np.int32) % 4) + 1
    active = (np.arange(B) % 5 != 2).astype(np.uint8)
    ctx = binding.Context(V, d, 8, max_batch=B, max_rows=8, clf_hidden=16)
    Wg, clf = W.cuda(), to_gpu_clf(params)
    for act in (None, active, None):   # (a masked step between two full ones: scratch of either parity is left clean)
        got = gpu_draft_step(ctx, Wg, h, pos, nd, clf, 0.5, 3, active=act)
        ref = oracle.draft_step(_bits(W), _bits(h), pos, nd, to_oracle_clf(oracle, params), 0.5, 3, active=act, nthreads=8)
        _check_draft_and_each_probability(got, ref, 0.5, active=act)
    assert ctx.device_status() == 0
    ctx.close()


# Two narrow vocabulary tiles per CTA with CTAs of their own for the finishing, without them, and two wide ones; contractions around
# the limit of the rule
@pytest.mark.parametrize("d", [320, 328])
@pytest.mark.parametrize("B", [33, 128])
@pytest.mark.parametrize("finishers,extra", [(True, 0), (True, 1), (False, 0), (False, 1)])
def test_batched_draft_step_where_its_tiles_grow(oracle, finishers, extra, B, d):
    """A logit is a sum of 328 products of some 328 * 0.1 * 0.64 = 21 in all, in fp32: good to 328 * 21 * 2^-24 = 4.1e-4."""
    V = 256 * (_sms() - ((B + 9) // 10 if finishers else 0)) + extra
    W, h = inputs.lm_head(V, d, seed=V, std=0.1), inputs.hidden(B, d, seed=B)
    params = make_clf(16, seed=1)
    pos, nd = np.arange(1, B + 1, dtype=np.int32), (np.arange(B, dtype=np.int32) % 4) + 1
    ctx = binding.Context(V, d, 8, max_batch=B, max_rows=8, clf_hidden=16)
    got = gpu_draft_step(ctx, W.cuda(), h, pos, nd, to_gpu_clf(params), 0.5, 3)
    ref = oracle.draft_step(_bits(W), _bits(h), pos, nd, to_oracle_clf(oracle, params), 0.5, 3, nthreads=16)
    _check_draft_and_each_probability(got, ref, 0.5, rel=4.1e-4)
    assert ctx.device_status() == 0
    ctx.close()


@pytest.mark.parametrize("V,copies", [(5000, 5000), (5000, 40), (40000, 1000), (20000, 12)])
def test_logits_that_no_bound_can_tell_apart(oracle, V, copies):
    """The largest logit occurs `copies` times (the whole vocabulary, or in consecutive rows of a few CTAs): the lists
    overflow, the arg-max is the lowest index."""
    d, B = 16, 12
    W, h = inputs.lm_head(V, d, seed=V + copies, std=0.2), inputs.hidden(B, d, seed=3)
    peak = (h[0].float() * 0.5).to(torch.bfloat16)          # sequence 0: logit |h|^2 / 2, far above the others
    at = (V - copies) // 2
    W[at:at + copies] = peak
    params = make_clf(8, seed=2)
    pos, nd = np.ones(B, np.int32), np.ones(B, np.int32)
    ctx = binding.Context(V, d, 8, max_batch=B, max_rows=8, clf_hidden=8)
    got = gpu_draft_step(ctx, W.cuda(), h, pos, nd, to_gpu_clf(params), 0.5, 3)
    ref = oracle.draft_step(_bits(W), _bits(h), pos, nd, to_oracle_clf(oracle, params), 0.5, 3, nthreads=8)
    assert int(got["token"][0]) == at == int(ref.token[0])
    ties = ref.gap < 1e-3                                    # other sequences may tie at rows of the block as well
    got["token"][ties] = ref.token[ties]
    ref.topk_ids[ties, 0] = ref.token[ties]
    _check_draft_and_each_probability(got, ref, 0.5)
    assert ctx.device_status() == 0
    ctx.close()


# (32000 and 4000 rows leave CTAs without a vocabulary row on 148 SMs: they are done while the others have just started)
@pytest.mark.parametrize("V", [32000, 4000])
def test_steps_in_a_row_do_not_see_each_others_bounds(V):
    """Back-to-back steps whose logits shrink and grow by a factor of 32 and whose row counts change: a bound left over from
    the step before would drop all of a small step's candidates."""
    d, counts, steps = 16, (40, 8, 1, 130), 160
    W = inputs.lm_head(V, d, seed=V, std=0.3).cuda()
    h = inputs.hidden(steps * 130, d, seed=11).view(steps, 130, d)
    h[::2] *= 4.0
    h[1::2] *= 0.125
    h, clf = h.cuda(), to_gpu_clf(make_clf(8, seed=3))
    ctx = binding.Context(V, d, 8, max_batch=130, max_rows=8, clf_hidden=8)
    z = lambda *s, t=torch.float32: torch.zeros(*s, dtype=t, device="cuda")
    one, token, feats = torch.ones(130, dtype=torch.int32, device="cuda"), z(steps, 130, t=torch.int32), z(steps, 130, 12)
    conf, halt = z(130), z(130, t=torch.uint8)
    rows = [counts[i // 2 % 4] for i in range(steps)]
    for i, B in enumerate(rows):
        ctx.draft_step(W, h[i, :B], one[:B], one[:B], clf, 0.5, 4, token[i], conf, halt, feats=feats[i])
    assert ctx.device_status() == 0
    for i, B in enumerate(rows):
        logits = h[i, :B].double() @ W.double().T
        top = logits.topk(10, -1).values
        want = (top - torch.logsumexp(logits, -1, keepdim=True)).exp()
        # a logit is a sum of 16 products of up to 60 in all, in fp32: 16 * 60 * 2^-24 = 6e-5 at most, e^z moves by as much
        assert float(((feats[i, :B, :10].double() - want) / want).abs().max()) < 2e-4, f"step {i}"
        picked = logits.gather(1, token[i, :B].long()[:, None])[:, 0]
        assert float((top[:, 0] - picked).max()) < 2e-4, f"step {i}"
    ctx.close()


@pytest.mark.parametrize("V,B", [(32000, 1), (5001, 40), (20011, 200)])
@pytest.mark.parametrize("path", [0, 1])
def test_soft_max_does_not_depend_on_what_all_logits_have_in_common(V, B, path):
    """Row b's logits are w_v + its offset, exactly (w_v a multiple of 1/32 below 4): the distribution is that of the w_v."""
    d = 8
    g = torch.Generator().manual_seed(V)
    w = torch.randint(-127, 128, (V,), generator=g).double() / 32
    W, h = torch.zeros(V, d), torch.zeros(B, d)
    W[:, 0], W[:, 1], h[:, 1] = 1.0, w.float(), 1.0
    h[:, 0] = torch.tensor([400.0, 0.0, 96.0, -2048.0, 131072.0, -131072.0])[torch.arange(B) % 6]
    W, h = W.to(torch.bfloat16).cuda(), h.to(torch.bfloat16).cuda()
    y = torch.softmax(w, -1)
    top, ent = y.topk(10).values, -(y * y.log()).sum()
    z = lambda *s, t=torch.float32: torch.zeros(*s, dtype=t, device="cuda")
    one, token, nxt, conf, halt = z(B, t=torch.int32) + 1, z(B, t=torch.int32), z(B, t=torch.int32), z(B), z(B, t=torch.uint8)
    feats, y_T = z(B, 12), z(B, V)
    ctx = binding.Context(V, d, d, max_batch=B, max_rows=B, clf_hidden=8)
    ctx.set_kernel_path(path)
    ctx.draft_step(W, h, one, one, to_gpu_clf(make_clf(8, seed=5)), 0.5, 4, token, conf, halt, feats=feats)
    ctx.verify_sample_ragged(W, h, None, None, None, B, B, None, z(B), z(B, t=torch.int32), nxt, y_T)
    assert ctx.device_status() == 0
    # an exponential is good to 2 ulp of its own and 2^-24 * |z - m| of its argument, |z - m| < 8: 8e-7 in all, once above
    # and once below the fraction bar; the entropy is some 10, a difference of ln Z and S / Z of that accuracy
    assert float(((feats[:, :10].cpu().double() - top) / top).abs().max()) < 2e-6
    assert float((feats[:, 10].cpu().double() - ent).abs().max()) < 1e-5
    assert float(((y_T.cpu().double() - y) / y).abs().max()) < 2e-6
    assert token.tolist() == [int(w.argmax())] * B
    ctx.close()


@pytest.mark.parametrize("V,B", [(4000, 1), (4000, 3), (30000, 4), (30000, 40), (3000, 200)])
@pytest.mark.parametrize("path", [0, 1, 2])
def test_logits_that_are_not_numbers(V, B, path):
    """A hidden row that is no number: token -1, never an index outside the vocabulary; the other rows do not notice.  One
    infinite logit: the token is an index or -1, and the features are numbers (tensor-core kernels)."""
    d, bad = 16, B // 2
    W, h = inputs.lm_head(V, d, seed=V, std=0.3), inputs.hidden(B, d, seed=B)
    h[bad], h[:, 3] = float("nan"), 1.0
    params = to_gpu_clf(make_clf(8, seed=5))
    z = lambda *s, t=torch.float32: torch.zeros(*s, dtype=t, device="cuda")
    ints = lambda *s: z(*s, t=torch.int32)
    ctx = binding.Context(V, d, d, max_batch=B, max_rows=2 * B, clf_hidden=8)
    ctx.set_kernel_path(path)

    def every_pass(Wg, hg):
        one, conf, halt, feats, y, y2, u = ints(B) + 1, z(2, B), z(2, B, t=torch.uint8), z(2, B, 12), z(B, V), z(B, V), z(B) + 0.5
        out = {}
        out["step"], out["loop"], out["drawn"], out["target"], out["feature"] = ints(B), ints(2, B), ints(B), ints(B), ints(B)
        ctx.draft_step(Wg, hg, one, one, params, 0.5, 4, out["step"], conf[0], halt[0], feats=feats[0])
        numbers = [torch.isfinite(feats[0][out["step"] >= 0]).all()]
        ctx.draft_loop(Wg, torch.stack([hg, hg]), one, params, 0.0, 2, out["loop"], conf, halt, ints(B), feats=feats)
        numbers.append(torch.isfinite(feats[out["loop"] >= 0]).all())
        # (the CUDA-core kernel leaves out the 32 logits beside an infinite one, but not that one: its features say so)
        assert all(map(bool, numbers)) or path == 1
        ctx.draft_step_sample(Wg, hg, one, one, params, 0.5, 4, u, out["drawn"], conf[0], halt[0], y)
        ctx.verify_sample_ragged(Wg, hg, None, None, None, B, B, None, u, ints(B), ints(B), y, target_ids=out["target"])
        ctx.extract_features(Wg, hg, Wg, hg, one, feats[0], feats[1], z(B), halt[0], out["feature"], ints(B), y, y2)
        assert ctx.device_status() == 0
        return out

    best = (h.double() @ W.double().T).argmax(-1).to(torch.int32)
    good = torch.arange(B) != bad
    for name, token in every_pass(W.cuda(), h.cuda()).items():
        token = token.cpu()
        assert bool((token[..., bad] == -1).all()), name
        if name != "drawn":
            assert torch.equal(token[..., good], best[good].expand_as(token[..., good])), name
    W[V // 3], W[V // 3, 3] = 0.0, float("inf")
    for name, token in every_pass(W.cuda(), h.cuda()).items():
        assert bool(((token >= -1) & (token < V)).all()), name
    ctx.close()


# slabs whose length is and is not a multiple of four, rows of V floats that are not 16-byte aligned, one to many CTAs a row, more
# rows than a grid's second dimension has room for
@pytest.mark.parametrize("V,B", [(7, 1), (4096, 1), (4099, 3), (30002, 2), (30000, 40), (5001, 150), (7, 65600)])
def test_draw_finds_the_entry_that_holds_the_target(V, B):
    d = 24
    W, h = inputs.lm_head(V, d, seed=V, std=0.3).cuda(), inputs.hidden(B, d, seed=B).cuda()
    clf = to_gpu_clf(make_clf(8, seed=4))
    ctx = binding.Context(V, d, 8, max_batch=B, max_rows=8, clf_hidden=8)
    i32 = dict(dtype=torch.int32, device="cuda")
    one, token = torch.ones(B, **i32), torch.zeros(B, **i32)
    conf, p_tok = torch.zeros(B, device="cuda"), torch.zeros(B, device="cuda")
    halt, probs = torch.zeros(B, dtype=torch.uint8, device="cuda"), torch.zeros(B, V, device="cuda")
    logits = h.double() @ W.double().T
    for u_all in (0.0, 0.37, float(np.nextafter(np.float32(1), np.float32(0)))):
        u = torch.full((B,), u_all, device="cuda")
        ctx.draft_step_sample(W, h, one, one, clf, 0.5, 4, u, token, conf, halt, probs, p_token=p_tok)
        torch.cuda.synchronize()
        y = torch.softmax(logits, -1)
        assert float((probs.double() - y).abs().max()) < 2e-3
        cdf = torch.cumsum(y, -1)
        t = token.long()[:, None]
        hi, lo = cdf.gather(1, t)[:, 0], (cdf.gather(1, t) - y.gather(1, t))[:, 0]
        # the running sums are of fp32 exponentials: 2e-5 of the total, the tolerance of every draw
        assert bool(((lo <= u_all + 2e-5) & (hi >= u_all - 2e-5)).all())
        assert torch.equal(p_tok, probs.gather(1, t)[:, 0])
    assert ctx.device_status() == 0
    ctx.close()


def _verification_agrees(oracle, V, B, R, d, path=0):
    sl = np.full(B, R // B - 1, dtype=np.int32)
    sl[-1] += R - int((sl + 1).sum())
    off = inputs.row_offsets(torch.from_numpy(sl)).numpy()
    W, H = inputs.lm_head(V, d, seed=R, std=0.1), inputs.hidden(R, d, seed=R + d)
    free = oracle.verify_ragged(_bits(W), _bits(H), np.zeros(R - B, np.int32), off, nthreads=8)
    clean = np.concatenate([free.target_ids[off[b]:off[b + 1] - 1] for b in range(B)]).astype(np.int32)
    draft = inputs.corrupt_ids(torch.from_numpy(clean), 0.02, V, seed=R).numpy()
    ref = oracle.verify_ragged(_bits(W), _bits(H), draft, off, nthreads=8)
    ctx = binding.Context(V, 8, d, max_batch=B, max_rows=R)
    if path:
        ctx.set_kernel_path(path)
    got = gpu_verify(ctx, W.cuda(), H, draft, row_off=off)
    check_verify(got, ref, off, draft, near_tie_ids(oracle, _bits(W), _bits(H), ref.gap))
    assert ctx.device_status() == 0
    ctx.close()


# 1, 2, 3, 4 and 5 tiles of hidden rows, each just full and with one row more; short and long contractions
@pytest.mark.parametrize("R", [127, 128, 129, 256, 257, 384, 385, 512, 513])
@pytest.mark.parametrize("d", [64, 2048])
def test_verification_at_the_edges_of_the_tiles_of_hidden_rows(oracle, R, d):
    _verification_agrees(oracle, 700, 7, R, d)


# as many tiles of hidden rows as SMs, one more (two tiles to a CTA), as many as that takes, and one more (CUDA cores)
@pytest.mark.parametrize("tiles_per_sm,extra", [(1, 0), (1, 1), (2, 0), (2, 1)])
@pytest.mark.parametrize("fixed_shape", [False, True])
def test_verification_of_more_rows_than_the_sms_have_tiles_for(tiles_per_sm, extra, fixed_shape):
    R, V, d, SL = 128 * _sms() * tiles_per_sm + extra, 300, 8, 3
    R = R if not fixed_shape else (R + SL) // (SL + 1) * (SL + 1)
    B = R // (SL + 1)
    W, H = inputs.lm_head(V, d, seed=1, std=0.3).cuda(), inputs.hidden(R, d, seed=2).cuda()
    logits = H.double() @ W.double().T
    free = logits.argmax(-1).to(torch.int32)
    z = lambda *s: torch.zeros(*s, dtype=torch.int32, device="cuda")
    ctx = binding.Context(V, 8, d, max_batch=B, max_rows=R)
    n_acc, nxt = z(B), z(B)
    if fixed_shape:
        sl = (torch.arange(B, device="cuda") % (SL + 1)).to(torch.int32)
        tids, off = torch.full((B, SL + 1), -1, dtype=torch.int32, device="cuda"), z(B + 1)
        ctx.verify_sl(W, H, free.view(B, SL + 1)[:, :SL].contiguous(), SL, 1, sl, B, SL, n_acc, nxt, target_ids=tids, row_off=off)
        counts = torch.arange(SL + 1, device="cuda")[None] <= sl[:, None]
        assert torch.equal(off[1:], torch.cumsum(sl + 1, 0).to(torch.int32))
    else:   # the last sequence takes the rows that are left over
        off = torch.arange(B + 1, dtype=torch.int32, device="cuda") * (SL + 1)
        off[-1] = R
        rows = torch.ones(R, dtype=torch.bool, device="cuda")
        rows[(off[1:] - 1).long()] = False
        tids = z(R)
        ctx.verify_ragged(W, H, free[rows], off, B, R, n_acc, nxt, tids)
        sl = off[1:] - off[:-1] - 1
        counts = torch.ones(R, dtype=torch.bool, device="cuda")
    assert ctx.device_status() == 0
    got = tids.reshape(-1)[counts.reshape(-1)].long()
    seen = logits[counts.reshape(-1)]
    # a logit is a sum of 8 products of up to 10 in all, in fp32: 8 * 10 * 2^-24 = 5e-6 at most
    assert float((seen.max(-1).values - seen.gather(1, got[:, None])[:, 0]).max()) < 1e-5
    gap = logits.topk(2, -1).values
    if float((gap[:, 0] - gap[:, 1]).min()) > 1e-5:
        assert torch.equal(n_acc, sl)
    else:   # (a row that ties may end its sequence's prefix)
        assert float((n_acc == sl).float().mean()) > 0.99
    ctx.close()


@pytest.mark.parametrize("B,SL", [(700, 0), (350, 1)])
def test_fixed_shape_verification_is_bounded_by_its_rows_alone(B, SL):
    """More sequences than the context's max_batch, which bounds the draft steps only; more than one tile of rows, so that the
    rows that count are packed and B + 1 offsets are kept in scratch."""
    V, d, R = 500, 16, B * (SL + 1)
    W, H = inputs.lm_head(V, d, seed=3, std=0.3).cuda(), inputs.hidden(R, d, seed=4).cuda()
    z = lambda *s: torch.zeros(*s, dtype=torch.int32, device="cuda")
    ctx = binding.Context(V, 8, d, max_batch=1, max_rows=R)
    n_acc, nxt, off, tids = z(B), z(B), z(B + 1), torch.full((B, SL + 1), -1, dtype=torch.int32, device="cuda")
    sl = (torch.arange(B, device="cuda") % (SL + 1)).to(torch.int32)
    ids = torch.full((B, max(SL, 1)), -1, dtype=torch.int32, device="cuda")   # no draft token is the target's
    for _ in range(2):
        ctx.verify_sl(W, H, ids if SL else None, SL, 1, sl, B, SL, n_acc, nxt, target_ids=tids, row_off=off)
    assert ctx.device_status() == 0
    assert torch.equal(off[1:], torch.cumsum(sl + 1, 0).to(torch.int32)) and not bool(n_acc.any())
    logits = (H.double() @ W.double().T).view(B, SL + 1, V)
    best = logits.max(-1).values
    # a logit is a sum of 16 products of up to 20 in all, in fp32: 16 * 20 * 2^-24 = 2e-5 at most
    for j in range(SL + 1):
        on = sl >= j
        got = tids[on, j].long()
        assert float((best[on, j] - logits[on, j].gather(1, got[:, None])[:, 0]).max()) < 2e-5
        assert bool((tids[~on, j] == -1).all())
    assert torch.equal(nxt, tids[:, 0])
    ctx.close()


# vocabulary rows on the lanes: a block of 128 not full, full, two of them, several tiles; 16 rows per column group and one more
@pytest.mark.parametrize("rows_per_sm", [2, 128, 129, 256, 257, 600])
@pytest.mark.parametrize("R", [2, 16, 17, 32, 33])
def test_verification_of_few_rows_at_the_edges_of_its_tiling(oracle, rows_per_sm, R):
    _verification_agrees(oracle, _sms() * rows_per_sm - 1, 1, R, 24, path=2)


# ... with a column per hidden row and the keys in shared memory: two tiles in flight and one, and the row counts around the rule
@pytest.mark.parametrize("rows_per_sm", [2, 128, 129, 600])
@pytest.mark.parametrize("R", [34, 64, 65, 129, 144, 160, 161])
def test_verification_with_a_column_per_row_at_the_edges_of_its_tiling(oracle, rows_per_sm, R):
    _verification_agrees(oracle, _sms() * rows_per_sm - 1, 3, R, 24, path=2)


# a box below 128 rows, exactly 128, both halves, two and four tiles of it, and beyond what the persistent kernel takes: the steps of a
# head each go to that kernel, in one launch, up to 1024 rows per SM, and those of one head share launches of the other one
@pytest.mark.parametrize("rows_per_sm", [3, 128, 129, 256, 257, 1024, 1025])
@pytest.mark.parametrize("B", [1, 2, 4])
@pytest.mark.parametrize("heads", [1, 3])
def test_draft_phase_at_the_edges_of_its_tiling(oracle, rows_per_sm, B, heads):
    V, d, S = _sms() * rows_per_sm - 1, 16, 3
    W, h = inputs.lm_head(V, d, seed=V, std=0.3), inputs.hidden(S * B, d, seed=B).view(S, B, d)
    params = make_clf(16, seed=6)
    ctx = binding.Context(V, d, 8, max_batch=B, max_rows=8, clf_hidden=16)
    z = lambda *s, t=torch.int32: torch.zeros(*s, dtype=t, device="cuda")
    token, conf, halt = z(S, B), z(S, B, t=torch.float32), z(S, B, t=torch.uint8)
    feats, sl, pos0 = z(S, B, binding.NFEAT, t=torch.float32), z(B), torch.arange(5, 5 + B, dtype=torch.int32)
    W_D = W.cuda() if heads == 1 else torch.stack([W] * S).cuda()
    ctx.draft_loop(W_D, h.cuda(), pos0.cuda(), to_gpu_clf(params), 0.0, S, token, conf, halt, sl, feats=feats,
                   w_step_stride=0 if heads == 1 else V * d * 2)
    torch.cuda.synchronize()
    assert sl.tolist() == [S] * B
    # scratch for eight rows: all three steps in a launch, or two and one
    assert ctx.launch_count() == ((1 if B < 4 else 2) if heads == 1 else (1 if rows_per_sm <= 1024 else S))
    for i in range(S):
        ref = oracle.draft_step(_bits(W), _bits(h[i]), pos0.numpy() + i + 1, np.full(B, i + 1, np.int32),
                                to_oracle_clf(oracle, params), 0.0, S, nthreads=8)
        got = dict(token=token[i].cpu().numpy(), conf=conf[i].cpu().numpy(), halt=halt[i].cpu().numpy(),
                   feats=feats[i].cpu().numpy(), probs=None)
        _check_draft_and_each_probability(got, ref, 0.0)
    assert ctx.device_status() == 0
    ctx.close()


@pytest.mark.parametrize("V,N", [(1000, 3), (1001, 130)])
def test_features_with_rows_that_are_and_are_not_aligned(oracle, V, N):
    d_D, d_T = 16, 24
    W_D, W_T = inputs.lm_head(V, d_D, seed=1, std=0.3), inputs.lm_head(V, d_T, seed=2, std=0.3)
    H_D, H_T = inputs.hidden(N, d_D, seed=3), inputs.hidden(N, d_T, seed=4)
    ctx = binding.Context(V, d_D, d_T, max_batch=1, max_rows=N)
    z = lambda *s, t=torch.float32: torch.zeros(*s, dtype=t, device="cuda")
    fD, fT, tv, lab = z(N, 12), z(N, 12), z(N), z(N, t=torch.uint8)
    tD, tT, yD, yT = z(N, t=torch.int32), z(N, t=torch.int32), z(N, V), z(N, V)
    ctx.extract_features(W_D.cuda(), H_D.cuda(), W_T.cuda(), H_T.cuda(), torch.ones(N, dtype=torch.int32, device="cuda"),
                         fD, fT, tv, lab, tD, tT, yD, yT)
    torch.cuda.synchronize()
    want = [torch.softmax(H.double() @ W.double().T, -1) for H, W in ((H_D, W_D), (H_T, W_T))]
    for y, w in zip((yD, yT), want):
        assert float((y.cpu().double() - w).abs().max()) < 2e-3
    # half a sum of V differences of fp32 probabilities (rows that sum to one): 1e-5
    assert float((tv.cpu().double() - 0.5 * (want[0] - want[1]).abs().sum(-1)).abs().max()) < 1e-5
    assert torch.equal(lab.cpu().bool(), tD.cpu() == tT.cpu())
    assert ctx.device_status() == 0
    ctx.close()


# Few hidden rows, the vocabulary on the lanes: the rows a warp holds (8, 16, 32), tiles of exactly 32 and 128 vocabulary rows
# and one more or less, more tiles than accumulators (2100 rows per SM: 17 tiles), CTAs without a vocabulary row
@pytest.mark.parametrize("rows_per_sm,extra,B", [(31, 0, 1), (32, 1, 8), (33, 0, 9), (127, 3, 16), (128, 1, 17), (129, 0, 32),
                                                 (257, -2, 33), (2100, 5, 3), (2100, 0, 20), (1, -100, 2)])
def test_few_rows_at_the_edges_of_their_tiling(oracle, rows_per_sm, extra, B):
    V, d = _sms() * rows_per_sm + extra, 40 if rows_per_sm < 1000 else 16
    W, h = inputs.lm_head(V, d, seed=V + B, std=0.3), inputs.hidden(B, d, seed=B)
    params = make_clf(16, seed=1)
    pos, nd = np.arange(1, B + 1, dtype=np.int32), (np.arange(B, dtype=np.int32) % 4) + 1
    active = (np.arange(B) % 5 != 2).astype(np.uint8)
    ctx = binding.Context(V, d, 8, max_batch=B, max_rows=8, clf_hidden=16)
    Wg, clf = W.cuda(), to_gpu_clf(params)
    for act in (None, active, None):
        got = gpu_draft_step(ctx, Wg, h, pos, nd, clf, 0.5, 3, active=act, want_probs=True)
        ref = oracle.draft_step(_bits(W), _bits(h), pos, nd, to_oracle_clf(oracle, params), 0.5, 3, active=act, want_probs=True, nthreads=8)
        _check_draft_and_each_probability(got, ref, 0.5, active=act)
    assert ctx.device_status() == 0
    ctx.close()


# Tiles of hidden rows in pairs of CTAs (test_host_rules.py has the sizes at which they are taken): full and part-filled pairs, a last
# pair with one tile, kept logits; one size at which the tiles stay single
@pytest.mark.parametrize("N,V,d", [(129, 8000, 2048), (256, 8000, 2048), (257, 401, 2056), (400, 8003, 2048), (520, 12300, 2048),
                                   (1000, 300, 2048)])
def test_feature_extraction_by_pairs_of_ctas(N, V, d):
    """The ten probabilities, the distribution and the token of every row against float64.  A logit is 128 additions of 16 products
    each: a partial sum is below 4 (standard deviation 0.02 * 2048 ^ 0.5 = 0.9) and loses at most 2^-23 of it per addition, 6.1e-5 in all;
    the products, below 0.4, lose at most 16 * 2^-24 of that, 4.9e-5 in all.  (Measured: 1.4e-5.)"""
    tol = 1.2e-4
    ctx = binding.Context(V, 64, d, max_batch=1, max_rows=N)
    W_D, H_D = inputs.lm_head(V, 64, seed=1).cuda(), inputs.hidden(N, 64, seed=2).cuda()
    W_T, H_T = inputs.lm_head(V, d, seed=3).cuda(), inputs.hidden(N, d, seed=4).cuda()
    z = lambda *s, t=torch.float32: torch.zeros(*s, dtype=t, device="cuda")
    pos, tv, label = torch.arange(N, dtype=torch.int32, device="cuda"), z(N), z(N, t=torch.uint8)
    fD, fT, tD, tT, yD, yT = z(N, 12), z(N, 12), z(N, t=torch.int32), z(N, t=torch.int32), z(N, V), z(N, V)
    for _ in range(2):
        ctx.extract_features(W_D, H_D, W_T, H_T, pos, fD, fT, tv, label, tD, tT, yD, yT)
    assert ctx.device_status() == 0
    ctx.close()
    for W, H, feats, token, y in ((W_D, H_D, fD, tD, yD), (W_T, H_T, fT, tT, yT)):
        logits = H.double() @ W.double().T
        want = torch.softmax(logits, -1)
        assert float((y.double() / want - 1).abs().max()) < tol
        assert float((feats[:, :10].double() / want.topk(10, -1).values - 1).abs().max()) < tol
        picked = logits.gather(1, token.long()[:, None])[:, 0]
        assert float((logits.max(-1).values - picked).max()) < 2 * tol
    assert float((tv.double() - 0.5 * (yD.double() - yT.double()).abs().sum(-1)).abs().max()) < 1e-5


def _ragged_verification(oracle, V, d, sls, seed, ctx):
    """One verification with look-aheads `sls`, most offered ids the target's own, against the oracle."""
    off = np.concatenate([[0], np.cumsum(np.asarray(sls) + 1)]).astype(np.int32)
    R, B = int(off[-1]), len(sls)
    W, H = inputs.lm_head(V, d, seed=seed, std=0.3), inputs.hidden(R, d, seed=seed + 1)
    free = oracle.verify_ragged(_bits(W), _bits(H), np.zeros(R - B, np.int32), off, nthreads=16)
    keep = np.ones(R, bool)
    keep[off[1:] - 1] = False
    draft = inputs.corrupt_ids(torch.from_numpy(free.target_ids[keep].astype(np.int32)), 0.2, V, seed=seed).numpy()
    ref = oracle.verify_ragged(_bits(W), _bits(H), draft, off, nthreads=16)
    got = gpu_verify(ctx, W.cuda(), H, draft, row_off=off)
    check_verify(got, ref, off, draft, near_tie_ids(oracle, _bits(W), _bits(H), ref.gap))


# CTAs that finish eight sequences each: one of them, full, one sequence more, the most there are and more than that; the
# second call of a context finds keys and counters as the first has left them
@pytest.mark.parametrize("B", [1, 8, 9, 33, 64, 65])
def test_verification_finished_by_ctas_of_their_own(oracle, B):
    ctx = binding.Context(3001, 8, 72, max_batch=B, max_rows=4 * B)
    for k in range(2):
        _ragged_verification(oracle, 3001, 72, [(b + k) % 4 for b in range(B)], 50 + B + k, ctx)
    assert ctx.device_status() == 0
    ctx.close()


# Pairs of CTAs (test_host_rules.py has the sizes at which they are taken): two tiles of 128 rows (the second nearly empty, full), four,
# ten and an odd number of them; one and several vocabulary tiles per pair; a pair with two tiles of 256 rows
@pytest.mark.parametrize("V,rows,d", [(300, 129, 1032), (300, 256, 1032), (2500, 500, 2056), (20000, 180, 1032), (400, 1160, 2056),
                                      (700, 1409, 2056), (9000, 1409, 1032), (4000, 1409, 4104)])
def test_verification_by_pairs_of_ctas(oracle, V, rows, d):
    _verification_agrees(oracle, V, rows // 8, rows, d)
