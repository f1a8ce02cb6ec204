"""What the performance of this framework is measured on.

A speculative decoder calls the library once per draft token (draft_step), once per verification (verify_ragged),
or once per iteration (iteration, iteration_host); decoding at temperature 1 takes the sampling variants of the two
tails, and training the halt classifier takes extract_features.  The listed cases are those calls at the head shapes
of inputs.WORKLOADS and of the benchmark, from one sequence to 256; draw() gives further ones of the same ranges
(vocabulary 4000 .. 49152, odd sizes included; hidden widths, multiples of 8, 256 .. 1024 for the draft model and
1024 .. 6144 for the target; 1 .. 256 sequences; look-aheads 1 .. 16).

Every look-ahead is decided by the halt classifier itself: one of its units watches the position feature and ends the
drafting of a sequence where the case wants it, the other units are the usual random initialisation.
"""
import math

import torch

from paper_2405_04304_b200 import binding, inputs

CLF_HIDDEN = 64
STOP_AT = 1000      # position at which the classifier's score falls below tau
TAU = 0.5


def listed():
    return [
        # One draft token of one sequence: the smallest call, made for every token a single-user decoder drafts.
        dict(name="draft_1", kind="draft", V=32000, d=768, B=1, active=1),
        # A handful of sequences and a vocabulary that is no round number (tokens added to a tokeniser).
        dict(name="draft_7_odd", kind="draft", V=40011, d=768, B=7, active=7),
        # A serving batch: some sequences have stopped drafting and are masked.
        dict(name="draft_64_masked", kind="draft", V=32000, d=768, B=64, active=48),
        # A drafted token at temperature 1: the distribution is kept for the verification.
        dict(name="draft_sample_8", kind="draft_sample", V=49152, d=768, B=8),
        # One verification of one sequence, full look-ahead.
        dict(name="verify_1", kind="verify", V=32000, d=5120, B=1, sl=10),
        # A small batch, every sequence with a look-ahead of its own, and the smaller target.
        dict(name="verify_20_ragged", kind="verify", V=32000, d=2048, B=20, sl=10),
        # Verification at temperature 1 of a few sequences.
        dict(name="verify_sample_4", kind="verify_sample", V=32000, d=5120, B=4, sl=8),
        # One whole iteration of one sequence on the device: four tokens drafted of ten allowed.
        dict(name="iteration_1", kind="iteration", V=32000, d_D=768, d_T=5120, B=1, sl_max=10, sl=4),
        # The same for a decoder whose hidden states arrive in host memory, with the larger heads.
        dict(name="iteration_host_1", kind="iteration_host", V=49152, d_D=768, d_T=6144, B=1, sl_max=10, sl=3),
        # A serving batch, look-aheads spread over 1 .. 10.
        dict(name="iteration_64", kind="iteration", V=32000, d_D=768, d_T=5120, B=64, sl_max=10, sl=10),
        # The largest batch, look-aheads spread over 1 .. 16.
        dict(name="iteration_256", kind="iteration", V=49152, d_D=768, d_T=6144, B=256, sl_max=16, sl=16),
        # Training data for the classifier: a thousand positions through both heads.
        dict(name="features_1000", kind="features", V=32000, d_D=768, d_T=5120, N=1000),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["draft", "draft", "draft_sample", "verify", "verify", "verify_sample", "iteration", "iteration",
                       "iteration_host", "features"])
    V = log_int(4000, 49152)
    d_D, d_T = 8 * rng.randint(32, 128), 8 * log_int(128, 768)
    if kind == "draft":
        B = log_int(1, 256)
        return dict(kind=kind, V=V, d=d_D, B=B, active=rng.choice([B, max(1, (3 * B) // 4)]))
    if kind == "draft_sample":
        return dict(kind=kind, V=V, d=d_D, B=log_int(1, 64))
    if kind == "verify":
        return dict(kind=kind, V=V, d=d_T, B=log_int(1, 256), sl=rng.randint(1, 16))
    if kind == "verify_sample":
        return dict(kind=kind, V=V, d=d_T, B=log_int(1, 16), sl=rng.randint(1, 16))
    if kind == "features":
        return dict(kind=kind, V=V, d_D=d_D, d_T=d_T, N=log_int(16, 1000))
    sl_max = rng.randint(2, 16)
    B = log_int(1, 256) if kind == "iteration" else log_int(1, 16)
    return dict(kind=kind, V=V, d_D=d_D, d_T=d_T, B=B, sl_max=sl_max, sl=rng.randint(1, sl_max))


# ------------------------------------------------------------------------------------------------ inputs
def look_aheads(B, sl):
    """Look-aheads of the sequences: sl, sl - 1, .. 1, sl, ..; prepare() shuffles them."""
    return [sl - b % sl for b in range(B)]


def _rows(B, sl):
    return sum(look_aheads(B, sl)) + B


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _shuffled_look_aheads(case, seed):
    sl = torch.tensor(look_aheads(case["B"], case["sl"]), dtype=torch.int32)
    g = torch.Generator()
    g.manual_seed(seed)
    return sl[torch.randperm(case["B"], generator=g)]


def _classifier(seed):
    """Random initialisation; the position feature goes to unit 0 alone, which lowers the score from +8 to -8 (plus
    what the other units say, about +-1) at position STOP_AT."""
    W1, b1, w2, b2 = inputs.classifier_params(CLF_HIDDEN, seed)
    W1[:, 11] = 0.0
    W1[0] = 0.0
    W1[0, 11], b1[0], w2[0], b2[0] = 1.0, -(STOP_AT - 1.0), -16.0, 8.0
    return binding.Classifier(W1.cuda(), b1.cuda(), w2.cuda(), b2.cuda())


def _logits(W, H, rows=1024):
    Wf = W.float()
    return torch.cat([H[r:r + rows].float() @ Wf.T for r in range(0, H.shape[0], rows)], 0)


def _greedy(W, H, rows=1024):
    Wf = W.float()
    return torch.cat([(H[r:r + rows].float() @ Wf.T).argmax(-1) for r in range(0, H.shape[0], rows)], 0).to(torch.int32)


def _corrupt(ids, p, V, g):
    """The ids a draft model would offer: each of the target's own tokens replaced by a random one with probability p."""
    coin = torch.rand(ids.shape, generator=g, device="cuda")
    other = torch.randint(0, V, ids.shape, generator=g, device="cuda", dtype=torch.int32)
    return torch.where(coin < p, other, ids)


def _out(shape, dtype):
    return torch.zeros(shape, dtype=dtype, device="cuda")


def prepare(case, seed):
    s = lambda *tags: inputs.sub_seed(seed, *tags)
    kind, V = case["kind"], case["V"]
    g = _gen(s(1))
    i32, f32, u8 = torch.int32, torch.float32, torch.uint8
    st = dict(kind=kind, case=case)

    if kind in ("draft", "draft_sample"):
        B, d = case["B"], case["d"]
        active = None
        if case.get("active", B) < B:
            active = torch.ones(B, dtype=u8, device="cuda")
            active[torch.randperm(B, generator=g, device="cuda")[case["active"]:]] = 0
        st.update(ctx=binding.Context(V, d, 8, max_batch=B, max_rows=B, clf_hidden=CLF_HIDDEN),
                  W=inputs.lm_head(V, d, s(2), device="cuda"), h=inputs.hidden(B, d, s(3), device="cuda"),
                  clf=_classifier(s(4)), active=active,
                  pos=torch.randint(1, 2 * STOP_AT, (B,), generator=g, device="cuda", dtype=i32),
                  n_drafted=torch.randint(1, 11, (B,), generator=g, device="cuda", dtype=i32),
                  token=_out(B, i32), conf=_out(B, f32), halt=_out(B, u8), feats=_out((B, binding.NFEAT), f32))
        if kind == "draft_sample":
            st.update(u=torch.rand(B, generator=g, device="cuda"), p_token=_out(B, f32), probs=_out((B, V), f32))
        return st

    if kind in ("verify", "verify_sample"):
        B, d, sl = case["B"], case["d"], case["sl"]
        sls = _shuffled_look_aheads(case, s(5))
        off = inputs.row_offsets(sls)
        R = int(off[-1])
        W, H = inputs.lm_head(V, d, s(2), device="cuda"), inputs.hidden(R, d, s(3), device="cuda")
        checked = torch.ones(R, dtype=torch.bool)
        checked[(off[1:] - 1).long()] = False            # the last row of a sequence has no draft token to check
        rows = checked.nonzero().flatten().cuda()
        st.update(ctx=binding.Context(V, 8, d, max_batch=B, max_rows=R), W=W, H=H, off=off.cuda(), B=B, R=R,
                  n_accept=_out(B, i32), next=_out(B, i32), target_ids=_out(R, i32))
        if kind == "verify":
            st["ids"] = _corrupt(_greedy(W, H[rows]), 0.2, V, g)
            return st
        # a draft distribution near the target's, and tokens drawn from it
        y = torch.softmax(_logits(W, H[rows]) + torch.randn((R - B, V), generator=g, device="cuda"), -1)
        probs = _out((sl, B, V), f32)
        b = torch.repeat_interleave(torch.arange(B), sls.long()).cuda()
        i = torch.cat([torch.arange(int(n)) for n in sls]).cuda()
        probs[i, b] = y
        st.update(ids=torch.multinomial(y, 1, generator=g).flatten().to(i32), probs=probs,
                  u_accept=torch.rand(R - B, generator=g, device="cuda"), u_sample=torch.rand(B, generator=g, device="cuda"),
                  y_T=_out((R, V), f32))
        return st

    if kind == "features":
        N = case["N"]
        st.update(ctx=binding.Context(V, case["d_D"], case["d_T"], max_batch=1, max_rows=N),
                  W_D=inputs.lm_head(V, case["d_D"], s(2), device="cuda"), H_D=inputs.hidden(N, case["d_D"], s(3), device="cuda"),
                  W_T=inputs.lm_head(V, case["d_T"], s(4), device="cuda"), H_T=inputs.hidden(N, case["d_T"], s(5), device="cuda"),
                  pos=torch.randint(1, 2 * STOP_AT, (N,), generator=g, device="cuda", dtype=i32),
                  feats_D=_out((N, binding.NFEAT), f32), feats_T=_out((N, binding.NFEAT), f32), tv=_out(N, f32),
                  label=_out(N, u8), token_D=_out(N, i32), token_T=_out(N, i32), y_D=_out((N, V), f32), y_T=_out((N, V), f32))
        return st

    # iteration, iteration_host
    B, S = case["B"], case["sl_max"]
    sls = _shuffled_look_aheads(case, s(5))
    W_T = inputs.lm_head(V, case["d_T"], s(4), device="cuda")
    H_T = inputs.hidden(B * (S + 1), case["d_T"], s(6), device="cuda")
    ids = _greedy(W_T, H_T).view(B, S + 1)[:, :S].contiguous()
    st.update(ctx=binding.Context(V, case["d_D"], case["d_T"], max_batch=B, max_rows=B * (S + 1), clf_hidden=CLF_HIDDEN),
              W_D=inputs.lm_head(V, case["d_D"], s(2), device="cuda"), W_T=W_T, S=S,
              h_D=inputs.hidden(S * B, case["d_D"], s(3), device="cuda").view(S, B, case["d_D"]),
              H_T=H_T.view(B, S + 1, case["d_T"]), ids=_corrupt(ids, 0.2, V, g), clf=_classifier(s(7)),
              pos0=(STOP_AT - sls).cuda(),
              token=_out((S, B), i32), conf=_out((S, B), f32), halt=_out((S, B), u8), sl=_out(B, i32),
              n_accept=_out(B, i32), bonus=_out(B, i32), pos_next=_out(B, i32))
    if kind == "iteration":
        st.update(feats=_out((S, B, binding.NFEAT), f32), target_ids=torch.full((B, S + 1), -1, dtype=i32, device="cuda"),
                  row_off=_out(B + 1, i32))
    else:   # the heads and the classifier stay on the device, everything else lives in pinned host memory
        for k in ("h_D", "H_T", "ids", "pos0", "token", "conf", "halt", "sl", "n_accept", "bonus", "pos_next"):
            st[k] = st[k].cpu().pin_memory()
    return st


# ------------------------------------------------------------------------------------------------ one pass
def run(st):
    kind, ctx = st["kind"], st["ctx"]
    if kind == "draft":
        ctx.draft_step(st["W"], st["h"], st["pos"], st["n_drafted"], st["clf"], TAU, 10, st["token"], st["conf"], st["halt"],
                       active=st["active"], feats=st["feats"])
        return st["token"], st["conf"], st["halt"], st["feats"]
    if kind == "draft_sample":
        ctx.draft_step_sample(st["W"], st["h"], st["pos"], st["n_drafted"], st["clf"], TAU, 10, st["u"], st["token"],
                              st["conf"], st["halt"], st["probs"], p_token=st["p_token"], feats=st["feats"])
        return st["token"], st["p_token"], st["conf"], st["halt"], st["feats"], st["probs"]
    if kind == "verify":
        ctx.verify_ragged(st["W"], st["H"], st["ids"], st["off"], st["B"], st["R"], st["n_accept"], st["next"],
                          st["target_ids"])
        return st["n_accept"], st["next"], st["target_ids"]
    if kind == "verify_sample":
        ctx.verify_sample_ragged(st["W"], st["H"], st["ids"], st["probs"], st["off"], st["B"], st["R"], st["u_accept"],
                                 st["u_sample"], st["n_accept"], st["next"], st["y_T"], target_ids=st["target_ids"])
        return st["n_accept"], st["next"], st["target_ids"], st["y_T"]
    if kind == "features":
        ctx.extract_features(st["W_D"], st["H_D"], st["W_T"], st["H_T"], st["pos"], st["feats_D"], st["feats_T"], st["tv"],
                             st["label"], st["token_D"], st["token_T"], st["y_D"], st["y_T"])
        return (st["feats_D"], st["feats_T"], st["tv"], st["label"], st["token_D"], st["token_T"], st["y_D"], st["y_T"])
    if kind == "iteration":
        ctx.iteration(st["W_D"], st["h_D"], st["W_T"], st["H_T"], st["pos0"], st["clf"], TAU, st["S"], st["token"],
                      st["conf"], st["halt"], st["sl"], st["n_accept"], st["bonus"], draft_ids=st["ids"], feats=st["feats"],
                      target_ids=st["target_ids"], row_off=st["row_off"], pos_next=st["pos_next"])
        return (st["token"], st["conf"], st["halt"], st["feats"], st["sl"], st["n_accept"], st["bonus"], st["target_ids"],
                st["row_off"], st["pos_next"])
    ctx.iteration_host(st["W_D"], st["h_D"], st["W_T"], st["H_T"], st["pos0"], st["clf"], TAU, st["S"], st["token"],
                       st["conf"], st["halt"], st["sl"], st["n_accept"], st["bonus"], draft_ids=st["ids"],
                       pos_next=st["pos_next"])
    return (st["token"], st["conf"], st["halt"], st["sl"], st["n_accept"], st["bonus"], st["pos_next"])


# ------------------------------------------------------------------------------------------------ floors
def work(case):
    """Heads and hidden states in bf16 read once (a batch of draft steps shares one head), fp32 distributions written
    once where the call returns them; two operations per multiply-add of the projections."""
    kind, V = case["kind"], case["V"]
    if kind in ("draft", "draft_sample"):
        B, d = case["B"], case["d"]
        n = case.get("active", B)
        kept = 4 * B * V if kind == "draft_sample" else 0
        return dict(bytes=2 * d * (V + n) + kept + 64 * n, flops=2 * n * V * d)
    if kind in ("verify", "verify_sample"):
        B, d = case["B"], case["d"]
        R = _rows(B, case["sl"])
        # y_T written; the draft distribution of the row a token is drawn from, read
        kept = 4 * V * (R + B) if kind == "verify_sample" else 0
        return dict(bytes=2 * d * (V + R) + kept + 12 * R, flops=2 * R * V * d)
    if kind == "features":
        N, d = case["N"], case["d_D"] + case["d_T"]
        return dict(bytes=2 * d * (V + N) + 8 * N * V + 128 * N, flops=2 * N * V * d)
    drafted = sum(look_aheads(case["B"], case["sl"]))
    R = drafted + case["B"]
    return dict(bytes=2 * case["d_D"] * (V + drafted) + 2 * case["d_T"] * (V + R) + 64 * R,
                flops=2 * V * (drafted * case["d_D"] + R * case["d_T"]))


def tolerance(case):
    """fp32 accumulation of bf16 products in any order, fast exponentials; two ids may change places where their logits
    agree to fp32 rounding, a drawn token where the uniform falls on the edge of its interval."""
    if case["kind"] == "verify":
        return dict(rel=0.0, differ=2e-3)
    return dict(rel=2e-5, max=1e-3, differ=5e-3 if "sample" in case["kind"] else 2e-3)
