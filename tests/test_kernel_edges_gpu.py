"""GPU parity at the sizes where a kernel or a branch of its dispatch can go wrong: edges of its
tiles, remainders, the smallest and the largest of its range.  Oracle, metrics and gates are those
of test_parity_gpu.py."""
import functools
import inspect
import sys
import threading

import pytest
import torch
from torch.utils._python_dispatch import TorchDispatchMode

import oracle
import paper_2409_18747_b200 as cott
from paper_2409_18747_b200 import synth
from test_parity_gpu import (DM_COND_BF16, DM_COND_F32, TOL_STATE_F32, dev, dm_condition, force_group, gate, gate_dm, option)  # noqa: F401
from _metrics import norm_max_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("N,group", [(1, 0), (31, 0), (33, 32), (64, 32), (97, 0), (500, 32), (545, 32), (300, 4096)])
@pytest.mark.parametrize("causal", [True, False])
def test_fp32_walk_chunk_and_group_edges(d, N, group, causal, force_group):
    """The fp32 walk (32 tokens a chunk): single rows, one row short of and one past a chunk, 16 groups
    (each walk sums the partial states before its own), 18 groups (a scan launch does), one group."""
    force_group(group)
    B, H = 2, 3
    c = synth.make_qkv(B, H, N, d, torch.float32, 7100 + N + d, row_lognormal=True, with_do=True)
    args = [dev(c[x]) for x in ("q", "k", "v")]
    o, st = cott.fwd(*args, dev(c["m"]), causal=causal, return_state=True)
    ref_o = oracle.fwd_quadratic(c["q"], c["k"], c["v"], c["m"], None, causal)
    _, ref_state = oracle.fwd_bidir_assoc(c["q"], c["k"], c["v"], c["m"], None)
    assert norm_max_err(st, ref_state) <= TOL_STATE_F32
    dq, dk, dv, dm = cott.bwd(*args, dev(c["d_o"]), dev(c["m"]), causal=causal)
    rq, rk, rv, rm = oracle.bwd_quadratic(c["q"], c["k"], c["v"], c["d_o"], c["m"], None, causal)
    if N > 1:
        for x, r in ((o, ref_o), (dq, rq), (dk, rk), (dv, rv)):
            gate(x, r, torch.float32)
        gate_dm(dm, rm, 1e-4, dm_condition(rv, c["v"], c["m"], None), DM_COND_F32)
        return
    # One token (c = 1, dm = 0): every row is one dot product of unit or raw rows times a row, and
    # where that dot product cancels the relative error has no bound.  Absolute: a dot product of d
    # terms is off by at most (d + 8) u |x| |y| (u = 2^-24, the norms and scalings included), and dq,
    # dk go through two of them and a division by the row's norm.
    u = (d + 8) * 2.0 ** -24
    nq, nk, nv, nd = (c[x].double().norm(dim=-1, keepdim=True).numpy() for x in ("q", "k", "v", "d_o"))
    for x, r, bound in ((o, ref_o, nv), (dv, rv, nd), (dq, rq, 2 * nd * nv / nq), (dk, rk, 2 * nd * nv / nk)):
        assert (abs(x.double().cpu().numpy() - r) <= u * bound).all()


def one_token_bounds(got, refs, c):
    """Gradients of a sequence of one token (c = 1), where the relative error of a row has no bound: the rows
    are one product of unit rows with raw rows, and dq, dk lose their part along q or k.  With u = 2^-9 (bf16
    rounding): dV' = (q^ . k^) dO has the roundings of q^, k^, the score and the result, 4 u |dO|; dq^ and dk^
    have two (score, unit row) of |dO| |v|, which the projection can double, and the result's."""
    nq, nk, nv, nd = (c[x].double().norm(dim=-1, keepdim=True).numpy() for x in ("q", "k", "v", "d_o"))
    nq, nk = nq.clip(1e-12), nk.clip(1e-12)
    u = 2.0 ** -9
    for x, r, bound in zip(got, refs, (6 * nd * nv / nq, 6 * nd * nv / nk, 4 * nd)):
        assert (abs(x.double().cpu().numpy() - r) <= u * bound).all()


@pytest.mark.parametrize("N,group", [(1, 0), (127, 0), (128, 0), (129, 0), (257, 0), (400, 128), (900, 256), (700, 128)])
@pytest.mark.parametrize("dk,dv", [(128, 128), (72, 128), (96, 40)])
@pytest.mark.parametrize("causal", [True, False])
def test_backward_d128_chunk_and_group_edges(N, group, dk, dv, causal, force_group):
    """The d = 128 backward (two walks in one launch): one to several chunks, a ragged last one, one
    group, up to four (summed by the walks) and six (scan launches), widths zero-filled to 128."""
    force_group(group)
    B, H = 2, 3
    c = synth.make_qkv(B, H, N, dk, torch.bfloat16, 7300 + N + dk, row_lognormal=True, with_do=True, d_v=dv)
    c["k"][0, 1, N // 2] = 0.0
    args = [dev(c[x]) for x in ("q", "k", "v", "d_o", "m")]
    dq, dk_, dv_, dm = cott.bwd(*args, causal=causal)
    rq, rk, rv, rm = oracle.bwd_quadratic(c["q"], c["k"], c["v"], c["d_o"], c["m"], None, causal)
    if N == 1:
        one_token_bounds((dq, dk_, dv_), (rq, rk, rv), c)
        assert (dm == 0).all() and (rm == 0).all()         # (c = 1: ln 1 = 0)
        return
    # the zero key row's gradient is that of the clamped formula, 1e12 times larger: gated on its own
    z = (0, 1, N // 2)
    assert norm_max_err(dk_[z], rk[z]) <= 1e-2
    dk_[z] = 0.0
    rk[z] = 0.0
    gate(dq, rq, torch.bfloat16); gate(dk_, rk, torch.bfloat16); gate(dv_, rv, torch.bfloat16)
    # dm's error scales with the sum of its absolute terms (see dm_condition): 3e-4 of it at worst
    # over random shapes of this size for bf16 operands
    cond = dm_condition(rv, c["v"], c["m"], None)
    assert (abs(dm.double().cpu().numpy() - rm) <= 1e-3 * cond).all()
    gate_dm(dm, rm, 1e-2, cond, DM_COND_BF16)


@pytest.mark.parametrize("T", [1, 8, 15, 16, 17, 32, 48, 49, 64])
@pytest.mark.parametrize("dk,dv", [(128, 128), (64, 64), (8, 8), (24, 104), (120, 72)])
def test_token_block_edges(T, dk, dv):
    """The token-block kernel (tiles of 16 tokens, strips of 32 value columns, steps of 16 key rows):
    edges of each, with and without a state on either side."""
    B, H = 2, 3
    c = synth.make_qkv(B, H, T, dk, torch.bfloat16, 7500 + T + dk, row_lognormal=True, d_v=dv)
    c["k"][1, 1, T // 2] = 0.0
    s = 300.0
    g = torch.Generator().manual_seed(3)
    state = torch.randn((B, H, dk, dv), generator=g)
    q, k, v, m = (dev(c[x]) for x in ("q", "k", "v", "m"))
    for st in (state, torch.zeros(B, H, dk, dv)):
        given = st is state
        if not given and (dk != dv or T == 1):     # (one token alone: a row of a single term, four roundings deep)
            continue
        o, st_out = cott.fwd_stateful(q, k, v, m, s, state_in=dev(st) if given else None)
        r_o, r_s = oracle.fwd_segment(c["q"], c["k"], c["v"], c["m"], st, torch.tensor([s] * B))
        gate(o, r_o, torch.bfloat16)
        assert norm_max_err(st_out, r_s) <= 1e-2
    o2 = cott.fwd_stateful(q, k, v, m, s, state_in=dev(state), return_state=False)
    assert torch.equal(o2, cott.fwd_stateful(q, k, v, m, s, state_in=dev(state))[0])


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("groups", [2, 4, 5, 9, 10])
def test_forward_walk_sums_or_scans_the_group_states(d, groups, force_group):
    """A causal forward in groups, with and without a state on either side: few groups are summed inside
    the walk (whose last group then writes the state), more by a scan launch."""
    force_group(128)
    B, H, N = 1, 3, 128 * groups - 39
    c = synth.make_qkv(B, H, N, d, torch.bfloat16, 7700 + N + d)
    state = torch.randn((B, H, d, d), generator=torch.Generator().manual_seed(5))
    q, k, v, m = (dev(c[x]) for x in ("q", "k", "v", "m"))
    s = torch.full((B,), 2.0 * N)
    for st in (state, torch.zeros_like(state)):
        o, st_out = cott.fwd_stateful(q, k, v, m, 2.0 * N, state_in=dev(st) if st is state else None)
        r_o, r_s = oracle.fwd_segment(c["q"], c["k"], c["v"], c["m"], st, s)
        gate(o, r_o, torch.bfloat16)
        assert norm_max_err(st_out, r_s) <= 1e-2


@pytest.mark.parametrize("BH,d,groups,given,summed", [
    (3, 64, 9, True, True), (3, 64, 10, True, False), (3, 128, 2, False, True), (3, 128, 2, True, False),
    (3, 128, 3, False, False), (16, 128, 3, False, True), (16, 128, 2, True, True), (16, 128, 3, True, False), (40, 128, 3, True, True),
    (40, 128, 4, True, False)])
def test_forward_walk_sums_states_where_that_is_faster(BH, d, groups, given, summed, force_group):
    """The rule that picks between the sum inside the walk (two launches) and a scan launch (three): by the
    number of states a CTA would read and, at d = 128, the number of heads."""
    force_group(128)
    B, H, N = 1, BH, 128 * groups - 5
    c = synth.make_qkv(B, H, N, d, torch.bfloat16, 8600 + BH + groups)
    state = torch.randn((B, H, d, d), generator=torch.Generator().manual_seed(6)) if given else torch.zeros(B, H, d, d)
    q, k, v, m = (dev(c[x]) for x in ("q", "k", "v", "m"))
    n0 = cott.cott.launch_count()
    o, st_out = cott.fwd_stateful(q, k, v, m, 2.0 * N, state_in=dev(state) if given else None)
    assert cott.cott.launch_count() - n0 == (2 if summed else 3)
    r_o, r_s = oracle.fwd_segment(c["q"], c["k"], c["v"], c["m"], state, torch.full((B,), 2.0 * N))
    gate(o, r_o, torch.bfloat16)
    assert norm_max_err(st_out, r_s) <= 1e-2


@pytest.mark.parametrize("B,H,N", [(2, 12, 500), (4, 16, 260), (1, 18, 1000), (1, 74, 200)])
def test_bidirectional_backward_d128_in_one_wave(B, H, N):
    """Where the plan's groups would give the two walks more CTAs than SMs: as many groups as fit."""
    c = synth.make_qkv(B, H, N, 128, torch.bfloat16, 8700 + N, with_do=True)
    q, k, v, d_o, m = (dev(c[x]) for x in ("q", "k", "v", "d_o", "m"))
    dq, dk, dv, dm = cott.bwd(q, k, v, d_o, m, causal=False)
    rq, rk, rv, rm = oracle.bwd_quadratic(c["q"], c["k"], c["v"], c["d_o"], c["m"], None, False)
    gate(dq, rq, torch.bfloat16); gate(dk, rk, torch.bfloat16); gate(dv, rv, torch.bfloat16)
    gate_dm(dm, rm, 1e-2, dm_condition(rv, c["v"], c["m"], None), DM_COND_BF16)


@pytest.mark.parametrize("B,H,T,d", [(64, 16, 16, 128), (64, 16, 20, 128), (72, 16, 40, 120), (37, 4, 17, 64), (15, 10, 17, 64), (15, 10, 32, 64)])
def test_token_blocks_of_many_heads(B, H, T, d):
    """States of more than the L2 (1024 heads of 64 KB and more) take the instances that mark them for early
    eviction, d = 64 with more than 148 (b, h) those of 32 tokens: as the same rows in calls on a quarter of
    the batch, bit for bit where the kernel is the same, and two heads against the definition."""
    g = torch.Generator(device="cuda").manual_seed(B + T)
    q, k, v = ((torch.randn((B, H, T, d), generator=g, device="cuda") + 0.2).to(torch.bfloat16) for _ in range(3))
    m, state = torch.randn(H, generator=g, device="cuda"), torch.randn((B, H, d, d), generator=g, device="cuda")
    o, st = cott.fwd_stateful(q, k, v, m, 300.0, state_in=state)
    for b0 in range(0, B, B // 4):
        sl = slice(b0, b0 + B // 4)
        o1, st1 = cott.fwd_stateful(q[sl].contiguous(), k[sl].contiguous(), v[sl].contiguous(), m, 300.0, state_in=state[sl].contiguous())
        if d != 64:
            assert torch.equal(o[sl], o1) and torch.equal(st[sl], st1)
        else:
            gate(o[sl], o1.double().cpu().numpy(), torch.bfloat16)
            assert norm_max_err(st[sl], st1) <= 1e-2
    for b in (0, B - 1):
        x = [t[b:b + 1, :2].contiguous().cpu() for t in (q, k, v)]
        r_o, r_s = oracle.fwd_segment(*x, m[:2].cpu(), state[b:b + 1, :2].cpu(), torch.tensor([300.0]))
        gate(o[b:b + 1, :2], r_o, torch.bfloat16)
        assert norm_max_err(st[b:b + 1, :2], r_s) <= 1e-2


@pytest.mark.parametrize("B,H,N", [(3, 16, 700), (3, 8, 1000), (1, 12, 900), (2, 20, 1300), (1, 40, 1100), (5, 15, 300)])
def test_backward_d128_groups_of_the_two_walks(B, H, N):
    """The d = 128 backward with the library's own choice of groups: the dK, dV walk cut finer than the
    dQ walk, both cut, state passes in parts, neither cut; ragged last chunks and groups."""
    c = synth.make_qkv(B, H, N, 128, torch.bfloat16, 7900 + N, with_do=True)
    q, k, v, d_o, m = (dev(c[x]) for x in ("q", "k", "v", "d_o", "m"))
    dq, dk, dv, dm = cott.bwd(q, k, v, d_o, m, causal=True)
    rq, rk, rv, rm = oracle.bwd_quadratic(c["q"], c["k"], c["v"], c["d_o"], c["m"], None, True)
    gate(dq, rq, torch.bfloat16); gate(dk, rk, torch.bfloat16); gate(dv, rv, torch.bfloat16)
    cond = dm_condition(rv, c["v"], c["m"], None)       # (as in the edge test above)
    assert (abs(dm.double().cpu().numpy() - rm) <= 1e-3 * cond).all()
    gate_dm(dm, rm, 1e-2, cond, DM_COND_BF16)


@pytest.mark.parametrize("N", [1025, 1152, 2175])
@pytest.mark.parametrize("packed", [False, True])
def test_bidirectional_backward_in_one_launch_beyond_eight_chunks(N, packed, force_group):
    """The one-launch bidirectional backward with nine, exactly nine and seventeen chunks (its ring has
    three stages), dense and as a packed batch with short neighbours."""
    force_group(4096)
    H, d = 2, 64
    lens = [N, 1, 130] if packed else [N]
    cs = [synth.make_qkv(1, H, n, d, torch.bfloat16, 7900 + n + H, with_do=True) for n in lens]
    m = dev(cs[0]["m"])
    n0 = cott.cott.launch_count()
    if packed:
        q, k, v, d_o = (torch.cat([dev(c[x])[0].permute(1, 0, 2) for c in cs]).contiguous() for x in ("q", "k", "v", "d_o"))
        cu = torch.tensor([0, N, N + 1, N + 131], dtype=torch.int32, device="cuda")
        *grads, dm = cott.bwd_varlen(q, k, v, d_o, m, cu, N, causal=False)
    else:
        *grads, dm = cott.bwd(*(dev(cs[0][x]) for x in ("q", "k", "v", "d_o")), m, causal=False)
    assert cott.cott.launch_count() - n0 == 1
    rm = cond = 0.0
    for i, (n, c) in enumerate(zip(lens, cs)):
        c["m"] = cs[0]["m"]
        own = [x[sum(lens[:i]):sum(lens[:i + 1])].permute(1, 0, 2)[None] for x in grads] if packed else grads
        *refs, r = oracle.bwd_quadratic(c["q"], c["k"], c["v"], c["d_o"], c["m"], None, False)
        rm, cond = rm + r, cond + dm_condition(refs[2], c["v"], c["m"], None)
        if n == 1:
            one_token_bounds(own, refs, c)
        else:
            for x, ref in zip(own, refs):
                gate(x.contiguous(), ref, torch.bfloat16)
    gate_dm(dm, rm, 1e-2, cond, DM_COND_BF16)


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("t", [0, 5, 31, 40, 69])
def test_fp32_causal_rows_do_not_see_infinities_of_masked_tokens(d, bad, t):
    """One token of v, k or dO is not finite: what does not depend on it stays what it is without it.  The
    walk masks pairs inside a chunk of 32 tokens, and a masked score of zero times infinity would be NaN."""
    B, H, N = 1, 2, 70
    c = synth.make_qkv(B, H, N, d, torch.float32, 8100 + d + t, with_do=True)
    m = dev(c["m"])
    clean = {x: dev(c[x]) for x in ("q", "k", "v", "d_o")}
    ref_o = oracle.fwd_quadratic(c["q"], c["k"], c["v"], c["m"], None, True)
    refs = oracle.bwd_quadratic(c["q"], c["k"], c["v"], c["d_o"], c["m"], None, True)
    for name in ("v", "k", "d_o"):
        x = {**clean, name: clean[name].clone()}
        x[name][0, 0, t] = bad
        o = cott.fwd(x["q"], x["k"], x["v"], m, causal=True)
        dq, dk, dv, _ = cott.bwd(x["q"], x["k"], x["v"], x["d_o"], m, causal=True)
        ok = torch.ones(B, H, N, dtype=torch.bool)
        if name == "d_o":                     # dk, dv of a token sum over the tokens from it on
            ok[0, 0, :t + 1] = False
            pairs = ((dk, refs[1]), (dv, refs[2]))
        else:                                 # o, dq of a token over the tokens up to it
            ok[0, 0, t:] = False
            pairs = ((o, ref_o), (dq, refs[0]))
        for got, r in pairs:
            got = got.cpu()
            assert got[ok].isfinite().all() and not got[~ok].isfinite().all()
            r = torch.from_numpy(r)
            assert (got[ok].double() - r[ok]).abs().max() <= 1e-5 * r.abs().max()


U32 = 2.0 ** -24


def _rel(x, r):
    x, r = x.double().cpu(), torch.as_tensor(r)
    return ((x - r).norm() / r.norm()).item()


@pytest.mark.parametrize("N", [1, 40, 500, 1024])
@pytest.mark.parametrize("d", [32, 64, 128])
def test_fp32_state_is_exact_to_a_few_roundings(d, N):
    """A caller's state and the tokens' sum, a small part of it here, meet in one addition of full size
    whatever the number of tokens and groups: off by u at most, and as much again for the smaller sum's
    own roundings (token by token onto the state it is 2.3 u to 3.8 u)."""
    B, H, s = 2, 4, 8192.0
    c = synth.make_qkv(B, H, N, d, torch.float32, 8300 + d + N, with_do=True)
    g = torch.Generator().manual_seed(9)
    st, ds = (3.0 * torch.randn((B, H, d, d), generator=g) for _ in range(2))
    q, k, v, d_o, m = (dev(c[x]) for x in ("q", "k", "v", "d_o", "m"))
    _, out = cott.fwd_stateful(q, k, v, m, s, state_in=dev(st))
    *_, ds_in, _ = cott.bwd_stateful(q, k, v, d_o, m, s, state_in=dev(st), d_state_out=dev(ds))
    unit = lambda x: x.double() / x.double().norm(dim=-1, keepdim=True)
    cf = s ** -torch.sigmoid(c["m"].double()).view(1, H, 1, 1)
    want = st.double() + unit(c["k"]).transpose(-1, -2) @ (cf * c["v"].double())
    want_ds = ds.double() + unit(c["q"]).transpose(-1, -2) @ c["d_o"].double()
    assert _rel(out, want) <= 2 * U32
    # (dO is not scaled by c: the tokens' sum is as large as the state, and its own chains of a group's
    # tokens, 128 at most, add sqrt(128) / 4 u)
    assert _rel(ds_in, want_ds) <= 4 * U32


@pytest.mark.parametrize("N", [500, 1024])
@pytest.mark.parametrize("causal", [True, False])
def test_fp32_rows_are_summed_in_short_chains(N, causal):
    """The products of a row with the 128 rows of a state, or with the tokens of a chunk, are summed four by
    four: 2.0 u to 2.4 u off 64 bits in the 2-norm, norms and scales included; one chain over all of them
    measured 3.1 u to 3.6 u."""
    B, H, d = 2, 4, 128
    g = torch.Generator().manual_seed(8400 + N)
    q, k, v = (torch.randn((B, H, N, d), generator=g) + 0.3 for _ in range(3))
    m = torch.randn(H, generator=g)
    o = cott.fwd(*(dev(x) for x in (q, k, v, m)), causal=causal)
    assert _rel(o, oracle.fwd_quadratic(q, k, v, m, None, causal)) <= 2.7 * U32


@pytest.mark.parametrize("path", ["walk", "short64", "short128", "backward128"])
def test_normalised_rows_are_rounded_once(path):
    """x / ||x|| as the tensor cores get it is bf16, rounded once from fp32: only elements whose exact quotient
    is within 3 u of the middle between two bf16 numbers may end on the other side, 3 u / 2^-9 = one in ten
    thousand; the gate is three times that.  (Products with a scale split in two bf16 terms measure 5 to 8.)
    Unit vectors as the other operands, with c = 1/2, make the call return the rows."""
    d = 64 if path == "short64" else 128
    B, H = 2, 3
    g = torch.Generator().manual_seed(11)
    x = torch.randn((B, H, d, d), generator=g).to(torch.bfloat16)
    eye = torch.eye(d, dtype=torch.bfloat16).expand(B, H, d, d).contiguous()
    m, s = torch.zeros(H), torch.full((B,), 4.0)               # 4^-sigma(0) = 1/2
    xd, ed = dev(x), dev(eye)
    if path == "walk":                                         # state = c sum_j x^_j e_j^T
        got = cott.fwd(ed, xd, ed, dev(m), dev(s), causal=True, return_state=True)[1].transpose(-1, -2)
    elif path == "backward128":                                # dk_j = c q^_j without its part along k_j = e_{d-1}
        k = torch.zeros_like(ed)
        k[..., d - 1] = 1
        got = cott.bwd(xd, k, ed, ed, dev(m), dev(s), causal=True)[1]
    else:                                                      # o_i = c sum_j <e_i, x^_j> e_j
        got = cott.fwd(ed, xd, ed, dev(m), dev(s), causal=False).transpose(-1, -2)
    want = (x.double() / x.double().norm(dim=-1, keepdim=True)).float().to(torch.bfloat16)
    got = (2.0 * got.float().cpu()).to(torch.bfloat16)
    cols = slice(0, d - 1) if path == "backward128" else slice(None)
    assert (got != want)[..., cols].double().mean().item() <= 3e-4


@pytest.mark.parametrize("dtype,BH,N", [(torch.float32, 4, 1024), (torch.float32, 16, 509), (torch.bfloat16, 50, 2048)])
@pytest.mark.parametrize("causal", [True, False])
def test_noalloc_takes_coarser_groups_where_the_finer_ones_do_not_fit(dtype, BH, N, causal):
    """cott_fwd's own plan for these d = 128 problems needs a little more or much more than the 8 MiB of the
    built-in scratch, a coarser one fits: the call is taken, and its rows are those of cott_fwd to rounding."""
    g = torch.Generator(device="cuda").manual_seed(N)
    q, k, v = (torch.randn((1, BH, N, 128), generator=g, device="cuda").to(dtype) for _ in range(3))
    m = torch.randn(BH, generator=g, device="cuda")
    lib = cott.cott
    dt = lib.F32 if dtype == torch.float32 else lib.BF16
    if causal or dt == lib.F32:
        assert cott.workspace_bytes(lib.OP_FWD, dt, 1, BH, N, 128, causal) > 8 << 20
    got, want = cott.fwd_noalloc(q, k, v, m, causal=causal), cott.fwd(q, k, v, m, causal=causal)
    gate(got, want.double().cpu().numpy(), dtype)
    assert lib.fwd_noalloc_status() == 0


@pytest.mark.parametrize("kind", ["head first", "token first", "wide rows", "every other token"])
@pytest.mark.parametrize("call", ["block", "backward128", "segment128", "fp32"])
def test_memory_orders_match_dense(call, kind):
    """Tensors stored [H,B,N,d] or [N,B,H,d], as columns of wider rows or as every other token of a longer tensor:
    the kernels that calls of these shapes take give the bits they give on dense tensors."""
    B, H, N, d, dtype = {"block": (2, 3, 16, 128, torch.bfloat16), "backward128": (2, 3, 300, 128, torch.bfloat16),
                         "segment128": (2, 3, 300, 128, torch.bfloat16), "fp32": (2, 3, 150, 64, torch.float32)}[call]

    def stored(x):
        if kind == "head first":
            return x.permute(1, 0, 2, 3).contiguous().permute(1, 0, 2, 3)
        if kind == "token first":
            return x.permute(2, 0, 1, 3).contiguous().permute(1, 2, 0, 3)
        if kind == "wide rows":
            y = torch.full((B, H, N, d + 24), 7.0, dtype=dtype, device="cuda")
            y[..., 8:8 + d] = x
            return y[..., 8:8 + d]
        y = torch.full((B, H, 2 * N + 1, d), 7.0, dtype=dtype, device="cuda")
        y[:, :, 1::2] = x
        return y[:, :, 1::2]

    g = torch.Generator(device="cuda").manual_seed(17)
    q, k, v, d_o = (torch.randn((B, H, N, d), generator=g, device="cuda").to(dtype) for _ in range(4))
    m = torch.randn(H, generator=g, device="cuda")
    st, ds = (torch.randn((B, H, d, d), generator=g, device="cuda") for _ in range(2))
    run = {"block": lambda *x: cott.fwd_stateful(*x[:3], m, 99.0, state_in=st),
           "backward128": lambda *x: cott.bwd(*x, m, causal=True), "fp32": lambda *x: (cott.fwd(*x[:3], m), *cott.bwd(*x, m)),
           "segment128": lambda *x: cott.bwd_stateful(*x, m, 999.0, state_in=st, d_state_out=ds)}[call]
    for got, want in zip(run(*(stored(x) for x in (q, k, v, d_o))), run(q, k, v, d_o)):
        assert torch.equal(got, want)


def _laid_out(x, layout):
    """x [B,H,N,d] on the GPU in another memory order: [B,N,H,d], or slices of a fused [B,N,3,H,d] buffer."""
    x = dev(x)
    if layout == "dense":
        return x
    B, H, N, d = x.shape
    if layout == "bnhd":
        return x.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
    buf = torch.full((B, N, 3, H, d), float("nan"), dtype=x.dtype, device=x.device)
    buf[:, :, 1] = x.permute(0, 2, 1, 3)
    return buf[:, :, 1].permute(0, 2, 1, 3)


def _short_cases(lengths):
    """(N, dk, dv, causal) of calls that the kernels for at most 128 tokens take: bidirectional ones at d = 64 up to 64
    tokens (with one sequence a tile two CTAs an SM of the one-launch bidirectional kernels are faster)."""
    return [(N, dk, dv, causal) for causal in (True, False) for dk, dv in ((64, 64), (128, 128), (32, 32), (96, 40), (64, 128))
            for N in lengths if causal or N <= 64 or max(dk, dv) > 64]


@pytest.mark.parametrize("N,dk,dv,causal", _short_cases([1, 2, 7, 8, 9, 24, 31, 64, 65, 100, 127, 128]))
def test_short_backward_tiles(N, dk, dv, causal):
    """The backward of at most 128 tokens: one to sixteen sequences a tile, places of whole eights of rows
    with and without rows to spare, a last tile that is not full, padded rows, every memory order."""
    B, H = 13, 23                                          # (enough for the rule to take this kernel)
    layout = ("dense", "bnhd", "fused")[N % 3]
    c = synth.make_qkv(B, H, N, dk, torch.bfloat16, 8100 + N + dk, row_lognormal=True, with_do=True, d_v=dv)
    c["k"][0, 1, N // 2] = 0.0
    args = [_laid_out(c[x], layout) for x in ("q", "k", "v", "d_o")]
    before = cott.cott.launch_count()
    dq, dk_, dv_, dm = cott.bwd(*args, dev(c["m"]), causal=causal)
    assert cott.cott.launch_count() - before == 1
    rq, rk, rv, rm = oracle.bwd_quadratic(c["q"], c["k"], c["v"], c["d_o"], c["m"], None, causal)
    if N == 1:
        one_token_bounds((dq, dk_, dv_), (rq, rk, rv), c)
        assert (dm == 0).all() and (rm == 0).all()
        return
    z = (0, 1, N // 2)                                     # (the clamped formula's gradient, gated on its own)
    assert norm_max_err(dk_[z], rk[z]) <= 1e-2
    dk_[z] = 0.0
    rk[z] = 0.0
    gate(dq, rq, torch.bfloat16); gate(dk_, rk, torch.bfloat16); gate(dv_, rv, torch.bfloat16)
    # dm: products of fp32 scores of the rows as they were given, summed in fp32: N terms a row in four
    # chains, each with a few roundings of 2^-24
    cond = dm_condition(rv, c["v"], c["m"], None)
    assert (abs(dm.double().cpu().numpy() - rm) <= 1e-5 * cond).all()
    again = cott.bwd(*args, dev(c["m"]), causal=causal)
    dk2 = again[1].clone(); dk2[z] = 0.0
    for x, y in zip((dq, dk_, dv_, dm), (again[0], dk2, again[2], again[3])):
        assert torch.equal(x, y)


@pytest.mark.parametrize("N", [1, 20, 65, 127, 128])
@pytest.mark.parametrize("d,causal", [(64, True), (128, True), (128, False), (96, False)])
def test_short_sequences_through_the_kernels_for_longer_ones(N, d, causal, option):
    """short_bwd = 0 and short_fwd = 0, the way back to the kernels for longer sequences, whose walks then have one
    chunk: the same call both ways against the definition."""
    B, H = 13, 23
    c = synth.make_qkv(B, H, N, d, torch.bfloat16, 8200 + N + d, with_do=True)
    args = [_laid_out(c[x], "bnhd") for x in ("q", "k", "v", "d_o")]
    m = dev(c["m"])
    ref_o = oracle.fwd_quadratic(c["q"], c["k"], c["v"], c["m"], None, causal)
    rq, rk, rv, rm = oracle.bwd_quadratic(c["q"], c["k"], c["v"], c["d_o"], c["m"], None, causal)
    seen = []
    for short in (0, 1):
        option("short_bwd", short)
        option("short_fwd", short)
        o = cott.fwd(*args[:3], m, causal=causal)
        dq, dk, dv, dm = cott.bwd(*args, m, causal=causal)
        seen.append((o, dq, dk, dv))
        if N == 1:
            one_token_bounds((dq, dk, dv), (rq, rk, rv), c)
            assert (dm == 0).all()
            continue
        for x, r in ((o, ref_o), (dq, rq), (dk, rk), (dv, rv)):
            gate(x, r, torch.bfloat16)
        gate_dm(dm, rm, 1e-2, dm_condition(rv, c["v"], c["m"], None), DM_COND_BF16)
    # (other roundings: another kernel ran)
    assert N == 1 or not all(torch.equal(x, y) for x, y in zip(*seen))


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), 3.0e38])
@pytest.mark.parametrize("which", ["q", "k", "v", "d_o"])
def test_short_backward_keeps_sequences_apart(d, bad, which):
    """A row that is not finite (or whose scores overflow) in one sequence: the sequences that share its tile
    get the bits that they get without it."""
    B, H, N = 60, 5, 20                                    # five sequences a tile of 24 rows each
    c = synth.make_qkv(B, H, N, d, torch.bfloat16, 8300 + d, with_do=True)
    m = dev(c["m"])
    ref = cott.bwd(*(dev(c[x]) for x in ("q", "k", "v", "d_o")), m)
    c[which][0, 2, 3] = bad
    got = cott.bwd(*(dev(c[x]) for x in ("q", "k", "v", "d_o")), m)
    keep = torch.ones(B, H, dtype=torch.bool)
    keep[0, 2] = False
    for x, y in zip(got[:3], ref[:3]):
        assert torch.equal(x[keep], y[keep])
    assert torch.equal(got[3][[0, 1, 3, 4]], ref[3][[0, 1, 3, 4]])
    if bad == 3.0e38 and which in "qk":                    # (too long for fp32, but finite: a unit row of zeros)
        assert all(torch.isfinite(x[0, 2].float()).all() for x in got[:3])
    else:
        assert not all(torch.isfinite(x[0, 2].float()).all() for x in got[:3])


@pytest.mark.parametrize("dk,dv,N,causal", [(64, 64, 20, True), (64, 64, 20, False), (64, 64, 128, True), (128, 128, 20, True),
                                            (128, 128, 20, False), (128, 128, 128, True), (128, 128, 128, False), (96, 40, 20, True)])
@pytest.mark.parametrize("value", [3.0e38, 1.0e25, "one"])
@pytest.mark.parametrize("which", ["q", "k"])
def test_short_backward_rows_too_long_for_fp32(which, value, causal, N, dk, dv):
    """Finite rows of q or k whose squared norm overflows fp32 (1 / norm = 0), one sequence a tile and five: the
    same as a row of zeros there for everybody else, as in the kernels that normalise the rows first, and a
    gradient of zeros for the row itself."""
    B, H, z = (30, 11, (0, 2, 3)) if N == 20 else (14, 11, (0, 2, 77))
    c = synth.make_qkv(B, H, N, dk, torch.bfloat16, 8400 + N + dk, with_do=True, d_v=dv)
    args = {x: dev(c[x]) for x in ("q", "k", "v", "d_o", "m")}
    args[which][z] = 0.0
    want = cott.bwd(*args.values(), causal=causal)
    if value == "one":
        args[which][z][5] = 3.0e38
    else:
        args[which][z] = value
    got = cott.bwd(*args.values(), causal=causal)
    own = 0 if which == "q" else 1
    assert (got[own][z] == 0).all()
    want[own][z] = 0.0                                     # (the zero row's is that of the clamped formula)
    for x, y in zip(got, want):
        assert torch.equal(x, y)


@pytest.mark.parametrize("form", ["plain", "orders", "given", "per item", "subclass", "unequal"])
def test_native_and_python_bindings_agree(form):
    """The native half of the binding and the Python code behind it, which takes what the native half leaves:
    the same bits, the same strides, the tensors that were given handed back, the same refusals.  The native half
    is called by itself, so that it is seen to take what it should take and to leave the rest."""
    native, native_takes = cott.cott._load_native(), form not in ("subclass", "unequal")

    def by_native(name, *args, **kw):
        call = inspect.signature(getattr(cott, name)).bind(*args, **kw)
        call.apply_defaults()
        return getattr(native, name)(*(x for key, x in call.arguments.items() if key != "stream"))

    B, H, N, d = 2, 3, 70, 64
    d_v = 96 if form == "unequal" else d
    order = (lambda x: _laid_out(x, "fused")) if form == "orders" else dev
    c = synth.make_qkv(B, H, N, d, torch.bfloat16, 8500, with_do=True, d_v=d_v)
    q, k, v, d_o = (order(c[x]) for x in ("q", "k", "v", "d_o"))
    m = dev(c["m"])
    if form == "subclass":
        class Tagged(torch.Tensor):
            pass
        q = q.as_subclass(Tagged)
    s = torch.tensor([100.0, 300.0], device="cuda") if form == "per item" else 300.0
    state = 0.1 * torch.randn(B, H, d, d_v, device="cuda")
    give = form == "given"
    new = torch.empty_like
    ws = torch.empty(1 << 24, dtype=torch.uint8, device="cuda") if give else None

    def flat(x):
        return [y for z in x for y in flat(z)] if isinstance(x, (tuple, list)) else [x]

    calls = [
        ("fwd", (q, k, v, m, s), dict(causal=False, out=new(v) if give else None, workspace=ws)),
        ("fwd", (q, k, v, m), dict(return_state=True)),
        ("fwd_stateful", (q, k, v, m, s), dict(state_in=state, out=new(v) if give else None, workspace=ws)),
        ("bwd", (q, k, v, d_o, m, s), dict(out=(new(q), new(k), new(v)) if give else None, workspace=ws)),
        ("bwd_stateful", (q, k, v, d_o, m, s), dict(state_in=state, d_state_out=state, out=[new(q), new(k), new(v)] if give else None)),
    ]
    if form != "unequal":
        cu = torch.tensor([0, 50, 70], dtype=torch.int32, device="cuda")
        rows = [x.permute(0, 2, 1, 3)[0].contiguous() for x in (q, k, v, d_o)]
        calls += [("fwd_varlen", (*rows[:3], m, cu, 50), dict(causal=False)), ("bwd_varlen", (*rows, m, cu, 50), {})]
    for name, args, kw in calls:
        a = by_native(name, *args, **kw)
        assert (a is not None) == native_takes, name
        a = flat(getattr(cott, name)(*args, **kw) if a is None else a)
        a = [x.clone(memory_format=torch.preserve_format) for x in a]
        b = flat(getattr(cott.cott, f"_{name}_any")(*args, **kw))
        assert len(a) == len(b)
        for x, y in zip(a, b):
            assert torch.equal(x, y) and x.stride() == y.stride() and x.dtype == y.dtype, name
    if give:
        got = cott.bwd(q, k, v, d_o, m, out=calls[3][2]["out"])
        assert all(x is y for x, y in zip(got, calls[3][2]["out"]))
    rows = [x[:, :, 0].contiguous() for x in (q, k, v)]
    s1, s2 = state.clone(), state.clone()
    o1, o2 = by_native("decode_step", *rows, s1, m, s), cott.cott._decode_step_any(*rows, s2, m, s)
    assert (o1 is not None) == native_takes
    o1 = cott.decode_step(*rows, s1, m, s) if o1 is None else o1
    assert torch.equal(o1, o2) and torch.equal(s1, s2)
    small = torch.empty(16, dtype=torch.uint8, device="cuda")
    # (what the library refuses comes back from the native half as its status, what the Python code refuses as None)
    for status, bad in ((None, lambda f: f(q, k.transpose(2, 3), v, m)), (None, lambda f: f(q.half(), k, v, m)),
                        (None, lambda f: f(q.cpu(), k, v, m)), (None, lambda f: f(q, k, v, m.cpu())),
                        (None, lambda f: f(q[0], k[0], v[0], m)), (torch.Tensor, lambda f: f(q, k, v, m, -1.0)),
                        (-3, lambda f: f(q, k, v, m, workspace=small))):
        answer = bad(functools.partial(by_native, "fwd"))
        answer = torch.Tensor if isinstance(answer, torch.Tensor) else answer
        assert answer == (status if native_takes else None)
        said = []
        for f in (cott.fwd, cott.cott._fwd_any):
            try:
                bad(f)
                said.append(None)
            except Exception as e:
                said.append((type(e), str(e)))
        assert said[0] == said[1]


def _native_and_python_calls(B=2, H=3, N=70, d=64):
    """(name, arguments) of every call that has a native form."""
    c = synth.make_qkv(B, H, N, d, torch.bfloat16, 8600, with_do=True)
    q, k, v, d_o, m = (dev(c[x]) for x in ("q", "k", "v", "d_o", "m"))
    state = 0.1 * torch.randn(B, H, d, d, device="cuda")
    cu = torch.tensor([0, 50, 70], dtype=torch.int32, device="cuda")
    rows = [x.permute(0, 2, 1, 3)[0].contiguous() for x in (q, k, v, d_o)]
    one = [x[:, :, 0].contiguous() for x in (q, k, v)]
    return [("fwd", (q, k, v, m, None, True, False, None, None)),
            ("fwd_stateful", (q, k, v, m, 300.0, state, True, None, None)),
            ("bwd", (q, k, v, d_o, m, None, True, None, None, None)),
            ("bwd_stateful", (q, k, v, d_o, m, 300.0, state, state, True, None, None)),
            ("fwd_varlen", (*rows[:3], m, cu, 50, None, True, None, None)),
            ("bwd_varlen", (*rows, m, cu, 50, None, True, None)),
            ("decode_step", (*one, state, m, 300.0, None))]


class _PassThrough(TorchDispatchMode):
    def __torch_dispatch__(self, func, types, args=(), kwargs=None):
        return func(*args, **(kwargs or {}))


@pytest.mark.parametrize("inside", ["grad", "jvp", "vmap", "dispatch mode", "function mode"])
def test_native_binding_leaves_transforms_and_modes_to_python(inside):
    """Tensors that a transform only captures look plain, but what is allocated inside a level of grad or jvp has
    no storage: the native half hands every call back, and the Python code answers as it does by itself."""
    native = cott.cott._load_native()

    def within(f):
        got = []
        body = lambda x: (got.append(f()), x.sum())[1]
        x = torch.ones(2, 2, device="cuda")
        if inside == "grad":
            torch.func.grad(body)(x)
        elif inside == "jvp":
            torch.func.jvp(body, (x,), (x,))
        elif inside == "vmap":
            torch.func.vmap(body)(x)
        elif inside == "dispatch mode":
            with _PassThrough():
                body(x)
        else:
            with torch.overrides.BaseTorchFunctionMode():
                body(x)
        return got[0]

    def said(f):
        try:
            return within(f)
        except Exception as e:
            return type(e), str(e)

    for name, args in _native_and_python_calls():
        assert within(lambda: getattr(native, name)(*args)) is None, name
        again = [x.clone() if i == 3 and name == "decode_step" else x for i, x in enumerate(args)]
        a, b = said(lambda: getattr(cott, name)(*args)), said(lambda: getattr(cott.cott, f"_{name}_any")(*again))
        assert type(a) is type(b)
        if isinstance(a, tuple) and isinstance(a[0], type):
            assert a == b, name
        else:
            for x, y in zip(a if isinstance(a, tuple) else [a], b if isinstance(b, tuple) else [b]):
                assert torch.equal(x, y), name
        assert getattr(native, name)(*args) is not None, name     # (and it takes the call outside)


def test_native_binding_holds_the_lock_after_a_refused_pointer():
    """torch refuses the data pointer of a workspace while the native half has the interpreter lock released: the
    lock is taken again and the Python code reports the refusal."""
    for name, args in _native_and_python_calls():
        if name == "decode_step":                          # (no workspace: the output, of which no reference stays behind)
            out = torch.empty_like(args[2])
            torch._C._set_throw_on_mutable_data_ptr(out)
            before = sys.getrefcount(out)
            with pytest.raises(RuntimeError):
                cott.decode_step(*args[:-1], out=out)
            assert sys.getrefcount(out) == before
            continue
        at = {"bwd": 7, "bwd_varlen": 9, "bwd_stateful": 9, "fwd_varlen": 9}.get(name, 8)
        ws = torch.empty(1 << 24, dtype=torch.uint8, device="cuda")
        assert getattr(cott.cott._load_native(), name)(*args[:at], ws, *args[at + 1:]) is not None
        torch._C._set_throw_on_mutable_data_ptr(ws)
        with pytest.raises(RuntimeError):
            getattr(cott, name)(*args[:at], workspace=ws)
        assert getattr(cott.cott._load_native(), name)(*args) is not None


def test_native_binding_uses_the_current_stream():
    """Two threads with a stream of their own as the current one: the calls run on it, behind what their inputs come
    from there (the stream is kept busy first, and the inputs hold something else until then)."""
    native = cott.cott._load_native()
    calls = _native_and_python_calls()
    want = {name: getattr(cott, name)(*(x.clone() if isinstance(x, torch.Tensor) else x for x in args)) for name, args in calls}
    torch.cuda.synchronize()
    said = []

    def work():
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(5):
                    for name, args in calls:
                        late = [torch.zeros_like(x) if isinstance(x, torch.Tensor) and x.dtype != torch.int32 else x for x in args]
                        torch.cuda.current_stream().synchronize()
                        torch.cuda._sleep(200000)          # (0.1 ms)
                        for x, y in zip(late, args):
                            if x is not y:
                                x.copy_(y)
                        got = getattr(native, name)(*late)
                        flat = lambda x: list(x) if isinstance(x, tuple) else [x]
                        for x, y in zip(flat(got), flat(want[name])):
                            assert torch.equal(x, y), name
        except BaseException as e:
            said.append(e)

    threads = [threading.Thread(target=work) for _ in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if said:
        raise said[0]


@pytest.mark.parametrize("name", ["bwd", "bwd_stateful"])
def test_native_binding_while_another_thread_changes_the_list(name):
    """`out` given as a list whose items another thread replaces during the call, which runs without the
    interpreter lock: the tensors that the gradients went to come back, whole."""
    args = dict(_native_and_python_calls())[name][:4 + 2 * (name == "bwd_stateful") + 1]
    want = getattr(cott, name)(*args)
    new = lambda: [torch.empty_like(x) for x in args[:3]]
    out, stop = new(), threading.Event()

    def replace():
        while not stop.is_set():
            out[:] = new()

    t = threading.Thread(target=replace)
    t.start()
    try:
        for _ in range(300):
            for x, y in zip(getattr(cott, name)(*args, out=out), want):
                assert torch.equal(x, y)
    finally:
        stop.set()
        t.join()


@pytest.mark.parametrize("N,dk,dv,causal", _short_cases([1, 2, 7, 8, 9, 31, 64, 65, 100, 128]))
def test_short_forward_memory_orders(N, dk, dv, causal):
    """The forward of at most 128 tokens in memory orders that are not dense: places of whole eights of rows,
    a last tile that is not full; against the dense tensors' kernel, whose tiles hold the same rows (the
    scores and the sums over a row's own columns do not depend on where in a tile a sequence lies)."""
    B, H = 13, 23                                          # (enough for the rule to take this kernel)
    c = synth.make_qkv(B, H, N, dk, torch.bfloat16, 8700 + N + dk, row_lognormal=True, d_v=dv)
    c["k"][0, 1, N // 2] = 0.0
    m = dev(c["m"])
    o = cott.fwd(*(dev(c[x]) for x in ("q", "k", "v")), m, causal=causal)
    if N > 1:
        gate(o, oracle.fwd_quadratic(c["q"], c["k"], c["v"], c["m"], None, causal), torch.bfloat16)
    for layout in ("bnhd", "fused"):
        out = torch.full((B, N, H, dv), 7.0, dtype=torch.bfloat16, device="cuda").permute(0, 2, 1, 3)
        before = cott.cott.launch_count()
        cott.fwd(*(_laid_out(c[x], layout) for x in ("q", "k", "v")), m, causal=causal, out=out)
        assert cott.cott.launch_count() - before == 1
        assert norm_max_err(out, o) <= 2.0 ** -8           # (one rounding of the output)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("which", ["q", "k", "v"])
@pytest.mark.parametrize("layout", ["dense", "bnhd"])
@pytest.mark.parametrize("N", [1, 20, 64])
def test_short_forward_keeps_sequences_apart(N, layout, d, bad, which):
    """Rows that are not finite in the last two sequences, which share a tile (with up to 42 more; in places of
    whole eights of rows with up to ten): every other sequence gets the bits that it gets without them, and each of
    the two those that it gets without the other."""
    B, H = 60, 5
    c = synth.make_qkv(B, H, N, d, torch.bfloat16, 8800 + d)
    m = dev(c["m"])
    rows = [(B - 1, H - 2, 0), (B - 1, H - 1, N - 1)]

    def call(which_rows):
        x = {n: y.clone() for n, y in c.items()}
        for r in which_rows:
            x[which][r] = bad
        return cott.fwd(*(_laid_out(x[n], layout) for n in ("q", "k", "v")), m)

    ref, got = call([]), call(rows)
    keep = torch.ones(B, H, dtype=torch.bool)
    for r in rows:
        keep[r[:2]] = False
        x, y = got[r[:2]], call([r])[r[:2]]
        assert torch.equal(x.isnan(), y.isnan()) and torch.equal(x.nan_to_num(), y.nan_to_num())
        assert not torch.isfinite(x.float()).all()
    assert torch.equal(got[keep], ref[keep])
