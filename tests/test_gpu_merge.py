"""The cross-CTA merge of the fused decode kernels: its edges and its values.

A slab over several CTAs is merged by its last CTA from words that are 0 while
empty, with one, two or three warps a (slab, column). Sizes here put it at its
edges: fewer rows than CTAs, one row a CTA, slabs that end on a CTA boundary, one
to many slabs a CTA; values that are exactly 0 (which must not read as "empty").
Outputs against the fp64 oracle within the suite's tolerance; the constant-value
cases against their closed form within 1e-5 (64 x the fp32 rounding of one sum).
"""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2609_32663_gb300.dkv as dkv
from paper_2609_32663_gb300 import inputs as I
from parity import Case, assert_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built(cuda):
    from paper_2609_32663_gb300 import build
    build.build_library()
    torch.cuda.set_device(cuda)


def wl(**kw):
    base = dict(L=1, H=4, Hkv=1, T=3000, B=1, D=2, W=2000, pattern="ones", rate=1.0, seed=7)
    base.update(kw)
    return I.Workload("merge", **base)


@pytest.mark.parametrize("G", [1, 4, 8])
@pytest.mark.parametrize("T", [3, 75, 76, 151, 152, 153, 152 * 16, 152 * 16 + 1, 5000])
def test_rows_around_the_cta_count(G, T):
    c = Case(wl(H=G, T=T), reserve=2)
    c.decode_steps(2, append=True)
    c.close()


@pytest.mark.parametrize("G,Hkv,B,T", [(4, 8, 1, 4096), (4, 2, 1, 4104), (7, 4, 4, 2000), (8, 1, 3, 1700),
                                       (2, 19, 1, 1216), (1, 16, 16, 1300), (3, 5, 40, 1170)])
def test_slabs_per_cta(G, Hkv, B, T):
    """From one slab over many CTAs to many slabs a CTA (teams of three, two and one warps a task)."""
    c = Case(wl(H=G * Hkv, Hkv=Hkv, B=B, T=T, seed=T), reserve=1)
    c.decode_steps(1, append=True)
    c.close()


@pytest.mark.parametrize("G", [4, 7])
@pytest.mark.parametrize("v", [0.0, 1.0])
def test_zero_scores_and_constant_values(G, v):
    """q = 0: every score and running max is exactly 0 and the output is V's mean."""
    c = Case(wl(H=2 * G, Hkv=2, T=9000, W=4000))
    q = torch.zeros((1, 2 * G, 128), dtype=torch.bfloat16, device=c.dev)
    c.Vc.fill_(v)
    out = torch.full((1, 2 * G, 128), float("nan"), device=c.dev)
    for _ in range(3):
        dkv.dkv_decode_attn(c.plan, 0, q, None, None, None, c.Kc, c.Vc, out)
        assert (out - v).abs().max().item() <= 1e-5
    assert dkv.dkv_plan_status(c.plan) == 0
    c.close()


def test_back_to_back_calls_are_identical():
    """The exchange is empty again after every launch: calls in a row, over two
    layers, with one and several queries, repeat their outputs bit for bit."""
    c = Case(wl(L=2, H=8, Hkv=2, T=9000, W=4000, B=2))
    q = I.decode_inputs(c.wl, 1)[0][0].to(c.dev)
    qm = torch.stack([q, -q], dim=2)  # [L][B][2][H][128]
    first = None
    for _ in range(20):
        outs = [torch.empty((2, 8, 128), device=c.dev) for _ in range(2)]
        multi = [torch.empty((2, 2, 8, 128), device=c.dev) for _ in range(2)]
        for l in range(2):
            dkv.dkv_decode_attn(c.plan, l, q[l], None, None, None, c.Kc, c.Vc, outs[l])
            dkv.dkv_decode_multi(c.plan, l, qm[l].contiguous(), 2, None, c.Kc, c.Vc, multi[l])
        got = torch.cat([t.reshape(-1) for t in outs + multi])
        first = got if first is None else first
        assert torch.equal(got, first)
    assert dkv.dkv_plan_status(c.plan) == 0
    c.close()


@pytest.mark.parametrize("Hkv,B,Q,T", [(8, 8, 5, 1800), (8, 9, 5, 1800), (1, 1, 16, 152 * 64 + 1), (1, 40, 5, 1500)])
def test_combine_on_both_sides_of_the_slab_limit(Hkv, B, Q, T):
    """17 or more columns: the combine kernel places a slab's partials itself up to
    64 slabs a layer and reads them from the partial kernel above; also a slab over
    every CTA (more partials than one batch)."""
    G = 4
    c = Case(wl(H=G * Hkv, Hkv=Hkv, B=B, T=T, W=T, seed=Q + T))
    gen = torch.Generator().manual_seed(T)
    q = torch.randn((B, Q, G * Hkv, 128), generator=gen).to(torch.bfloat16)
    out = torch.full((B, Q, G * Hkv, 128), float("nan"), device=c.dev)
    for _ in range(2):
        dkv.dkv_decode_multi(c.plan, 0, q.to(c.dev), Q, None, c.Kc, c.Vc, out)
    got = out.double().cpu().numpy()
    for i in sorted({0, Q - 1}):
        want = O.decode(c.om, 0, B, G * Hkv, Hkv, I.bf16_bits(q[:, i].contiguous()), c.oKc, c.oVc)
        assert_close(np.ascontiguousarray(got[:, i]), want, f"query {i}")
    assert dkv.dkv_plan_status(c.plan) == 0
    c.close()


def test_plans_of_other_sizes_side_by_side():
    """A plan keeps working after plans of the same group size but fewer sequences
    or KV heads were made (a kernel's shared-memory limit is the kernel's, not a
    plan's)."""
    big = Case(wl(H=4 * 16, Hkv=16, T=1300, B=20), reserve=2)
    small = [Case(wl(H=4 * h, Hkv=h, T=1300, B=b), reserve=2) for h, b in ((1, 1), (8, 1), (2, 3))]
    q = torch.zeros((20, 5, 64, 128), dtype=torch.bfloat16, device=big.dev)
    for c in [big] + small:
        c.decode_steps(1, append=True)
    for Q in (1, 2, 4, 5):  # every multi-query kernel
        qq = q[:, :Q].contiguous()
        out = torch.empty(qq.shape, device=big.dev)
        dkv.dkv_decode_multi(big.plan, 0, qq, Q, None, big.Kc, big.Vc, out)
    big.decode_steps(1, append=False)
    for c in [big] + small:
        c.close()


@pytest.mark.parametrize("G,Q", [(4, 1), (7, 1), (4, 2), (4, 4)])
def test_a_partial_that_came_late_is_gone_after_the_status_is_cleared(monkeypatch, G, Q):
    """DKV_FAULT=late: every exchange word is full after the call, as if partials had
    arrived after their merge gave up. Once the status word is cleared, the next call
    of any kind is exact."""
    w = wl(L=1, H=2 * G, Hkv=2, T=9000, W=4000, B=2, seed=G)
    c = Case(w, reserve=4)
    gen = torch.Generator().manual_seed(G)
    q = torch.randn((2, Q, 2 * G, 128), generator=gen).to(torch.bfloat16)
    dq = q.to(c.dev)
    out = torch.full((2, Q, 2 * G, 128), float("nan"), device=c.dev)
    scratch = torch.empty((2, 2 * G, 128), device=c.dev)
    monkeypatch.setenv("DKV_FAULT", "late")
    dkv.dkv_decode_attn(c.plan, 0, dq[:, 0].contiguous(), None, None, None, c.Kc, c.Vc, scratch)
    monkeypatch.delenv("DKV_FAULT")
    assert dkv.dkv_plan_status(c.plan, clear=True) == dkv.DKV_DEV_MERGE_TIMEOUT
    dkv.dkv_decode_multi(c.plan, 0, dq, Q, None, c.Kc, c.Vc, out)
    got = out.double().cpu().numpy()
    for i in sorted({0, Q - 1}):
        want = O.decode(c.om, 0, 2, 2 * G, 2, I.bf16_bits(q[:, i].contiguous()), c.oKc, c.oVc)
        assert_close(np.ascontiguousarray(got[:, i]), want, f"query {i}")
    c.decode_steps(2, append=True)
    c.close()


@pytest.mark.parametrize("Hkv,B,Q,T", [(2, 2, 5, 9000), (2, 2, 16, 9000), (8, 9, 5, 1800)])
def test_outputs_of_a_timed_out_multi_query_call_stay_unwritten(monkeypatch, Hkv, B, Q, T):
    """DKV_FAULT=copy, 17 or more columns, up to and above 64 slabs: the combine
    kernel writes nothing from the partials that an earlier call left behind."""
    G = 4
    c = Case(wl(H=G * Hkv, Hkv=Hkv, B=B, T=T, W=T, seed=Q))
    gen = torch.Generator().manual_seed(T)
    q = torch.randn((B, Q, G * Hkv, 128), generator=gen).to(torch.bfloat16).to(c.dev)
    first, out, again = (torch.full(q.shape, -7.0, device=c.dev) for _ in range(3))
    dkv.dkv_decode_multi(c.plan, 0, q, Q, None, c.Kc, c.Vc, first)
    torch.cuda.synchronize()
    monkeypatch.setenv("DKV_FAULT", "copy")
    dkv.dkv_decode_multi(c.plan, 0, q, Q, None, c.Kc, c.Vc, out)
    torch.cuda.synchronize()
    monkeypatch.delenv("DKV_FAULT")
    assert dkv.dkv_plan_status(c.plan, clear=True) & dkv.DKV_DEV_TMA_TIMEOUT
    assert (out == -7.0).all()
    dkv.dkv_decode_multi(c.plan, 0, q, Q, None, c.Kc, c.Vc, again)
    assert torch.equal(again, first)
    assert dkv.dkv_plan_status(c.plan) == 0
    c.close()


@pytest.mark.parametrize("Q", [1, 2, 4, 5, 16])
def test_values_of_plans_of_other_sizes_side_by_side(Q):
    """Every multi-query kernel of a large plan after plans of fewer sequences and KV
    heads were made: with q = 0 an output is the mean of its slab's V rows."""
    big = Case(wl(H=4 * 16, Hkv=16, T=1300, B=20), reserve=2)
    small = [Case(wl(H=4 * h, Hkv=h, T=1300, B=b), reserve=2) for h, b in ((1, 1), (8, 1), (2, 3))]
    for c in [big] + small:
        B, H, Hkv = c.wl.B, c.wl.H, c.wl.Hkv
        out = torch.full((B, Q, H, 128), float("nan"), device=c.dev)
        q = torch.zeros(out.shape, dtype=torch.bfloat16, device=c.dev)
        dkv.dkv_decode_multi(c.plan, 0, q, Q, None, c.Kc, c.Vc, out)
        off = c.om.off[:-1].reshape(B, Hkv)
        ln = c.om.len.reshape(B, Hkv)
        for b in range(B):
            for g in range(Hkv):
                mean = c.Vc[int(off[b, g]):int(off[b, g] + ln[b, g])].double().mean(dim=0)
                got = out[b, :, 4 * g:4 * g + 4].double()
                assert (got - mean).abs().max().item() <= 1e-5
        assert dkv.dkv_plan_status(c.plan) == 0
    for c in [big] + small:
        c.close()
