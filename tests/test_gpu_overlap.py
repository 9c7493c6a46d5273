"""Decode calls that follow each other without an ordinary kernel between them: a
call may start before the previous one has stored its appended rows, and has to
attend to them all the same. n_appended comes from buffers prepared beforehand, one
a count, so no dkv_advance separates the calls. Rows that were never appended are
NaN. Outputs against the fp64 oracle within the suite's tolerance."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2609_32663_gb300.dkv as dkv
from paper_2609_32663_gb300 import inputs as I
from parity import Case, assert_close

pytestmark = pytest.mark.gpu
STEPS = 5


@pytest.fixture(scope="module", autouse=True)
def _built(cuda):
    from paper_2609_32663_gb300 import build
    build.build_library()
    torch.cuda.set_device(cuda)


def wl(G, T, Hkv=2, B=2):
    return I.Workload("overlap", L=1, H=G * Hkv, Hkv=Hkv, T=T, B=B, D=2, W=T, pattern="ones", rate=1.0, seed=G + T)


class Run:
    """A case whose inputs of STEPS appends are on the device, with the oracle's caches."""

    def __init__(self, G, T):
        w = wl(G, T)
        self.c = c = Case(w, reserve=STEPS + 1)
        self.q, self.kn, self.vn = I.decode_inputs(w, STEPS)
        self.dq, self.dk, self.dv = (t[:, 0].to(c.dev) for t in (self.q, self.kn, self.vn))
        self.napp = [torch.full((w.B,), s, dtype=torch.int32, device=c.dev) for s in range(STEPS + 1)]
        self.out = torch.full((STEPS, w.B, w.H, 128), float("nan"), device=c.dev)
        torch.cuda.synchronize()

    def append(self, s):
        c = self.c
        dkv.dkv_decode_attn(c.plan, 0, self.dq[s], self.dk[s], self.dv[s], self.napp[s], c.Kc, c.Vc, self.out[s])

    def oracle_append(self, s):
        c, w = self.c, self.c.wl
        O.append(c.om, 0, w.B, w.Hkv, c.reserve, np.full(w.B, s, np.int32), I.bf16_bits(self.kn[s, 0]),
                 I.bf16_bits(self.vn[s, 0]), c.oKc, c.oVc)

    def want(self, q, rows):
        c, w = self.c, self.c.wl
        return O.decode(c.om, 0, w.B, w.H, w.Hkv, I.bf16_bits(q), c.oKc, c.oVc, n_rows_app=np.full(w.B, rows, np.int32))

    def check_appends(self):
        got = self.out.double().cpu().numpy()
        for s in range(STEPS):
            self.oracle_append(s)
            assert_close(got[s], self.want(self.q[s, 0], s + 1), f"append {s}")


@pytest.mark.parametrize("G", [4, 7])
@pytest.mark.parametrize("T", [40, 1200, 30000])
def test_appends_in_a_row_on_one_layer(G, T):
    r = Run(G, T)
    for s in range(STEPS):
        r.append(s)
    r.check_appends()
    assert dkv.dkv_plan_status(r.c.plan) == 0
    r.c.close()


@pytest.mark.parametrize("G,Q", [(4, 2), (4, 4), (4, 5), (4, 16), (7, 4), (8, 1)])
@pytest.mark.parametrize("T", [40, 1200, 30000])
def test_multi_query_right_after_an_append(G, Q, T):
    r = Run(G, T)
    c, w = r.c, r.c.wl
    gen = torch.Generator().manual_seed(Q)
    mq = torch.randn((w.B, Q, w.H, 128), generator=gen).to(torch.bfloat16)
    dmq = mq.to(c.dev)
    multi = torch.full((STEPS, w.B, Q, w.H, 128), float("nan"), device=c.dev)
    torch.cuda.synchronize()
    for s in range(STEPS):
        r.append(s)
        dkv.dkv_decode_multi(c.plan, 0, dmq, Q, r.napp[s + 1], c.Kc, c.Vc, multi[s])
    r.check_appends()
    got = multi[-1].double().cpu().numpy()
    assert torch.isfinite(multi).all()
    for i in sorted({0, Q - 1}):
        assert_close(np.ascontiguousarray(got[:, i]), r.want(mq[:, i].contiguous(), STEPS), f"query {i}")
    assert dkv.dkv_plan_status(c.plan) == 0
    c.close()


@pytest.mark.parametrize("G", [2, 4, 7])
@pytest.mark.parametrize("T", [40, 1200, 30000])
def test_allocation_free_appends_in_a_row(G, T):
    r = Run(G, T)
    c, w, info = r.c, r.c.wl, r.c.info
    status = torch.zeros(1, dtype=torch.int32, device=c.dev)
    torch.cuda.synchronize()
    for s in range(STEPS):
        dkv.dkv_decode_attn_noalloc(c.sh, w.B, 0, c.reserve, info.d_len, info.d_off, info.d_ioff, r.dq[s], r.dk[s],
                                    r.dv[s], r.napp[s], c.Kc, c.Vc, r.out[s], status=status)
    r.check_appends()
    assert status.item() == 0
    c.close()


def test_allocation_free_call_without_rows_waits_for_the_one_before():
    """A layer with no rows: its zeros are written after the previous call's outputs."""
    r = Run(4, 30000)
    c, w, info = r.c, r.c.wl, r.c.info
    none = torch.zeros(w.B * w.Hkv + 1, dtype=torch.int64, device=c.dev)
    out = torch.full((20, w.B, w.H, 128), float("nan"), device=c.dev)
    torch.cuda.synchronize()
    for o in out:
        dkv.dkv_decode_attn_noalloc(c.sh, w.B, 0, c.reserve, info.d_len, info.d_off, info.d_ioff, r.dq[0], None, None,
                                    None, c.Kc, c.Vc, o)
        dkv.dkv_decode_attn_noalloc(c.sh, w.B, 0, c.reserve, none, none, none, r.dq[0], None, None, None, c.Kc, c.Vc, o)
    assert not out.any()
    c.close()


@pytest.mark.parametrize("T", [1200, 30000])
def test_export_of_what_the_previous_call_writes(T):
    """A decode call signals early; the export that follows reads its outputs as
    probabilities, in one buffer that every step rewrites."""
    r = Run(4, T)
    c, w = r.c, r.c.wl
    n = w.B * w.H * 128
    P = torch.full((w.B, w.H, 128), float("nan"), device=c.dev)
    kept = torch.empty_like(P).expand(STEPS, *P.shape).clone()
    M = torch.full((STEPS, n), 7, dtype=torch.uint8, device=c.dev)
    work = torch.empty(dkv.dkv_topk_workspace_bytes(), dtype=torch.uint8, device=c.dev)
    torch.cuda.synchronize()
    for s in range(STEPS):
        dkv.dkv_decode_attn(c.plan, 0, r.dq[s], None, None, None, c.Kc, c.Vc, P)
        dkv.dkv_topk_mask(P, n // 3, M[s], work)
        dkv.dkv_decode_attn(c.plan, 0, r.dq[s], None, None, None, c.Kc, c.Vc, kept[s])
    for s in range(STEPS):
        assert np.array_equal(M[s].cpu().numpy(), O.topk_mask(kept[s].cpu().numpy(), n // 3).reshape(-1)), f"step {s}"
    c.close()
