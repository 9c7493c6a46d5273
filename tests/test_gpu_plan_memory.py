"""A released plan's memory serves the next plan and is given back with the last one."""
import threading

import numpy as np
import pytest
import torch

import paper_2609_32663_gb300.dkv as dkv
from paper_2609_32663_gb300 import inputs as I
from parity import Case, check_map

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built(cuda):
    from paper_2609_32663_gb300 import build
    build.build_library()
    torch.cuda.set_device(cuda)


def wl(seed, **kw):
    base = dict(L=2, H=8, Hkv=2, T=6000, B=2, D=8, W=606, pattern="profile", rate=0.4, ragged=(1500, 6000))
    return I.Workload("memory", **{**base, "seed": seed, **kw})


def test_reused_memory_and_what_is_left():
    cases = [Case(wl(1), reserve=3), Case(wl(2), reserve=3)]
    for c in cases:  # loads the kernels, fills the exchange words' memory once
        c.decode_steps(1, append=True)
    for seed in range(3, 9):
        cases.pop(0).close()  # its memory is kept: another plan is alive
        cases.append(Case(wl(seed, B=1 + seed % 3), reserve=3))
        check_map(cases[-1].plan, cases[-1].om)
        cases[-1].decode_steps(2, append=True)
    cases[0].decode_steps(1, append=False)
    torch.cuda.synchronize()
    alive = torch.cuda.mem_get_info()[0]
    for c in cases:
        c.close()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    assert free > alive  # given back with the last plan
    plan = Case(wl(20)).plan
    plan.close()
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= free - (64 << 20)  # nothing grows (torch's own blocks aside)


def test_plans_made_and_released_by_several_threads():
    w = wl(30)
    first = Case(w)
    errors = []

    def work(k):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for _ in range(10):
                    p = dkv.dkv_map_pattern(first.M, first.Tc, first.sh, reserve_rows=0)
                    ln, off, ioff, idx = dkv.dkv_plan_read(p)
                    assert np.array_equal(ln, first.om.len) and np.array_equal(idx, first.om.idx)
                    p.close()
        except Exception as e:  # noqa: BLE001 (reported by the main thread)
            errors.append((k, e))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    first.close()


def test_memory_of_a_plan_of_many_slabs():
    """What a plan of 512 sequences x 32 KV heads takes: the partials' workspace (one
    record of 64 columns a CTA and a slab, one of 16 a warp), 16 columns a CTA for the
    fused merge, and the metadata. Not a fused-merge slot a slab (136 MB)."""
    import gc
    B, Hkv = 512, 32
    NH, rec = B * Hkv, 130 * 4
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sh = dkv.Shape(L=1, H=Hkv, H_kv=Hkv, D=1, bin_width=1)
    gc.collect()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    plan = dkv.dkv_plan_dense(np.full(B, 3, np.int32), sh, 16)
    torch.cuda.synchronize()
    taken = free - torch.cuda.mem_get_info()[0]
    plan.close()
    bound = (sms + NH) * 64 * rec + sms * 16 * 16 * rec + sms * 16 * rec + 64 * NH
    assert taken <= bound + (4 << 20)  # allocations come in pages of 2 MB
