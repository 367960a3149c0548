"""Failure detection on the device without a fault: a bounded wait inside a kernel is made to run out
(acache_debug_expire_next_wait gives one grid-wide barrier a target it cannot reach and a short poll
limit), and the test checks what the library promises for that case: the kernel returns, the status word
carries ACACHE_FLAG_WAIT_EXPIRED, acache_poll_status answers ACACHE_ERR_TIMEOUT and re-arms the barrier,
and the very next call on the same context gives the bits of a clean run."""
import numpy as np
import pytest
import torch

from oracle import acache_oracle as orc
from paper_2608_26140_b200 import binding as ab
from paper_2608_26140_b200 import workloads as wl

from helpers import DEV, DeviceCase
from test_gpu_parity import MID128, dev_i32

pytestmark = pytest.mark.gpu


# q/k/v of few rows and a long K: cut between the CTAs of a cluster, which pass their barriers whatever ran out
DEEP128 = wl.LayerShape(3584, 4, 1, 128, 256, 1e-6, True, 1e6, "deep-d128")
WIDE_Q128 = wl.LayerShape(256, 40, 5, 128, 256, 1e-5, True, 5e5, "wide-q-d128")
LONG128 = wl.LayerShape(2560, 6, 3, 128, 256, 1e-6, True, 1e6, "long-d128")


@pytest.mark.parametrize("shape,B,L,extra,kernel", [
    (wl.TINY, 1, 300, "none", "gemm_rows_kernel<1, 0, true>"),       # 60 rows: one CTA per tile, ring stages filled with weights
    (MID128, 1, 300, "none", "gemm_rows_kernel<2, 0, true>"),        # before the barrier; two and four CTAs per tile
    (LONG128, 1, 160, "none", "gemm_rows_kernel<2, 0, false>"),
    (DEEP128, 1, 300, "none", "gemm_rows_kernel<4, 0, false>"),
    (MID128, 2, 400, "all", "gemm_tc2_kernel"),                      # several 128-row tiles: the two-SM projection kernel
    (WIDE_Q128, 2, 400, "all", "gemm_wm_kernel<0>"),                 # the same, more columns: weights as the product's M
])
def test_a_wait_that_runs_out_is_reported_and_the_context_stays_usable(shape, B, L, extra, kernel):
    lay = wl.make_layout(B, 4, L, 40, 32, 32, extra)
    case = wl.make_case(shape, lay, 0.2, cfg_id=17)
    dc = DeviceCase(case)
    K = orc.k_from_ratio(L, 0.2)
    n = K + lay.n_extra
    g = np.random.default_rng(1)
    anchors = dev_i32(np.stack([np.sort(g.choice(L, K, replace=False)) for _ in range(B)]))

    def step():
        y = torch.zeros((B, n, shape.hidden), dtype=torch.bfloat16, device=DEV)
        dc.ctx.layer_step(dc.lw, dc.req, dc.kv(), dc.x, 0, 0.2, 0, None, anchors, y)
        torch.cuda.synchronize()                     # returns: no kernel of the step is stuck
        return ab.to_host_bits(y), ab.to_host_bits(dc.ck), ab.to_host_bits(dc.cv)

    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        clean = step()
    names = [e.key for e in prof.key_averages()]
    assert any(kernel in name for name in names), names              # the projection whose barrier runs out is this kernel
    assert dc.ctx.poll_status_code() == (ab.OK, 0)
    dc.reset_cache()
    dc.ctx.debug_expire_next_wait()
    step()                                           # its outputs are meaningless; only that it ends matters
    code, flags = dc.ctx.poll_status_code()
    assert code == ab.ERR_TIMEOUT and (flags & ab.FLAG_WAIT_EXPIRED)
    assert dc.ctx.poll_status_code() == (ab.OK, 0)   # the poll cleared the word
    dc.reset_cache()
    again = step()
    assert dc.ctx.poll_status_code() == (ab.OK, 0)
    for a, b in zip(clean, again):
        assert np.array_equal(a, b)


# Up to 64 rows of up to 256 columns the clean steps take a kernel without a grid-wide barrier; the step that is to run out takes the one
# that has it, as the clean steps of more rows do.
@pytest.mark.parametrize("L,kernel", [(300, "acache::own_gemm_rows_kernel<1, 0, true>"), (400, "acache::gemm_rows_kernel<1, 0, true>")])
def test_a_wait_that_runs_out_with_and_without_the_barrier_in_clean_steps(L, kernel):
    test_a_wait_that_runs_out_is_reported_and_the_context_stays_usable(wl.TINY, 1, L, "none", kernel)
