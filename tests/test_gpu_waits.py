"""The kernels' bounded waits: a wait that runs out ends the launch with a status, not a hang.

kvx_debug_stall_next_translate makes the first CTA of the identity kernel, or of the row-gather kernel, stop
issuing its source copies at a chosen work unit, with every on-chip wait bounded at 2 ms.  The launch must come
back (well within a second), record KVX_DEV_WAIT_TIMEOUT, and leave the context usable: the
next call, with the normal bounds, equals the oracle.
"""
import dataclasses
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2608_30963_gb300 as kvx
from paper_2608_30963_gb300 import synth

from harness import compare, make_case, oracle_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("unit", [0, 1])
def test_wait_that_runs_out_returns_a_status_and_the_next_call_is_correct(unit):
    from gpu_harness import DeviceCase
    kvx.build()
    spec = synth.config_specs()["qwen7b_to_qwen1p5b_4k"]
    spec = dataclasses.replace(spec, src=dataclasses.replace(spec.src, num_layers=4),
                               dst=dataclasses.replace(spec.dst, num_layers=4))
    c = make_case(spec, [4096])   # 256 K and 256 V units over the SMs: CTA 0 walks at least two
    g = DeviceCase(c, path=kvx.KVX_PATH_AUTO)
    assert g.tr.device_status() == 0
    g.tr.debug_stall_next_translate(unit, 2000)
    t0 = time.perf_counter()
    g.run()
    torch.cuda.synchronize()
    took = time.perf_counter() - t0
    bits = g.tr.device_status()
    assert bits & kvx.KVX_DEV_WAIT_TIMEOUT, f"status 0x{bits:x}"
    assert took < 1.0, took
    # the context is usable and the next call (normal bounds) is complete and correct
    for t in g.dst_k + g.dst_v:
        t.fill_(float("nan"))
    g.run()
    torch.cuda.synchronize()
    assert g.tr.device_status() == 0
    ok, ov = oracle_problem(c).translate()
    gk, gv = g.gather()
    compare(gk, ok, "bf16", "after a timed-out call K")
    compare(gv, ov, "bf16", "after a timed-out call V")


@pytest.mark.parametrize("unit", [0, 1, 3])
@pytest.mark.parametrize("kl", [1, 2])
def test_row_gather_wait_that_runs_out_returns_a_status_and_the_next_call_is_correct(kl, unit):
    """Spans of 1..3 rows, 256 input channels (resident weights) and 512 (two K groups, weights streamed): the
    first CTA stops with copies of earlier units, further rows and weights in flight.  Only its own units miss
    rows; a call before, the stalled one and the one after follow one another on the stream."""
    kvx.build()
    L, Hs, Ht, d, T = 8, 4, 2, 128, 4096       # 1024 units over the SMs: CTA 0 walks at least six
    rng = np.random.default_rng(3)
    n = rng.integers(1, 4, size=T)
    hi = np.cumsum(n)
    S = int(hi[-1])
    i32 = lambda x: torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(8)
    rnd = lambda *sh: torch.randn(sh, device="cuda", generator=gen).to(torch.bfloat16)
    src = [[rnd(1, Hs, S, d) for _ in range(L * kl)] for _ in range(2)]
    w = [rnd(L, Ht, kl * 2 * d, d) for _ in range(2)]
    tr = kvx.Translator(synth.ModelGeom(L * kl, Hs, d, 1e4), synth.ModelGeom(L, Ht, d, 1e6), w[0], w[1],
                        layer_map=[[j * kl + k for k in range(kl)] for j in range(L)], layers_per_target=kl)
    dst = [[[torch.full((1, Ht, T, d), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(L)] for _ in range(2)]
           for _ in range(3)]
    sl, so, lo, hi = i32([S]), i32([0, T]), i32(hi - n), i32(hi)
    run = lambda k: tr.translate(src[0], src[1], sl, so, T, dst[k][0], dst[k][1], span_lo=lo, span_hi=hi)
    run(0)
    torch.cuda.synchronize()
    assert tr.device_status() == 0
    tr.debug_stall_next_translate(unit, 2000)
    t0 = time.perf_counter()
    run(1)
    run(2)
    torch.cuda.synchronize()
    took = time.perf_counter() - t0
    assert tr.device_status() == kvx.KVX_DEV_WAIT_TIMEOUT
    assert took < 1.0, took
    missing = written = 0
    for kv in range(2):
        for j in range(L):
            good = dst[0][kv][j]
            assert not good.isnan().any()
            gone = dst[1][kv][j].isnan().all(-1)
            missing += int(gone.sum())
            written += int((~gone).sum())
            for k, rows in ((1, ~gone), (2, torch.ones_like(gone))):
                err = (dst[k][kv][j][rows].double() - good[rows].double()).norm()
                assert err <= 2.0 ** -8 * 1.5 * good.double().norm(), (k, kv, j, err)
    assert 0 < missing < written
