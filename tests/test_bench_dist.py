"""The N > 1 logic of bench.py on CPU: two gloo ranks (one GPU per rank on a
GB300 node runs the same code over NCCL).  The path has no data exchange
(replicas: every rank splits its own copy), so what must hold is the
timing rule -- the job time is the slowest rank's -- and the whole-job
rate, plus the reference arm's "rank 0 only" rule."""
from __future__ import annotations

import io
import os
import socket
import sys
from contextlib import redirect_stdout

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def _free_port() -> int:
    with socket.socket() as s:
        s.bind(("127.0.0.1", 0))
        return s.getsockname()[1]


def _rank_main(rank: int, world: int, port: int, times, out):
    import torch.distributed as dist
    import bench
    os.environ.update(MASTER_ADDR="127.0.0.1", MASTER_PORT=str(port), RANK=str(rank),
                      WORLD_SIZE=str(world), LOCAL_RANK=str(rank))
    dist.init_process_group("gloo", rank=rank, world_size=world)
    try:
        w, r, _ = bench.dist_env()
        assert (w, r) == (world, rank)
        dist.barrier()
        t = bench.max_over_ranks(times[rank], dist, device="cpu")
        out[rank] = (t, bench.whole_job_rate(world, 1000, t))
        dist.barrier()
    finally:
        dist.destroy_process_group()


def test_max_over_ranks_and_whole_job_rate_gloo():
    import torch.multiprocessing as mp
    world = 2
    times = [0.25, 0.75]
    ctx = mp.get_context("spawn")
    with ctx.Manager() as m:
        out = m.dict()
        port = _free_port()
        procs = [ctx.Process(target=_rank_main, args=(r, world, port, times, out)) for r in range(world)]
        for p in procs:
            p.start()
        for p in procs:
            p.join(timeout=120)
        assert all(p.exitcode == 0 for p in procs), [p.exitcode for p in procs]
        res = dict(out)
    for r in range(world):
        t, rate = res[r]
        assert t == max(times)  # the job takes as long as its slowest rank
        assert rate == world * 1000 / max(times)  # all ranks' units over that time


def test_single_rank_helpers():
    import bench
    assert bench.max_over_ranks(1.5) == 1.5
    assert bench.whole_job_rate(1, 524288, 0.5) == 1048576.0


def test_reference_arm_runs_on_rank_zero_only(monkeypatch):
    import bench
    args = type("A", (), {"steps": 1, "warmup": 0, "gpus": 2})()
    monkeypatch.setenv("RANK", "1")
    monkeypatch.setenv("WORLD_SIZE", "2")
    buf = io.StringIO()
    with redirect_stdout(buf):
        bench.run_reference(args, bench.CONFIGS["hyp12"])
    assert buf.getvalue() == ""  # other ranks exit without work or output
    monkeypatch.setenv("RANK", "0")
    with redirect_stdout(buf):
        bench.run_reference(args, bench.CONFIGS["hyp12"])
    import json
    line = json.loads(buf.getvalue().strip().splitlines()[-1])
    assert line["impl"] == "reference" and line["value"] > 0
    assert line["e2e"]["h2d_bytes_per_step"] == 0 and line["cpu_baseline"]["kind"] == "oracle"


@pytest.mark.parametrize("cfg", ["hyp12", "hyp20", "hyp24mixed", "hyp28dd", "mis16"])
def test_configs_are_well_formed(cfg):
    import bench
    kind, l, n, prec = bench.CONFIGS[cfg]
    assert kind in ("hyp", "mis", "misbatch") and prec in ("fp64", "mixed", "dd")
    assert 1 <= n <= 40


def _stats(**kw):
    st = {"ms_walk": 2.0, "ms_seeds": 0.5, "ms_descend": 3.0, "walk_newton": 1000, "seed_newton": 100,
          "desc_newton": 2000, "desc_fp32": 0, "steps_fp32": 0, "finish_newton": 0, "n_starts": 4096,
          "ms_k_walk": 1.5, "ms_k_desc64": 3.0, "ms_k_desc32": 0.0, "ms_k_finish": 0.0, "desc_orbit_steps": 0}
    st.update(kw)
    return st


def test_kernel_rooflines_arithmetic():
    """achieved = counted steps x flops per step / the kernel's own time; frac
    = achieved / the measured rate of the kernel's pipe; the kernel with the
    largest time is the line's roofline."""
    import bench
    pk = {"fp64": 1.2, "fp32": 75.0}
    ks = bench.kernel_rooflines("hyp", 0, 20, [_stats()], pk)
    by = {k["kernel"]: k for k in ks}
    flops = 2000 * (13 * 20 + 24)
    assert abs(by["k_descend"]["achieved"] - flops / 3e-3 / 1e12) < 1e-12
    assert abs(by["k_descend"]["frac"] - by["k_descend"]["achieved"] / 1.2) < 1e-12
    assert by["k_walk"]["flops_per_launch"] == 900 * (13 * 20 + 24) and by["k_walk"]["pipe"] == "fp64"
    assert bench.roofline_of(ks, "x")["kernel"] == "k_descend"
    # the mixed tier: binary32 descents against the binary32 rate, the finish against binary64
    st = _stats(ms_k_desc64=0.0, desc_fp32=1500, steps_fp32=1600, finish_newton=500, ms_k_desc32=1.0,
                ms_k_finish=2.5, n_starts=(1 << 23) + 1)
    by = {k["kernel"]: k for k in bench.kernel_rooflines("hyp", 0, 20, [st], pk)}
    assert set(by) == {"k_descend_mixed", "k_finish_f64", "k_walk_mixed"}
    assert by["k_descend_mixed"]["launches"] == 2 and by["k_descend_mixed"]["peak"] == 75.0
    flops32 = 1500 * (19 * 19 + 25) + ((1 << 23) + 1) * (65 * 20 + 28)  # Newton steps + anchor orbits
    assert abs(by["k_descend_mixed"]["achieved"] - flops32 / 1e-3 / 1e12) < 1e-12
    assert abs(by["k_finish_f64"]["achieved"] - 500 * (7 * 20 + 2) / 2.5e-3 / 1e12) < 1e-12
    assert bench.roofline_of(list(by.values()), "x")["kernel"] == "k_finish_f64"
    # the binary64 descents of the mixed tier (the tip redo): desc_newton less
    # the binary32 steps and the finish steps
    st = _stats(ms_k_desc64=0.5, desc_newton=2100, desc_fp32=1500, steps_fp32=1600, finish_newton=500,
                ms_k_desc32=1.0, ms_k_finish=2.5, n_finish=300)
    by = {k["kernel"]: k for k in bench.kernel_rooflines("hyp", 0, 20, [st], pk)}
    assert by["k_descend"]["flops_per_launch"] == 100 * (13 * 20 + 24)
    # DRAM traffic per launch: the captured bytes per unit x this launch's units
    assert by["k_descend"]["traffic"] is None  # the tip redo (a list), not captured
    assert abs(by["k_descend_mixed"]["traffic"] - 32.1 * 4096) < 1e-6
    assert abs(by["k_finish_f64"]["traffic"] - 118.5 * st["n_finish"]) < 1e-6
    st = _stats(n_starts=1 << 20)
    by = {k["kernel"]: k for k in bench.kernel_rooflines("hyp", 0, 20, [st], pk)}
    assert by["k_descend"]["traffic"] == 16 * (1 << 20)
    # the batched split: orbit lengths differ per polynomial, counted by the kernel
    st = _stats(desc_orbit_steps=30000)
    k = bench.kernel_rooflines("mis", 0, 15, [st], pk)[0]
    assert k["kernel"] == "k_descend_batch" and k["flops_per_launch"] == 13 * 30000 + 24 * 2000


def test_stratified_windows():
    """One window centred in each of the equal parts of the upper half of
    the level line, aligned to whole turns, inside the line, together
    covering the requested fraction."""
    import bench
    n = 20
    J = 8 * 2 ** (n - 1) // 2
    w = bench.windows(n, 0.1, 64)
    assert len(w) == 64
    for i, (what, nn, a, b) in enumerate(w):
        assert what == "window" and nn == n and 0 <= a < b <= J and a % 8 == 0
        assert i * J // 64 <= a and b <= (i + 1) * J // 64  # inside its own part
    cover = sum(b - a for _, _, a, b in w) / J
    assert 0.09 < cover <= 0.1


def test_error_vs_oracle_on_the_host():
    """The bench's error report: the oracle's own roots of p_10 move by less
    than binary64 rounding under its binary128 polish; one root moved by
    1e-9 shows as a 1e-9 error."""
    import numpy as np
    import bench
    import oracle
    z = oracle.split("hyp", 10, want_types=False)["roots"]
    e = bench.error_vs_oracle("hyp", 0, 10, z)
    assert e["checked_fp64"] == z.size and e["max_abs"] < 1e-15 and e["within_tol"]
    z2 = z.copy()
    z2[100] += 1e-9
    e = bench.error_vs_oracle("hyp", 0, 10, z2)
    assert abs(e["max_abs"] - 1e-9) < 1e-12 and not e["within_tol"]
    zl = np.zeros_like(z2)
    zl[5] = 1e-17  # a double-double root: checked with its low part, against the dd tolerance
    e = bench.error_vs_oracle("hyp", 0, 10, z, zl, sample=64)
    assert e["checked_dd"] == 1 and e["checked_fp64"] >= 64 and e["max_abs_dd_roots"] > 5e-18


def test_the_line_stays_short():
    """The printed line with every part it can have and numbers of full length:
    short enough that a reader of the last 8 KB of the output gets it whole."""
    import json
    import math
    import bench
    x = math.pi * 1e8
    kern = [dict(bench._kernel("k_descend_mixed_%d" % i, "fp32", x, x, 3, x, x, "a description " * 8), traffic=x,
                 traffic_unit="bytes per launch " * 4) for i in range(5)]
    err = {k: x for k in ("max_abs", "max_abs_fp64_roots", "max_abs_dd_roots", "tol_fp64", "tol_dd", "checked_fp64",
                          "checked_dd", "roots", "polish_last_step_max", "host_s")}
    err.update(within_tol=True, how="binary128 " * 40)
    rec = {"config_name": "c", "workload": "p_28 hyperbolic centres, " * 5, "value": x, "unit": "roots/s",
           "ms_per_step": x, "steps": 20, "precision": "dd",
           "e2e": {"value": x, "unit": "roots/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 4294968320,
                   "ms_per_step": x, "call_ms": [x] * 500, "copy_ms": [x] * 500, "note": "n" * 320},
           "roofline": bench.roofline_of(kern, "measured in this run " * 8), "kernels": kern, "gpu_launches": 100000,
           "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 100},
           "detail": {"ms_k_something_%d" % i: x for i in range(24)}, "max_abs_err_vs_oracle": err,
           "compare": {"mixed": {"value": x, "ms_per_step": x, "all_certified": True, "speedup_vs_fp64": x, "kernels": kern}},
           "cpu_baseline": {"value": x, "unit": "roots/s", "cores": 16, "kind": "oracle", "sample": "s" * 300},
           "separation": {"ms": x, "set": "Hyp(28)", "roots": 1 << 27, "roots_per_s": x, "min_dist": x, "law": 118.4}}
    line = bench.line_of(rec, {n: rec for n in bench.DEFAULT_SUB.split(",")}, 20, 5, 1,
                         {"fp64": x, "fp32": x})
    text = json.dumps(line)
    assert len(text) < 8000, len(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline"):
        assert key in line, key
    assert abs(line["value"] / x - 1) < 1e-5 and set(line["configs"]) == set(bench.DEFAULT_SUB.split(","))


def test_rooflines_name_the_pipe_that_runs():
    """With the integer rate measured, fixed-point kernels are held against it,
    19 multiply-adds an orbit step (7 for the finish's value), and the
    polynomials kept in binary64 against binary64; launches as timed."""
    import bench
    pk = {"fp64": 1.25, "fp32": 78.0, "imad": 9.0}
    by = lambda *a: {k["kernel"]: k for k in bench.kernel_rooflines(*a, pk)}
    k = by("hyp", 0, 20, [_stats()])
    assert k["k_descend"]["pipe"] == "imad" and abs(k["k_descend"]["frac"] - 19 * 20 * 2000 / 3e-3 / 9e12) < 1e-12
    assert abs(k["k_descend"]["fp64_equiv"] - 2000 * (13 * 20 + 24) / 3e-3 / 1.25e12) < 1e-12
    assert k["k_walk"]["pipe"] == "imad"
    k = by("mis", 2, 14, [_stats()])  # roots 0, +-i: binary64
    assert k["k_descend"]["pipe"] == k["k_walk"]["pipe"] == "fp64" and "binary64" in k["k_walk"]["work"]
    k = by("q", 9, 8, [_stats()])
    assert k["k_descend_q"]["pipe"] == k["k_walk"]["pipe"] == "fp64"
    k = by("q", 9, 9, [_stats()])
    assert k["k_descend_q"]["pipe"] == "fp64" and k["k_walk"]["pipe"] == "imad"
    assert bench.kernel_rooflines("mis", 0, 15, [_stats(desc_orbit_steps=30000)], pk)[0]["pipe"] == "imad"
    st = dict(desc_fp32=1500, steps_fp32=1600, finish_newton=400, ms_k_desc32=1.0, ms_k_finish=2.5, n_finish=300,
              n_starts=(1 << 24) + 1)
    k = by("hyp", 0, 24, [_stats(n_k_timed=5, **st)])
    assert k["k_descend_mixed"]["launches"] == 2 and k["k_finish_f64"]["pipe"] == "imad"
    assert abs(k["k_finish_f64"]["achieved"] - 7 * 24 * 400 / 2.5e-3 / 1e12) < 1e-12
    k = by("hyp", 0, 22, [_stats(n_k_timed=4, **st)])
    assert k["k_descend_mixed"]["launches"] == 1 and k["k_finish_f64"]["pipe"] == "fp64"
    assert k["k_descend"]["pipe"] == "fp64"  # the tip redo of a short orbit
    assert by("mis", 8, 10, [_stats(n_k_timed=4, **st)])["k_descend_mixed"]["launches"] == 1
