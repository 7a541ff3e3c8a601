"""The bench's synthetic workloads are seeded and have the stated shapes (no GPU needed)."""
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402

E, NU = 1.0, 0.3


def test_uneven_batch_is_seeded_and_spans_the_stated_mix():
    a = bench.batch_problems()
    b = bench.batch_problems()
    assert len(a) == 64
    for p, q in zip(a, b):
        assert (p["n"], p["nz"], p["rough"]) == (q["n"], q["nz"], q["rough"])
        assert np.array_equal(p["h"], q["h"]) and p["loads"] == q["loads"]
    assert {p["n"] for p in a} == {64, 128, 256, 512}
    assert {p["nz"] for p in a} == {8, 16, 32}
    assert 16 < sum(p["rough"] for p in a) < 48
    es = E / (1 - NU * NU)
    for p in a:
        n, h, z = p["n"], p["h"], p["z"]
        assert h.shape == (n, n) and z[0] == 0.0 and z.size == p["nz"]
        # five equal increments; the total load lies in the decade below the 10 % area load
        loads = np.array(p["loads"])
        assert np.allclose(np.diff(loads), loads[0])
        if p["rough"]:
            w10 = 0.1 * es * 0.1 / 2.0
            assert abs(z[-1] - 0.05) < 1e-12 and abs(h.mean()) < 1e-12
        else:
            w10 = 4.0 * es * np.sqrt(0.1 / np.pi) ** 3 / (3.0 * 0.5)
            assert abs(z[-1] - 0.5) < 1e-12
        assert 0.1 * w10 * (1 - 1e-12) <= loads[-1] <= w10 * (1 + 1e-12)


def test_rough_surfaces_of_the_batch_have_the_stated_slope():
    """Spectral rms slope sqrt(mean |grad h|^2) = 0.1 for the self-affine surfaces among the first
    twelve problems."""
    for p in bench.batch_problems()[:12]:
        if not p["rough"]:
            continue
        n, h = p["n"], p["h"]
        k = np.fft.fftfreq(n, 1.0 / n)
        K2, K1 = np.meshgrid(k, k, indexing="ij")
        g = np.fft.fft2(h)
        slope = np.sqrt(np.sum(((2 * np.pi) ** 2) * (K1 ** 2 + K2 ** 2) * np.abs(g) ** 2)) / (n * n)
        assert abs(slope - 0.1) < 1e-9


def test_reference_arm_line_keeps_the_contract():
    """`bench.py --impl reference` (the oracle on the host cores, no GPU) prints one JSON line
    with the GPU arm's metric and unit, a measured step time that the run can account for, and
    the extrapolated one-core apply time beside it."""
    import json
    import subprocess

    r = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--steps", "1",
                        "--warmup", "3"], capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [x for x in r.stdout.splitlines() if x.startswith("{")]
    assert len(lines) == 1
    d = json.loads(lines[0])
    assert d["impl"] == "reference" and d["metric"] == bench.METRIC and d["unit"] == bench.UNIT
    assert d["higher_is_better"] is True and d["value"] > 0 and d["steps"] == 1 and d["warmup"] == 3
    assert 0 < d["ms_per_step"] < 600e3
    assert d["ms_per_apply_one_core_extrapolated"] > d["ms_per_step"]
    assert d["cpu_baseline"]["kind"] == "oracle" and d["cpu_baseline"]["cores"] >= 1
    assert d["e2e"]["h2d_bytes_per_step"] == 0 and d["e2e"]["d2h_bytes_per_step"] == 0


def test_batch_runs_every_problem_with_the_carried_relaxation():
    for pb in bench.batch_problems(64, 1814):
        assert pb["relax_mode"] == 1
        assert pb["relax"] == (0.3 if pb["rough"] else 0.5)


def test_result_line_is_short_and_keeps_the_contract():
    """The line printed on stdout stays below bench.LINE_MAX characters with every workload's metrics in
    it (a 23 KB line did not survive a captured output's tail); contract keys pass unchanged."""
    import json

    keys = {"metric": bench.METRIC, "value": 1.25e10, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 0.65123456789, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32", "data": "synthetic", "gpu_launches": 100, "config": {"workload": "w", "n1": 512},
            "e2e": {"value": 6.5e9, "h2d_bytes_per_step": 402653184, "d2h_bytes_per_step": 402653184},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}}
    rec = [{"n": 512, "nz": 32, "ms": 3444.142112000, "iters": [3, 13, 24, 30, 30]} for _ in range(64)]
    big = dict(keys, solves={"batch": {"solves_per_s": 1.23456789, "per_problem": rec, "grids": [64, 128, 256, 512]}},
               scaling_sweep={"ms": {"fp32_%d" % n: 0.1234567891 for n in (4, 8, 16)}})
    out = bench.short_line(big)
    assert {k: out[k] for k in keys} == keys
    assert out["solves"]["batch"] == {"solves_per_s": 1.23457, "grids": [64, 128, 256, 512]}
    assert out["scaling_sweep"]["ms"]["fp32_8"] == 0.123457
    many = dict(big, solves={"m%d" % i: {"x%d" % j: 0.123456789 for j in range(40)} for i in range(40)})
    assert len(json.dumps(bench.short_line(many))) <= bench.LINE_MAX
    assert {k: bench.short_line(many)[k] for k in keys} == keys
