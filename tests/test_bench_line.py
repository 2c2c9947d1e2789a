"""The benchmark's line on stdout: complete for the keys that readers of it need, short, and the last
thing printed; the record of every leg goes to a file or to stderr."""
import json

import bench


def _record():
    legs = {"per_mass": {str(m): {"iterations": 814, "median_ms": 77.278} for m in range(40)}}
    return {
        "metric": bench.METRIC, "value": 42.147, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
        "ms_per_step": 94.907, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32+bf16 (V-cycle), f32 (Krylov iteration) / f64 (reliable updates, solution, true residual, coarsest)",
        "data": "synthetic: seeded quenched U(1) Metropolis configuration, Gaussian source",
        "config": {"workload": "L128_b6_massweep", "lattice": [128, 128], "beta": 6.0, "levels": 3,
                   "blocks": [[4, 4], [2, 2]], "Nv": [8, 8], "masses": [-2.078905765905, -0.05, 0.0, 0.1],
                   "m_crit": -2.0809057659048835, "tol": 1e-10, "rhs_per_solve": 1, "solves_per_step": 4,
                   "step": "setup at m_nc + 4 x (re-Galerkin/coarsest inverse, b = D^dag chi, solve)",
                   "coarsest_reuse": 12, "parallelism": "replicas x1", "l2": "flushed between timed steps (256 MiB write)"},
        "latency_ms": {"p50": 1.097, "p99": 77.353, **legs}, "plain_fp64": {"value": 20.583, "unit": "solves/s", **legs},
        "mixed_vs_plain_fp64": 2.048, "solver": "mixed", "batched_configs": [legs] * 20, "serving": [legs] * 20,
        "stencil": {"gbs": 6227.6, "frac_hbm": 0.9187}, "gpu_launches": 123456,
        "e2e": {"value": 42.889, "unit": "solves/s", "steps": 3, "h2d_bytes_per_step": 8912896, "d2h_bytes_per_step": 2097152},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 4}}


def test_line_is_short_and_complete(capsys, tmp_path):
    rec = _record()
    bench.report(rec, str(tmp_path / "full.json"))
    out = capsys.readouterr()
    assert out.err == "" and json.loads((tmp_path / "full.json").read_text()) == rec
    (line,) = out.out.strip().splitlines()
    assert len(line) <= bench.LINE_MAX
    got = json.loads(line)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
        assert got[key] == rec[key]
    assert got["latency_ms"] == {"p50": 1.097, "p99": 77.353} and got["stencil_gbs"] == 6227.6


def test_inverse_counts_its_own_tile_products():
    """The 4096-unknown coarsest level: the counts stated in kernels_inverse.cu.  One site per
    block (n = 64) on 3 x 3 sites couples every pair: the dense sweep's sum over pivots."""
    assert bench.inverse_tile_products(16, 16, 16) == (25840, 28)
    assert bench.inverse_tile_products(3, 3, 64) == (9 * 8 * 9 // 2, 9)


def test_record_goes_to_stderr_by_default(capsys):
    rec = _record()
    bench.report(rec, "")
    out = capsys.readouterr()
    assert json.loads(out.err) == rec and len(out.out.strip().splitlines()) == 1
