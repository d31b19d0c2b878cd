"""bench.py prints one line that fits the last 2000 characters of its output, with the figures the metric names; the rest of
the record goes to the file of --details."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _record():
    """A record as run_ours makes it, with long figures and notes everywhere."""
    x = 1234.567890123456
    stage = {"kernel": "blend_bwd", "bound": "alu", "achieved": x, "peak": x, "unit": "TFLOP/s", "frac": x, "note": "n" * 500, "kernels": "k" * 200}
    decode = {f"{m}_{n}M": {"fwd_ms": x, "bwd_ms": x, "GBps": x, "frac_of_hbm_peak": x, "bytes_per_primitive": 660}
              for m in ("neural", "neural_half", "sh", "sv") for n in (1, 3, 10)}
    decode["cache"] = "c" * 100
    e2e = {"value": x, "unit": "ms/iter (8 views, fwd+bwd)", "h2d_bytes_per_step": 99_836_928, "d2h_bytes_per_step": 99_836_928, "what": "w" * 900}
    return dict(
        metric="fwd+bwd rasterizer ms/iter @1M Gaussians; appearance-decode GB/s vs HBM peak", value=x, unit="ms/iter (8 views, fwd+bwd)",
        n_gpus=8, steps=1000, warmup=1000, ms_per_step=x, higher_is_better=False, scaling="weak", vs_baseline=None, dtype="f32", data="synthetic",
        config={"workload": "w" * 240, "appearance": "neural", "n": 1_000_000, "width": 1256, "height": 828, "views": 8, "cache": "c" * 90,
                "multi_gpu": "replicas only"},
        gprimitives_per_s=x, ms_per_step_single_stream=x, ms_per_step_streams_no_graph=x, cuda_graph={"ms_per_step": x, "captured": True}, streams=4,
        clocks=dict(sm_mhz=1965.0, sm_max_mhz=1965.0, reasons=["sw_power_cap"], samples=99), e2e=e2e, e2e_gradients_to_host=e2e,
        gpu_launches=160_000, roofline=stage, rooflines={"blend_bwd": stage}, sh={"ms_per_step": x}, sv={"ms_per_step": x},
        appearance_decode=decode, cpu_baseline={"value": x, "unit": "ms/iter (8 views, fwd+bwd)", "cores": 16, "kind": "oracle", "sample": "s" * 100})


def test_the_line_fits_and_holds_the_figures():
    sys.path.insert(0, ROOT)
    import bench
    out = _record()
    text = json.dumps(bench.headline(out))
    assert len(text) < 2000 and "\n" not in text
    line = json.loads(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype",
                "data", "config", "clocks", "gpu_launches"):
        assert line[key] == out[key], key
    assert line["e2e"]["h2d_bytes_per_step"] == out["e2e"]["h2d_bytes_per_step"] and line["e2e"]["value"] > 0
    assert line["appearance_decode"]["neural_1M"]["frac_of_hbm_peak"] > 0


def test_parts_that_were_skipped():
    sys.path.insert(0, ROOT)
    import bench
    out = _record()
    del out["cpu_baseline"]
    out.update(e2e=None, appearance_decode=None, sh=None, sv=None, clocks=None)
    line = json.loads(json.dumps(bench.headline(out)))
    assert line["e2e"] is None and line["appearance_decode"] == {} and line["value"] == out["value"]
