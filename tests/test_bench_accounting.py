"""The benchmark's roofline numerators (algorithmic bytes per launch) against the weight and cache
sizes computed independently from the drafter's shape: every GEMM streams its weights once, the
attention reads the context keys/values once, the argmax reads the logits once."""
import numpy as np
import pytest

import bench
import synth

GEMMS = {"gemm_qkv": "D", "gemm_o": "D", "gemm_gate_up": "D", "gemm_down": "D",
         "gemm_kv_ctx": 1, "gemm_lm_head": 1}


def _weight_bytes(s):
    e = 2 if s.dtype == "bf16" else 4
    per_layer = (s.d_q + 2 * s.d_kv) * s.d + s.d * s.d_q + 3 * s.d * s.ffn + 2 * s.d_kv * s.d
    return e * (s.n_draft_layers * per_layer + s.vocab * s.d)


@pytest.mark.parametrize("name", ["qwen3_4b", "qwen3_8b_b4", "gptoss_20b_b2"])
def test_gemm_bytes_are_the_weights_plus_small_activations(name):
    w = synth.preset(name)
    s = w.shape
    tau = 6.0
    total = 0.0
    for k, n in GEMMS.items():
        launches = s.n_draft_layers if n == "D" else n
        total += launches * bench.algorithmic_bytes(w, k, tau)
    weights = _weight_bytes(s)
    # activations (inputs, outputs, the fp32 residual) add a few per cent at 16..64 token rows
    assert weights <= total <= 1.05 * weights, (total, weights)


def test_qwen3_4b_step_bytes_and_lower_bound():
    """The Qwen3-4B-shaped step: 1.858 GB of GEMM bytes (weights 1.857 GB), 1.91 GB in all, so
    0.28 ms at the measured 6785 GB/s copy bandwidth."""
    w = synth.preset("qwen3_4b")
    s = w.shape
    tau = 6.4
    gemm = sum((s.n_draft_layers if n == "D" else n) * bench.algorithmic_bytes(w, k, tau)
               for k, n in GEMMS.items())
    assert abs(gemm - 1.858e9) < 0.002e9
    kv = bench.algorithmic_bytes(w, "attention", tau)
    # context keys and values of one layer: (L + B) positions x 2 x d_kv x 2 bytes, plus Q and O
    L = float(np.mean(w.ctx_lens))
    assert kv == pytest.approx((L + s.block) * 2 * s.d_kv * 2 + 2 * s.block * s.d_q * 2)
    step = gemm + s.n_draft_layers * kv + bench.algorithmic_bytes(w, "argmax", tau) + \
        bench.algorithmic_bytes(w, "fuse_layers", tau)
    assert abs(step - 1.91e9) < 0.01e9
    assert abs(step / 6785.2e9 * 1e3 - 0.282) < 0.002


def test_argmax_reads_the_mask_rows_logits_once():
    w = synth.preset("qwen3_4b")
    s = w.shape
    assert bench.algorithmic_bytes(w, "argmax", 6.0) == w.batch * (s.block - 1) * s.vocab * 4


def test_event_timed_gemms_are_held_against_the_traced_step():
    """The fp32 drafter's GEMMs, timed by event pairs: their sum holds the launches' latencies, so it may exceed
    the step without events (153.9 us of pairs were seen beside a step of 132.9), but not the traced one."""
    pairs = {"gemm_qkv": [0.0101] * 8, "gemm_o": [0.0095] * 8, "gemm_gate_up": [0.0092] * 8, "gemm_down": [0.00967] * 8}
    us = bench.event_gemm_us(pairs, traced_ms=0.31, nb=2)
    assert us == pytest.approx(1e3 * sum(sum(t) for t in pairs.values()) / 2) and us > 132.9
    with pytest.raises(RuntimeError, match="traced step"):
        bench.event_gemm_us(pairs, traced_ms=0.13, nb=2)


def test_a_failed_configuration_leaves_the_headline(monkeypatch, capsys):
    """One JSON line with the headline's value also when a further configuration's measurement fails."""
    import json
    import sys

    import torch

    def measure(w, *a, **kw):
        if w.name == "tiny_f32":
            raise RuntimeError("GEMM time exceeds the step")
        return {"value": 1.5, "unit": bench.UNIT, "config": {"workload": w.name}}

    monkeypatch.setattr(torch.cuda, "set_device", lambda i: None)
    monkeypatch.setattr(bench, "measure", measure)
    monkeypatch.setattr(sys, "argv", ["bench.py"])
    assert bench.main() in (0, None)
    out = capsys.readouterr().out.strip().splitlines()
    line = json.loads(out[0])
    assert len(out) == 1 and line["value"] == 1.5
    assert "GEMM time" in line["configs"]["tiny_f32"]["error"]
    assert all(line["configs"][n]["value"] == 1.5 for n in bench.CONFIG_SET if n not in ("tiny_f32", bench.HEADLINE))


def test_launches_behind_the_fp32_attention():
    """One launch up to three 64-key tiles (184 cached positions and a block of 8), a combine launch beyond, none
    when 304 query tiles fill 152 SMs twice; bf16 always one."""
    s = synth.preset("tiny_f32").shape
    assert [bench.kernels_per_trace(s, 1, n, 152)["attention"] for n in (128, 184, 185, 4000)] == [1, 1, 2, 2]
    assert bench.kernels_per_trace(s, 152, 4000, 152)["attention"] == 1
    assert bench.kernels_per_trace(synth.preset("qwen3_4b").shape, 1, 4000, 152)["attention"] == 1


@pytest.mark.parametrize("changed", [None, "gemm_tc.cu", "epilogue.cuh", "umma.cuh"])
def test_gemm_traffic_belongs_to_the_sources_it_was_measured_on(tmp_path, monkeypatch, changed):
    """The committed DRAM bytes are reported only while every source of the kernel is the one they came from."""
    import hashlib
    import json
    csrc = tmp_path / "paper_2606_02091_gb300" / "csrc"
    csrc.mkdir(parents=True)
    (tmp_path / "profiles").mkdir()
    files = ("gemm_tc.cu", "epilogue.cuh", "umma.cuh")
    for f in files:
        (csrc / f).write_text(f + "\n")
    h = hashlib.sha256(b"".join((csrc / f).read_bytes() for f in files)).hexdigest()[:16]
    (tmp_path / "profiles" / "gemm_tc_traffic_qwen3_4b.json").write_text(
        json.dumps({"dram_bytes_per_step": 7.0, "source_sha256_16": h}))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    if changed:
        (csrc / changed).write_text("other\n")
    assert bench.gemm_traffic(synth.preset("qwen3_4b")) == (None if changed else 7.0)
