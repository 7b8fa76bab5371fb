"""bench.py's CPU-only modes run without a GPU: the reference arm (the oracle timed on the C2
workload) and the per-configuration oracle suite."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_cpu_suite_prints_one_line_per_configuration_and_thread_count():
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--cpu-suite", "--cpu-seconds", "0.1"],
                         capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert out.returncode == 0, out.stderr[-2000:]
    rows = [json.loads(l) for l in out.stdout.splitlines() if l.startswith("{")]
    assert {r["cfg"] for r in rows} == {"C1", "C2", "C3", "C4", "C5"}
    assert all(r["impl"] == "cpu-oracle" and r["us"] > 0 and r["eff_gbs"] > 0 for r in rows)
    assert 1 in {r["threads"] for r in rows}


def test_reference_arm_prints_the_contract_line():
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--steps", "1", "--warmup", "1"],
                         capture_output=True, text=True, timeout=900, cwd=ROOT)
    assert out.returncode == 0, out.stderr[-2000:]
    lines = [l for l in out.stdout.splitlines() if l.startswith("{")]
    assert len(lines) == 1
    r = json.loads(lines[0])
    assert r["impl"] == "reference" and r["metric"] == "effective collective GB/s" and r["unit"] == "GB/s"
    assert r["higher_is_better"] is True and r["n_gpus"] == 1 and r["steps"] == 1 and r["warmup"] == 1
    assert r["value"] > 0 and r["ms_per_step"] > 0 and r["vs_baseline"] is None
    assert r["cpu_baseline"]["kind"] == "oracle" and r["cpu_baseline"]["cores"] >= 1 and r["cpu_baseline"]["value"] == r["value"]
    assert r["e2e"] == {"value": r["value"], "unit": "GB/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}
    assert "workload" in r["config"]


def test_the_printed_line_is_short(tmp_path, capsys):
    """Whoever keeps the last 3 KB of the output must find the whole line in them; every configuration goes to a file."""
    sys.path.insert(0, ROOT)
    import bench
    text = "x" * 60
    entry = {f"number_{i}": 1234.56789012345 + i for i in range(12)}
    line = {"metric": "effective collective GB/s", "value": 714.123456789012, "unit": "GB/s", "config": {k: text * 3 for k in "abcd"},
            "clocks": {"sm_mhz": 1965, "reasons": []}, "e2e": dict(entry, api=text), "roofline": dict(entry, kernel=text), "cpu_baseline": dict(list(entry.items())[:3], sample=text),
            "small_allreduce": {"metric": text, "p50_us": 1.23456789, "all": {"oneshot": entry, "fused": entry}}, "detail": {str(i): entry for i in range(100)}}
    bench.emit(line, str(tmp_path / "detail.json"))
    out = capsys.readouterr().out
    assert out.count("\n") == 1 and len(out) < 2800
    short, full = json.loads(out), json.loads((tmp_path / "detail.json").read_text())
    assert full == line and "detail" not in short and "all" not in short["small_allreduce"]
    assert set(line) - set(short) == {"detail"} and abs(short["value"] / line["value"] - 1) < 1e-5


def test_a_ring_whose_partial_sums_stay_on_the_sms_moves_inputs_and_outputs():
    """The op list of a ring counts every hop: bytes that a folded ring, or one with its hops in shared memory, never moves."""
    import types

    import bench_suite as S
    from paper_2609_36954_b200 import binding as B
    R, n, es = 8, 1 << 20, 2
    comm = B.pl_comm_create_planner(R, B.PL_BF16)  # on the op queues: hops through memory
    s = B.pl_schedule_build(comm, B.PL_REDUCE_SCATTER, B.PL_ALGO_RING, n, 65536, None)
    try:
        info = B.pl_schedule_info(s)
        ins, outs = R * n * es, n * es
        assert info.bytes_written > 4 * outs
        for algo in ("ring", "ring_folded"):
            assert S.moved_bytes(info, algo, R) == (info.bytes_read, info.bytes_written)
            # what a GPU communicator reports for the same schedule
            on_sms = types.SimpleNamespace(bytes_read=info.bytes_read, bytes_written=info.bytes_written, hbm_bytes=ins + outs,
                                           in_bytes=info.in_bytes, out_bytes=info.out_bytes)
            assert S.moved_bytes(on_sms, algo, R) == (ins, outs)
    finally:
        B.pl_schedule_destroy(s)
        B.pl_comm_destroy(comm)
