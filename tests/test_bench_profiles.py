"""bench.py's link between the committed ncu summaries and the kernel sources
(CPU only): a summary's DRAM bytes per launch are reported as the roofline's
`traffic` only while the kernel source the counters were taken on is
unchanged -- a comment edit keeps them, any code change drops them."""
import os

import bench


def test_fingerprint_ignores_comments_and_blank_lines(tmp_path):
    a, b, c = tmp_path / "a.cu", tmp_path / "b.cu", tmp_path / "c.cu"
    a.write_text("int f() {\n  return 1;  // one\n}\n")
    b.write_text("// a header\n\nint f() {\n  return 1;\n}\n\n")
    c.write_text("int f() {\n  return 2;\n}\n")
    fa, fb, fc = (bench.code_fingerprint(str(p)) for p in (a, b, c))
    assert fa == fb != fc
    assert len(fa) == 16 and int(fa, 16) >= 0


def test_traffic_only_for_an_unchanged_kernel(tmp_path, monkeypatch):
    src = tmp_path / "paper_1612_08608_gb300" / "csrc"
    src.mkdir(parents=True)
    prof = tmp_path / "profiles"
    prof.mkdir()
    kernel = src / "k.cu"
    kernel.write_text("__global__ void k() {}\n")
    fp = bench.code_fingerprint(str(kernel))
    (prof / "k.txt").write_text("metric   value\n"
                                "dram_bytes_per_launch: 12345\n"
                                f"kernel_code_sha256_16: {fp}\n")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    monkeypatch.setitem(bench.TRAFFIC, ("w", "k"), ("k.txt", "k.cu"))
    assert bench.traffic_per_launch("w", "k") == 12345.0
    kernel.write_text("__global__ void k() {}  // a comment only\n")
    assert bench.traffic_per_launch("w", "k") == 12345.0
    kernel.write_text("__global__ void k() { int x = 0; }\n")
    assert bench.traffic_per_launch("w", "k") is None
    assert bench.traffic_per_launch("w", "not_mapped") is None


def test_committed_summaries_match_the_committed_kernels():
    # every summary the bench reads carries its DRAM figure and the
    # fingerprint of the kernel source it was captured on, and that source
    # has not changed since
    for (workload, kernel), (summary, source) in bench.TRAFFIC.items():
        path = os.path.join(bench.ROOT, "profiles", summary)
        txt = open(path).read()
        assert "dram_bytes_per_launch:" in txt and "kernel_code_sha256_16:" in txt, summary
        assert os.path.exists(os.path.join(bench.ROOT, "paper_1612_08608_gb300", "csrc", source))
        traffic = bench.traffic_per_launch(workload, kernel)
        assert traffic is not None and traffic > 0, (summary, source)


def test_kernel_bytes_follow_the_layout_not_the_workload(monkeypatch):
    # 2 workers x 8 rows of 5 entries in distinct columns, in 100 (128 stored) columns
    import numpy as np
    from paper_1612_08608_gb300 import inputs
    N, B, d = 2, 8, 100
    sh = inputs.sparse_custom(seed=0, N=N, d=d, rows=B, lengths=[np.full(B, 5)] * N)
    for i in range(N):
        sh.col[i][:] = np.arange(40)
    monkeypatch.setattr(bench, "WORKLOAD", dict(name="sparse_logistic_hashed", N=N, B=B, d=d, loss="logistic"))
    E = N * B * 5                                          # entries, and columns touched
    bytes_of = lambda **kw: {k: v[1] for k, v in bench.kernel_work(sh, kw).items()}
    lists = bytes_of(entries=False, entry_bytes=12, streams=False)
    assert lists == {"local_step": 20 * E + 4 * N * B, "reduce": 8 * N * 128, "apply": 16 * E, "gather": 12 * E}
    touched = bytes_of(entries=True, entry_bytes=10, streams=False)
    assert touched == {"local_step": 4 * E + 10 * N * B, "reduce": 8 * N * 128, "gather": 18 * E,
                       "apply": 16 * E + 4 * N * B}
    streamed = bytes_of(entries=True, entry_bytes=8, streams=True)
    assert streamed["apply"] == (8 + 4 + 8 + 4) * E + 4 * N * B + 4 * N * 128
