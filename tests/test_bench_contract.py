"""bench.py's reference arm (the oracle timed on the host cores) prints one
JSON line with the keys of the bench contract; it needs no GPU."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reference_arm_prints_the_contract_line():
    out = subprocess.run([sys.executable, "bench.py", "--impl", "reference", "--steps", "1", "--warmup", "0"],
                         cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert out.returncode == 0, out.stderr[-500:]
    line = json.loads(out.stdout.strip().splitlines()[-1])
    assert line["impl"] == "reference"
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
                "scaling", "vs_baseline", "dtype", "data", "config", "cpu_baseline", "e2e"):
        assert key in line, key
    assert line["value"] > 0 and line["unit"] == "DOFs/s" and line["higher_is_better"] is True
    assert line["steps"] == 1 and line["n_gpus"] == 1
    assert line["e2e"]["value"] == line["value"]
    assert line["e2e"]["h2d_bytes_per_step"] == 0 and line["e2e"]["d2h_bytes_per_step"] == 0
    cb = line["cpu_baseline"]
    assert cb["kind"] == "oracle" and cb["cores"] >= 1 and cb["value"] == line["value"] and cb["sample"]
    assert "workload" in line["config"]


def test_roofline_byte_model():
    """The algorithmic bytes the bench divides by launch time: stored stencil
    words per unknown (the FP32 scalar kernels read the symmetric half, 14 of
    27 in 3D and 5 of 9 in 2D; FP64 data the full stencil; 81 for
    elasticity) and the per-unknown figures of the block kernels."""
    sys.path.insert(0, ROOT)
    import bench
    assert bench.stencil_words(3, 4) == 14 and bench.stencil_words(2, 4) == 5
    assert bench.stencil_words(3, 8) == 27 and bench.stencil_words(2, 8) == 9
    assert bench.stencil_words(3, 4, vector=True) == 81
    n, C, w = 1000, 6, 4
    b, f = bench.kernel_work("spmm", n, C, 0, w, S=14)
    assert b == (14 + 2 * C) * w * n and f == 2 * (27 * C + C) * n   # products of the full stencil
    b, f = bench.kernel_work("spmm", n, C, 0, 8, S=27)
    assert b == (27 + 2 * C) * 8 * n and f == 2 * (27 * C + C) * n
    b, _ = bench.kernel_work("orth_update", n, C, 5, w)
    assert b == (2 * 5 * C + 4 * C + 1) * w * n
    assert bench.bmin_per_iteration(1, n, C, 5, w, 14) == ((2 * C + 4) * w + 14 * w) * n
    # one MG chain of two grids with fused nu = 2 Jacobi: (S + 3) w per unknown of each grid
    ns = [10, 100]
    trace = [("init", 0.0), ("jacobi", 1.0), ("jacobi", 1.0), ("check", 0.0)]
    dom, rl, share, tot = bench.roofline(trace, ns, 2, 5, 4, {"hbm_gbs": 1000.0}, None, S=14)
    assert dom == "jacobi" and rl["launches"] == 2
    assert rl["algorithmic_bytes_per_launch"] == (14 + 3) * 4 * (ns[1] + ns[0]) / 2


def test_work_of_the_launches_as_they_are():
    """A P by the block SpMM of P: the orthogonalisation reads Z and the window's
    P_j alone, the Gram sums go with the product or in a launch of their own; large
    grids of 8-byte words smooth in two launches; a 2D restriction chain takes two or
    three grids a launch and ends above the grids of the single-block tail."""
    sys.path.insert(0, ROOT)
    import bench
    n, C, w, cnt = 1000, 6, 4, 5
    kw = dict(recurrence=False)
    assert bench.kernel_work("orth_update", n, C, cnt, w, **kw) == ((cnt + 2) * C * w * n, 2 * cnt * C * C * n)
    assert bench.kernel_work("orth_gram", n, C, cnt, w, **kw) == ((2 * C + 1) * w * n, 2 * 27 * n)
    assert bench.kernel_work("spmm", n, C, cnt, w, 14, **kw) == ((14 + 2 * C) * w * n, 2 * 27 * C * n)
    assert bench.kernel_work("spmm", n, C, cnt, w, 14, fused=True, **kw) == \
        ((15 + 2 * C) * w * n, 2 * (27 * C + 27) * n)
    # 129^3: grids of 7^3 and 3^3 unknowns in the tail, three restrictions before it
    assert bench.padded_points(127 ** 3, 3) == 128 ** 3 and bench.padded_points(95 ** 3, 3) == 96 ** 3
    assert bench.restrict_launches([1, 27, 343, 3375, 29791, 250047, 2048383][1:], 3) == [1, 1, 1]
    # 1025^2, nine grids: 15^2 and smaller in the tail, five restrictions in two launches
    ns = [(2 ** k - 1) ** 2 for k in range(2, 11)]
    assert bench.restrict_launches(ns, 2) == [2, 3]
    per = [("restrict", 1.0), ("restrict", 1.0)]
    dom, rl, _, _ = bench.roofline([("init", 0.0)] + per + [("check", 0.0)] + per, ns, 9, 5, 4, {"hbm_gbs": 1e3}, None, S=5)
    assert dom == "restrict" and rl["launches"] == 4
    assert rl["algorithmic_bytes_per_launch"] == 4 * (sum(ns[-3:]) + sum(ns[-6:-2])) / 2
    # FP64, 65^3: the fine grid takes two launches, the next one; one MG chain
    ns = [343, 3375, 29791, 250047]
    trace = [("init", 0.0)] + [("jacobi", 1.0)] * 4 + [("check", 0.0)]
    _, rl, _, _ = bench.roofline(trace, ns, 5, 5, 8, {"hbm_gbs": 1e3}, None, S=27)
    assert rl["algorithmic_bytes_per_launch"] == 8 * ((3 + 31) * ns[3] + 30 * (ns[2] + ns[1])) / 4
