"""Host logic without a GPU: the chunking of the staged plan (tn_chunk_bounds), the bench's
JSON line of the reference arm (the FP64 oracle on the host cores) and its clock record."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def built():
    from paper_1905_01330_gb300 import build
    return build.build()


@pytest.mark.parametrize("weights,chunks,bounds", [
    ([1] * 8, 4, [0, 2, 4, 6, 8]),
    ([1] * 7, 3, [0, 2, 5, 7]),
    ([10, 1, 1, 1], 3, [0, 1, 2, 4]),       # a heavy first item ends a run by itself
    ([1, 1, 1, 10], 3, [0, 3, 4]),          # a heavy last item: fewer runs
    ([5.68e6, 8.2e5] + [4e4] * 20, 3, [0, 1, 2, 22]),   # the staged-plan GPU test's specs
    ([5], 8, [0, 1]),
    ([], 4, [0, 0]),
])
def test_chunk_bounds(built, weights, chunks, bounds):
    from paper_1905_01330_gb300.tn import chunk_bounds
    got = chunk_bounds(weights, chunks)  # tn_chunk_bounds, host code of libtn.so
    assert got == bounds
    assert all(a < b for a, b in zip(got, got[1:])) or not weights


def test_chunk_bounds_properties_on_random_weights(built):
    """On random weights (zeros and heavy items included): the bounds start at
    0, end at n, rise strictly, give at most `chunks` runs, and no run of more
    than one item exceeds the ideal share by more than twice the largest item
    (each cut lands within one item of its ideal place)."""
    import random
    from paper_1905_01330_gb300.tn import chunk_bounds
    rnd = random.Random(5)
    for _ in range(300):
        n = rnd.randint(1, 60)
        w = [rnd.choice([0.0, rnd.random(), 10 * rnd.random(), 1000 * rnd.random()]) for _ in range(n)]
        chunks = rnd.randint(1, 12)
        b = chunk_bounds(w, chunks)
        assert b[0] == 0 and b[-1] == n
        assert all(x < y for x, y in zip(b, b[1:]))
        assert len(b) - 1 <= chunks
        share, big = sum(w) / chunks, max(w)
        for lo, hi in zip(b, b[1:]):
            if hi - lo > 1:
                assert sum(w[lo:hi]) <= share + 2 * big + 1e-9, (w, chunks, b)


def test_reference_arm_json_line():
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--steps", "1",
                          "--warmup", "0"], capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert out.returncode == 0, out.stderr[-2000:]
    line = json.loads([l for l in out.stdout.splitlines() if l.startswith("{")][-1])
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
                "scaling", "vs_baseline", "dtype", "data", "config", "cpu_baseline", "e2e"):
        assert key in line, key
    assert line["impl"] == "reference" and line["dtype"] == "f64"
    assert line["cpu_baseline"]["kind"] == "oracle" and line["cpu_baseline"]["value"] == line["value"]
    assert line["e2e"] == {"value": line["value"], "unit": line["unit"], "h2d_bytes_per_step": 0,
                           "d2h_bytes_per_step": 0}


def test_clock_sampler_keeps_samples_of_the_timed_region(tmp_path, monkeypatch):
    """The bench's clock record: samples taken between start() and stop()
    only, with the throttle reasons parsed from nvidia-smi's CSV. A stand-in
    nvidia-smi on PATH prints one CSV line every 50 ms."""
    fake = tmp_path / "nvidia-smi"
    fake.write_text("#!/bin/sh\nwhile true; do\n"
                    "  echo '0, 2070, 2070, 512.3, 0x4, Not Active, Not Active, Not Active, Active'\n"
                    "  sleep 0.05\ndone\n")
    fake.chmod(0o755)
    monkeypatch.setenv("PATH", str(tmp_path) + os.pathsep + os.environ.get("PATH", ""))
    sys.path.insert(0, ROOT)
    try:
        import bench
    finally:
        sys.path.remove(ROOT)
    import time
    s = bench.ClockSampler(0)
    s.start()
    time.sleep(0.4)
    c = s.stop()
    assert c is not None
    assert c["sm_mhz"] == 2070.0 and c["sm_max_mhz"] == 2070.0
    assert c["reasons"] == ["sw_power_cap"]
    assert 3 <= c["samples"] <= 12
    # without nvidia-smi there is no record (and no error)
    monkeypatch.setenv("PATH", str(tmp_path / "none"))
    s = bench.ClockSampler(0)
    s.start()
    assert s.stop() is None


PLANS = r"""
#include <chrono>
#include <cstdio>
#include <cstring>
#include "tn_internal.h"
using namespace tn;
int main(int argc, char** argv) {
  const bool group = !strcmp(argv[1], "group");
  const SimtPlan how = group ? SimtPlan::group : !strcmp(argv[1], "sweep") ? SimtPlan::sweep : SimtPlan::alone;
  long long M, N, K, ta, tb;
  while (scanf("%lld %lld %lld %lld %lld", &M, &N, &K, &ta, &tb) == 5) {
    tn_tensor A{}, B{}, C{};
    A.data = B.data = C.data = (void*)4096;
    A.rank = B.rank = C.rank = 2;
    A.dtype = B.dtype = C.dtype = TN_F32;
    A.shape[0] = ta ? K : M; A.shape[1] = ta ? M : K;
    B.shape[0] = tb ? N : K; B.shape[1] = tb ? K : N;
    C.shape[0] = M; C.shape[1] = N;
    const int la = ta ? 0 : 1, lb = tb ? 1 : 0;
    ContractDesc d;
    if (plan_contract(&A, &la, &B, &lb, 1, &C, &d) != TN_OK) return 1;
    plan_units(&d, group ? 1 : 304);
    const long long ranges = d.splits, range = d.k_per_split;
    const auto t0 = std::chrono::steady_clock::now();
    plan_simt(&d, how, group ? 4 : 1);
    const double us = std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now() - t0).count();
    printf("%lld %lld %d %lld %d %.2f\n", ranges, range, (int)d.splits, (long long)d.k_per_split, (int)d.chunk, us);
  }
}
"""


def simt_plans(built, tmp_path, how, cases):
    """(k ranges of plan_units, their length, k ranges and length of plan_simt, its chunk, microseconds) per (M, N, K, A
    transposed, B transposed)."""
    src, exe = tmp_path / "plans.cpp", tmp_path / "plans"
    src.write_text(PLANS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_1905_01330_gb300", "csrc"),
                    "-I", "/usr/local/cuda/include", str(src), built, "-Wl,-rpath," + os.path.dirname(built),
                    "-o", str(exe)], check=True, timeout=300)
    out = subprocess.run([str(exe), how], input="".join("%d %d %d %d %d\n" % c for c in cases), capture_output=True,
                         text=True, check=True, timeout=300).stdout.split("\n")
    return [[float(x) for x in line.split()] for line in out if line]


def test_sweep_results_are_sums_of_the_k_ranges_one_by_one(built, tmp_path):
    """A float32 contraction of a sweep adds the chains of plan_units' k ranges
    (at most 2048 shared indices each) to a result one by one: a unit runs one
    of them, or all in ascending order. Sums of sums, which no order of such
    additions gives, are for lone contractions only. Over the bonds an energy
    or norm sweep meets, rising, level and falling, and MPO bonds 1 to 5."""
    bonds = [(a, b) for c in (100, 256, 300, 383, 384, 400, 512, 640, 1024) for a, b in ((c, c), (c, c // 2), (c // 2, c))]
    cases = []
    for a, b in bonds:
        for d in (2, 3):
            cases += [(a, d * b, a, 1, 0), (b, b, d * a, 1, 0)]                       # norm
            for w in (2, 4, 6):
                cases += [(w * a, d * b, a, 1, 0), (w * b, b, d * a, 0, 0)]           # energy
    several = 0
    for case, (ranges, rng, units, per, chunk, _) in zip(cases, simt_plans(built, tmp_path, "sweep", cases)):
        assert chunk * 64 == min(rng, 2048) and per % (chunk * 64) == 0, case
        assert units == 1 or (units == ranges and per == rng), case
        several += ranges > 2
    assert several >= 20


def test_planning_a_long_shared_index_is_quick(built, tmp_path):
    """A lone float32 contraction's plan takes microseconds whatever the length
    of its shared index (tens of thousands of k ranges), and covers it."""
    cases = [(m, n, k, 0, 0) for m, n in ((1, 1), (2, 5), (3, 1)) for k in (10 ** 6, 10 ** 7, 10 ** 8, 2 * 10 ** 8 + 1)]
    plans = simt_plans(built, tmp_path, "alone", cases * 5)
    for case, (_, _, units, per, chunk, _) in zip(cases * 5, plans):
        assert units * per >= case[2] > (units - 1) * per and per % (64 * chunk) == 0, (case, units, per)
    assert min(max(p[5] for p in plans[i * len(cases):(i + 1) * len(cases)]) for i in range(5)) <= 100.0


def test_a_group_keeps_the_lengths_of_its_chains(built, tmp_path):
    """A large float32 group runs up to four k ranges of a tile in one unit, as
    chains of the lengths plan_units gave them (even ones: 36 slabs are 18 + 18,
    not 32 + 4, whose longer chain rounds worse)."""
    cases = [(640, 512, k, 0, 0) for k in (40, 64, 2048, 2049, 2304, 4200, 6145, 9000, 50000)]
    for case, (ranges, rng, units, per, chunk, _) in zip(cases, simt_plans(built, tmp_path, "group", cases)):
        assert chunk * 64 == rng and per == min(4, ranges) * rng and units == -(-case[2] // per), case


def test_lone_contractions_spread_a_long_shared_index(built, tmp_path):
    """A lone float32 contraction of a few dozen tiles cuts its shared index
    into as many ranges as the SMs take, not two at most."""
    cases = [(885, 150, 2862, 0, 0), (150, 885, 2862, 1, 1), (1951, 367, 1797, 0, 1), (640, 640, 5000, 0, 1),
             (128, 2048, 4000, 0, 0), (118, 1361, 1417, 1, 1)]
    for case, (_, _, units, *_) in zip(cases, simt_plans(built, tmp_path, "alone", cases)):
        assert units >= 3, case


@pytest.mark.parametrize("sweeps", [13, -40])
def test_split_node_warns_at_the_sweep_limit(monkeypatch, sweeps):
    """The binding says so when the library reports that the sweeps ran out
    (a negative count), whether or not the caller asked for the count."""
    import ctypes
    import warnings
    import torch
    from paper_1905_01330_gb300 import tn

    class Lib:
        def tn_split_node_workspace_bytes(self, *a):
            return 256

        def tn_split_node(self, *a):
            ctypes.cast(a[12], ctypes.POINTER(ctypes.c_int64))[0] = 2
            ctypes.cast(a[13], ctypes.POINTER(ctypes.c_int32))[0] = sweeps
            return 0

    monkeypatch.setattr(tn, "load", lambda: Lib())
    monkeypatch.setattr(tn, "tensor_desc", lambda t: ctypes.c_int(0))
    monkeypatch.setattr(tn, "_workspace", lambda n, dev: torch.empty(n, dtype=torch.uint8))
    monkeypatch.setattr(tn, "_stream", lambda s: None)
    with warnings.catch_warnings(record=True) as got:
        warnings.simplefilter("always")
        u, vh, dropped = tn.split_node(torch.ones(3, 4), [0], [1])
    assert u.shape == (3, 2) and vh.shape == (2, 4) and dropped.shape == (1,)
    assert [w.category for w in got] == ([RuntimeWarning] if sweeps < 0 else [])


@pytest.mark.parametrize("n", [1, 2, 15, 16, 40])
def test_chain_descriptions_short_and_long(n):
    """Both ways of filling a chain's arrays hold the bonds and pointers."""
    import torch
    from paper_1905_01330_gb300 import tn
    bonds = [1] + [2 + i % 5 for i in range(n - 1)] + [1]
    cores = [torch.zeros(bonds[i], 3, bonds[i + 1]) for i in range(n)]
    ch, keep = tn._chain(cores, bonds, 3)
    assert (ch.n, ch.d) == (n, 3) and keep[2] is cores
    assert [ch.bond[i] for i in range(n + 1)] == bonds
    assert [ch.cores[i] for i in range(n)] == [c.data_ptr() for c in cores]
