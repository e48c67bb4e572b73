"""The rule that sends an FP64 product to the digit engine picks the engine that was
measured faster (GB300, us: digits, FP64), batches of small products included,
whose tiles are mostly padding."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))

# M, N, batches, K per group, digits us, FP64 us
TIMES = [
    (16, 16, 4096, [16], 227, 44), (16, 16, 2048, [16], 108, 25), (16, 16, 192, [256], 56, 41),
    (16, 16, 768, [256], 156, 119), (16, 256, 64, [16] * 5, 80, 47), (16, 256, 256, [16] * 5, 271, 170),
    (256, 16, 256, [16], 39, 44), (32, 32, 512, [32], 35, 43), (32, 32, 2048, [32], 109, 143),
    (32, 32, 1024, [32], 57, 74), (32, 32, 48, [256], 29, 51), (32, 32, 192, [256], 57, 127),
    (32, 256, 16, [32] * 5, 45, 68), (32, 1024, 16, [32] * 5, 72, 182), (32, 32, 48, [1024], 52, 143),
    (1024, 32, 16, [32], 14, 43), (64, 64, 64, [64], 18, 59), (64, 4096, 1, [64] * 17, 113, 619),
    (128, 128, 128, [128] * 3, 102, 1621), (128, 16384, 1, [128], 37, 557), (128, 128, 1, [16384], 56, 479),
    (96, 80, 1, [10007], 54, 253), (17, 31, 1, [40007], 57, 107), (16, 16, 1, [32768], 43, 55),
    (16, 16, 1, [262144], 186, 375), (24, 24, 1, [16384], 29, 51), (64, 16, 1, [16384], 31, 51),
]


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path_factory.mktemp("ozrule") / "driver")
    subprocess.run([gxx, "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "oz_rule_driver.cpp")], check=True)

    def run(rows):
        text = "".join(f"{m} {n} {b} {len(k)} {' '.join(map(str, k))}\n" for m, n, b, k in rows)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return [int(x) for x in out.split()]
    return run


def test_faster_engine_is_chosen(rule):
    got = rule([t[:4] for t in TIMES])
    for (m, n, b, k, dig, f64), use in zip(TIMES, got):
        assert use == (dig < f64), (m, n, b, k)


def test_small_products_stay_on_the_fp64_kernel(rule):
    assert rule([(128, 128, 1, [128]), (64, 64, 16, [64]), (16, 16, 1, [16])]) == [0, 0, 0]
