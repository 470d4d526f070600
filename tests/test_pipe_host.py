"""The tensor-core pipeline's roles on host threads (tests/host/pipe.cpp): every
tile meets its own decoder's weights and its own slots, whatever the runs of
decoders, the images in shared memory and the order in which roles get on; and
when a role never starts, the others' waits run out without an MMA or a commit
that was never prepared."""
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_27888_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture(scope="module")
def pipe(tmp_path_factory):
    d = tmp_path_factory.mktemp("pipe") / "csrc"
    d.mkdir()
    (d.parent / "include").symlink_to(os.path.join(ROOT, "include"))
    shutil.copy(os.path.join(CSRC, "decode_pipe.cuh"), d)
    for f in ("pipe.cpp", "tcgen05.cuh"):
        shutil.copy(os.path.join(ROOT, "tests", "host", f), d)
    src = open(os.path.join(CSRC, "ntc_internal.cuh")).read()
    parts = [re.search(rf"^struct (?:alignas\(16\) )?{n} {{.*?^}};", src, re.M | re.S).group(0)
             for n in ("GridDesc", "Buckets", "TileWalk")]
    (d / "parts.cuh").write_text("namespace ntc {\n" + "\n".join(parts) + "\n}\n")
    exe = str(d / "pipe")
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", os.path.join(CUDA, "include"), str(d / "pipe.cpp"), "-o", exe],
                   check=True)

    def run(*args):
        return subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=300).stdout
    return run


RUNS = {"one decoder": [70], "every tile another": [1] * 70, "runs of one to three": [1, 3, 2, 0, 1, 1, 2, 3] * 5,
        "empty decoders, long runs": [0, 0, 17, 0, 40, 1, 0, 9]}
SHAPES = [(64, 0, 2), (128, 0, 2), (64, 8, 3), (64, 16, 1), (128, 8, 4), (128, 16, 3)]  # H; 0 or latent channels; layers


@pytest.mark.parametrize("runs", RUNS)
@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_every_tile_meets_its_decoder(pipe, shape, runs):
    H, general, layers = shape
    for grid, cta in ((1, 0), (3, 2)):
        out = pipe("run", H, general, layers, grid, cta, 7, 2, *RUNS[runs])
        assert out.endswith("status 0\ndone\n"), out


@pytest.mark.parametrize("silent", ["dispatcher", "loader", "producer"])
@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_waits_that_run_out_leave_memory_alone(pipe, shape, silent):
    H, general, layers = shape
    out = pipe("silent-" + silent, H, general, layers, 2, 1, 3, 1, *[3] * 12)
    assert out.endswith("status 1\ndone\n"), out


def test_bias_blocks_add_up_to_the_fp32_bias(pipe):
    rng = np.random.default_rng(3)
    b = (rng.uniform(1, 2, 4000) * 2.0 ** rng.integers(-30, 30, 4000) * rng.choice([-1, 1], 4000)).astype(np.float32)
    b = np.concatenate([b, np.array([0, 1, -1, 0.1, 65504, 65536, 70000, -2.0 ** 30, 65519.0 * 2 ** 15, 2.0 ** -15, 2.0 ** -40, np.inf,
                                     -np.inf, np.nan], np.float32)])
    got = np.array([[float(x) for x in line.split()] for line in pipe("bias", *(f"{x:08x}" for x in b.view(np.uint32))).splitlines()])
    half, bf16 = got.T
    exact = np.abs(b) >= 2.0 ** -15
    assert np.array_equal(half[exact], b[exact].astype(np.float64))
    small = np.abs(b) < 2.0 ** -15
    assert np.abs(half[small] - b[small]).max() <= 2.0 ** -39
    assert np.array_equal(bf16, b.astype(np.float64), equal_nan=True) and np.isnan(half[-1])
