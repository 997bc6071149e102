"""Device functions and kernels called directly, by small CUDA programs that are
compiled here (each says in its header what it compares with what)."""
import os
import subprocess
import tempfile

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _run(source, *flags):
    from paper_2002_09603_gb300 import build
    with tempfile.TemporaryDirectory() as d:
        exe = os.path.join(d, "check")
        r = subprocess.run([build.nvcc(), "-std=c++17", "-O2", "--expt-relaxed-constexpr", *build.ARCH,
                            os.path.join(HERE, source), "-o", exe, *flags],
                           capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
        r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout[-2000:] + r.stderr[-2000:]


def test_conversions_over_every_branch():
    _run("conversion_check.cu")


def test_sweeps_under_every_schedule():
    from paper_2002_09603_gb300 import LIB_PATH
    lib = os.path.dirname(os.path.abspath(LIB_PATH))
    _run("sweep_check.cu", "-L" + lib, "-lmhfp", "-Xlinker", "-rpath=" + lib)


def test_registered_bytes_of_the_float_float_operator():
    import bench
    import mhfp_inputs as mi
    from paper_2002_09603_gb300 import default_options, prepare
    o = default_options()
    o.precision, o.autotune = 1, 0
    s = prepare(mi.random_small(5, 5, 5, seed=3), o)
    x = torch.ones(s.n, dtype=torch.float64, device="cuda")
    s.timing(True)
    s.apply_operator_ff(x)
    torch.cuda.synchronize()
    t = s.timing_read(6)
    s.timing(False)
    assert t["launches"] == 1 and t["bytes_per_launch"] == bench.ff_operator_bytes(5)
    s.close()
