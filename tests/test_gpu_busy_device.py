"""Calls whose blocks wait for one another while a long kernel holds all SMs but
one (tests/gpu_hog.cu, two seconds at most): with only a few of their blocks on
the GPU at a time they take longer, and give the same results."""
import contextlib
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")
torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def hog(tmp_path_factory):
    so = tmp_path_factory.mktemp("hog") / "libhog.so"
    subprocess.check_call([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_103a,code=sm_103a", "-O2",
                           "-shared", "-Xcompiler", "-fPIC", "-o", str(so), os.path.join(ROOT, "tests", "gpu_hog.cu")])
    return ctypes.CDLL(str(so))


@contextlib.contextmanager
def held(hog, ms):
    """All SMs but one held for ms milliseconds; checks that the body finished meanwhile."""
    assert hog.hog_start(1, ms) > 0
    try:
        yield
        assert hog.hog_running()
    finally:
        assert hog.hog_wait() == 0


@pytest.mark.parametrize("n", [32 * 4096, 3_000_001, (1 << 24) + 4097])
def test_filter_with_few_blocks_at_a_time(hog, n):
    v = torch.arange(n, dtype=torch.int32, device="cuda") % 1000
    out = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    want = np.nonzero(v.cpu().numpy() < 137)[0]

    def call():
        st, cnt = vx.vx_filter_device_static([v.data_ptr()], [(0, vx.VX_LT, 137, 0)], n, 0, out.data_ptr(), n,
                                             stream.cuda_stream)
        assert st == vx.VX_OK and cnt == len(want)

    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    call()  # loads the kernel
    out.fill_(-1)
    torch.cuda.synchronize()
    with held(hog, 2000):
        call()
    got = out.cpu().numpy()
    assert np.array_equal(got[:len(want)], want) and (got[len(want):] == -1).all()
