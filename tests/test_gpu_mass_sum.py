"""The mass sum, the first step of every call, takes nothing from the call
before: whatever its workspace holds -- here a pattern in every byte, in use what
an earlier call or two overlapping ones left -- it writes the same sum, in the
same order of additions, sets the ray pass's work counter to zero and clears the
cell counts.  The sum is compared bit for bit with that order in numpy."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2204_10871_gb300 import build as libbuild
from gpu_common import require_gpu

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
BLOCKS, THREADS = 128, 256


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    require_gpu()
    lib = libbuild.build()
    ctypes.CDLL(lib, mode=ctypes.RTLD_GLOBAL)
    so = str(tmp_path_factory.mktemp("probe") / "probe.so")
    subprocess.run([libbuild._nvcc()] + libbuild._flags() + ["-I", libbuild.CSRC, "-shared", "-o", so,
                   os.path.join(HERE, "mass_sum_probe.cu"), lib, "-lcudart"], check=True)
    fn = ctypes.CDLL(so).probe_mass_sum
    fn.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p]
    return fn


def _ordered_sum(m):
    """Each thread adds its masses, BLOCKS * THREADS apart; a block halves its
    threads' sums; the blocks' sums are added in order."""
    rows = -(-max(1, m.size) // (BLOCKS * THREADS))
    a = np.zeros(rows * BLOCKS * THREADS)
    a[:m.size] = m
    t = np.zeros((BLOCKS, THREADS))
    for r in a.reshape(rows, BLOCKS, THREADS):
        t += r
    w = THREADS // 2
    while w:
        t = t[:, :w] + t[:, w:2 * w]
        w //= 2
    s = 0.0
    for v in t[:, 0]:
        s += v
    return s


@pytest.mark.parametrize("pattern", [0x00, 0xA5, 0x01])
@pytest.mark.parametrize("n", [0, 1, 256, 257, 1000, 32768, 32769, 100000])
def test_whatever_the_workspace_holds(probe, n, pattern):
    torch = require_gpu()
    m = np.random.default_rng(n).uniform(0.1, 1.0, n)
    dm = torch.from_numpy(m).cuda()
    scratch = torch.full((4096,), pattern, dtype=torch.uint8, device="cuda")
    cells = torch.full((9001,), 7, dtype=torch.int32, device="cuda")
    for call in range(2):
        assert probe(dm.data_ptr(), n, scratch.data_ptr(), cells.data_ptr(), cells.numel(),
                     torch.cuda.current_stream().cuda_stream) == 0
        torch.cuda.synchronize()
        assert scratch[:8].cpu().numpy().view(np.float64)[0] == _ordered_sum(m), f"call {call}"
        assert scratch[8:16].cpu().numpy().view(np.uint64)[0] == 0
        assert not cells.any()
