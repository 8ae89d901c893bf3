"""The W4A16_DEBUG build on the GPU: every kernel runs its index checks (TMA
coordinates and destinations, tensor-memory columns, store rows) on ragged
shapes of every dispatch path, no check fails, and the results still match
the oracle.  Runs in child processes that load libw4a16_debug.so, one per way of
forcing the kernels that shapes of this size would not reach."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_CHILD = r"""
import sys
import numpy as np, torch
sys.path.insert(0, {root!r})
from oracle import oracle as O
from paper_2608_30877_gb300 import synthetic as S
from paper_2608_30877_gb300 import w4a16 as W
from tests.gpu_helpers import assert_close, bf16_to_f64, host_case, to_device
assert W.LIB_PATH.endswith("libw4a16_debug.so"), W.LIB_PATH
for (M, N, K, g) in {cases!r}:
    assert W.route(M, N, K, g)[0] == {kernel!r}, (M, N, K, g, W.route(M, N, K, g))
    x, xb, packed, scales = host_case(M, N, K, g, M + 1, N + 2)
    xd, wd, sd = to_device(x, packed, scales)
    out = W.linear(xd, wd, sd, g)
    torch.cuda.synchronize()
    ref = O.linear_rows(xb, packed, scales, N, K, g, nthreads=O.max_threads())
    assert_close(bf16_to_f64(out), ref, f"debug build {{M}}x{{N}}x{{K}} g{{g}}")
    assert W.get_device_error() == W.OK, (M, N, K, g)
# attention over ragged sequences
H = 2
st = torch.tensor([0, 100, 300, 301, 700], dtype=torch.int32)
qkv = S.make_x(700, 3 * H * 128, 4, "cpu")
out = W.attention_prefill(qkv.cuda(), st.cuda(), H, 160)
torch.cuda.synchronize()
assert W.get_device_error() == W.OK
bits = S.bf16_bits(qkv)
ref = O.attention_rows(bits, H, 128, st.numpy().astype(np.int64), 160)
v = O.bf16_bits_to_f32(bits[:, 2 * H * 128:]).astype(np.float64)
v_rms = float(np.sqrt(np.mean(v * v)))
err = np.abs(bf16_to_f64(out) - ref)
# the attention tests' bound: P rounded to bf16 for PV, one bf16 store
assert float(np.max(err / (2.0 ** -8 * np.abs(ref) + 2.0 ** -7 * v_rms))) <= 1.0
print("ok")
"""


GEMM_CASES = [(300, 1000, 1024, 128), (520, 384, 512, 128), (129, 257, 576, 192), (900, 130, 320, 64)]


@pytest.mark.parametrize("kernel,env,cases", [
    # 32, 64, 96, 112 and 128 token columns, K split and whole, K ending inside a stage, token tiles
    ("stream", {"W4A16_SMALL_M": "tc"}, [(8, 2000, 1280, 128), (24, 1234, 640, 128), (48, 1234, 4096, 128),
                                         (90, 300, 1088, 64), (100, 1234, 640, 128), (128, 60010, 256, 128),
                                         (5, 200, 256, 64), (300, 1000, 1024, 128)]),
    ("rows", {"W4A16_SMALL_M": "mma"}, [(1, 300, 128, 128), (8, 2000, 1280, 128), (13, 60010, 256, 128)]),
    ("head", {}, [(64, 2, 1024, 128), (700, 8, 192, 64)]),
    ("gemm", {"W4A16_GEMM_WIDE": "1"}, GEMM_CASES),
    ("gemm", {"W4A16_GEMM_WIDE": "0"}, GEMM_CASES),
    ("gemm", {"W4A16_GEMM_PAIR": "0"}, GEMM_CASES),
])
def test_debug_build_checks_pass_and_results_match(kernel, env, cases):
    from paper_2608_30877_gb300 import build as B
    B.build(debug=True)
    env = dict(os.environ, W4A16_DEBUG="1", **env)
    r = subprocess.run([sys.executable, "-c", _CHILD.format(root=ROOT, cases=cases, kernel=kernel)],
                       env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]


_ABORT = r"""
import sys
sys.path.insert(0, {root!r})
import torch
from paper_2608_30877_gb300 import w4a16 as W
from paper_2608_30877_gb300 import synthetic as S
from tests.test_gpu_failure import check_abort_forced, _linear_still_correct
assert W.LIB_PATH.endswith("libw4a16_debug.so"), W.LIB_PATH
check_abort_forced({kernel!r}, *{cases!r})
H = 8
qkv = S.make_x(4096, 3 * H * 128, 9, "cuda")
st = torch.arange(0, 4097, 1024, dtype=torch.int32, device="cuda")
want = W.attention_prefill(qkv, st, H)
W.set_wait_limit(1)
got = W.attention_prefill(qkv, st, H)
assert W.get_device_error() == W.ERR_TIMEOUT
W.set_wait_limit(0)
rows = lambda t: t.view(4096, H, 128)
assert ((rows(got) == rows(want)).all(-1) | (rows(got) == 0).all(-1)).all()
_linear_still_correct()
print("ok")
"""


@pytest.mark.parametrize("kernel,env,cases", [
    ("stream", {"W4A16_SMALL_M": "tc"}, [(8, 8192, 4096, 128), (96, 8192, 4096, 128),
                                         (24, 49152, 2048, 128), (300, 25600, 2048, 128, 1, True)]),
    ("rows", {"W4A16_SMALL_M": "mma"}, [(8, 8192, 4096, 128), (16, 60000, 1024, 128)]),
    ("gemm", {"W4A16_GEMM_WIDE": "1"}, [(900, 12800, 2048, 128), (300, 25600, 2048, 128, 1, True)]),
    ("gemm", {"W4A16_GEMM_WIDE": "0"}, [(900, 12800, 2048, 128), (300, 25600, 2048, 128, 1, True)]),
    ("gemm", {"W4A16_GEMM_PAIR": "0"}, [(900, 12800, 2048, 128), (300, 25600, 2048, 128, 1, True)]),
])
def test_any_role_may_give_up_first(kernel, env, cases):
    """With a lowered wait limit the debug build's waits poll without suspending, in every
    role, so the first to give up is not only the producer."""
    from paper_2608_30877_gb300 import build as B
    B.build(debug=True)
    env = dict(os.environ, W4A16_DEBUG="1", **env)
    r = subprocess.run([sys.executable, "-c", _ABORT.format(root=ROOT, cases=cases, kernel=kernel)],
                       env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]
