"""EOD_FP32_GEMM and EOD_FP64_GEMM (read once per process): simt keeps every
product on the FMA kernels, emulated and no value use the digits here."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import sys, torch
sys.path.insert(0, {root!r})
import paper_2506_22713_gb300 as eod
g = torch.Generator(device="cuda").manual_seed(1)
L, R = (torch.randn(400, n, generator=g, device="cuda", dtype=torch.float64) for n in (1900, 1500))
A = (R.t() @ L).to(torch.{dtype}).t()
eod.eod_abe_debug_profile(1)
f = eod.factor(A, 1e-3, 5, tol_mode="rel", block_k=128)
print("rank", f.rank, "digits", eod.profile_read(5)["launches"])
"""


@pytest.mark.parametrize("dtype,name", [("float32", "EOD_FP32_GEMM"), ("float64", "EOD_FP64_GEMM")])
@pytest.mark.parametrize("value", ["simt", "emulated", None])
def test_switch(dtype, name, value):
    import __graft_entry__ as g
    g.build()
    env = {k: v for k, v in os.environ.items() if k not in ("EOD_FP32_GEMM", "EOD_FP64_GEMM")}
    if dtype == "float32":
        env["EOD_FP64_GEMM"] = "simt"   # the wide Grams of FP32 data are FP64 products
    if value:
        env[name] = value
    out = subprocess.run([sys.executable, "-c", CODE.format(root=ROOT, dtype=dtype)], env=env, capture_output=True,
                         text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    words = out.stdout.split()
    assert words[0] == "rank" and words[1] == "400"
    assert (int(words[3]) == 0) == (value == "simt")
