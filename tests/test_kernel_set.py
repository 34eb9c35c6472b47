"""The library holds the fused multigrid kernels its launches can choose, and no
others: every unreachable instantiation costs build time (a few seconds of
device compilation each) and size.  Read from the names of the compiled
kernels; no GPU needed."""
import re
import shutil
import subprocess

import pytest


def test_only_reachable_fused_kernels_are_compiled():
    from paper_2301_10041_gb300 import build
    if shutil.which("nm") is None:
        pytest.skip("nm not available")
    try:
        path = build.build()
    except RuntimeError as e:   # no toolkit on this machine
        pytest.skip(str(e))
    out = subprocess.run(["nm", "-C", path], capture_output=True, text=True, check=True).stdout
    fused = set(re.findall(r"\b(k_mf[up]_(?:down|up))<(\w+), (\d+), (\d+), \d+, (\d+)>", out))
    degrees = "1234"
    want = set()
    for d in degrees:
        for k in ("k_mfu_down", "k_mfu_up"):         # 4-, 8- and 16-node velocity tiles
            want |= {(k, "float", "4", d, "1"), (k, "float", "8", d, "2"), (k, "float", "16", d, "2")}
        # pressure: 4-cell tiles up to 128 cells and above, 8-cell tiles from 512
        want |= {("k_mfp_down", "float", "4", d, m) for m in "16"} | {("k_mfp_down", "float", "8", d, "6")}
        want |= {("k_mfp_up", "float", "4", d, m) for m in "18"} | {("k_mfp_up", "float", "8", d, "6")}
    assert fused == want
    # the per-level matrix-free products exist for the FP64 levels only
    assert set(re.findall(r"\b(?:k_mfv|k_mfp|k_mfv_start)<(\w+)", out)) == {"double"}
