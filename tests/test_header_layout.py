"""The table header's layout is part of the binary interface: kernels of a user's
module, built with their own copy of include/, read and write it beside the library's.
Its fields stay where ABI version 2 has them."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FIELDS = {"live": 0, "used": 8, "err": 16, "side_present": 20, "side_lock": 28, "side_val": 32, "dump_count": 48,
          "claim_key_at": 64}


def test_header_fields_stay_in_place(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "layout.cu"
    src.write_text('#include <cstddef>\n#include "hc_core.cuh"\n' + "".join(
        f'static_assert(offsetof(hc::Header, {f}) == {at}, "{f}");\n' for f, at in FIELDS.items()))
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", f"-I{ROOT}/include", "-c",
                        str(src), "-o", str(tmp_path / "layout.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
