"""A launcher that can refuse (a tensor map that cannot be encoded, a size it
does not take) says so in its result, and the library does not build with
that result dropped: a product left out silently would leave a wrong inverse."""
import os
import subprocess

import pytest

from paper_2309_05435_gb300 import build

CALLS = {
    "spd_inverse": "qsel::spd_inverse<double>(s, qsel::SweepBatch<double>{}, 64, nullptr);",
    "launch_oz_gemm": "qsel::launch_oz_gemm(s, qsel::OzGemmBatch{}, 64, 64, 64, 64, false, -1, nullptr);",
    "launch_oz_split_cols": "qsel::launch_oz_split_cols(s, nullptr, 0, 64, 32, 32);",
    "launch_tc_gemm": "qsel::launch_tc_gemm(s, qsel::GemmBatch<float>{}, 64, 64, 64, 64, 64, 64, false, 3, nullptr);",
    "launch_tc_gemm_split":
        "qsel::launch_tc_gemm_split(s, qsel::SplitGemmBatch{}, 64, 64, 64, 64, 64, 64, false, nullptr);",
    "launch_tc_update": "qsel::launch_tc_update(s, qsel::UpdateBatch{}, 64, 64, 64, -1.0f, 1.0f, nullptr, 0);",
}


@pytest.mark.parametrize("name", list(CALLS))
def test_a_dropped_result_does_not_compile(tmp_path, name):
    if not os.path.exists(build.NVCC):
        pytest.skip("needs nvcc")

    def compiles(statement):
        src = tmp_path / "probe.cu"
        src.write_text(f'#include "kernels.cuh"\nvoid probe(cudaStream_t s) {{ {statement} }}\n')
        r = subprocess.run([build.NVCC, *build.FLAGS, "-c", str(src), "-o", str(tmp_path / "probe.o")],
                           capture_output=True, text=True)
        return r.returncode == 0, r.stderr

    kept, log = compiles("if (!" + CALLS[name][:-1] + ") return;")
    assert kept, log
    dropped, log = compiles(CALLS[name])
    assert not dropped and "nodiscard" in log
