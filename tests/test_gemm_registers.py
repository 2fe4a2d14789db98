"""The matrix products' epilogues use all registers that their launch can have; what the compiler says of each instance."""
import os
import re
import subprocess

import pytest

from paper_2512_04939_b200.build import CFLAGS, CSRC, NVCC


@pytest.fixture(scope="module")
def spills(tmp_path_factory):
    """(epilogue, columns, CTAs of a tile) -> bytes of spill stores and loads."""
    if not os.path.exists(NVCC):
        pytest.skip("no nvcc")
    obj = str(tmp_path_factory.mktemp("registers") / "linear.o")
    log = subprocess.run([NVCC, *CFLAGS, "-c", os.path.join(CSRC, "linear.cu"), "-o", obj], check=True, capture_output=True, text=True).stderr
    found = re.findall(r"function '_ZN2lv14gemm_tc_kernelINS_\d+(\w+?)ELi(\d+)ELi(\d)E\w+'.*?(\d+) bytes spill stores, (\d+) bytes spill loads",
                       re.sub(r"\s+", " ", log))
    return {(epilogue, int(columns), int(ctas)): (int(stores), int(loads)) for epilogue, columns, ctas, stores, loads in found}


@pytest.mark.parametrize("columns,ctas", [(64, 2), (128, 2), (160, 2), (192, 2), (224, 2), (256, 2), (256, 1)])
@pytest.mark.parametrize("epilogue", ["LinearEpilogue", "MlpEpilogue"])
def test_no_instance_spills(spills, epilogue, columns, ctas):
    assert spills[epilogue, columns, ctas] == (0, 0)
