"""The fixed-point helpers of the FP64 kernels (csrc/fixed.cuh), compiled for
the host and checked against long double."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.skipif(not shutil.which('g++'), reason='needs g++')
def test_digits_and_scaling(tmp_path):
    exe = str(tmp_path / 'fixed_check')
    subprocess.run(['g++', '-O2', '-std=c++17', '-I', os.path.join(ROOT, 'paper_2509_11424_gb300', 'csrc'),
                    os.path.join(ROOT, 'tests', 'fixed_check.cpp'), '-o', exe], check=True)
    assert subprocess.run([exe]).returncode == 0
