"""The fingerprint that ties a profile to the sources covers every CUDA source and header."""
import os

import bench
from paper_0908_4421_gb300 import build as cuda_build


def test_fingerprint_covers_all_sources():
    sources = {f for f in os.listdir(cuda_build.CSRC) if f.endswith((".cu", ".cuh", ".h"))}
    assert set(bench.SOURCE_FILES) == sources and set(cuda_build.SOURCES) <= sources
