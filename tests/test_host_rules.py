"""Host-side decisions (csrc/host_rules.h), compiled alone with the host compiler."""
import ctypes
import os
import subprocess

import pytest

from paper_0908_4421_gb300 import build as cuda_build

WRAPPERS = """
#include "host_rules.h"
extern "C" int may_use(int where, int owner, int dev) {
    return imrt::kernels_may_use(static_cast<imrt::Memory>(where), owner, dev);
}
extern "C" int chunk_rows(int m, int n, int sm_count) { return imrt::transpose_chunk_rows(m, n, sm_count); }
extern "C" long long table_bytes(int m, int n, int rows) { return imrt::count_table_bytes(m, n, rows); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_rules")
    src, lib = d / "rules.cpp", d / "rules.so"
    src.write_text(WRAPPERS)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", cuda_build.CSRC, "-o", str(lib), str(src)])
    return ctypes.CDLL(str(lib))


def test_kernels_use_only_their_own_devices_memory(rules):
    host, device, managed = 0, 1, 2
    for dev in (0, 3):
        assert not rules.may_use(host, -1, dev)
        assert rules.may_use(device, dev, dev)
        assert not rules.may_use(device, dev + 1, dev)  # another GPU's: through a copy
        assert rules.may_use(managed, 0, dev)


def test_every_array_of_a_caller_that_a_kernel_takes_in_place_passes_the_rule():
    text = open(os.path.join(cuda_build.CSRC, "api.cu")).read()
    assert "direct_z = usable_on(z_out, p->device)" in text
    assert "direct_g = is_memory_of(g_out, p->device)" in text
    assert "is_memory_of(x, p->device)" in text
    assert "usable_on(structures, p->device)" in text


@pytest.mark.parametrize("n", [1, 620, 3140, 20000, 28000])
@pytest.mark.parametrize("m", [1, 31, 2000, 24000, 100000, 305000, 1048576, 16777216, 2 ** 31 - 1025])
def test_count_table_stays_within_the_admission_estimate(rules, m, n):
    from paper_0908_4421_gb300 import serve
    rules.table_bytes.restype = ctypes.c_longlong
    coarse = min(rules.table_bytes(m, n, 512), 256 << 20)
    for sm_count in (1, 76, 152, 4096):
        rows = rules.chunk_rows(m, n, sm_count)
        table = rules.table_bytes(m, n, rows)
        assert rows >= 32 and rows & (rows - 1) == 0
        # smaller chunks never cost more than 32 MiB beyond what chunks of 512 rows take
        assert table <= max(coarse, 32 << 20)
        assert table <= serve.count_table_bytes(m, n) <= serve.plan_footprint_bytes(m, n, 0, 0) - (64 << 20)
