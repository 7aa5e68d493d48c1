"""The CUDA-core recurrence's launch rule through gtr_gla_simt_plan (host arithmetic, no GPU): the cluster
that shares a sequence, and what it falls to on a device that cannot place that cluster."""
import ctypes

import pytest
import torch

from paper_2609_26590_gb300 import build as gbuild
from paper_2609_26590_gb300 import gla

GB300_SMS = 152


@pytest.fixture(scope="module", autouse=True)
def lib():
    gbuild.build()
    return gla.load()


def rule(B, H, gh, gw, Dk, Dv, n_sm, max_cluster):
    """The rule restated: the largest cluster that keeps every CTA resident, two blocks a group at least."""
    units = B * H * -(-Dv // 64)
    blocks = -(-gh * gw // 8)
    groups = 4 if Dk <= 32 else 2 if Dk <= 64 else 1
    for c in (16, 8, 4, 3, 2):
        if c <= max_cluster and units * c <= (n_sm if c == 16 else 2 * n_sm) and blocks >= 2 * groups * c:
            return c
    return 0


# the clusters of the shapes in tests/test_gpu_simt_segments.py on 152 SMs
SHAPES = [
    ((1, 2, 33, 31, 64, 64), 16), ((1, 3, 29, 25, 40, 72), 16), ((1, 1, 20, 27, 33, 50), 16),
    ((2, 6, 13, 20, 20, 24), 4), ((3, 11, 19, 23, 64, 61), 8), ((5, 9, 11, 12, 128, 128), 3),
    ((5, 18, 11, 12, 96, 64), 3), ((11, 13, 9, 10, 64, 64), 2), ((19, 9, 6, 7, 64, 64), 0),
    ((1, 1, 5, 5, 32, 8), 0),
]


@pytest.mark.parametrize("shape,cluster", SHAPES)
def test_cluster_on_gb300(shape, cluster):
    assert gla.simt_plan(*shape, torch.float32, GB300_SMS)[0] == cluster


@pytest.mark.parametrize("max_cluster", [16, 15, 8, 7, 4, 3, 2, 1, 0])
def test_falls_to_smaller_clusters(max_cluster):
    for shape, _ in SHAPES:
        for n_sm in (1, 8, 76, 132, 152):
            got = gla.simt_plan(*shape, torch.float32, n_sm, max_cluster)[0]
            assert got == rule(*shape, n_sm, max_cluster) and (got == 0 or got <= max_cluster)


# whole sequences (no cluster): 16 columns a CTA for narrow values, for up to 32 key channels while those
# CTAs are few, for short sequences and for long 16-bit ones; tiles of 64 columns otherwise
COLUMNS = [
    ((1, 200, 40, 40, 32, 16), "f32", 16), ((1, 4000, 16, 16, 32, 16), "f32", 16),
    ((1, 380, 16, 16, 32, 17), "f32", 16), ((1, 381, 16, 16, 32, 17), "f32", 64),
    ((1, 912, 40, 40, 20, 20), "f16", 16), ((1, 913, 40, 40, 20, 20), "f16", 64),
    ((1, 608, 16, 16, 20, 20), "f16", 16), ((1, 609, 16, 16, 20, 20), "f16", 64),
    ((1, 304, 16, 16, 33, 16), "f32", 16), ((1, 304, 16, 17, 64, 16), "f32", 64), ((1, 305, 16, 17, 64, 16), "f32", 16),
    ((1, 304, 40, 40, 61, 14), "f16", 16), ((1, 400, 16, 16, 65, 16), "f32", 64),
    ((1, 24, 6, 8, 64, 64), "f32", 16), ((1, 76, 6, 8, 64, 64), "f32", 16), ((1, 77, 6, 8, 64, 64), "f32", 64),
    ((1, 24, 7, 7, 64, 64), "f32", 64),
    ((1, 304, 32, 32, 61, 20), "f16", 16), ((1, 305, 32, 32, 61, 20), "f16", 64), ((1, 200, 32, 32, 61, 33), "f16", 64),
    ((1, 200, 31, 33, 61, 20), "f16", 64), ((1, 200, 32, 32, 61, 20), "f32", 64), ((1, 400, 40, 40, 64, 64), "f32", 64),
]


@pytest.mark.parametrize("shape,dtype,columns", COLUMNS, ids=str)
def test_columns_of_whole_sequences(shape, dtype, columns):
    dt = {"f32": torch.float32, "f16": torch.float16}[dtype]
    assert gla.simt_plan(*shape, dt, GB300_SMS) == (0, columns)


def test_invalid_arguments(lib):
    a, b = ctypes.c_int(-7), ctypes.c_int(-7)
    pa, pb = ctypes.byref(a), ctypes.byref(b)
    assert lib.gtr_gla_simt_plan(1, 1, 8, 8, 64, 64, 0, 0, 16, pa, pb) == 1
    assert lib.gtr_gla_simt_plan(1, 1, 0, 8, 64, 64, 0, 152, 16, pa, pb) == 1
    assert lib.gtr_gla_simt_plan(1, 1, 8, 8, 64, 300, 0, 152, 16, pa, pb) == 1
    assert lib.gtr_gla_simt_plan(1, 1, 8, 8, 64, 64, 5, 152, 16, pa, pb) == 1
    assert lib.gtr_gla_simt_plan(1, 1, 8, 8, 64, 64, 0, 152, 16, None, pb) == 1
    assert a.value == b.value == -7
