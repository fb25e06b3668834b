"""What the rerank's launcher refuses, without a GPU: LVQ-8 secondaries need their mean, which the kernel reads
for every query."""
import ctypes

import kernel_unit

LV_ERR_STATE = -8


def test_lvq_secondaries_need_their_mean():
    lib = kernel_unit.load("rerank_unit")
    null, one = ctypes.c_void_p(0), ctypes.c_int64(1)
    for metric in (0, 1):
        rc = lib.rerank_unit(null, ctypes.c_int64(96), 4, 8, metric, null, one, 64, null, null, null, 32, 1, null, null, 1,
                             null, 0, null)
        assert rc == LV_ERR_STATE
