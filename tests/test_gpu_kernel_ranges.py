"""Edges of the size ranges the kernel variants are chosen by, against the fp64 oracle (rules and tolerances of
tests/parity.py, every chunk)."""
import pytest
import torch

import paper_2411_19870_b200 as demo
from paper_2411_19870_b200 import inputs
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["tensor_scaled", "student_t_ties"])
@pytest.mark.parametrize("k", [48, 49, 64, 65, 128, 192, 193])
def test_s64_list_and_dense_row_stage(k, kind):
    """s = 64: k = 48 is the last with a listed row stage, k = 192 the last bounded by quarter rows; an all-zero tile and a
    single non-zero element among ordinary ones."""
    wl = inputs.Workload("s64k", [(3 * 64, 4 * 64), (64, 64)], chunk=64, topk=k, num_workers=2, grad_kind=kind,
                         grad_dtype=torch.float32 if k % 2 else torch.bfloat16)
    r = parity.Runner(wl, max_chunks=10**9, seed=k)
    for step in range(2):
        grads = [st.next() for st in r.streams]
        for g in grads:
            g[0][:64, :64] = 0
            g[0][64:128, :64] = 0
            g[0][70, 5] = 0.5
        r.step(grads=grads)
    r.close()
