"""Window attention at the edges of its M tiles: window rows that leave whole
softmax warps without rows, that just fill one M tile, that need a second one
for a few rows, and that fill both, over sequences of less than one 64-key unit,
of exactly one and two, and of a ragged last unit, so that a CTA's range holds
pieces of one unit after longer ones (the queries in tensor memory are replaced
at each).  Against the fp64 oracle at the bounds of test_gpu_attention.
"""
import dataclasses

import pytest
import torch

from paper_2606_01790_gb300 import starkv as sk
from paper_2606_01790_gb300 import synthetic as syn

import harness as H

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import test_gpu_attention as A


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("rows,w", [(8, 8), (64, 16), (104, 8), (128, 32), (136, 8), (160, 32), (224, 32), (256, 32)])
def test_rows_at_the_edges_of_the_m_tiles(rows, w):
    G = 2
    base = dataclasses.replace(syn.WORKLOADS["tiny"], n_heads=rows // w * G, n_kv_heads=G, window=w, n_layers=24)
    texts = [w + 1, w + 64, w + 65, w + 128, w + 449, w]   # L_p = 1, 64, 65, 128, 449 and 0
    st = sk.init_state(H.gpu_config(base, H.hyper(), max_seqs=len(texts)))
    sis, dss = [], []
    for i, text in enumerate(texts):
        wl = dataclasses.replace(base, name=f"t{i}", cfg_id=300 + i, n_shots=0, n_text=text)
        si = syn.make_sequence(wl)
        assert si.L == text
        sis.append((si, wl))
        dss.append(A._attach(H.device_seq(si, wl, slot=i), si, wl))
    A._run_attention(st, dss)
    for (si, wl), ds in zip(sis, dss):
        for layer in (0, 11, 23):
            A.check_layer(ds, si, wl, layer)
    st.close()
