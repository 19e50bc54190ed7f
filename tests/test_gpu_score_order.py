"""Scoring pass 2 over the tiles in reverse order: taken when one M tile holds
the window rows and the launch's K exceeds the L2 (more than 4096 128-key tiles).
Sizes around that line, with ragged last tiles and sequences of one tile between
long ones, so that a CTA's range ends and begins inside rows.  S of the whole
step against the softmax sums in 64 bits (Eqs. 2-4) to 1e-5, and against the
per-layer calls, whose launches are below the line, to 2e-6: the two differ
only in where the normalisers' partial sums are cut, a few units of 2^-24 each.
"""
import dataclasses
import math

import pytest
import torch

from paper_2606_01790_gb300 import starkv as sk
from paper_2606_01790_gb300 import synthetic as syn

import harness as H

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _reference(q, k, w, pool):
    """S [G][Lp] of one layer in float64."""
    G, L, d = k.shape
    lp, rows = L - w, q.shape[0] // G * w
    z = torch.bmm(q.double().reshape(G, rows, d), k[:, :lp].double().transpose(1, 2)) / math.sqrt(d)
    a = torch.softmax(z, dim=2).sum(1)                                     # [G][Lp]
    a = torch.nn.functional.avg_pool1d(a[:, None], pool, 1, pool // 2, count_include_pad=True)[:, 0]
    return a * G / q.shape[0]


@pytest.mark.parametrize("texts", [[16399, 30, 16100], [16399, 30, 17, 16100]], ids=["at_the_line", "above"])
def test_pass_2_backwards(texts):
    w, G, nl = 8, 4, 4
    base = dataclasses.replace(syn.WORKLOADS["tiny"], n_heads=8, n_kv_heads=G, window=w, n_layers=nl)
    tiles = nl * G * sum((t - w + 127) // 128 for t in texts)
    assert tiles == (4096 if len(texts) == 3 else 4112)
    hyper = H.hyper()
    sts = [sk.init_state(H.gpu_config(base, hyper, max_seqs=len(texts))) for _ in range(2)]
    runs, sis = [], []
    for i, text in enumerate(texts):
        wl = dataclasses.replace(base, name=f"o{i}", cfg_id=400 + i, n_shots=0, n_text=text)
        si = syn.make_sequence(wl)
        sis.append(si)
        runs.append([H.device_seq(si, wl, slot=i) for _ in range(2)])
    whole, layered = ([r[j].seq for r in runs] for j in range(2))
    sk.step(sts[0], whole, sk.workspace(sts[0], whole))
    ws = sk.workspace(sts[1], layered)
    for layer in range(nl):
        sk.score_layer(sts[1], layer, layered, ws)
    torch.cuda.synchronize()
    for st in sts:
        sk.check_device_error(st)
    for si, a, b in zip(sis, whole, layered):
        if si.L == w:
            continue
        lp = si.L - w
        for layer in range(nl):
            got = a.S.reshape(nl, G, lp)[layer].double()
            ref = _reference(si.q[layer].cuda(), si.k[layer].cuda(), w, 5)
            assert ((got - ref).abs() / ref.clamp_min(1e-30)).max().item() <= 1e-5
            other = b.S.reshape(nl, G, lp)[layer].double()
            assert ((got - other).abs() / other.clamp_min(1e-30)).max().item() <= 2e-6
    for st in sts:
        st.close()
