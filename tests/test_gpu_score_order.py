"""Scoring pass 2 over the tiles in reverse order: taken when one M tile holds
the window rows and the launch's K exceeds the device's L2.  Sizes on both sides of
that line, with ragged last tiles and sequences of one tile between long ones, so
that a CTA's range ends and begins inside rows; every number of 16-column chunks
a warp can hold there; and a row spread over more than eight CTAs, whose normalisers
two threads merge.  The state's counter shows which order ran.

S of the whole step against the softmax sums in 64 bits (Eqs. 2-4) to 1e-5, and
against the per-layer calls, whose launches are below the line, to 2e-6: the two
differ only in where the normalisers' partial sums are cut, a few units of 2^-24
each.
"""
import math

import pytest
import torch

from paper_2606_01790_gb300 import starkv as sk

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

D = 128
TILE = 128   # keys


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


# heads, groups, window, layers, tiles of the short sequences between the long ones
SHAPES = [(8, 4, 8, 4, [1]),       # 16 window rows: chunks 1, 0, 0, 0 of the four warpgroups
          (8, 4, 8, 4, [1, 1]),
          (12, 4, 31, 4, [3]),     # 93 rows: 2, 2, 1, 1
          (16, 4, 32, 4, [1]),     # 128 rows: 2, 2, 2, 2
          (4, 1, 8, 4, [])]        # one sequence: rows of 40 CTAs


@pytest.mark.parametrize("above", [False, True], ids=["at_the_line", "above"])
@pytest.mark.parametrize("heads,G,w,nl,short", SHAPES)
def test_pass_2_backwards(heads, G, w, nl, short, above):
    line = torch.cuda.get_device_properties(0).L2_cache_size // (TILE * D * 2)   # tiles that fit
    n = line // (nl * G) + above - sum(short)    # of the long sequences, per row
    lens = ([n // 2 * TILE - 17] + [t * TILE - 106 for t in short] + [(n - n // 2) * TILE - 28]) if short else [n * TILE - 5]
    tiles = nl * G * sum(-(-lp // TILE) for lp in lens)
    assert (tiles > line) == above and abs(tiles - line) <= nl * G
    gen = torch.Generator(device="cuda")
    gen.manual_seed(heads + above)

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda").to(torch.bfloat16)

    def room(lp):
        return dict(k_out=torch.empty(nl, G, 1 + w, D, dtype=torch.bfloat16, device="cuda"),
                    v_out=torch.empty(nl, G, 1 + w, D, dtype=torch.bfloat16, device="cuda"),
                    meta_out=torch.empty(nl, 1 + w, dtype=torch.int32, device="cuda"),
                    idx=torch.empty(nl, 1, dtype=torch.int32, device="cuda"), S=torch.empty(nl, G, lp, device="cuda"))

    whole, layered = [], []
    for i, lp in enumerate(lens):
        k, q = normal(nl, G, lp + w, D), normal(nl, heads, w, D)
        meta = torch.zeros(lp + w, dtype=torch.int32, device="cuda")
        for seqs in (whole, layered):
            seqs.append(sk.Seq(k=k, v=k, q=q, meta=meta, L=lp + w, budget=1, slot=i, **room(lp)))
    sts = [sk.init_state(sk.Config(n_layers=nl, n_heads=heads, n_kv_heads=G, window=w, max_seqs=len(lens))) for _ in range(2)]
    sk.step(sts[0], whole, sk.workspace(sts[0], whole))
    ws = sk.workspace(sts[1], layered)
    for layer in range(nl):
        sk.score_layer(sts[1], layer, layered, ws)
    torch.cuda.synchronize()
    for st in sts:
        sk.check_device_error(st)
    assert [sk.backward_launches(st) for st in sts] == [int(above), 0]
    for a, b in zip(whole, layered):
        for layer in range(nl):
            got, other = a.S[layer].double(), b.S[layer].double()
            ref = _reference(a.q[layer], a.k[layer], w, 5)
            assert ((got - ref).abs() / ref.clamp_min(1e-30)).max().item() <= 1e-5
            assert ((got - other).abs() / other.clamp_min(1e-30)).max().item() <= 2e-6
    for st in sts:
        st.close()
