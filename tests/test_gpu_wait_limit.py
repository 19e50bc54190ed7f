"""The wait limit of a state bounds each device-side wait of a kernel, not the time a
kernel spends behind the one before it.  Scoring pass 2 starts while pass 1's
last CTAs still run, and at 28 layers x 28 groups x 14,000 tokens these end tens of
microseconds after the first; no wait inside either pass takes that long, so a limit
of 20 microseconds must not run out."""
import pytest
import torch

from paper_2606_01790_gb300 import starkv as sk

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def test_a_short_wait_limit_does_not_count_the_previous_kernel():
    nl, G, w, L, B = 28, 28, 32, 14032, 1000
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    k = torch.empty(nl, G, L, 128, dtype=torch.bfloat16, device="cuda").normal_(generator=gen)
    q = torch.empty(nl, G, w, 128, dtype=torch.bfloat16, device="cuda").normal_(generator=gen)
    out = torch.empty(2, nl, G, B + w, 128, dtype=torch.bfloat16, device="cuda")
    seq = sk.Seq(k=k, v=k, q=q, meta=torch.zeros(L, dtype=torch.int32, device="cuda"), L=L, budget=B, k_out=out[0],
                 v_out=out[1], meta_out=torch.empty(nl, B + w, dtype=torch.int32, device="cuda"),
                 idx=torch.empty(nl, B, dtype=torch.int32, device="cuda"))
    st = sk.init_state(sk.Config(n_layers=nl, n_heads=G, n_kv_heads=G, window=w))
    ws = sk.workspace(st, [seq])
    sk.step(st, [seq], ws)
    sk.check_device_error(st)
    sk.set_wait_limit(st, 20_000)
    for _ in range(10):
        sk.step(st, [seq], ws)
        sk.check_device_error(st)
    st.close()
