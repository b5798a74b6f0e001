"""What a contract keeps of a model goes with the model: a contract priced on
ever new markets holds the entries of the live ones only, whichever of the two
is destroyed first."""
import pytest

from gpu_common import torch
import paper_2108_03076_gb300 as pc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("jit", [False, True], ids=["interpreted", "specialised"])
def test_a_contract_forgets_destroyed_models(jit):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_03076_gb300 import build
    build.build()
    st = torch.cuda.Stream()
    ctx = pc.pc_create(0, st.cuda_stream)
    pc.pc_set_jit(ctx, jit)
    w, c = pc.pc_assemble("(mult (max (sub (model 0 2) 1.0) 0.0) (payoff 2 0 1))")
    a, b = pc.pc_load_payoff(ctx, w, c), pc.pc_load_payoff(ctx, w, c)

    def model(s):
        return pc.pc_model_create(ctx, [s], [0.2], [[1.0]], 0.01, [30, 60])
    kept = model(1.0)
    want = pc.pc_price(kept, a, 4096, 1)
    for i in range(20):
        m = model(1.0 + 0.01 * i)
        price = pc.pc_price(m, a, 4096, 1)
        assert (price == want) == (i == 0)
        assert pc.pc_price(m, b, 4096, 1) == price
        assert (pc.pc_debug_contract_models(a), pc.pc_debug_contract_models(b)) == (2, 1)
        pc.pc_model_destroy(m)
        assert (pc.pc_debug_contract_models(a), pc.pc_debug_contract_models(b)) == (1, 0)
    assert pc.pc_price(kept, a, 4096, 1) == want
    last = model(1.2)
    pc.pc_price(last, a, 4096, 1)
    pc.pc_price(last, b, 4096, 1)
    pc.pc_contract_destroy(b)  # contract first, then the model that it was priced on
    pc.pc_model_destroy(last)
    assert pc.pc_debug_contract_models(a) == 1
    pc.pc_model_destroy(kept)
    assert pc.pc_debug_contract_models(a) == 0
    pc.pc_contract_destroy(a)
    pc.pc_destroy(ctx)
