"""The two forms of the FP32 travel-time network (tiles of 64 and of 32 pairs) at
the pair counts where the launch changes form and at ragged tile tails, against
the FP64 network.  Both forms add in the same order, so a pair's result does not
depend on the launch it is part of."""
import numpy as np
import pytest

from oracle import spider_oracle as O
from paper_2508_12117_gb300 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [32, 64, 128, 256])
def test_forms_agree_and_match_the_oracle(H):
    torch = pytest.importorskip("torch")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    net = synth.strong_mlp_weights(H, 900 + H)
    nd = binding.NetDevice(binding.Net(binding.TT_MLP, mlp=net))
    top = 64 * sms * 4 + 33
    rng = np.random.default_rng(H)
    src = np.c_[rng.uniform(0, 60, top), rng.uniform(0, 60, top), rng.uniform(2, 16, top), np.zeros(top)]
    rcv = np.c_[rng.uniform(-10, 70, top), rng.uniform(-10, 70, top), np.zeros((top, 2))]
    s4, r4 = (torch.from_numpy(a.astype(np.float32)).cuda() for a in (src, rcv))

    def run(n):
        hi, lo, J = torch.full((n,), np.nan, device="cuda"), torch.full((n,), np.nan, device="cuda"), \
            torch.full((n, 4), np.nan, device="cuda")
        nd.spider_tt_pairs(n, s4.data_ptr(), r4.data_ptr(), hi.data_ptr(), lo.data_ptr(), J.data_ptr())
        torch.cuda.synchronize()
        return hi, lo, J

    want = run(top)
    s64, r64 = s4[:, :3].double().cpu().numpy(), r4[:, :3].double().cpu().numpy()
    T, dT = O.tt_mlp(s64, r64, net)
    got = want[0].double().cpu().numpy() + want[1].double().cpu().numpy()
    rel_t = np.linalg.norm(got - T) / np.linalg.norm(T)
    rel_j = np.linalg.norm(want[2][:, :3].double().cpu().numpy() - dT) / np.linalg.norm(dT)
    print(f"H {H}: T rel-L2 {rel_t:.2e}, J rel-L2 {rel_j:.2e}")
    # H terms a chain, rounded once each, over six products
    assert rel_t <= 1e-5 and rel_j <= 1e-5
    for n in (1, 31, 33, 63, 65, 32 * sms, 32 * sms + 1, 64 * sms, 64 * sms + 1, 128 * sms, 128 * sms + 1):
        for a, b in zip(run(n), want):
            assert torch.equal(a, b[:n]), n
    nd.close()


@pytest.mark.parametrize("kind,precision", [("homogeneous", "FP32"), ("mlp", "FP32"), ("mlp", "BF16")])
def test_times_may_overlap_the_inputs(kind, precision):
    """T_hi and T_lo written over the source positions (and over each other's
    neighbour) are those of separate arrays: every pair is read before any time
    that lies on an input is written."""
    torch = pytest.importorskip("torch")
    net = binding.Net(binding.TT_MLP, mlp=synth.mlp_weights(64, 5)) if kind == "mlp" else \
        binding.Net(binding.TT_HOMOGENEOUS, v0=6.0)
    nd = binding.NetDevice(net, precision=getattr(binding, precision))
    n = 20_001
    torch.manual_seed(1)
    s4, r4 = torch.rand(n, 4, device="cuda") * 40, torch.rand(n, 4, device="cuda") * 40
    hi, lo, J = torch.empty(n, device="cuda"), torch.empty(n, device="cuda"), torch.empty(n, 4, device="cuda")
    nd.spider_tt_pairs(n, s4.data_ptr(), r4.data_ptr(), hi.data_ptr(), lo.data_ptr(), J.data_ptr())
    only = torch.empty(n, device="cuda")
    nd.spider_tt_pairs(n, s4.data_ptr(), r4.data_ptr(), only.data_ptr(), 0, 0)
    s, J2 = s4.clone(), torch.empty(n, 4, device="cuda")
    over = s.view(-1)
    nd.spider_tt_pairs(n, s.data_ptr(), r4.data_ptr(), over.data_ptr(), over.data_ptr() + 4 * n, J2.data_ptr())
    torch.cuda.synchronize()
    assert torch.equal(only, hi)
    assert torch.equal(over[:n], hi) and torch.equal(over[n:2 * n], lo) and torch.equal(J2, J)
    nd.close()
