"""Travel times from positions in rows of three: the same bits as the padded
entry point, for every travel-time form, at tile edges and ragged tails."""
import numpy as np
import pytest

from paper_2508_12117_gb300 import binding, synth

pytestmark = pytest.mark.gpu

FORMS = [("homogeneous", 0, "FP32"), ("mlp", 32, "FP32"), ("mlp", 128, "FP32"), ("mlp", 64, "BF16"),
         ("mlp", 256, "BF16"), ("mlp", 128, "FP8"), ("mlp", 256, "FP8")]


def _netdev(kind, H, precision):
    net = binding.Net(binding.TT_MLP, mlp=synth.strong_mlp_weights(H, 3)) if kind == "mlp" else \
        binding.Net(binding.TT_HOMOGENEOUS, v0=6.0)
    return binding.NetDevice(net, precision=getattr(binding, precision))


def _positions(torch, n):
    g = torch.Generator(device="cuda").manual_seed(n)
    u = torch.rand(n, 6, device="cuda", generator=g)
    return 60 * u[:, :3].contiguous() + 2, (80 * u[:, 3:] - 10).contiguous()


@pytest.mark.parametrize("kind,H,precision", FORMS)
def test_rows_equal_the_padded_entry(kind, H, precision):
    torch = pytest.importorskip("torch")
    nd = _netdev(kind, H, precision)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n in (1, 47, 127, 128, 129, 128 * sms + 1, 3 * 128 * sms + 77):
        s3, r3 = _positions(torch, n)
        s4, r4 = (torch.cat([x, torch.zeros(n, 1, device="cuda")], 1).contiguous() for x in (s3, r3))
        hi, lo, T = (torch.full((n,), np.nan, device="cuda") for _ in range(3))
        J4, J3 = (torch.full((n, 4), np.nan, device="cuda") for _ in range(2))
        nd.spider_tt_pairs(n, s4.data_ptr(), r4.data_ptr(), hi.data_ptr(), lo.data_ptr(), J4.data_ptr())
        nd.spider_tt_pairs_rows(n, s3.data_ptr(), r3.data_ptr(), T.data_ptr(), J3.data_ptr())
        torch.cuda.synchronize()
        assert torch.equal(T, hi + lo) and torch.equal(J3, J4), n
        assert torch.isfinite(T).all() and torch.isfinite(J3).all()
    nd.close()


def test_autograd_takes_any_layout_and_type():
    torch = pytest.importorskip("torch")
    from paper_2508_12117_gb300.autograd import travel_time
    nd = _netdev("mlp", 64, "FP32")
    for n in (0, 1, 300):
        s, r = _positions(torch, n)
        want = []
        for recompute in ("auto", True):
            x = s.clone().requires_grad_(True)
            T = travel_time(x, r, nd, recompute=recompute)
            (g,) = torch.autograd.grad(T.sum(), x)
            want.append((T.detach(), g))
        assert all(torch.equal(a, b) for a, b in zip(*want))
        wide = torch.zeros(n, 5, device="cuda")
        wide[:, 1:4] = s
        forms = [wide[:, 1:4], s.t().contiguous().t(), s.double(), torch.view_as_complex(
            torch.stack([s, -s], 2)).conj().imag]
        for f in forms:
            x = f.detach().requires_grad_(True)
            T = travel_time(x, r, nd)
            (g,) = torch.autograd.grad(T.sum(), x)
            assert torch.equal(T.detach(), want[0][0]) and torch.equal(g.float(), want[0][1])
    nd.close()
