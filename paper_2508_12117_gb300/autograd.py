"""torch.autograd.Function over the library's travel-time kernel.

forward(src, rcv) returns T(src; rcv) for P pairs (FP32, T_hi + T_lo rounded);
backward(dL/dT) returns dL/dsrc = dL/dT * dT/dsrc, where dT/dsrc comes from
the same fused launch (reverse sweep through the MLP, Sec. 3.2).  The Jacobian
(16 B per pair) is kept for backward, or, when it would not fit in the free
device memory with headroom to spare, recomputed by a second launch.

With the Jacobian kept, the kernel reads the caller's rows of three and writes
T rounded: padded copies, a low part and its sum were seven launches around it,
and the free memory was asked of the driver each time (47 pairs: 317 -> 174 us a
pass).  A Jacobian of up to 64 MB is simply allocated: it is half of the positions
that a recomputing backward keeps."""
from __future__ import annotations

import torch

from .binding import FP32, Net, NetDevice


def _pack4(x: torch.Tensor) -> torch.Tensor:
    out = torch.zeros(x.shape[0], 4, device=x.device, dtype=torch.float32)
    out[:, :3] = x
    return out


_ASK = 64 << 20            # bytes of Jacobian from which the free memory is looked up


def _rows(x: torch.Tensor) -> torch.Tensor:
    x = x.detach()
    if x.dtype != torch.float32 or not x.is_contiguous() or x.is_neg():
        x = torch.empty(x.shape, device=x.device, dtype=torch.float32).copy_(x)
    return x


class TravelTime(torch.autograd.Function):
    @staticmethod
    def forward(ctx, src, rcv, netdev: NetDevice, recompute: str = "auto"):
        assert src.is_cuda and rcv.is_cuda and src.shape == rcv.shape and src.shape[1] == 3
        P = src.shape[0]
        need_grad = ctx.needs_input_grad[0]
        if recompute == "auto":
            recompute_now = P * 16 > _ASK and P * 16 > torch.cuda.mem_get_info(src.device)[0] // 4
        else:
            recompute_now = bool(recompute)
        stream = torch.cuda.current_stream(src.device).cuda_stream
        T = torch.empty(P, device=src.device, dtype=torch.float32)
        J = None
        if need_grad and not recompute_now:
            try:
                J = torch.empty(P, 4, device=src.device, dtype=torch.float32)
            except torch.cuda.OutOfMemoryError:
                if recompute != "auto":
                    raise
        ctx.netdev = netdev
        ctx.recompute = J is None and need_grad
        if ctx.recompute:
            s4, r4 = _pack4(src.detach()), _pack4(rcv.detach())
            Tlo = torch.empty(P, device=src.device, dtype=torch.float32)
            netdev.spider_tt_pairs(P, s4.data_ptr(), r4.data_ptr(), T.data_ptr(), Tlo.data_ptr(), 0, stream)
            ctx.save_for_backward(s4, r4)
            return T + Tlo
        s3, r3 = _rows(src), _rows(rcv)
        netdev.spider_tt_pairs_rows(P, s3.data_ptr(), r3.data_ptr(), T.data_ptr(),
                                    J.data_ptr() if J is not None else 0, stream)
        if J is not None:
            ctx.save_for_backward(J)
        return T

    @staticmethod
    def backward(ctx, gT):
        if ctx.recompute:
            s4, r4 = ctx.saved_tensors
            P = s4.shape[0]
            T = torch.empty(P, device=s4.device)
            J = torch.empty(P, 4, device=s4.device)
            stream = torch.cuda.current_stream(s4.device).cuda_stream
            ctx.netdev.spider_tt_pairs(P, s4.data_ptr(), r4.data_ptr(), T.data_ptr(), 0,
                                       J.data_ptr(), stream)
        else:
            (J,) = ctx.saved_tensors
        return gT[:, None] * J[:, :3], None, None, None


def travel_time(src, rcv, netdev: NetDevice, recompute: str = "auto"):
    return TravelTime.apply(src, rcv, netdev, recompute)
