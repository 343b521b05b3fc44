"""The surrogate's convolutions beyond the small images of
test_gpu_surrogate.py: wide output slices, streamed weights and several tiles
per block against FP64 sums on BF16 data, and what its calls report when a
device wait runs out."""
import ctypes

import numpy as np
import pytest

from paper_2604_21128_gb300 import qla

pytestmark = pytest.mark.gpu


def bf16(rng, shape, scale=1.0):
    import torch
    return torch.tensor(rng.standard_normal(shape) * scale, dtype=torch.float32).bfloat16().cuda()


def conv64(x, w):
    """FP64 periodic convolution on the GPU: x (B, H, W, ci), w (co, 9, ci)."""
    import torch
    x, w = x.double(), w.double()
    out = torch.zeros(x.shape[:3] + (w.shape[0],), dtype=torch.float64, device="cuda")
    for tap in range(9):
        shifted = torch.roll(x, (1 - tap // 3, 1 - tap % 3), (1, 2))
        out += torch.matmul(shifted, w[:, tap].T)
    return out


def accumulation_bound(steps):
    """Relative error of a sum in `steps` K = 16 tensor-core steps: products of
    BF16 values are exact, each step may truncate the FP32 running sum (on the
    mean half of 2^-23 of it, the sum growing as the root of the step)."""
    return 1e-6 + steps * 2.0 ** -24


def conv_raw(x, w):
    import torch
    B, H, W, cin = x.shape
    out = torch.empty((B, H, W, w.shape[0]), dtype=torch.float32, device="cuda")
    st = qla.load().surr_conv3x3_raw(ctypes.c_void_p(x.data_ptr()), B, H, W, cin,
                                     ctypes.c_void_p(w.data_ptr()), w.shape[0],
                                     ctypes.c_void_p(out.data_ptr()), None)
    return st, out


# widths that are no multiple of 128 need a tile's patches resident: with 16
# of them (cin = 512), 256-channel weight slices do not fit beside
@pytest.mark.parametrize("B,H,W,cin,cout", [(2, 64, 100, 512, 256), (1, 112, 112, 512, 512),
                                            (1, 16, 24, 512, 256), (1, 16, 24, 544, 32)])
def test_wide_inputs_are_taken(B, H, W, cin, cout):
    import torch
    rng = np.random.default_rng(cin + cout + W)
    x, w = bf16(rng, (B, H, W, cin)), bf16(rng, (cout, 9, cin), 0.1)
    st, out = conv_raw(x, w)
    assert st == 0
    want = conv64(x, w)
    # products of BF16 values are exact; the FP32 accumulation of 9 cin terms
    # rounds (~sqrt(9 cin) 6e-8 relative)
    assert float(torch.linalg.norm(out - want) / torch.linalg.norm(want)) <= 1e-5


# (on 152 SMs) slices of 256, 128 and 64 channels, weights resident and streamed
# in units of one, two and four patches, one tile per block and several, ragged
# tile edges; widths of 128 take the patches in the outer loop
@pytest.mark.parametrize("B,H,W,cin,cout", [(8, 64, 64, 256, 256), (3, 100, 90, 128, 256),
                                            (4, 96, 96, 64, 128), (2, 130, 104, 32, 64),
                                            (8, 128, 128, 128, 64), (2, 64, 128, 256, 128),
                                            (1, 40, 384, 96, 160), (5, 33, 72, 160, 96),
                                            (8, 32, 32, 128, 256), (8, 64, 64, 256, 512)])
def test_convolution_layouts_of_large_images(B, H, W, cin, cout):
    import torch
    rng = np.random.default_rng(B + H + W)
    x, w = bf16(rng, (B, H, W, cin)), bf16(rng, (cout, 9, cin), 0.1)
    st, out = conv_raw(x, w)
    assert st == 0
    want = conv64(x, w)
    assert float(torch.linalg.norm(out - want) / torch.linalg.norm(want)) <= \
        accumulation_bound(9 * cin / 16)


def small_net(seed=3):
    import torch
    from paper_2604_21128_gb300 import surrogate
    net = surrogate.Surrogate(32, 48, max_batch=2, seed=seed)
    rng = np.random.default_rng(seed)
    x = torch.tensor(rng.standard_normal((2, 32, 48, 6)), dtype=torch.float32, device="cuda")
    t = torch.tensor(rng.standard_normal((2, 32, 48, 3)) * 0.1, dtype=torch.float32, device="cuda")
    return net, x, t


def test_wait_that_runs_out_in_the_backward_pass_is_reported():
    """The loss is out before the backward pass: a wait that runs out there
    leaves the parameters alone, is reported when they are read, does not
    count as a step and does not touch another network."""
    lib = qla.load()
    net, x, t = small_net()
    other, _, _ = small_net()
    want, _, _ = small_net()
    for n in (net, want):
        n.train_step(x, t, 1e-3)
    before = net.params()
    assert lib.surr_test_stall_conv(2) == 0        # input gradients only
    try:
        loss = net.train_step(x, t, 1e-3)
        other_before = other.params()              # no timeout of its own
        with pytest.raises(qla.QLAError) as e:
            net.params()
    finally:
        assert lib.surr_test_stall_conv(0) == 0
    assert e.value.status == 5                     # QLA_ETIMEOUT
    assert np.array_equal(net.params(), before)
    # the next step is the second again
    assert net.train_step(x, t, 1e-3) == loss == want.train_step(x, t, 1e-3)
    assert np.array_equal(net.params(), want.params())
    assert np.array_equal(other.params(), other_before)


def test_gradient_with_a_wait_that_ran_out_is_refused():
    lib = qla.load()
    net, x, t = small_net()
    want = net.loss_grad(x, t)
    assert lib.surr_test_stall_conv(2) == 0
    try:
        with pytest.raises(qla.QLAError) as e:
            net.loss_grad(x, t)
    finally:
        assert lib.surr_test_stall_conv(0) == 0
    assert e.value.status == 5                     # QLA_ETIMEOUT
    got = net.loss_grad(x, t)
    assert got[0] == want[0] and np.array_equal(got[1], want[1])


def weight_grad_raw(dz, x, B, H, W, splits=2):
    """dz (.., cout) and x (.., cin) hold at least B H W pixels."""
    import torch
    cout, cin = dz.shape[-1], x.shape[-1]
    part = torch.full((splits * cout * 9 * cin,), 7.0, device="cuda")
    dw = torch.full((cout, 9, cin), 7.0, device="cuda")
    st = qla.load().surr_weight_grad_raw(ctypes.c_void_p(dz.data_ptr()),
                                         ctypes.c_void_p(x.data_ptr()), B, H, W, cout, cin, splits,
                                         ctypes.c_void_p(part.data_ptr()),
                                         ctypes.c_void_p(dw.data_ptr()), None)
    torch.cuda.synchronize()
    return st, dw


# widths of part segments (48, 80, 112, 208), whole rows per stage (16, 32, with
# heights that do and do not divide into stages), other widths; splits that end
# within a row; 32, 16 and 8 input channels per block
@pytest.mark.parametrize("B,H,W,cout,cin,splits", [(2, 9, 48, 32, 32, 3), (1, 17, 80, 64, 64, 5),
                                                   (3, 11, 112, 256, 32, 2), (1, 8, 208, 32, 96, 4),
                                                   (2, 12, 16, 64, 128, 2), (2, 6, 16, 32, 64, 3),
                                                   (1, 10, 32, 128, 256, 3), (3, 7, 32, 96, 32, 2),
                                                   (2, 6, 24, 64, 96, 2),
                                                   (8, 64, 64, 256, 256, 8),
                                                   (2, 128, 128, 64, 32, 128)])
def test_weight_gradient_at_ragged_widths(B, H, W, cout, cin, splits):
    import torch
    rng = np.random.default_rng(W + cout + splits)
    dz, x = bf16(rng, (B, H, W, cout)), bf16(rng, (B, H, W, cin))
    st, dw = weight_grad_raw(dz, x, B, H, W, splits)
    assert st == 0
    want = torch.empty((cout, 9, cin), dtype=torch.float64, device="cuda")
    z = dz.double().reshape(-1, cout).T
    for tap in range(9):
        shifted = torch.roll(x.double(), (1 - tap // 3, 1 - tap % 3), (1, 2))
        want[:, tap] = z @ shifted.reshape(-1, cin)
    assert float(torch.linalg.norm(dw - want) / torch.linalg.norm(want)) <= \
        accumulation_bound(B * H * W / splits / 16 + 4)


# deepest levels of one and of two pixels, sides that are no powers of two, and
# images large enough for the wide slices; bounds: those of the small images in
# test_gpu_surrogate.py
@pytest.mark.parametrize("B,H,W", [(1, 16, 16), (2, 32, 16), (2, 48, 80), (1, 112, 144),
                                   (2, 256, 128)])
def test_network_matches_fp64_reference(B, H, W):
    import torch
    from oracle import surrogate as ref
    from paper_2604_21128_gb300 import surrogate
    net = surrogate.Surrogate(H, W, max_batch=B, seed=1)
    rng = np.random.default_rng(H + W)
    theta = (rng.standard_normal(net.nparams) * 0.05).astype(np.float32)
    net.set_params(theta)
    x, t = rng.standard_normal((B, H, W, 6)), 0.1 * rng.standard_normal((B, H, W, 3))
    xd, td = (torch.tensor(v, dtype=torch.float32, device="cuda") for v in (x, t))
    got = net.forward(xd).cpu().numpy()
    want = ref.forward(theta.astype(np.float64), xd.cpu().numpy())
    assert np.linalg.norm(got - want) <= 3e-2 * np.linalg.norm(want)
    loss, g = net.loss_grad(xd, td)
    rloss, rg = ref.loss_grad(theta.astype(np.float64), xd.cpu().numpy(), td.cpu().numpy())
    assert abs(loss / rloss - 1) <= 3e-2
    assert np.linalg.norm(g - rg) <= 5e-2 * np.linalg.norm(rg)


@pytest.mark.parametrize("B,H,W", [(0, 4, 16), (2, 0, 16), (2, 4, 0)])
def test_weight_gradient_over_no_pixels_is_zero(B, H, W):
    rng = np.random.default_rng(1)
    dz, x = bf16(rng, (64, 32)), bf16(rng, (64, 64))
    st, dw = weight_grad_raw(dz, x, B, H, W)
    assert st == 0 and not dw.any()


@pytest.mark.parametrize("W", [16, 128])
def test_tensors_off_16_byte_boundaries_are_refused(W):
    rng = np.random.default_rng(2)
    x, z = bf16(rng, (2 * W + 1, 32)), bf16(rng, (2 * W, 32))
    off = x.reshape(-1)[1:1 + 2 * W * 32].reshape(1, 2, W, 32)
    assert off.data_ptr() % 16 == 2
    assert conv_raw(off, bf16(rng, (32, 9, 32)))[0] == 4          # QLA_ECUDA
    off = off.reshape(-1, 32)
    assert weight_grad_raw(z, off, 1, 2, W)[0] == 4
    assert weight_grad_raw(off, z, 1, 2, W)[0] == 4
