"""The length of the weight gradients' FP32 sums on a large batch: a thread's
sum goes to its block's partial every 256 terms, so the error does not grow
with the batch.

The bias gradient of the last 3x3 layer is a sum of known terms: its output
gradient is dy times the 1x1 layer's bfloat16 weight, in FP32. Equal terms of
one sign are the worst case (the roundings of a running sum go one way).
Bound: 256 terms of a thread, one addition to the block's partial per 256 x 4
x (resident blocks: at least one per SM) pixels, 3 groups, and per output 8 lanes
of at most (blocks / 8) partials with at most 8 blocks an SM, each addition
within 2^-24 of the sum.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h,w", [(12, 256, 256), (64, 512, 512)])
def test_bias_sum_of_equal_terms(n, h, w):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required")
    from paper_2303_10499_gb300 import build as B
    B.build()
    from paper_2303_10499_gb300 import gea as G, learned
    at, where = 0, {}
    for i, (cin, cout, k, *_) in enumerate(G.net_layout()):
        where[i] = (at, at + cout * k * k * cin, cout)
        at += cout * k * k * cin + cout
    net = G.Net(n, h, w, relu=False)
    theta = learned.initial_params(5)
    net.set_params(theta)
    r = torch.randn((n, h, w), device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    y, grad = torch.empty_like(r), torch.empty(G.net_param_count(), device="cuda")
    net.forward(r, y)
    net.backward(torch.full_like(r, 0.1), grad)
    o = where[14][0]
    wq = torch.tensor(theta[o:o + 16], device="cuda", dtype=torch.float32).bfloat16().float()
    want = (torch.tensor(0.1, device="cuda") * wq).double() * (n * h * w)
    _, b, cout = where[13]
    err = ((grad[b:b + cout].double() - want).abs() / want.abs()).max().item()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    additions = 256 + int(np.ceil(n * h * w / (256 * 4 * sms))) + 3 + sms + 8
    print(n, h, w, "error", err, "bound", additions * 2.0 ** -24)
    assert err <= additions * 2.0 ** -24
    net.close()
