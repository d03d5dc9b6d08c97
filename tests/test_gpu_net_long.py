"""The network on a lattice with more tiles along z than a grid has blocks in
its third dimension (131,072 planes of 8 x 8 sites): its last planes against
a network on the last 128 planes alone.  The arithmetic of a site depends on its
surroundings only, so the outputs and stored activations are equal; the
activation gradients differ by the ratio of the sites, a power of two."""

import numpy as np
import pytest

import test_gpu_net as N
from paper_2105_00448_gb300 import hca

pytestmark = pytest.mark.gpu

LONG, SHORT, TAIL = 131072, 128, 32   # planes; TAIL of them feel no other plane (a site reaches 32 planes each way)


def test_many_planes():
    import torch

    rng = np.random.default_rng(11)
    x = torch.zeros((LONG, 8, 8, 16), dtype=torch.bfloat16, device=N.dev())
    x[-SHORT:] = N.to_bf16_dev(rng.standard_normal((SHORT, 8, 8, 16)) * 0.7)
    target = torch.zeros((LONG, 8, 8), device=N.dev())
    target[-SHORT:] = torch.from_numpy(rng.standard_normal((SHORT, 8, 8)).astype(np.float32)).to(N.dev())
    flat = N.random_params(12)
    got = []
    for planes in (LONG, SHORT):
        net = hca.Net(planes, 8, 8, trainable=True)
        net.set_params(flat)
        xs, ts = x[-planes:].contiguous(), target[-planes:].contiguous()
        out = torch.empty((planes, 8, 8), device=N.dev())
        hca.hca_net_forward_x(net.handle, xs, out)
        grads = torch.empty(hca.hca_net_param_count(), device=N.dev())
        hca.hca_net_gradients_x(net.handle, xs, ts, grads=grads)
        assert bool(torch.isfinite(grads).all())
        tails = [out[-TAIL:].clone()]
        for which, lvl, ch in ((0, 0, 16), (1, 1, 32), (4, 2, 64), (5, 1, 32), (6, 0, 16)):
            g = torch.empty((planes >> lvl, 8 >> lvl, 8 >> lvl, ch), dtype=torch.bfloat16, device=N.dev())
            hca.hca_net_read_gradient(net.handle, which, g)
            tails.append(g[-(TAIL >> lvl):].float() * (planes / SHORT))
        got.append(tails)
        net.close()
    for a, b in zip(*got):
        assert bool((b != 0).any()) and torch.equal(a, b)
