"""The training gradients' sums have a stated order, so a training run repeats
itself bit for bit on every version of the kernels: each gradient tensor over
six Adam steps against recorded checksums (tests/golden/net_gradient_bits.txt,
one line per lattice, loss and step: the CRC-32 of every tensor's FP32 words).

The order: a weight gradient sums 16 consecutive sites of x per matrix
instruction, the rows and tiles of its partial in order, then the partials in
order; the other sums go per thread, by a binary tree over the block's threads
(bias gradients of the inner layers: threads in order), then over the blocks in
order.  The checksums hold for 152 multiprocessors (the numbers of blocks and
partials follow that count).  Adam divides by sqrt(v), so a last bit of a small
gradient grows from step to step: equality is what is asked.

Lattices: one tile and one partial; widths that are no multiple of a tile's 16
sites; more tiles than partials at every level; a long thin one.
"""

import os
import zlib

import numpy as np
import pytest

from paper_2105_00448_gb300 import hca

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "net_gradient_bits.txt")
CONVS = (("enc0", 16, 16), ("enc1", 16, 32), ("enc2", 32, 64), ("enc3", 64, 64), ("dec2", 64, 64), ("dec1", 64, 32),
         ("dec0", 32, 16))
SHAPES = [(8, 8, 8), (16, 24, 40), (24, 8, 56), (48, 56, 72), (64, 64, 64), (8, 8, 400), (104, 96, 120)]
STEPS = 6


def inputs(shape):
    """Weights, one recorded solve and one feature tensor, from uniform draws alone."""
    rng = np.random.default_rng(sum(shape))
    parts = []
    for _, ci, co in CONVS:
        parts += [(rng.random(27 * co * ci) - 0.5) * np.sqrt(24.0 / (27 * ci)), 0.1 * (rng.random(co) - 0.5)]
    params = np.concatenate(parts + [rng.random(17) - 0.5]).astype(np.float32)
    state = rng.integers(0, 6, shape).astype(np.uint8)
    perf = (0.5 + rng.random(shape)).astype(np.float32)
    K_prev = (2.0 + 16.0 * rng.random(shape)).astype(np.float32)
    K_new = (K_prev + rng.random(shape).astype(np.float32) - np.float32(0.5)).astype(np.float32)
    x = (rng.random((*shape, 16)) - 0.5).astype(np.float32)
    target = (rng.random(shape) - 0.5).astype(np.float32)
    return params, state, perf, K_prev, K_new, x, target


def checksums(shape, residual):
    """[step][tensor] CRC-32 of the gradients (the loss last) of STEPS training steps."""
    import torch

    def dev(a):
        return torch.from_numpy(a).cuda()

    nz, ny, nx = shape
    params, state, perf, K_prev, K_new, x, target = inputs(shape)
    net = hca.Net(nz, ny, nx, trainable=True)
    net.set_params(params)
    n = hca.hca_net_param_count()
    grads, loss = torch.empty(n, device="cuda"), torch.empty(1, device="cuda")
    cfg = hca.make_config(nx, ny, nz, precision="f32")
    held = [dev(a) for a in (state, perf, K_prev, K_new, target)]
    xb = dev(x).to(torch.bfloat16).contiguous()
    out = []
    for _ in range(STEPS):
        if residual:
            hca.hca_net_gradients(net.handle, cfg, *held[:4], w_mse=1.0, w_res=0.03, grads=grads, loss=loss)
        else:
            hca.hca_net_gradients_x(net.handle, xb, held[4], grads=grads, loss=loss)
        torch.cuda.synchronize()
        flat = grads.cpu().numpy()
        o, row = 0, []
        for _, ci, co in CONVS:
            for k in (27 * co * ci, co):
                row.append(zlib.crc32(flat[o:o + k].tobytes()))
                o += k
        row += [zlib.crc32(flat[o:].tobytes()), zlib.crc32(loss.cpu().numpy().tobytes())]
        out.append(row)
        hca.hca_net_adam(net.handle, 1e-3)
    net.close()
    return out


def line(shape, residual, step, row):
    return " ".join(["x".join(map(str, shape)), "residual" if residual else "mse", str(step)] + ["%08x" % c for c in row])


@pytest.mark.parametrize("residual", [True, False])
@pytest.mark.parametrize("shape", SHAPES)
def test_gradients_keep_their_bits(shape, residual):
    import torch

    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the checksums hold for 152 multiprocessors")
    golden = [s.strip() for s in open(GOLDEN) if not s.startswith("#")]
    for step, row in enumerate(checksums(shape, residual)):
        assert line(shape, residual, step, row) in golden, (step, row)


if __name__ == "__main__":   # prints the checksums of the library at hand
    for s in SHAPES:
        for res in (True, False):
            for k, r in enumerate(checksums(s, res)):
                print(line(s, res, k, r))
