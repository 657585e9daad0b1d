"""Kernels at the sizes where they can go wrong: edges of tiles, remainders, the ends of their ranges.
Oracle and acceptance rules as in test_gpu_parity.py."""
import numpy as np
import pytest
import torch

import __graft_entry__ as entry
from oracle import prox_oracle as po
from paper_2607_27591_b200 import inputs
from tests.gpu_common import Problem, dev_bf16

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pb():
    entry.build()
    from paper_2607_27591_b200 import binding
    return binding


@pytest.mark.parametrize("D,F", [(128, 64), (256, 192), (640, 448)])
@pytest.mark.parametrize("bits,group", [(4, 0), (4, 128), (8, 0), (8, 128)])
def test_packer_tiles_ties_and_repacking(pb, D, F, bits, group):
    """Half and odd tiles; weights whose quotient is an exact half (integer multiples of half a scale, the row's
    largest weight being qmax scales), tiny weights (fp16-subnormal and zero scales); packing again in place."""
    wg, wu, wd, x = inputs.make_small(D, F, 1, seed=D + F + bits)
    rng = np.random.default_rng(7)
    qmax = (1 << (bits - 1)) - 1
    halves = rng.integers(-2 * qmax, 2 * qmax + 1, size=(F // 2, D)).astype(np.float32) / 2
    halves[:, ::128] = qmax                                        # every group's scale is exactly 2^-7
    wg[: F // 2] = inputs.f32_to_bf16_bits(halves * 2.0 ** -7)
    wu[3] = inputs.f32_to_bf16_bits(rng.standard_normal(D).astype(np.float32) * 1e-6)
    wu[5] = inputs.f32_to_bf16_bits(rng.standard_normal(D).astype(np.float32) * 1e-9)
    p = Problem(pb, wg, wu, wd, x)
    try:
        for again in range(2):
            if again:                                              # other weights in the same buffers
                wg, wu, wd = wg[::-1].copy(), wu[:, ::-1].copy(), wd[::-1].copy()
                for t, b in ((p.t_wg, wg), (p.t_wu, wu), (p.t_wd, wd)):
                    t.copy_(dev_bf16(b))
            pb.prox_quantize_proxy(p.h, bits, group)
            ng = 1 if group == 0 else D // group
            for which, w in enumerate((wg, wu)):
                q_ref, s_ref = po.quantize_proxy(inputs.bf16_bits_to_f32(w), bits, group)
                q, s = np.empty((F, D), dtype=np.int8), np.empty((F, ng), dtype=np.float32)
                pb.prox_proxy_export(p.h, which, q, s)
                assert np.array_equal(s, s_ref.astype(np.float32)) and np.array_equal(q, q_ref)
            # the channel-major copy of W_down: one kept channel at a time, y = h_j W_down[:, j]
            y = p.y_empty()
            for j in (0, 1, F // 2 + 1, F - 1):
                pb.prox_stage2_ffn(p.h, p.t_x, 1, torch.tensor([[j]], dtype=torch.int32, device="cuda"), 1, y)
                y_ref, _ = po.stage2(po.bf16_to_f64(x[0]), [j], *(inputs.bf16_bits_to_f32(w) for w in (wg, wu, wd)))
                # fp32 sums of D products against fp64: sqrt(D) 2^-24 relative, times a few
                assert np.linalg.norm(y.cpu().numpy()[0] - y_ref) <= 1e-4 * np.linalg.norm(y_ref) + 1e-20
    finally:
        p.close()
