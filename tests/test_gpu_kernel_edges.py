"""Kernels at the sizes where they can go wrong: edges of tiles, remainders, the ends of their ranges.
Oracle and acceptance rules as in test_gpu_parity.py."""
import numpy as np
import pytest
import torch

import __graft_entry__ as entry
from oracle import prox_oracle as po
from paper_2607_27591_b200 import inputs
from tests.gpu_common import Problem, dev_bf16
from tests.test_gpu_parity import _check_fused_stage1

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


@pytest.mark.parametrize("D,F,bits,group", [(512, 1536, 4, 128), (512, 1536, 8, 0), (1024, 4096, 4, 0), (256, 19136, 4, 128)])
@pytest.mark.parametrize("grid", [1, 7, 100])
def test_persistent_kernel_with_part_of_its_grid(pb, D, F, bits, group, grid):
    """Blocks that do not run are replaced by those that do: the same masks and results with a part of the grid, in the
    plain, the threshold and the layer form in place (19136 channels: a line and sometimes half a line of the proxy
    rows each)."""
    k1, k2 = D // 3, F // 4 + 1
    wg, wu, wd, x = inputs.make_small(D, F, 1, seed=D + F + bits)
    p = Problem(pb, wg, wu, wd, x)
    try:
        pb.prox_quantize_proxy(p.h, bits, group)
        nw = torch.ones(D, dtype=torch.bfloat16, device="cuda")

        def run():
            y, yt = p.y_empty(), p.y_empty()
            sel, idx = torch.empty(1, k2, dtype=torch.int32, device="cuda"), torch.empty(k1, dtype=torch.int32, device="cuda")
            sc = torch.empty(F, dtype=torch.float32, device="cuda")
            pb.prox_ffn_forward(p.h, p.t_x, 1, k1, k2, y)
            pb.prox_ffn_last_mask(p.h, 1, k2, sel)
            pb.prox_ffn_last_stage1(p.h, k1, idx, sc)
            tau_x = float(p.t_x[0].float().abs().sort(descending=True).values[k1 - 1])
            tau_s = float(sc.sort(descending=True).values[k2 - 1])
            pb.prox_runtime_sparsity(p.h, reset=True)
            pb.prox_ffn_forward_threshold(p.h, p.t_x, 1, tau_x, tau_s, yt)
            kept = pb.prox_runtime_sparsity(p.h)
            xr = p.t_x.float().contiguous()
            pb.prox_ffn_block_forward(p.h, xr, nw, 1e-6, 1, k1, k2, xr)
            torch.cuda.synchronize()
            assert pb.prox_last_device_status(p.h) == 0
            return [t.cpu().numpy() for t in (sel, idx, sc)], [t.cpu().numpy() for t in (y, yt, xr)], kept

        whole, part = run(), None
        pb.prox_debug_set_grid(p.h, grid)
        for _ in range(3):                                         # both sets of counters
            part = run()
            for a, b in zip(whole[0], part[0]):
                assert np.array_equal(a, b)
            assert whole[2] == part[2]
            # the same products, summed in fp32 in another order
            for a, b in zip(whole[1], part[1]):
                assert np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(a)
        pb.prox_debug_set_grid(p.h, 0)
        again = run()
        for a, b in zip(whole[0], again[0]):
            assert np.array_equal(a, b)
    finally:
        p.close()


@pytest.mark.parametrize("F,bits", [(9536, 4), (19008, 4), (28672, 4), (38016, 4), (9472, 8), (9536, 8), (14336, 8), (15872, 8)])
def test_shares_of_the_proxy_columns(pb, F, bits):
    """Proxy scores with less than a 128-byte line of the packed rows per SM, with one or two lines and halves or wholes of
    the lines left over, with a last line that is half a line, against the oracle."""
    p = Problem(pb, *inputs.make_small(256, F, 2, seed=F + bits))
    try:
        p.quantize(bits, 128)
        for t, k1 in ((0, 85), (1, 256)):
            _check_fused_stage1(pb, p, p.t_x[t], p.x[t], k1, F // 4)
        assert pb.prox_last_device_status(p.h) == 0
    finally:
        p.close()


@pytest.mark.parametrize("F", [64, 192, 2048, 4160, 65536])
@pytest.mark.parametrize("B,shared", [(1, False), (3, False), (8, True)])
def test_channel_mask_is_the_exact_topk_of_the_scores(pb, F, B, shared):
    """Few and many channels per block of a cluster, ties (repeated channels: equal scores), every k at the ends; the
    scores at an address that is not a multiple of 16."""
    D = 128
    g = torch.Generator(device="cuda").manual_seed(F + B)
    w = [(torch.randn(F, D, device="cuda", generator=g) * 0.1).to(torch.bfloat16) for _ in range(2)]
    for t in w:
        t[F // 2:] = t[:F - F // 2]                                 # every score twice
    wd = torch.zeros(D, F, dtype=torch.bfloat16, device="cuda")
    x = torch.randn(B, D, device="cuda", generator=g).to(torch.bfloat16)
    h = pb.prox_ffn_create(D, F, max(B, 2), 1, *w, wd)
    try:
        pb.prox_quantize_proxy(h, 4, 128)
        pb.prox_ffn_set_mask_policy(h, int(shared))
        buf = torch.empty(B * F + 1, dtype=torch.float32, device="cuda")
        for k2 in (1, 2, F // 3, F // 2 + 1, F - 1, F):
            for off in (0, 1):
                sc = buf[off:off + B * F].view(B, F)
                sel = torch.empty(B, k2, dtype=torch.int32, device="cuda")
                pb.prox_stage1_mask(h, x, B, 50, k2, sel, sc)
                rank = sc
                if shared:                                          # added token after token in fp32, as the library does
                    rank = torch.zeros(1, F, device="cuda")
                    for b in range(B):
                        rank = rank + sc[b]
                    rank = rank.expand(B, F)
                order = torch.sort(rank, dim=1, descending=True, stable=True).indices[:, :k2]
                assert torch.equal(sel.long(), order.sort(dim=1).values), (k2, off)
            # nothing but ties: the first k2 channels
            pb.prox_stage1_mask(h, torch.zeros_like(x), B, 50, k2, sel, sc)
            assert torch.equal(sel, torch.arange(k2, dtype=torch.int32, device="cuda").expand(B, k2))
        assert pb.prox_last_device_status(h) == 0
    finally:
        pb.prox_ffn_destroy(h)


@pytest.mark.parametrize("D,F", [(128, 64), (640, 1600), (2176, 2048), (3584, 1472), (4224, 1472), (8192, 704)])
@pytest.mark.parametrize("B", [2, 8])
def test_batch_stage2_rows_in_sections(pb, D, F, B):
    """One to four sections of a row, the last one short; unions smaller than the grid, ragged tiles and all channels."""
    wg, wu, wd, x = inputs.make_small(D, F, B, seed=D + F)
    p = Problem(pb, wg, wu, wd, x, max_batch=B)
    try:
        pb.prox_quantize_proxy(p.h, 4, 128)
        rng = np.random.default_rng(B)
        for k2 in (1, 13, F // 2, F):
            sel = np.stack([np.sort(rng.choice(F, size=k2, replace=False)) for _ in range(B)]).astype(np.int32)
            y = p.y_empty(B)
            pb.prox_stage2_ffn(p.h, p.t_x[:B], B, torch.from_numpy(sel).cuda(), k2, y)
            for b in range(B):
                y_ref, _ = po.stage2(p.x[b], sel[b], p.wg, p.wu, p.wd)
                # h enters the down projection as a bf16 pair (2^-17 relative), sums in fp32
                assert np.linalg.norm(y.cpu().numpy()[b] - y_ref) <= 1e-4 * np.linalg.norm(y_ref)
        assert pb.prox_last_device_status(p.h) == 0
    finally:
        p.close()


@pytest.mark.parametrize("D,F,bits,group", [(128, 64, 4, 0), (640, 4992, 8, 128), (8192, 704, 4, 128), (10240, 192, 4, 128), (1024, 2048, 16, 0)])
def test_stages_one_by_one(pb, D, F, bits, group):
    """The stages called alone (persistent kernel up to its scores, and on a given list; wider layers and 16-bit proxies:
    step-wise kernels) against the whole path on the same masks, with repeated calls; bad channel ids are skipped."""
    wg, wu, wd, x = inputs.make_small(D, F, 2, seed=D + F)
    p = Problem(pb, wg, wu, wd, x)
    try:
        pb.prox_quantize_proxy(p.h, bits, group)
        for k1, k2 in ((D // 3, F // 3), (1, 1), (D, F)):
            for t in (0, 1, 0):
                y, y1 = p.y_empty(), p.y_empty()
                sel, sel1 = (torch.empty(1, k2, dtype=torch.int32, device="cuda") for _ in range(2))
                sc, sc1 = (torch.empty(F, dtype=torch.float32, device="cuda") for _ in range(2))
                pb.prox_ffn_forward(p.h, p.t_x[t], 1, k1, k2, y)
                pb.prox_ffn_last_mask(p.h, 1, k2, sel)
                pb.prox_ffn_last_stage1(p.h, k1, None, sc)
                pb.prox_stage1_mask(p.h, p.t_x[t], 1, k1, k2, sel1, sc1)
                pb.prox_stage2_ffn(p.h, p.t_x[t], 1, sel1, k2, y1)
                torch.cuda.synchronize()
                assert torch.equal(sc, sc1) and torch.equal(sel, sel1)
                # the same products in another order of summation
                assert float((y - y1).norm()) <= 1e-5 * float(y.norm())
        n = min(F, 40)
        ids = torch.arange(F, dtype=torch.int32, device="cuda").view(1, F).contiguous()
        cnt = torch.tensor([n], dtype=torch.int32, device="cuda")
        y, y1 = p.y_empty(), p.y_empty()
        pb.prox_stage2_ffn_var(p.h, p.t_x, 1, ids, cnt, y)
        assert pb.prox_last_device_status(p.h) == 0
        bad = torch.cat([ids[0, :n], torch.tensor([F, -1], dtype=torch.int32, device="cuda")]).view(1, -1).contiguous()
        pb.prox_stage2_ffn(p.h, p.t_x, 1, bad, n + 2, y1)
        assert pb.prox_last_device_status(p.h) == 1
        assert float((y - y1).norm()) <= 1e-5 * float(y.norm())
    finally:
        p.close()


@pytest.mark.parametrize("D,F,B", [(128, 512, 2), (256, 768, 8), (1024, 3072, 5), (4224, 1472, 3), (9216, 320, 8)])
def test_batch_layer_form_rounds_the_residual_stream_once(pb, D, F, B):
    """x_res + y with one rounding to fp32 per element, in place or not, few or many blocks per column tile: a residual
    stream a thousand times y, against the y that the plain call gives for the same normalised input."""
    wg, wu, wd, x = inputs.make_small(D, F, B, seed=D + F)
    p = Problem(pb, wg, wu, wd, x, max_batch=B)
    try:
        pb.prox_quantize_proxy(p.h, 4, 128)
        k1, k2 = D // 2, F // 2
        nw = torch.ones(D, dtype=torch.bfloat16, device="cuda")
        xr = (p.t_x[:B].float() * 1e3 + 1.0).contiguous()
        xn = torch.empty(B, D, dtype=torch.bfloat16, device="cuda")
        pb.prox_rmsnorm(p.h, xr, nw, 1e-6, B, xn)
        y, out = p.y_empty(B), torch.empty_like(xr)
        pb.prox_ffn_forward(p.h, xn, B, k1, k2, y)
        for again in range(2):                                     # the accumulator is back at zero
            pb.prox_ffn_block_forward(p.h, xr, nw, 1e-6, B, k1, k2, out)
            inplace = xr.clone()
            pb.prox_ffn_block_forward(p.h, inplace, nw, 1e-6, B, k1, k2, inplace)
            exact = xr.double().cpu().numpy() + y.double().cpu().numpy()
            # half a unit in the last place, and what two orders of y's fp32 sums differ by
            bound = 0.5 * np.spacing(np.abs(exact).astype(np.float32)).astype(np.float64) + 1e-5 * float(y.double().pow(2).mean().sqrt())
            for got in (out, inplace):
                assert np.all(np.abs(got.double().cpu().numpy() - exact) <= bound)
        assert pb.prox_last_device_status(p.h) == 0
    finally:
        p.close()


@pytest.mark.parametrize("D,F", [(128, 12288), (640, 3136), (128, 65536)])
@pytest.mark.parametrize("grid", [1, 18, 56])
def test_batch_gateup_on_fewer_sms(pb, D, F, grid):
    """A block's share of the union is bounded whatever the number of SMs: every channel in the union, fewer blocks than
    a share's bound allows for."""
    B = 2
    g = torch.Generator(device="cuda").manual_seed(F)
    w = [torch.empty(s, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.1, generator=g) for s in ((F, D), (F, D), (D, F))]
    x = torch.randn(B, D, device="cuda", generator=g).to(torch.bfloat16)
    h = pb.prox_ffn_create(D, F, B, 1, *w)
    try:
        pb.prox_quantize_proxy(h, 4, 128)
        sel = torch.arange(F, dtype=torch.int32, device="cuda").repeat(B, 1)
        whole, part = (torch.empty(B, D, device="cuda") for _ in range(2))
        pb.prox_stage2_ffn(h, x, B, sel, F, whole)
        pb.prox_debug_set_grid(h, grid)
        pb.prox_stage2_ffn(h, x, B, sel, F, part)
        y64 = [(lambda gt, up: w[2].double() @ (up * gt / (1 + torch.exp(-gt))))(w[0].double() @ x[b].double(), w[1].double() @ x[b].double())
               for b in range(B)]
        for b in range(B):                                         # h enters the down projection as a bf16 pair: 2^-17
            for y in (whole, part):
                assert float((y[b].double() - y64[b]).norm()) <= 1e-4 * float(y64[b].norm())
        assert pb.prox_last_device_status(h) == 0
    finally:
        pb.prox_ffn_destroy(h)


@pytest.mark.parametrize("bits,group", [(4, 128), (8, 0)])
def test_expired_wait_inside_stage1_is_reported(pb, bits, group):
    """The wait for the code offsets runs out in one block, in Stage 1 called alone and in the whole path: the status says
    so (the scores of that block are not valid), y is untouched, and the next calls are ordinary."""
    D, F, k1, k2 = 512, 1536, 200, 300
    p = Problem(pb, *inputs.make_small(D, F, 1, seed=3))
    try:
        pb.prox_quantize_proxy(p.h, bits, group)

        def stage1(tau=False):
            sel, cnt = torch.empty(1, F if tau else k2, dtype=torch.int32, device="cuda"), torch.empty(1, dtype=torch.int32, device="cuda")
            sc = torch.empty(F, device="cuda")
            if tau:
                pb.prox_stage1_mask_threshold(p.h, p.t_x, 1, 0.5, 0.1, sel, cnt, sc)
            else:
                pb.prox_stage1_mask(p.h, p.t_x, 1, k1, k2, sel, sc)
            return sc

        y = p.y_empty()
        good = [stage1().cpu(), stage1(True).cpu()]
        pb.prox_debug_set_wait(p.h, 500, 1 << 31)
        try:
            for tau in (False, True):
                stage1(tau)
                status, code = pb.prox_last_device_status_raw(p.h)
                assert status == 6 and code == 4          # PROX_ERR_TIMEOUT
            y.fill_(7.0)
            pb.prox_ffn_forward(p.h, p.t_x, 1, k1, k2, y)
            status, code = pb.prox_last_device_status_raw(p.h)
            assert status == 6 and code == 4 and torch.all(y == 7.0)
            nw, xr = torch.ones(D, dtype=torch.bfloat16, device="cuda"), p.t_x.float().contiguous()
            for form in (lambda: pb.prox_ffn_block_forward(p.h, xr, nw, 1e-6, 1, k1, k2, xr),
                         lambda: pb.prox_ffn_block_forward_threshold(p.h, xr, nw, 1e-6, 1, 0.5, 0.1, xr)):
                form()                                    # in place: nothing of the call has reached the residual stream
                status, code = pb.prox_last_device_status_raw(p.h)
                assert status == 6 and code == 4 and torch.equal(xr, p.t_x.float())
        finally:
            pb.prox_debug_set_wait(p.h, 0, 0)
        assert torch.equal(stage1().cpu(), good[0]) and torch.equal(stage1(True).cpu(), good[1])
        pb.prox_ffn_forward(p.h, p.t_x, 1, k1, k2, y)
        assert pb.prox_last_device_status(p.h) == 0 and not torch.any(y == 7.0)
    finally:
        p.close()


@pytest.mark.parametrize("stale", [-1.0, float("nan"), float("-inf")])
def test_topk_of_a_stage1_that_gave_up_stays_in_its_list(pb, stale):
    """One block, which gives up in its first share: most scores are whatever the caller's buffer held.  The call reports
    it, and the list still has k2 valid channels and nothing behind them."""
    D, F, k1, k2 = 512, 12288, 200, 1000
    p = Problem(pb, *inputs.make_small(D, F, 1, seed=5))
    try:
        pb.prox_quantize_proxy(p.h, 4, 128)
        sc = torch.full((F,), stale, device="cuda")
        sel = torch.full((F,), -7, dtype=torch.int32, device="cuda")
        pb.prox_debug_set_grid(p.h, 1)
        pb.prox_debug_set_wait(p.h, 500, 1 << 31)
        try:
            pb.prox_stage1_mask(p.h, p.t_x, 1, k1, k2, sel, sc)
            status, code = pb.prox_last_device_status_raw(p.h)
        finally:
            pb.prox_debug_set_wait(p.h, 0, 0)
            pb.prox_debug_set_grid(p.h, 0)
        assert status == 6 and code == 4
        got = sel.cpu().numpy()
        assert np.all(got[k2:] == -7) and np.all(got[1:k2] > got[:k2 - 1]) and got[0] >= 0 and got[k2 - 1] < F
    finally:
        p.close()


@pytest.mark.parametrize("shared", [0, 1])
@pytest.mark.parametrize("bits", [4, 8])
def test_overflowed_scales_leave_nothing_behind(pb, bits, shared):
    """Finite weights whose scale overflows fp16 in one channel (its scores are not numbers), a call with two tokens; then
    ordinary weights and a call with eight: the masks are those of a handle that never saw the first weights."""
    D, F, k1, k2 = 256, 512, 100, 200
    wg, wu, wd, x = inputs.make_small(D, F, 8, seed=11)
    p, fresh = Problem(pb, wg, wu, wd, x, max_batch=8), Problem(pb, wg, wu, wd, x, max_batch=8)
    try:
        good = p.t_wg[17].clone()
        p.t_wg[17] = 3e38
        for q in (p, fresh):
            pb.prox_ffn_set_mask_policy(q.h, shared)
            pb.prox_quantize_proxy(q.h, bits, 128)
        y = p.y_empty(8)
        pb.prox_ffn_forward(p.h, p.t_x, 2, k1, k2, y)
        p.t_wg[17] = good
        pb.prox_quantize_proxy(p.h, bits, 128)
        sel = [torch.empty(8, k2, dtype=torch.int32, device="cuda") for _ in range(2)]
        for q, s in zip((p, fresh), sel):
            pb.prox_ffn_forward(q.h, q.t_x, 8, k1, k2, y)
            pb.prox_ffn_last_mask(q.h, 8, k2, s)
        assert torch.equal(sel[0], sel[1])
    finally:
        p.close()
        fresh.close()


@pytest.mark.parametrize("F", [64, 1600, 4160])
@pytest.mark.parametrize("B,bits", [(2, 4), (5, 8), (8, 4)])
def test_batch_stage1_scores_asked_for_or_not(pb, F, B, bits):
    """The scores that the caller asks for are the same with either mask policy and those of the tokens alone (up to the
    16 bits to which a batch's inputs are rounded), and asking for them changes no mask."""
    D, k1, k2 = 384, 200, F // 3
    p = Problem(pb, *inputs.make_small(D, F, B, seed=F + B), max_batch=B)
    try:
        pb.prox_quantize_proxy(p.h, bits, 128)
        got = []
        for shared in (0, 1):
            pb.prox_ffn_set_mask_policy(p.h, shared)
            sel, sel1 = (torch.empty(B, k2, dtype=torch.int32, device="cuda") for _ in range(2))
            sc = torch.full((B, F), -1.0, device="cuda")
            pb.prox_stage1_mask(p.h, p.t_x, B, k1, k2, sel, sc)
            pb.prox_stage1_mask(p.h, p.t_x, B, k1, k2, sel1)
            assert torch.equal(sel, sel1)
            got.append(sc)
        # sums of two or three parts of a tile's units, added in any order
        assert float((got[0] - got[1]).norm()) <= 1e-5 * float(got[0].norm())
        alone = torch.empty(F, device="cuda")
        for b in range(B):
            pb.prox_stage1_mask(p.h, p.t_x[b], 1, k1, k2, sel[0], alone)
            assert float((got[0][b] - alone).norm()) <= 2e-3 * float(alone.norm())
        assert pb.prox_last_device_status(p.h) == 0
    finally:
        p.close()


def test_last_mask_of_a_shared_mask_call(pb):
    """The one list of a shared-mask call for every token, after other calls on the handle, and per-token lists again."""
    D, F, B, k1, k2 = 384, 4160, 5, 200, 700
    p = Problem(pb, *inputs.make_small(D, F, B, seed=9), max_batch=B)
    try:
        pb.prox_quantize_proxy(p.h, 4, 128)
        y = p.y_empty(B)
        want = {}
        for shared in (0, 1):
            pb.prox_ffn_set_mask_policy(p.h, shared)
            want[shared] = torch.empty(B, k2, dtype=torch.int32, device="cuda")
            pb.prox_stage1_mask(p.h, p.t_x, B, k1, k2, want[shared])
        assert all(torch.equal(want[1][0], want[1][b]) for b in range(B)) and not torch.equal(want[0][0], want[0][1])

        def last():
            got = torch.full((B, k2), -1, dtype=torch.int32, device="cuda")
            pb.prox_ffn_last_mask(p.h, B, k2, got)
            return got

        for shared in (1, 0, 1):
            pb.prox_ffn_set_mask_policy(p.h, shared)
            pb.prox_ffn_forward(p.h, p.t_x, B, k1, k2, y)
            assert torch.equal(last(), want[shared])
            other = torch.empty(B, k2, dtype=torch.int32, device="cuda")
            pb.prox_stage1_mask(p.h, p.t_x, B, k1, k2, other)      # Stage 1 alone leaves the forward call's mask
            pb.prox_stage2_ffn(p.h, p.t_x, B, other, k2, y)
            assert torch.equal(last(), want[shared])
        pb.prox_ffn_forward_proxy_values(p.h, p.t_x, B, k1, k2, y)  # (always per token)
        assert not torch.equal(last()[0], last()[1])
        assert pb.prox_last_device_status(p.h) == 0
    finally:
        p.close()


@pytest.mark.parametrize("F,B,shared", [(12288, 1, False), (12352, 1, False), (10240, 3, False), (10304, 3, False), (12288, 2, True),
                                        (12352, 2, True)])
def test_channel_mask_at_the_lines_of_its_dispatch(pb, F, B, shared):
    """One block per list up to 12288 channels (10240 for several lists), a cluster above."""
    test_channel_mask_is_the_exact_topk_of_the_scores(pb, F, B, shared)


@pytest.mark.parametrize("bits,group", [(4, 128), (8, 0)])
def test_forms_mixed_on_one_handle(pb, bits, group):
    """Plain, threshold, layer and staged calls in any order on one handle: the score histograms that some forms fill and
    others only clear leave every mask, count and score as on a handle that saw that form alone."""
    D, F, k1, k2 = 512, 1600, 170, 400
    g = torch.Generator(device="cuda").manual_seed(bits)
    w = [torch.empty(s, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.04, generator=g) for s in ((F, D), (F, D), (D, F))]
    x = torch.randn(4, D, device="cuda", generator=g).to(torch.bfloat16)
    nw = torch.ones(D, dtype=torch.bfloat16, device="cuda")

    def call(h, form, t):
        y, sel = torch.empty(1, D, device="cuda"), torch.empty(1, k2, dtype=torch.int32, device="cuda")
        if form == "plain":
            pb.prox_ffn_forward(h, x[t], 1, k1, k2, y)
            pb.prox_ffn_last_mask(h, 1, k2, sel)
            return [sel]
        if form == "layer":
            xr = x[t].float()
            pb.prox_ffn_block_forward(h, xr, nw, 1e-6, 1, k1, k2, y)
            pb.prox_ffn_last_mask(h, 1, k2, sel)
            torch.cuda.synchronize()
            return [sel]
        if form == "threshold":
            pb.prox_runtime_sparsity(h, reset=True)
            pb.prox_ffn_forward_threshold(h, x[t], 1, 0.9, 0.05, y)
            tokens, s1, s2, e = pb.prox_runtime_sparsity(h)
            return [torch.tensor([float(tokens), s1, s2])]
        sc = torch.empty(F, device="cuda")
        if form == "stage1":
            pb.prox_stage1_mask(h, x[t], 1, k1, k2, sel, sc)
            return [sel, sc]
        cnt, lst = torch.empty(1, dtype=torch.int32, device="cuda"), torch.zeros(1, F, dtype=torch.int32, device="cuda")
        pb.prox_stage1_mask_threshold(h, x[t], 1, 0.9, 0.05, lst, cnt, sc)
        n = int(cnt)
        pb.prox_stage2_ffn_var(h, x[t], 1, lst, cnt, y)
        return [cnt, lst[:, :n], sc]

    forms = ["plain", "layer", "threshold", "stage1", "staged threshold"]
    hs = []
    try:
        alone = {}
        for f in forms + [None]:
            hs.append(pb.prox_ffn_create(D, F, 1, 1, *w))
            pb.prox_quantize_proxy(hs[-1], bits, group)
            if f:
                for t in range(4):                                 # (four calls: both sets of histograms)
                    alone[f, t] = [v.cpu() for v in call(hs[-1], f, t)]
        rng = np.random.default_rng(0)
        for _ in range(60):
            f, t = forms[rng.integers(len(forms))], int(rng.integers(4))
            assert all(torch.equal(a, b.cpu()) for a, b in zip(alone[f, t], call(hs[-1], f, t))), (f, t)
        assert pb.prox_last_device_status(hs[-1]) == 0
    finally:
        for h in hs:
            pb.prox_ffn_destroy(h)


@pytest.mark.parametrize("F,bits", [(64, 8), (512, 4), (4160, 4), (16384, 8), (16448, 8), (33344, 4), (50048, 8), (65536, 4)])
@pytest.mark.parametrize("distinct", [0, 8, 200])
def test_persistent_kernel_mask_is_the_exact_topk_of_its_scores(pb, F, bits, distinct):
    """The channel mask of the whole path against the scores it was made from (ties: lower channel first): one and several
    groups of half scores per thread, and with few distinct channels many equal scores in the threshold bin, so that its
    members do not fit the index list and are cut by their channels (the rows are short here: the list lies behind the ring);
    and the threshold form at the k-th score."""
    D, k1 = 128, 50
    g = torch.Generator(device="cuda").manual_seed(F + distinct)
    w = [(torch.randn(F, D, device="cuda", generator=g) * 0.1).to(torch.bfloat16) for _ in range(2)]
    if 0 < distinct < F:
        for t in w:
            t.copy_(t[torch.arange(F, device="cuda") % distinct])
    wd = (torch.randn(D, F, device="cuda", generator=g) * 0.1).to(torch.bfloat16)
    x = torch.randn(1, D, device="cuda", generator=g).to(torch.bfloat16)
    h = pb.prox_ffn_create(D, F, 1, 1, *w, wd)
    try:
        pb.prox_quantize_proxy(h, bits, 128)
        y, ref, sc = (torch.empty(n, dtype=torch.float32, device="cuda") for n in (D, D, F))
        for k2 in (1, F // 7 + 1, F // 2 + 1, F - 1, F):
            sel = torch.empty(1, k2, dtype=torch.int32, device="cuda")
            pb.prox_ffn_forward(h, x, 1, k1, k2, y)
            pb.prox_ffn_last_mask(h, 1, k2, sel)
            pb.prox_ffn_last_stage1(h, k1, None, sc)
            order = torch.sort(sc, descending=True, stable=True).indices[:k2]
            assert torch.equal(sel[0].long(), order.sort().values), k2
            pb.prox_stage2_ffn(h, x, 1, sel, k2, ref)
            # the same products, summed in fp32 in another order
            assert (y - ref).norm() <= 1e-5 * ref.norm(), k2
            kth, xa = sc[order[-1]], float(x[0].float().abs().sort(descending=True).values[k1 - 1])
            below = sc[sc < kth]
            nxt = below.max() if below.numel() else torch.zeros_like(kth)
            # between two scores (1e-5 apart or more), and with the same inputs, hence the same scores
            if kth - nxt > 1e-5 * kth and int((x[0].float().abs() >= xa).sum()) == k1:
                kept = torch.empty(1, int((sc >= kth).sum()), dtype=torch.int32, device="cuda")
                pb.prox_ffn_forward_threshold(h, x, 1, xa, float((kth + nxt) / 2), y)
                pb.prox_ffn_last_mask(h, 1, kept.shape[1], kept)
                assert torch.equal(kept[0].long(), (sc >= kth).nonzero()[:, 0]), k2
        assert pb.prox_last_device_status(h) == 0
    finally:
        pb.prox_ffn_destroy(h)


@pytest.mark.parametrize("bits", [4, 8])
def test_packer_keeps_what_is_not_a_number_to_its_channel(pb, bits):
    """A channel with an infinite weight or a scale beyond fp16 leaves the codes of the channels in the same words alone."""
    D, F = 128, 64
    wg, wu, wd, x = inputs.make_small(D, F, 1, seed=bits)
    bad = wg.copy()
    bad[5, 9] = 0x7F80                                              # inf
    bad[6, :] = inputs.f32_to_bf16_bits(np.full(D, 1e30, dtype=np.float32))
    p = Problem(pb, bad, wu, wd, x)
    try:
        pb.prox_quantize_proxy(p.h, bits, 128)
        q, s = np.empty((F, D), dtype=np.int8), np.empty((F, 1), dtype=np.float32)
        pb.prox_proxy_export(p.h, 0, q, s)
        q_ref, s_ref = po.quantize_proxy(inputs.bf16_bits_to_f32(wg), bits, 128)
        others = [j for j in range(F) if j not in (5, 6)]
        assert np.array_equal(q[others], q_ref[others]) and np.array_equal(s[others], s_ref.astype(np.float32)[others])
    finally:
        p.close()


def _mask_is_the_exact_topk(pb, D, F, bits, group, distinct, zero):
    """Forward calls on repeated channels (`distinct` different ones, 0 = all): the mask against a stable sort of the scores
    that it was made from, y against Stage 2 on that mask."""
    g = torch.Generator(device="cuda").manual_seed(D + F + distinct)
    w = [torch.empty(F, D, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.5 / D ** 0.5, generator=g) for _ in range(2)]
    if distinct:
        for t in w:
            t.copy_(t[torch.arange(F, device="cuda") % distinct])
    wd = torch.empty(D, F, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.1, generator=g)
    x = torch.zeros(1, D, device="cuda") if zero else torch.randn(1, D, device="cuda", generator=g)
    x, k1 = x.to(torch.bfloat16), D // 3
    h = pb.prox_ffn_create(D, F, 1, 1, *w, wd)
    try:
        pb.prox_quantize_proxy(h, bits, group)
        y, ref, sc = (torch.empty(n, dtype=torch.float32, device="cuda") for n in (D, D, F))
        for k2 in (1, F // 3 + 1, F - 1):
            assert pb.prox_fused_kernel_info(h, k1, k2)["usable"] == 1
            sel = torch.empty(1, k2, dtype=torch.int32, device="cuda")
            pb.prox_ffn_forward(h, x, 1, k1, k2, y)
            pb.prox_ffn_last_mask(h, 1, k2, sel)
            pb.prox_ffn_last_stage1(h, k1, None, sc)
            order = torch.sort(sc, descending=True, stable=True).indices[:k2]
            assert torch.equal(sel[0].long(), order.sort().values), k2
            pb.prox_stage2_ffn(h, x, 1, sel, k2, ref)
            # the same products, summed in fp32 in another order
            assert (y - ref).norm() <= 1e-5 * ref.norm(), k2
        assert pb.prox_last_device_status(h) == 0
    finally:
        pb.prox_ffn_destroy(h)


@pytest.mark.parametrize("zero", [False, True])
@pytest.mark.parametrize("D,F,bits,group,distinct", [(128, 40960, 4, 128, 1), (128, 65536, 4, 0, 2), (128, 65536, 8, 128, 1), (8192, 28672, 4, 0, 1)])
def test_threshold_bin_too_long_for_its_list(pb, D, F, bits, group, distinct, zero):
    """So many equal scores that the list of the threshold bin's members has no room in shared memory (20928 members at
    128 x 65536, 33216 at 128 x 40960, 23232 at 8192 x 28672): radix steps over all channels, in blocks that have had
    several tiles of the proxy rows each."""
    _mask_is_the_exact_topk(pb, D, F, bits, group, distinct, zero)


@pytest.mark.parametrize("D,F,distinct", [(512, 1536, 0), (512, 1536, 1), (128, 65536, 1)])
def test_whole_scores_that_do_not_come_are_reported(pb, D, F, distinct):
    """Where the threshold is settled by ranking, by radix steps over the list and by radix steps over all channels: a wait for
    a whole score that runs out ends the call without y and with its status; the threshold form has no such wait, and the next
    call is ordinary."""
    g = torch.Generator(device="cuda").manual_seed(F)
    w = [torch.empty(F, D, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.04, generator=g) for _ in range(3)]
    if distinct:
        for t in w[:2]:
            t.copy_(t[torch.arange(F, device="cuda") % distinct])
    x = torch.randn(1, D, device="cuda", generator=g).to(torch.bfloat16)
    h = pb.prox_ffn_create(D, F, 1, 1, w[0], w[1], w[2].view(D, F))
    try:
        pb.prox_quantize_proxy(h, 4, 128)
        k1, k2 = D // 3, F // 3 + 1
        y, again = (torch.full((1, D), 7.0, device="cuda") for _ in range(2))
        pb.prox_debug_set_wait(h, 300, 1 << 30)
        pb.prox_ffn_forward(h, x, 1, k1, k2, y)
        status, code = pb.prox_last_device_status_raw(h)
        assert code & 4 and status == 6 and torch.all(y == 7.0)         # PROX_ERR_TIMEOUT
        pb.prox_ffn_forward_threshold(h, x, 1, 0.5, 1e-3, y)
        assert pb.prox_last_device_status(h) == 0 and not torch.any(y == 7.0)
        pb.prox_debug_set_wait(h, 0, 0)
        sel = torch.empty(1, k2, dtype=torch.int32, device="cuda")
        pb.prox_ffn_forward(h, x, 1, k1, k2, y)
        pb.prox_ffn_last_mask(h, 1, k2, sel)
        pb.prox_stage2_ffn(h, x, 1, sel, k2, again)
        # the same products, summed in fp32 in another order
        assert (y - again).norm() <= 1e-5 * again.norm()
        assert pb.prox_last_device_status(h) == 0
    finally:
        pb.prox_ffn_destroy(h)


@pytest.mark.parametrize("bits,group", [(4, 0), (4, 128), (8, 0), (8, 128)])
def test_channels_that_are_not_finite(pb, bits, group):
    """Weights that are infinite or not a number, of either sign: their channels rank by the bits of their scores (not a number
    above infinity above the rest), the other channels and the call are as ever, and the threshold form keeps them."""
    D, F, k1 = 512, 1536, 170
    wg, wu, wd, x = inputs.make_small(D, F, 1, seed=bits + group)
    for row, value in ((5, 0x7F80), (6, 0xFF80), (700, 0x7FC0), (1535, 0xFFC0), (40, 0x7F80)):      # inf, -inf, nan, -nan, inf
        wg[row, :] = value
    wu[41, 3], wu[900, :] = 0x7F80, 0xFFFF
    h_args = [dev_bf16(t) for t in (wg, wu, wd)]
    h = pb.prox_ffn_create(D, F, 1, 1, *h_args)
    try:
        pb.prox_quantize_proxy(h, bits, group)
        t_x, y, sc = dev_bf16(x), torch.empty(1, D, device="cuda"), torch.empty(F, device="cuda")
        for k2 in (1, 3, 8, F // 3, F):
            sel = torch.empty(1, k2, dtype=torch.int32, device="cuda")
            pb.prox_ffn_forward(h, t_x, 1, k1, k2, y)
            pb.prox_ffn_last_mask(h, 1, k2, sel)
            pb.prox_ffn_last_stage1(h, k1, None, sc)
            keys = sc.view(torch.int32)
            assert int(keys.min()) >= 0 and not bool(torch.isfinite(sc[[5, 6, 40, 700, 900, 1535]]).any())
            order = torch.sort(keys, descending=True, stable=True).indices
            assert torch.equal(sel[0].long(), order[:k2].sort().values), k2
            tau_x = float(t_x[0].float().abs().sort(descending=True).values[k1 - 1])
            if int((t_x[0].float().abs() >= tau_x).sum()) == k1:          # the same inputs, hence the same scores
                kept = (keys >= torch.tensor(0.01, device="cuda").view(torch.int32)).nonzero()[:, 0]
                got = torch.empty(1, kept.numel(), dtype=torch.int32, device="cuda")
                pb.prox_ffn_forward_threshold(h, t_x, 1, tau_x, 0.01, y)
                pb.prox_ffn_last_mask(h, 1, kept.numel(), got)
                assert torch.equal(got[0].long(), kept), k2
        assert pb.prox_last_device_status(h) == 0
    finally:
        pb.prox_ffn_destroy(h)


@pytest.mark.parametrize("bits", [4, 8])
def test_many_scores_that_agree_in_their_upper_halves(pb, bits):
    """Four channels repeated, with the scale of one group a bit or none at all different: thousands of scores that share their
    upper 16 bits, equal ones and different ones among them, are cut by their lower halves and then by their channels."""
    D, F, base = 1024, 16384, 4
    g = torch.Generator(device="cuda").manual_seed(bits)
    w = [torch.empty(F, D, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.03, generator=g) for _ in range(2)]
    ch = torch.arange(F, device="cuda")
    for t in w:
        t.copy_(t[ch % base])
    up, variant = w[1].view(F, D // 128, 128), (ch // base) % 9
    for v in range(8):                                              # the group's largest weight one step up
        rows = (variant == v).nonzero()[:, 0]
        at = up[rows, v].abs().argmax(dim=1)
        up.view(torch.int16)[rows, v, at] += 1
    wd = torch.empty(D, F, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.1, generator=g)
    x, k1 = torch.randn(1, D, device="cuda", generator=g).to(torch.bfloat16), 341
    h = pb.prox_ffn_create(D, F, 1, 1, *w, wd)
    try:
        pb.prox_quantize_proxy(h, bits, 128)
        y, sc = torch.empty(1, D, device="cuda"), torch.empty(F, device="cuda")
        reached = 0
        for k2 in (500, 2048, 3000, 4097, 7000, 12000, 16000):
            sel = torch.empty(1, k2, dtype=torch.int32, device="cuda")
            pb.prox_ffn_forward(h, x, 1, k1, k2, y)
            pb.prox_ffn_last_mask(h, 1, k2, sel)
            pb.prox_ffn_last_stage1(h, k1, None, sc)
            order = torch.sort(sc, descending=True, stable=True).indices[:k2]
            assert torch.equal(sel[0].long(), order.sort().values), k2
            keys = sc.view(torch.int32)
            alike = keys[(keys >> 16) == (keys[order[-1]] >> 16)]
            reached += int(alike.numel() > 256 and alike.unique().numel() > 1)
        assert reached > 0
        assert pb.prox_last_device_status(h) == 0
    finally:
        pb.prox_ffn_destroy(h)


@pytest.mark.parametrize("F,B", [(1536, 8), (1600, 5), (14336, 8), (19136, 1)])
def test_sixteen_bit_scores_on_a_new_handle(pb, F, B):
    """The split-K tickets of 16-bit proxies (strips of 128 channels, the most per token) all start at zero, whatever the memory
    of a new handle held before."""
    D, k1, k2 = 512, 256, F // 3
    for words in (64, 128, 256, 1024, 4096):                        # pieces of memory that come back from the driver full of ones
        held = [torch.full((words,), -1, dtype=torch.int32, device="cuda") for _ in range(64)]
        del held
    torch.cuda.empty_cache()
    p = Problem(pb, *inputs.make_small(D, F, B, seed=F), max_batch=B)
    try:
        p.quantize(16, 0)
        sel, sc = torch.empty(B, k2, dtype=torch.int32, device="cuda"), torch.empty(B, F, device="cuda")
        for again in range(2):
            pb.prox_stage1_mask(p.h, p.t_x, B, k1, k2, sel, sc)
            for b in range(B):
                _, score, _, thr = p.oracle_stage1(b, k1, k2)
                assert float(np.max(np.abs(sc[b].cpu().numpy() - score)) / thr) < 2e-4, (again, b)      # as everywhere for scores
        assert pb.prox_last_device_status(p.h) == 0
    finally:
        p.close()


@pytest.mark.parametrize("zero", [False, True])
@pytest.mark.parametrize("D,F,bits,group,distinct", [(4096, 12288, 4, 128, 2), (4096, 14336, 8, 0, 1), (8192, 16384, 4, 0, 1)])
def test_threshold_bin_listed_over_the_ring(pb, D, F, bits, group, distinct, zero):
    """The list of the threshold bin's members (more than d_model / 2 of them) lies over slots of the ring that the first weight rows
    would go to: no row may get there before the list has been read."""
    _mask_is_the_exact_topk(pb, D, F, bits, group, distinct, zero)


@pytest.mark.parametrize("bits,distinct", [(4, 0), (8, 3)])
def test_half_scores_that_do_not_fit(pb, bits, distinct):
    """65536 half scores beside a d_model of 12288: no room in shared memory, the blocks read them where the others put them."""
    _mask_is_the_exact_topk(pb, 12288, 65536, bits, 0, distinct, False)
