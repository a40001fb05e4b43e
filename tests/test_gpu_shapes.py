"""Sizes at the edges of the kernels' tiles and dispatch rules, against the oracle or an fp64 restatement of the op."""
import numpy as np
import pytest

from paper_2405_10951_b200 import synth
from paper_2405_10951_b200.synth import Config

import parity as P

pytestmark = pytest.mark.gpu

MINI = Config("mini_shapes", 64, 8, 128, 2, 6, 256, (10,), 6, (3, 4, 5), (1, 3, 4), 7, 10, dtype="bf16", seed=1)


@pytest.mark.parametrize("batch", [1, 3, 5, 7])
def test_bf16_step_with_odd_row_counts(batch):
    """Weight gradients reduce over batch x tokens rows, which no tile divides here; same tolerance as every bf16 step."""
    cfg = MINI.with_(batch=batch, trainable=(1, 3, 5))
    images, labels, task_ids, params = synth.make_workload(cfg, peaked=False)
    gpu = P.run_gpu_step(cfg, images, labels, task_ids, params)
    P.compare_step(cfg, images, labels, task_ids, params, gpu, P.BF16_TOL, P.BF16_EXACT_MARGIN, P.BF16_SCORE_TOL)


@pytest.mark.parametrize("with_score_grad", [False, True])
@pytest.mark.parametrize("B,T,H", [(1, 257, 1), (2, 290, 3), (1, 384, 2), (1, 385, 1), (2, 577, 2), (1, 1025, 1)])
def test_attention_backward_beyond_256_tokens(B, T, H, with_score_grad):
    """dQ, dK, dV of the kernel pair that walks the other side in blocks of 64, last blocks of 1 to 64 columns and last
    row tiles of 1 to 128 rows; same bf16 inputs and tolerance as the shorter kernels."""
    import ctypes as C

    import torch
    from oracle import bsr_oracle as O
    from paper_2405_10951_b200 import binding as Bd
    d = 64
    rng = np.random.default_rng(T * 7 + B)
    qkv = synth.round_to_bf16(rng.standard_normal((B, T, 3, H, d)))
    do = synth.round_to_bf16(rng.standard_normal((B, T, H * d)))
    sg = rng.standard_normal((B, T - 1)) * 3.0 if with_score_grad else None
    q, k, v = (qkv[:, :, i].transpose(0, 2, 1, 3) for i in range(3))

    class Cfg:
        heads = H
        dim = H * d
    _, A = O.attention_fwd(Cfg, q, k, v)
    dA_cls = None
    if sg is not None:
        dA_cls = np.zeros((B, T))
        dA_cls[:, 1:] = sg / H
    want = np.stack(O.attention_bwd(Cfg, A, q, k, v, do.reshape(B, T, H, d).transpose(0, 2, 1, 3), dA_cls), axis=0).transpose(1, 3, 0, 2, 4)
    dev = torch.as_tensor(qkv.astype(np.float32)).cuda().bfloat16()
    dod = torch.as_tensor(do.astype(np.float32)).cuda().bfloat16()
    sgd = None if sg is None else torch.as_tensor(sg.astype(np.float32)).cuda()
    _, _, lse = Bd.bsr_attention_forward(dev, H, use_tensor_cores=True, want_lse=True)
    out, delta = torch.empty_like(dev), torch.empty(B * H * T, device="cuda")
    p = lambda t: None if t is None else C.c_void_p(t.data_ptr())
    rc = Bd.lib().bsr_attention_backward(p(dev), p(dod), p(lse), p(sgd), Bd.DTYPE_BF16, B, T, H, d, p(out), p(delta), 1,
                                         C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == Bd.BSR_OK
    torch.cuda.synchronize()
    got = out.float().cpu().numpy().astype(np.float64)
    for i, name in enumerate(("dq", "dk", "dv")):
        assert P.rel_err(got[:, :, i], want[:, :, i]) < 8e-3, name


@pytest.mark.parametrize("shift", [0, 1, 8])
def test_eval_replay_equals_launch_by_launch(shift):
    """Inference replayed from its graph (third call on: new input and output buffers every time) against the same calls
    enqueued kernel by kernel; `shift` moves the images off a 16-byte boundary, where they are read directly."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    cfg = MINI
    eng = Bd.Engine(cfg)
    _, _, _, params = synth.make_workload(cfg, peaked=True)
    eng.set_params(params)
    n = 4 * cfg.in_chans * cfg.image_size ** 2
    for stream in (torch.cuda.Stream(), torch.cuda.default_stream()):
        with torch.cuda.stream(stream):
            store = torch.randn(5, n + 64, device="cuda").bfloat16()
            inputs = [s[shift: shift + n].view(4, cfg.in_chans, cfg.image_size, cfg.image_size) for s in store]
            runs = []
            for graphs in (False, True):
                eng.set_graph_mode(graphs)
                runs.append([eng.eval_forward(x) for x in inputs])
            eng.sync_status()
            for (l0, k0), (l1, k1) in zip(*runs):
                assert torch.equal(l0, l1) and all(torch.equal(a, b) for a, b in zip(k0, k1))
            assert not torch.equal(runs[0][0][0], runs[0][1][0])
    eng.close()


@pytest.mark.parametrize("dtype,tol", [("fp32", 2e-6), ("bf16", 4e-3)])
@pytest.mark.parametrize("m,n,k", [(1, 8, 8), (64, 64, 64), (65, 60, 63), (520, 192, 768), (33, 30, 1030), (2080, 576, 40)])
def test_fma_contraction_forward_and_backward(m, n, k, dtype, tol):
    """The FP32-FMA contraction at tile remainders and at one to eight splits of the reduction over a cluster, all three operand
    orders: y = x W^T, dx = dy W, dW = dy^T x.  Tolerance: fp32 sums of up to 2080 products, or one bf16 rounding."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    rng = np.random.default_rng(m + n + k)
    mk = lambda *s: synth.round_to_bf16(rng.standard_normal(s)) if dtype == "bf16" else rng.standard_normal(s).astype(np.float32).astype(np.float64)
    x, w, dy = mk(m, k), mk(n, k), mk(m, n)
    dev = lambda a: torch.as_tensor(a.astype(np.float32)).cuda().to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    y = Bd.bsr_linear_forward(dev(x), dev(w))
    dx, dw = Bd.bsr_linear_backward(dev(x), dev(w), dev(dy))
    torch.cuda.synchronize()
    for got, want in ((y, x @ w.T), (dx, dy @ w), (dw, dy.T @ x)):
        assert P.rel_err(got.float().cpu().numpy(), want) < tol


@pytest.mark.parametrize("m,n,k", [(129, 64, 64), (256, 256, 64), (300, 200, 72), (19200, 768, 128), (18944, 2304, 64), (12001, 2048, 192), (12800, 2056, 64)])
def test_linear_on_cta_pairs(m, n, k):
    """The CTA-pair kernel at remainders of its 256-row tiles and with a last wave cut into parts of 64 to 256 columns: forward with
    bias, GELU and residual; the gradients, which CTA pairs do not take, as with single CTAs.  One bf16 rounding of the output."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    gen = torch.Generator(device="cuda").manual_seed(m + n + k)
    mk = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    x, w, dy, res, bias = mk(m, k), mk(n, k) / k ** 0.5, mk(m, n), mk(m, n), torch.randn(n, generator=gen, device="cuda")
    rel = lambda a, b: float((a.double() - b).norm() / b.norm())
    z = x.double() @ w.double().T + bias.double()
    assert rel(Bd.bsr_linear_forward(x, w, bias, use_tensor_cores=2), z) < 4e-3
    want = torch.nn.functional.gelu(z) + res.double()
    assert rel(Bd.bsr_linear_forward(x, w, bias, res, act_gelu=True, use_tensor_cores=2), want) < 4e-3
    if m % 8 == 0:
        dx, dw = Bd.bsr_linear_backward(x, w, dy, use_tensor_cores=2)
        assert rel(dx, dy.double() @ w.double()) < 4e-3 and rel(dw, dy.double().T @ x.double()) < 1e-4


@pytest.mark.parametrize("m,n,k", [(1, 64, 64), (130, 1152, 384), (200, 72, 200), (1576, 1152, 384), (1576, 384, 1544), (6304, 384, 384), (4096, 1536, 64), (2500, 3072, 128)])
def test_linear_over_tile_widths(m, n, k):
    """Sizes that take tiles of 64, 128, 192 and 256 columns, and weight gradients with one to sixteen shares of the reduction: the
    residual path and the input and weight gradients.  One bf16 rounding of the output, fp32 sums for the weight gradient."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    gen = torch.Generator(device="cuda").manual_seed(m + n + k)
    mk = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    x, w, dy, res, bias = mk(m, k), mk(n, k) / k ** 0.5, mk(m, n), mk(m, n), torch.randn(n, generator=gen, device="cuda")
    rel = lambda a, b: float((a.double() - b).norm() / b.norm())
    want = x.double() @ w.double().T + bias.double()
    assert rel(Bd.bsr_linear_forward(x, w, bias, res, use_tensor_cores=True), want + res.double()) < 4e-3
    if m % 8 == 0:
        ws = torch.empty(160 * 128 * 256, device="cuda")
        dx, dw = Bd.bsr_linear_backward(x, w, dy, use_tensor_cores=True, workspace=ws)
        assert rel(dx, dy.double() @ w.double()) < 4e-3 and rel(dw, dy.double().T @ x.double()) < 1e-4


@pytest.mark.parametrize("B,T,H", [(1, 257, 2), (2, 319, 1), (1, 320, 3), (1, 321, 1), (5, 577, 12), (1, 4096, 1)])
def test_long_attention_forward_at_block_edges(B, T, H):
    """Output, log-sum-exp and classification row of the single-walk kernel with last key blocks of 1, 63 and 64 keys, last query
    tiles of 1 to 128 rows and the longest sequence it takes; several CTAs per SM.  bf16 rounding of P and of the output."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    gen = torch.Generator(device="cuda").manual_seed(T + B)
    qkv = torch.randn(B, T, 3, H, 64, generator=gen, device="cuda").bfloat16()
    out, cp, lse = Bd.bsr_attention_forward(qkv, H, use_tensor_cores=True, want_lse=True)
    q, k, v = (qkv[:, :, i].transpose(1, 2).double() for i in range(3))
    s = q @ k.transpose(-1, -2) / 8.0
    rel = lambda a, b: float((a.double() - b).norm() / b.norm())
    assert rel(out, (s.softmax(-1) @ v).transpose(1, 2).reshape(B, T, H * 64)) < 6e-3
    assert rel(lse, s.logsumexp(-1)) < 1e-5
    assert rel(cp, s.softmax(-1)[:, :, 0, 1:]) < 2e-5


@pytest.mark.parametrize("optimizer", ["adamw", "sgd"])
@pytest.mark.parametrize("trainable", [(0, 5), (2, 4), (5,)])
def test_updates_beside_the_backward_pass(trainable, optimizer):
    """Blocks updated while the backward pass goes on (frozen blocks between them, a head of 7 classes whose bias is no
    multiple of four) equal one update after it bit for bit: every parameter, over a direct and two replayed steps."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    cfg = MINI.with_(trainable=trainable, optimizer=optimizer, num_classes=(7,))
    images, labels, task_ids, params = synth.make_workload(cfg, peaked=False)
    whole, split = Bd.Engine(cfg), Bd.Engine(cfg)
    with torch.cuda.stream(torch.cuda.Stream()):
        for e in (whole, split):
            e.set_params(params)
        img, lab = whole.images_to_device(images), torch.as_tensor(labels).cuda()
        for _ in range(3):
            whole.train_step(img, lab)
            split.forward_backward(img, lab)
            split.optimizer_step()
        whole.sync_status()
        split.sync_status()
        for n, shape in synth.param_shapes(cfg).items():
            assert torch.equal(whole.get_tensor(n, shape), split.get_tensor(n, shape)), n
    whole.close()
    split.close()


@pytest.mark.parametrize("experts,top_k,batch,classes", [(32, 4, 7, (10,)), (32, 1, 5, (10, 6)), (8, 3, 9, (10,)), (1, 1, 8, (5,) * 4)])
def test_expert_routing_and_row_sums_at_their_limits(experts, top_k, batch, classes):
    """One expert and the most, one slot and the most, token counts no multiple of a counting group, experts with fewer
    rows than a cluster has row lanes and one with all of them; tolerance of every bf16 step."""
    cfg = Config("mini_moe_shapes", 64, 8, 128, 2, 4, 256, classes, batch, (1, 2, 3), (1,), 7, 10, dtype="bf16", seed=4,
                 moe_experts=experts, moe_top_k=top_k, moe_blocks=(0, 2))
    images, labels, task_ids, params = synth.make_workload(cfg, peaked=False)
    gpu = P.run_gpu_step(cfg, images, labels, task_ids, params)
    P.compare_step(cfg, images, labels, task_ids, params, gpu, P.BF16_TOL, P.BF16_EXACT_MARGIN, P.BF16_SCORE_TOL)


@pytest.mark.parametrize("m,n,k", [(1, 768, 768), (7, 1152, 1152), (127, 776, 776), (129, 1160, 3080), (200, 768, 1600), (600, 1152, 3072), (1000, 1160, 1216)])
def test_linear_split_over_clusters(m, n, k):
    """Few-tile products whose reduction is split over 2, 4 and 8 CTAs: rows and columns past the last tile, shares of rows that do
    not divide a tile, reductions that are no multiple of a slab; forward with bias, GELU and residual, and the input gradient."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    gen = torch.Generator(device="cuda").manual_seed(m + n + k)
    mk = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    x, w, dy, res, bias = mk(m, k), mk(n, k) / k ** 0.5, mk(m, n), mk(m, n), torch.randn(n, generator=gen, device="cuda")
    rel = lambda a, b: float((a.double() - b).norm() / b.norm())
    z = x.double() @ w.double().T + bias.double()
    assert rel(Bd.bsr_linear_forward(x, w, bias, use_tensor_cores=True), z) < 4e-3
    want = torch.nn.functional.gelu(z) + res.double()
    assert rel(Bd.bsr_linear_forward(x, w, bias, res, act_gelu=True, use_tensor_cores=True), want) < 4e-3
    if m % 8 == 0:
        dx, _ = Bd.bsr_linear_backward(x, w, dy, use_tensor_cores=True)
        assert rel(dx, dy.double() @ w.double()) < 4e-3


@pytest.mark.parametrize("scale,with_score_grad", [(0.3, True), (1.0, False), (2.0, True)])
@pytest.mark.parametrize("B,T,H", [(2, 290, 3), (2, 577, 6)])
def test_long_attention_backward_is_as_exact_as_fp32_probabilities(B, T, H, scale, with_score_grad):
    """dQ, dK and dV beyond 256 tokens against 64 bits, beside the FP32-FMA kernels on the same inputs.  P and dS enter the products
    with 16 bits of mantissa (2^-17 lost), which adds (2^-17 / 1.66e-3)^2 / 2 = 1e-5 of itself to the error that the rounding of
    the outputs leaves; 1 % covers scores and sums in another order.  P and dS rounded to bf16 once give 1.4 times that error."""
    import ctypes as C

    import torch
    from paper_2405_10951_b200 import binding as Bd
    gen = torch.Generator(device="cuda").manual_seed(T + B)
    qkv = (torch.randn(B, T, 3, H, 64, generator=gen, device="cuda") * scale).bfloat16()
    do = torch.randn(B, T, H * 64, generator=gen, device="cuda").bfloat16()
    sg = 3.0 * torch.randn(B, T - 1, generator=gen, device="cuda") if with_score_grad else None
    q, k, v = (qkv[:, :, i].transpose(1, 2).double() for i in range(3))
    s = q @ k.transpose(-1, -2) / 8.0
    lse = s.logsumexp(-1)
    prob, dov = (s - lse.unsqueeze(-1)).exp(), do.double().view(B, T, H, 64).transpose(1, 2)
    dp = dov @ v.transpose(-1, -2)
    if sg is not None:
        dp[:, :, 0, 1:] += sg.double().unsqueeze(1) / H
    ds = prob * (dp - (prob * dp).sum(-1, keepdim=True)) / 8.0
    want = (ds @ k, ds.transpose(-1, -2) @ q, prob.transpose(-1, -2) @ dov)
    lse32, delta, p = lse.float().contiguous(), torch.empty(B * H * T, device="cuda"), lambda t: None if t is None else C.c_void_p(t.data_ptr())
    err = []
    for mode in (0, 1):
        out = torch.empty_like(qkv)
        assert Bd.lib().bsr_attention_backward(p(qkv), p(do), p(lse32), p(sg), Bd.DTYPE_BF16, B, T, H, 64, p(out), p(delta), mode,
                                               C.c_void_p(torch.cuda.current_stream().cuda_stream)) == Bd.BSR_OK
        torch.cuda.synchronize()
        got = out.permute(2, 0, 3, 1, 4).double()
        err.append([float((got[i] - w).norm() / w.norm()) for i, w in enumerate(want)])
    for name, fma, tensor in zip(("dq", "dk", "dv"), *err):
        assert tensor <= 1.01 * fma, (name, fma, tensor)


@pytest.mark.parametrize("m,n,k", [(1, 3072, 768), (7, 1536, 768), (128, 3072, 768), (200, 5000, 520), (256, 384, 1536)])
@pytest.mark.parametrize("bias", [0.0, -3.0, -3.8])
def test_gelu_of_few_row_products_is_exact(m, n, k, bias):
    """GELU where products of few rows and a long reduction apply it, down to the tail where a polynomial for Phi fails: nothing but
    the rounding of the outputs, at most 2^-9 of each (and fp32 sums, a hundredth of that)."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    gen = torch.Generator(device="cuda").manual_seed(m + n)
    x = torch.randn(m, k, generator=gen, device="cuda").bfloat16()
    w = (0.02 * torch.randn(n, k, generator=gen, device="cuda")).bfloat16()
    b = torch.full((n,), bias, device="cuda")
    z = x.double() @ w.double().T + b.double()
    want = 0.5 * z * torch.special.erfc(-z / 2 ** 0.5)
    got = Bd.bsr_linear_forward(x, w, b, act_gelu=True, use_tensor_cores=True).double()
    assert float((got - want).norm() / want.norm()) < 1.01 * 2 ** -9


def test_attention_backward_of_more_pairs_than_a_grid_dimension():
    """Up to 256 tokens the tensor-core kernels take any number of (image, head) pairs: 65544 of them, bit for bit as in small batches."""
    import ctypes as C

    import torch
    from paper_2405_10951_b200 import binding as Bd
    B, T, H = 5462, 5, 12
    gen = torch.Generator(device="cuda").manual_seed(3)
    qkv = torch.randn(B, T, 3, H, 64, generator=gen, device="cuda").bfloat16()
    do = torch.randn(B, T, H * 64, generator=gen, device="cuda").bfloat16()
    _, _, lse = Bd.bsr_attention_forward(qkv, H, use_tensor_cores=True, want_lse=True)
    p = lambda t: C.c_void_p(t.data_ptr())

    def backward(a, b):
        out = torch.empty_like(qkv[a:b])
        rc = Bd.lib().bsr_attention_backward(p(qkv[a:b]), p(do[a:b]), p(lse[a:b]), None, Bd.DTYPE_BF16, b - a, T, H, 64, p(out), None, 1,
                                             C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == Bd.BSR_OK
        return out
    whole = backward(0, B)
    assert torch.equal(whole[:7], backward(0, 7)) and torch.equal(whole[-7:], backward(B - 7, B))


def test_more_keys_than_graphs_capture_no_more_than_the_cache_holds():
    """Ten sets of step buffers and ten batch sizes of inference in turn: eight graphs of each kind, the rest enqueued, results as
    without graphs.  A batch size that stays alone long enough then takes the place of an idle one."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    cfg = MINI.with_(optimizer="sgd", lr=0.0, weight_decay=0.0)
    images, labels, _, params = synth.make_workload(cfg, peaked=True)
    eng = Bd.Engine(cfg, max_batch=12)
    eng.set_params(params)
    with torch.cuda.stream(torch.cuda.Stream()):
        img, lab = eng.images_to_device(images), torch.as_tensor(labels).cuda()
        loss, bufs = torch.zeros(1, device="cuda"), [torch.roll(img, i, 0).clone() for i in range(10)]
        evals = [torch.randn(b, *img.shape[1:], device="cuda").to(img.dtype) for b in range(1, 11)]
        runs = []
        for graphs in (False, True):
            eng.set_graph_mode(graphs)
            for _ in range(4):
                got = [eng.train_step(b, lab, out=(loss, None))[0].clone() for b in bufs] + [eng.eval_forward(x, want_kept=False)[0] for x in evals]
            runs.append(got)
        assert all(torch.equal(a, b) for a, b in zip(*runs))
        assert eng.profile_read()["graph_captures"] == 16
        for _ in range(300):
            eng.eval_forward(evals[9], want_kept=False)
        eng.sync_status()
        assert eng.profile_read()["graph_captures"] == 17
    eng.close()


def test_a_step_refused_half_way_leaves_nothing_in_flight():
    """730 tokens fit the attention backward on the tensor cores but not the one on FMAs, which refuses while reductions and weight
    gradients of the block above are on their lanes, here inside a capture.  The next step equals that of a new handle."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    cfg = Config("mini_730", 432, 16, 128, 2, 3, 256, (10,), 1, (0, 1, 2), (), 1, 1, dtype="bf16", seed=2)
    images, labels, _, params = synth.make_workload(cfg, peaked=False)
    shapes = synth.param_shapes(cfg)
    got = []
    with torch.cuda.stream(torch.cuda.Stream()):
        for refused in (True, False):
            eng = Bd.Engine(cfg)
            eng.set_params(params)
            img, lab = eng.images_to_device(images), torch.as_tensor(labels).cuda()
            if refused:
                eng.set_gemm_mode(0)
                for _ in range(2):
                    with pytest.raises(Bd.BsrError) as e:
                        eng.train_steps(img.expand(3, *img.shape).contiguous(), lab.expand(3, -1).contiguous(), total_steps=3)
                    assert e.value.status == -2          # BSR_ERR_UNSUPPORTED
                eng.set_gemm_mode(1)
            loss = eng.train_step(img, lab)[0]
            eng.sync_status()
            got.append([loss.clone()] + [eng.get_tensor("grad/" + n, shapes[n]) for n in shapes if n.startswith(("blocks", "head"))])
            eng.close()
    assert all(torch.equal(a, b) for a, b in zip(*got))


@pytest.mark.parametrize("mean", [0.0, 1.0])
@pytest.mark.parametrize("m,n,k", [(64, 72, 384), (200, 384, 1536), (328, 200, 256), (1024, 128, 256), (1032, 1152, 384), (4040, 768, 3072), (25216, 320, 768)])
def test_weight_gradients_are_summed_to_fp32(m, n, k, mean):
    """Reductions of one slab to hundreds, around the lines between 1, 2, 4 and 8 slabs a sum, split and unsplit.  An accumulator loses
    at most a unit of its last place (2^-23 of it, half of that on average) with each of its additions, four a slab.  The sums
    of the sums are rounded: 2^-24 each, of up to a hundred in random order.  One accumulator over 25216 rows: 1.4e-5."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    gen = torch.Generator(device="cuda").manual_seed(m + n)
    mk = lambda *s: (torch.randn(*s, generator=gen, device="cuda") + mean).bfloat16()
    x, w, dy = mk(m, k), mk(n, k), mk(m, n)
    want = dy.double().T @ x.double()
    additions = 4 if m <= 320 else 8 if m <= 1024 else 16 if m <= 4096 else 32
    for ws in (None, torch.empty(160 * 128 * 256, device="cuda")):
        _, dw = Bd.bsr_linear_backward(x, w, dy, use_tensor_cores=True, workspace=ws)
        assert float((dw.double() - want).norm() / want.norm()) < (additions + 10) * 2 ** -24


@pytest.mark.parametrize("drop", [(), (2,)])
@pytest.mark.parametrize("classes,dim,batch", [((1,), 64, 2), ((16, 31, 33), 64, 7), ((32, 100), 1024, 33), ((9000,), 128, 3), ((10,), 8, 1)])
def test_head_over_numbers_of_classes(classes, dim, batch, drop):
    """One, two, four and eight CTAs an image, slices beyond shared memory, several tasks, narrow and wide rows; with a drop location in the
    last block the head reads one row of many."""
    cfg = Config("mini_head", 16, 4, dim, max(1, dim // 64), 3, 2 * dim, classes, batch, (1, 2), drop, 1, 2, dtype="fp32", seed=len(classes))
    images, labels, task_ids, params = synth.make_workload(cfg, peaked=dim >= 64)
    gpu = P.run_gpu_step(cfg, images, labels, task_ids, params)
    P.compare_step(cfg, images, labels, task_ids, params, gpu, P.FP32_TOL, P.EXACT_MARGIN, P.FP32_TOL)


@pytest.mark.parametrize("dtype,grid,keep,fuse,dim,heads,batch", [
    ("fp32", 16, (1, 2), 1, 64, 4, 3), ("fp32", 17, (3, 10), 2, 192, 3, 1), ("fp32", 25, (7, 10), 0, 64, 4, 2), ("fp32", 26, (1, 100), 1, 128, 8, 1),
    ("fp32", 31, (99, 100), 2, 64, 4, 1), ("fp32", 32, (1, 2), 1, 64, 4, 1), ("fp32", 3, (1, 3), 1, 1024, 16, 9),
    ("bf16", 16, (1, 2), 2, 128, 2, 3), ("bf16", 26, (7, 10), 1, 64, 1, 2)])
def test_selection_compaction_and_layernorm_in_one_launch(dtype, grid, keep, fuse, dim, heads, batch):
    """Register counts of the selection (256, 640 tokens) and the longest row it takes (1023; 1024 go the general way), one kept
    token, few dropped ones, no fused token, rows of 64 to 1024 columns; a frozen and a trainable drop location."""
    cfg = Config("mini_select", 4 * grid, 4, dim, heads, 3, 2 * dim, (10,), batch, (1, 2), (0, 1), keep[0], keep[1], dtype=dtype, fuse_mode=fuse, seed=grid)
    images, labels, task_ids, params = synth.make_workload(cfg, peaked=dtype == "fp32")
    gpu = P.run_gpu_step(cfg, images, labels, task_ids, params)
    if dtype == "fp32":
        P.compare_step(cfg, images, labels, task_ids, params, gpu, P.FP32_TOL, P.EXACT_MARGIN, P.FP32_TOL)
    else:
        P.compare_step(cfg, images, labels, task_ids, params, gpu, P.BF16_TOL, P.BF16_EXACT_MARGIN, P.BF16_SCORE_TOL)


@pytest.mark.parametrize("T", [1, 5, 16, 33, 64, 65, 128, 129, 160, 161, 192, 193, 224, 256])
def test_attention_forward_of_an_image_does_not_depend_on_the_batch(T):
    """One image's tiles fit the SMs at once, those of 300 images do not: two kernels, the same bits, whichever turn of its CTA an image is."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    g = torch.Generator(device="cuda").manual_seed(T)
    qkv = torch.randn(300, T, 3, 2, 64, generator=g, device="cuda").bfloat16()
    many = Bd.bsr_attention_forward(qkv, 2, use_tensor_cores=True, want_lse=True)
    assert len(many) == 3                                            # output, classification row, log-sum-exp
    for i in (299, 150, 77, 1, 0):
        one = Bd.bsr_attention_forward(qkv[i: i + 1].contiguous(), 2, use_tensor_cores=True, want_lse=True)
        for a, b in zip(one, many):
            assert torch.equal(a, b[i: i + 1])
    o = torch.nn.functional.scaled_dot_product_attention(*qkv[:1].double().permute(2, 0, 3, 1, 4)).transpose(1, 2).reshape(1, T, 128)
    # P and the output are rounded to bf16 (2^-9 each), the rest is 32-bit
    assert float((one[0].double() - o).norm() / o.norm()) < 6e-3


@pytest.mark.parametrize("m,n,k", [(1, 4, 4), (31, 36, 60), (32, 32, 64), (33, 68, 260), (100, 192, 516), (7, 200, 2052), (9000, 512, 512)])
def test_fp32_products_in_small_tiles(m, n, k):
    """Edges of the 32 x 32 tiles and 64-deep slabs, one to eight parts of k, and the number of tiles beyond which tiles of 64 take over; sums of at
    most a few hundred fp32 additions in a row keep a relative error below 2e-6."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    g = torch.Generator(device="cuda").manual_seed(m + n + k)
    x, w, dy = (torch.randn(s, generator=g, device="cuda") for s in ((m, k), (n, k), (m, n)))
    bias, res = torch.randn(n, generator=g, device="cuda"), torch.randn(m, n, generator=g, device="cuda")
    rel = lambda a, b: float((a.double() - b).norm() / b.norm())
    z = x.double() @ w.double().T + bias.double()
    assert rel(Bd.bsr_linear_forward(x, w, bias, res), z + res.double()) < 2e-6
    assert rel(Bd.bsr_linear_forward(x, w, bias, act_gelu=True), torch.nn.functional.gelu(z)) < 2e-6
    dx, dw = Bd.bsr_linear_backward(x, w, dy)
    assert rel(dx, dy.double() @ w.double()) < 2e-6 and rel(dw, dy.double().T @ x.double()) < 2e-6


@pytest.mark.parametrize("H", [1, 3])
@pytest.mark.parametrize("with_score_grad", [False, True])
@pytest.mark.parametrize("T", [129, 143, 144, 145, 160, 192, 193, 255, 256])
def test_attention_backward_of_few_and_of_many_pairs(T, with_score_grad, H):
    """Two CTAs a pair, as long as all fit the SMs, against one: the same sums, parts of delta and dQ added up in another order in 32 bits, so
    that after rounding to bf16 values differ by a unit of their last place at most now and then."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    g = torch.Generator(device="cuda").manual_seed(T)
    qkv, do = torch.randn(80, T, 3, H, 64, generator=g, device="cuda").bfloat16(), torch.randn(80, T, H * 64, generator=g, device="cuda").bfloat16()
    sg = torch.randn(80, T - 1, generator=g, device="cuda") if with_score_grad else None
    _, _, lse = Bd.bsr_attention_forward(qkv, H, use_tensor_cores=True, want_lse=True)
    many = Bd.bsr_attention_backward(qkv, do, lse, sg, use_tensor_cores=True).float()
    for part in (slice(0, 3), slice(77, 80)):
        few = Bd.bsr_attention_backward(qkv[part].contiguous(), do[part].contiguous(), lse[part].contiguous(), None if sg is None else sg[part].contiguous(),
                                        use_tensor_cores=True).float()
        assert float((few - many[part]).norm() / many[part].norm()) < 1e-3


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_drop_location_that_keeps_all_but_one_token_fuses_it(dtype):
    """Nine patches, one kept and one fused; two tokens, one of them kept: the sequence keeps its length, but its last token is the fused one."""
    cfg = Config("mini_last_token", 12, 4, 128, 2, 3, 256, (10,), 5, (1, 2), (0, 1), 1, 9, dtype=dtype, seed=2)
    images, labels, task_ids, params = synth.make_workload(cfg, peaked=dtype == "fp32")
    gpu = P.run_gpu_step(cfg, images, labels, task_ids, params)
    tol = P.FP32_TOL if dtype == "fp32" else P.BF16_TOL
    P.compare_step(cfg, images, labels, task_ids, params, gpu, tol, P.EXACT_MARGIN if dtype == "fp32" else P.BF16_EXACT_MARGIN,
                   P.FP32_TOL if dtype == "fp32" else P.BF16_SCORE_TOL)


@pytest.mark.parametrize("n,k,rows", [(1536, 384, 4000), (192, 768, 13000), (768, 260, 3000), (4, 8, 2097121 + 40)])
def test_fp32_rows_do_not_depend_on_how_many_others_there_are(n, k, rows):
    """Small and wide tiles, and more rows than a grid of small ones has: one sum for an output, bit for bit."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    g = torch.Generator(device="cuda").manual_seed(n)
    x, w, bias = (torch.randn(s, generator=g, device="cuda") for s in ((rows, k), (n, k), (n,)))
    for gelu in (False, True):
        many = Bd.bsr_linear_forward(x, w, bias, act_gelu=gelu)
        for m in (1, 33, 65, 520, 788, 1576):
            assert torch.equal(Bd.bsr_linear_forward(x[:m], w, bias, act_gelu=gelu), many[:m])
            assert torch.equal(Bd.bsr_linear_forward(x[-m:], w, bias, act_gelu=gelu), many[-m:])


@pytest.mark.parametrize("grid,fuse", [(8, 0), (8, 1), (8, 2), (17, 1), (17, 2)])
def test_fp32_logits_of_an_image_do_not_depend_on_its_batch(grid, fuse):
    """64 and 289 patches, drop locations in one launch and in three, products in small and in wide tiles."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    cfg = Config("mini_alone", 4 * grid, 4, 384, 6, 3, 1536, (10,), 50, (2,), (0, 1), 1, 2, dtype="fp32", fuse_mode=fuse, seed=grid)
    images, _, _, params = synth.make_workload(cfg, peaked=True)
    eng = Bd.Engine(cfg)
    eng.set_params(params)
    img = eng.images_to_device(images)
    many, kept = eng.eval_forward(img)
    for part in (slice(0, 1), slice(49, 50), slice(0, 9), slice(0, 32), slice(17, 50), slice(1, 50)):
        logits, k = eng.eval_forward(img[part].contiguous())
        assert torch.equal(logits, many[part])
        assert all(torch.equal(a, b[part]) for a, b in zip(k, kept))
    eng.sync_status()
    eng.close()


def test_head_of_more_classes_than_a_grid_has_rows_of_sixteen():
    """1048560 classes and more are beyond 65535 groups of 16: loss, logits and the gradients of the head against 64 bits."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    n = 16 * 65535 + 21
    cfg = Config("mini_million", 8, 4, 8, 1, 1, 16, (n,), 2, (), (), 1, 2, dtype="fp32")
    g = torch.Generator(device="cuda").manual_seed(5)
    eng = Bd.Engine(cfg)
    params = {}
    for name, shape in synth.param_shapes(cfg).items():
        params[name] = torch.randn(shape, generator=g, device="cuda") * (0.02 if "norm" not in name else 1.0)
        eng.set_param(name, params[name])
    images = torch.randn(2, 3, 8, 8, generator=g, device="cuda")
    labels = torch.tensor([3, n - 1], dtype=torch.int32, device="cuda")
    loss = eng.forward_backward(images, labels, want_kept=False)[0]
    logits = eng.get_tensor("logits", (2, n)).double()
    dw, db, dbeta = (eng.get_tensor("grad/" + name, params[name].shape).double() for name in ("head.0.weight", "head.0.bias", "norm.bias"))
    eng.sync_status()
    assert torch.equal(eng.eval_forward(images, want_kept=False)[0].double(), logits)
    eng.close()
    w = params["head.0.weight"].double()
    xn = torch.linalg.solve(w.T @ w, w.T @ (logits - params["head.0.bias"].double()).T).T        # the normalised rows, from a million logits
    rel = lambda a, b: float((a - b).norm() / b.norm())
    assert rel(xn @ w.T + params["head.0.bias"].double(), logits) < 1e-6
    want = torch.nn.functional.cross_entropy(logits, labels.long())
    d = torch.softmax(logits, 1)
    d[torch.arange(2), labels.long()] -= 1
    d /= 2
    # sums of eight products and of a million terms in at most a few thousand fp32 additions in a row
    assert abs(float(loss[0]) - float(want)) < 1e-5 * float(want)
    assert rel(db, d.sum(0)) < 1e-5 and rel(dw, d.T @ xn) < 1e-5 and rel(dbeta, (d @ w).sum(0)) < 1e-4


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("classes", [(127,), (128,), (1000, 40), (9001,), (21841,)])
def test_logits_of_inference_are_those_of_training(classes, dtype):
    """Inference spreads an image's classes over more CTAs than a cluster has, as far as the SMs have room; the sums stay the same."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    cfg = Config("mini_many_classes", 16, 4, 64, 1, 2, 128, classes, 70, (1,), (0,), 1, 2, dtype=dtype, seed=3)
    images, labels, task_ids, params = synth.make_workload(cfg, peaked=False)
    eng = Bd.Engine(cfg)
    eng.set_params(params)
    img, lab = eng.images_to_device(images), torch.as_tensor(labels.astype(np.int32)).cuda()
    tid = torch.as_tensor(task_ids.astype(np.int32)).cuda() if len(classes) > 1 else None
    for B in (1, 7, 18, 70):
        part = lambda t: None if t is None else t[:B].contiguous()
        eng.forward_backward(part(img), part(lab), part(tid))
        logits = eng.get_tensor("logits", (70, max(classes)))[:B]
        assert torch.equal(eng.eval_forward(part(img), part(tid))[0], logits)
    eng.sync_status()
    eng.close()


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("classes,masked", [(100, (20, 80)), (128, (0, 16)), (1000, (100, 1000)), (10, (3, 9))])
def test_classes_masked_by_a_bias_of_minus_infinity(classes, masked, dtype):
    """A CTA all of whose classes are masked has the maximum -inf and adds nothing to the softmax's sum; masked classes get no gradient."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    cfg = Config("mini_masked", 16, 4, 64, 1, 2, 128, (classes,), 5, (1,), (0,), 1, 2, dtype=dtype, seed=3)
    images, _, _, params = synth.make_workload(cfg, peaked=False)
    a, b = masked
    params["head.0.bias"][a:b] = -np.inf
    eng = Bd.Engine(cfg)
    eng.set_params(params)
    labels = torch.tensor([c for c in range(classes) if not a <= c < b][:5] * 5, dtype=torch.int32, device="cuda")[:5].contiguous()
    loss = eng.train_step(eng.images_to_device(images), labels, want_kept=False)[0]
    eng.sync_status()
    logits = eng.get_tensor("logits", (5, classes)).double()
    assert bool((logits[:, a:b] == -float("inf")).all())
    want = torch.nn.functional.cross_entropy(logits, labels.long())
    assert abs(float(loss[0]) - float(want)) < 1e-5 * float(want)
    d = torch.softmax(logits, 1)
    d[torch.arange(5), labels.long()] -= 1
    db = eng.get_tensor("grad/head.0.bias", (classes,)).double()
    assert float((db - d.sum(0) / 5).norm() / d.sum(0).norm()) < 1e-5 and not bool(db[a:b].any())
    assert bool(eng.grad_buffer().isfinite().all())
    eng.close()


@pytest.mark.parametrize("graph", [False, True])
def test_step_outputs_in_pinned_memory(graph):
    """Loss and kept positions go where a copy can take them, not only where a kernel can write: pinned host memory as device memory."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    cfg = MINI.with_(optimizer="sgd", lr=0.0, weight_decay=0.0)
    images, labels, _, params = synth.make_workload(cfg, peaked=True)
    eng = Bd.Engine(cfg)
    eng.set_params(params)
    with torch.cuda.stream(torch.cuda.Stream()):
        eng.set_graph_mode(graph)
        img, lab = eng.images_to_device(images), torch.as_tensor(labels).cuda()
        loss, kept = eng.train_step(img, lab)
        out = torch.zeros(1).pin_memory(), torch.full((sum(k.numel() for k in kept),), -1, dtype=torch.int32).pin_memory()
        for call in (eng.train_step, eng.train_step, eng.train_step, eng.forward_backward):
            out[0].zero_(), out[1].fill_(-1)
            call(img, lab, out=out)
            torch.cuda.current_stream().synchronize()
            assert torch.equal(out[0], loss.cpu()) and torch.equal(out[1], torch.cat([k.flatten() for k in kept]).cpu())
        eng.sync_status()
    eng.close()


def test_step_in_a_graph_of_the_callers():
    """A caller may capture the step into a graph of its own (in the strictest capture mode); replays equal calls."""
    import torch
    from paper_2405_10951_b200 import binding as Bd
    cfg = MINI.with_(optimizer="sgd", lr=0.0, weight_decay=0.0)
    images, labels, _, params = synth.make_workload(cfg, peaked=True)
    eng = Bd.Engine(cfg)
    eng.set_params(params)
    img, lab = eng.images_to_device(images), torch.as_tensor(labels).cuda()
    loss, kept = eng.train_step(img, lab)
    want = [loss.clone(), torch.cat([k.flatten() for k in kept]), eng.grad_buffer().clone()]
    out = torch.zeros(1, device="cuda"), torch.full_like(want[1], -1)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        eng.train_step(img, lab, out=out)
    for _ in range(2):
        out[0].zero_(), out[1].fill_(-1), eng.grad_buffer().zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, [*out, eng.grad_buffer()]))
    eng.sync_status()
    eng.close()
