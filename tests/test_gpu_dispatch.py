"""GPU parity at the edges of the size rules by which calls are sent to one
kernel or another: the smallest and largest sizes, remainders and ragged ends
of each kernel's tiles, against the CPU oracle."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

import oracle as O
from paper_2608_02438_gb300 import workloads as W

from _parity import compare_accept, compare_blocks, device_inputs, oracle_model, run_oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def X():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_02438_gb300 import binding, build
    build.build()
    binding.load()
    return binding


def _refiner(X, cfg, weights):
    dt = X.XPRESS_BF16 if cfg.dtype == W.BF16 else X.XPRESS_F32
    return X.Refiner({k: X.to_device(v, dt) for k, v in weights.items()}, cfg.H, cfg.V, cfg.r, cfg.B, dt), dt


# Y^(0) = argmax s outside the persistent kernel (k_rowmax): fewer pieces than
# threads, one round and a remainder, several rounds; both storage types.
@pytest.mark.parametrize("dtype", [W.F32, W.BF16])
@pytest.mark.parametrize("V", [32, 2088, 36872])
def test_argmax_seed(X, dtype, V):
    cfg = W.tiny_config("seed", b=5, B=8, H=64, V=V, r=256, dtype=dtype, temps=(0.0, 1.0), seed=71)
    w = W.make_weights(cfg.H, cfg.V, cfg.r, cfg.B, cfg.dtype, 72, "strong")
    inp = W.make_inputs(cfg)
    inp["s"][:, :, V // 2] = inp["s"].max(axis=-1) if dtype == W.F32 else inp["s"][:, :, V // 2]   # an exact tie
    ref, dt = _refiner(X, cfg, w)
    d = device_inputs(dt, inp)
    out = ref.refine_block(d["h"], d["s"], None, d["anchor"], d["temperature"], d["seed"], inp["offset"], cfg.K_max)
    torch.cuda.synchronize()
    m = oracle_model(cfg, w)
    for i in range(cfg.b):
        o = O.jacobi(m, inp["h"][i], inp["s"][i], int(inp["anchor"][i]), None, float(inp["temperature"][i]),
                     int(inp["seed"][i]), inp["offset"], cfg.K_max)
        assert out["tokens"][i].cpu().numpy().tolist() == o["tokens"].tolist()
        assert int(out["iters"][i]) == o["iters"]


# Acceptance: empty and one-piece row chunks (V = 32), ragged last batches, a
# masked prefix that fills whole pieces (its log-sum-exp must not see it), both
# storage types, and the draws of one sweep, a partial second one and many.
@pytest.mark.parametrize("b,V,dtype,masked", [(1, 32, W.BF16, 0), (3, 2088, W.F32, 0), (9, 40008, W.BF16, 33000),
                                              (17, 1032, W.BF16, 64), (33, 296, W.BF16, 0), (70, 264, W.BF16, 0)])
def test_accept_row_and_draw_edges(X, b, V, dtype, masked):
    cfg = W.tiny_config("acce", b=b, B=4, H=64, V=V, r=256, dtype=dtype, temps=(1.0, 1.0, 0.0), seed=81 + b,
                        logits="gauss4_spike", draft="sample")
    w = W.make_weights(cfg.H, cfg.V, cfg.r, cfg.B, cfg.dtype, 82 + b, "strong")
    inp = W.make_inputs(cfg)
    if masked:
        inp["target"][:, :, :masked] = W.to_storage(np.float32([-np.inf]), dtype)[0]
    ref, dt = _refiner(X, cfg, w)
    d = device_inputs(dt, inp)
    o = ref.refine_block(d["h"], d["s"], d["draft"], d["anchor"], d["temperature"], d["seed"], inp["offset"], cfg.K_max)
    acc = ref.accept(d["target"], d["s"], o["tokens"], o["lse"], o["logit_sel"], o["z_final"], d["temperature"],
                     d["seed"], inp["offset"])
    torch.cuda.synchronize()
    assert ref.device_status("accept", b) == X.XPRESS_OK
    m = oracle_model(cfg, w)
    expect = {}
    for i in range(b):
        j = O.jacobi(m, inp["h"][i], inp["s"][i], int(inp["anchor"][i]), inp["draft"][i],
                     float(inp["temperature"][i]), int(inp["seed"][i]), inp["offset"], cfg.K_max)
        assert o["tokens"][i].cpu().numpy().tolist() == j["tokens"].tolist()
        n, out, _, gaps = O.accept(m, inp["target"][i], inp["s"][i], j["tokens"], j["lse"], j["sel"], j["z_final"],
                                   float(inp["temperature"][i]), int(inp["seed"][i]), inp["offset"], with_gaps=True)
        expect[i] = (n, out, gaps)
    compare_accept(acc["accept_len"].cpu().numpy(), acc["out_tokens"].cpu().numpy(), expect, list(range(b)),
                   inp["temperature"])


# More row tiles than SMs: dL/dl is held for one group of row tiles at a time,
# each with its own dz pass and dW_r product.  The step is the sum of the steps
# of its two halves (one group each, checked against the oracle elsewhere) up
# to the fp32 order of the sums, which moves a bf16 operand rounding (2^-8 of an
# element) in fewer than 2^-10 of the elements: below 2^-8 * 2^-5 = 2^-13 for
# each of the at most six operand roundings of a backward chain.
def test_train_row_tile_groups(X):
    cfg = W.Config("train_groups", b=310, B=32, H=64, V=264, r=256, dtype=W.BF16, K_max=32, logits="gauss4_spike",
                   seed=91)
    assert (cfg.b * cfg.B + 63) // 64 > torch.cuda.get_device_properties(0).multi_processor_count
    w = W.make_weights(cfg.H, cfg.V, cfg.r, cfg.B, cfg.dtype, 92, "paper")
    inp = W.make_train_inputs(cfg)
    ref, dt = _refiner(X, cfg, w)
    d = {k: X.to_device(inp[k], dt) for k in ("h", "s", "target")}
    d.update({k: torch.from_numpy(inp[k]).cuda() for k in ("ystar", "anchor")})
    loss, grads = ref.train_step(*(d[k] for k in ("h", "s", "target", "ystar", "anchor")))
    n = cfg.b // 2
    halves = ref.alloc_grads()
    parts = [ref.train_step(*(d[k][j].contiguous() for k in ("h", "s", "target", "ystar", "anchor")), grads=halves)[0]
             for j in (slice(0, n), slice(n, cfg.b))]
    torch.cuda.synchronize()
    assert ref.device_status("train", cfg.b) == X.XPRESS_OK
    assert torch.allclose(loss, torch.cat(parts), rtol=1e-5, atol=1e-4)
    for k, g in grads.items():
        assert float((g - halves[k]).norm() / halves[k].norm()) < 6 * 2.0 ** -13, k


# A sampling row whose every logit is NaN has no group to draw from: the
# reduction's member draw stays in bounds and the call reports it.
def test_nan_logits_are_reported(X):
    cfg = W.tiny_config("nan", b=5, B=8, H=64, V=2080, r=256, dtype=W.BF16, temps=(1.0,), seed=75)
    w = W.make_weights(cfg.H, cfg.V, cfg.r, cfg.B, cfg.dtype, 76, "paper")
    inp = W.make_inputs(cfg)
    inp["s"][2, 3] = 0x7FC0                             # bf16 NaN
    ref, dt = _refiner(X, cfg, w)
    d = device_inputs(dt, inp)
    out = ref.refine_block(d["h"], d["s"], d["draft"], d["anchor"], d["temperature"], d["seed"], inp["offset"], cfg.K_max)
    torch.cuda.synchronize()
    assert ref.device_status("refine", cfg.b) == X.XPRESS_ERR_DEVICE_CHECK
    tok = out["tokens"].cpu().numpy()
    assert (tok >= 0).all() and (tok < cfg.V).all()


# fp32 refiners (CUDA cores): hidden sizes of one short, one whole and three
# K slices, token tiles of 1, 32, 33 and 96 tokens, one group and several per
# vocabulary range, a last group of 8 ids; every activation.  Weights at 4-byte
# boundaries take the scalar loads.
@pytest.mark.parametrize("b,B,H,V,act,shift", [(1, 1, 8, 32, O.RELU, 0), (1, 32, 512, 1032, O.SILU, 0),
                                               (3, 11, 1288, 2088, O.GELU, 1), (3, 32, 256, 20008, O.SILU, 0)])
def test_fp32_refine_edges(X, b, B, H, V, act, shift):
    cfg = W.tiny_config("f32e", b=b, B=B, H=H, V=V, r=256, dtype=W.F32, temps=(0.0, 1.0), seed=111 + B)
    w = W.make_weights(cfg.H, cfg.V, cfg.r, cfg.B, cfg.dtype, 112 + B, "strong")
    inp = W.make_inputs(cfg)
    dev = {}
    for k, v in w.items():
        flat = torch.empty(v.size + shift, dtype=torch.float32, device="cuda")
        flat[shift:] = torch.from_numpy(v).cuda().flatten()
        dev[k] = flat[shift:].view(v.shape)
    ref = X.Refiner(dev, cfg.H, cfg.V, cfg.r, cfg.B, X.XPRESS_F32, act)
    d = device_inputs(X.XPRESS_F32, inp)
    out = ref.refine_block(d["h"], d["s"], d["draft"], d["anchor"], d["temperature"], d["seed"], inp["offset"],
                           cfg.K_max, want_logits=True, want_traj=True)
    torch.cuda.synchronize()
    assert ref.device_status("refine", b) == X.XPRESS_OK
    m = O.Model(w, cfg.H, cfg.V, cfg.r, cfg.B, O.F32, act)
    orc = {i: run_oracle(m, inp, i, cfg.K_max) for i in range(b)}
    g = {k: (v.cpu().numpy() if v is not None else None) for k, v in out.items()}
    compare_blocks(g, orc, list(range(b)), cfg.dtype, check_logits=g["refined_logits"], m=m, inp=inp)


# The LM head's token chunks and vocabulary items: the last size of each chunk
# width and the first of the next, an item count that leaves CTAs idle, two
# tiles per item (the second past V, or partly), three chunks over the CTAs.
@pytest.mark.parametrize("N,V,H", [(32, 136, 72), (33, 520, 200), (128, 2088, 264), (129, 2088, 136), (256, 78000, 72),
                                   (257, 39000, 72), (600, 26000, 136)])
def test_lm_head_shapes(X, N, V, H):
    g = torch.Generator(device="cuda").manual_seed(N)
    Wl = (torch.randn((V, H), generator=g, device="cuda") * 0.05).bfloat16()
    h = torch.randn((N, H), generator=g, device="cuda").bfloat16()
    s = torch.full((N, V), float("nan"), dtype=torch.bfloat16, device="cuda")
    am = torch.full((N,), -1, dtype=torch.int32, device="cuda")
    X.lm_head(Wl, h, s, am)
    torch.cuda.synchronize()
    exact = h.double() @ Wl.double().T
    # half a bf16 ulp of the value, and fp32 sums of H exact products
    bound = exact.abs() * 2.0 ** -8 + H * 2.0 ** -23 * (h.double().abs() @ Wl.double().abs().T)
    assert bool(((s.double() - exact).abs() <= bound).all())
    ids = torch.arange(V, device="cuda")
    sf = s.float()
    first = torch.where(sf == sf.amax(1, keepdim=True), ids, V).amin(1)
    assert torch.equal(am.long(), first)


# p = q at every id (W_r = 0 and target = s, with one id holding all the mass, so
# that both log-sum-exps are the same float): the subgradient is 0 there, by the
# passes' tie branch; V = 2088 also has a last tile of 40 ids.
def test_train_ties(X):
    cfg = W.Config("ties", b=2, B=8, H=64, V=2088, r=256, dtype=W.BF16, K_max=8, logits="gauss4_spike", seed=121)
    w = W.make_weights(cfg.H, cfg.V, cfg.r, cfg.B, cfg.dtype, 122, "paper")
    w["W_r"] = np.zeros_like(w["W_r"])
    inp = W.make_train_inputs(cfg)
    rng = np.random.default_rng(5)
    s = np.zeros((cfg.b, cfg.B, cfg.V), np.float32)
    np.put_along_axis(s, rng.integers(0, cfg.V, (cfg.b, cfg.B, 1)), 60.0, axis=2)
    inp["s"] = inp["target"] = W.to_storage(s, cfg.dtype)
    ref, dt = _refiner(X, cfg, w)
    d = {k: X.to_device(inp[k], dt) for k in ("h", "s", "target")}
    loss, grads = ref.train_step(d["h"], d["s"], d["target"], torch.from_numpy(inp["ystar"]).cuda(),
                                 torch.from_numpy(inp["anchor"]).cuda(), a_ce=0.5, a_l1=2.0)
    torch.cuda.synchronize()
    assert ref.device_status("train", cfg.b) == X.XPRESS_OK
    m = oracle_model(cfg, w)
    tot = None
    for i in range(cfg.b):
        lo, go = O.train_step(m, inp["h"][i], inp["s"][i], inp["target"][i], inp["ystar"][i], int(inp["anchor"][i]),
                              a_ce=0.5, a_l1=2.0)
        np.testing.assert_allclose(loss[i].cpu().numpy(), lo, rtol=2e-3, atol=2e-3)
        tot = go if tot is None else {k: tot[k] + go[k] for k in go}
    g = grads["W_r"].cpu().numpy()
    assert np.linalg.norm(g - tot["W_r"]) <= 2.0 ** -5 * np.linalg.norm(tot["W_r"])


# The graph path's tcgen05 Read: one to five token tiles and their ragged ends
# (the warp-wide copies of s meet missing tokens), over ranges of one and two
# vocabulary tiles per CTA, the last tile 8 ids wide; and a pass whose blocks are
# packed in two rounds of k_reduce16's 512 threads.
@pytest.mark.parametrize("b,B,V", [(11, 3, 20488), (10, 13, 20488), (12, 32, 20488), (25, 16, 2056), (65, 8, 20488),
                                   (9, 15, 40968), (20, 13, 20488), (33, 17, 20488), (515, 4, 2056)])
def test_read_token_tiles(X, b, B, V):
    cfg = W.tiny_config("readt", b=b, B=B, H=64, V=V, r=256, dtype=W.BF16, temps=(0.0, 1.0, 0.7), seed=101 + b,
                        logits="gauss4_spike", draft="sample")
    w = W.make_weights(cfg.H, cfg.V, cfg.r, cfg.B, cfg.dtype, 102 + b, "strong")
    inp = W.make_inputs(cfg)
    ref, dt = _refiner(X, cfg, w)
    d = device_inputs(dt, inp)
    out = ref.refine_block(d["h"], d["s"], d["draft"], d["anchor"], d["temperature"], d["seed"], inp["offset"],
                           cfg.K_max, want_traj=True)
    torch.cuda.synchronize()
    assert ref.device_status("refine", b) == X.XPRESS_OK
    m = oracle_model(cfg, w)
    with ThreadPoolExecutor(16) as ex:
        orc = dict(enumerate(ex.map(lambda i: run_oracle(m, inp, i, cfg.K_max, False), range(b))))
    g = {k: (v.cpu().numpy() if v is not None else None) for k, v in out.items()}
    compare_blocks(g, orc, list(range(b)), cfg.dtype, m=m, inp=inp)


# The hidden projection of the graph path (k_pre_tc), alone: W_in picks
# F = W_h + 2^-8 (W_h one row on), exact in the hi and lo terms, and everything
# after it is zero, so z = F h.  An accumulation step in tensor memory cuts the sum
# off by up to 2^-23 of it, 2^-24 on average; with 16 slices of 256 and two
# accumulators each takes n = 8 steps of 16 products of the hi term (the lo terms'
# sums are 2^-8 of it), and its sum grows to the end: below n 2^-24.
@pytest.mark.parametrize("b,B,n", [(3, 16, 8), (9, 16, 8), (16, 32, 8)])
def test_hidden_projection_accuracy(X, b, B, n):
    H, V, r = 4096, 64, 256
    g = torch.Generator(device="cuda").manual_seed(b)

    def zeros(*shape):
        return torch.zeros(shape, dtype=torch.bfloat16, device="cuda")

    W_h = (torch.randint(8, 16, (r, H), generator=g, device="cuda").float() / 8).bfloat16()
    W_in = zeros(r, 3 * r)
    W_in[:, :r] = (torch.eye(r) + torch.roll(torch.eye(r), 1, 1) * 2.0 ** -8).cuda()
    ref = X.Refiner(dict(W_e=zeros(V, r), W_h=W_h, W_g=zeros(r, H), W_in=W_in, L=zeros(r, B, B), W1=zeros(2 * r, r),
                         W2=zeros(r, 2 * r), W_r=zeros(V, r)), H, V, r, B, X.XPRESS_BF16)
    h = torch.randn((b, B, H), generator=g, device="cuda").bfloat16()
    s = torch.randn((b, B, V), generator=g, device="cuda").bfloat16()
    i32 = dict(dtype=torch.int32, device="cuda")
    out = ref.refine_block(h, s, torch.zeros((b, B), **i32), torch.zeros(b, **i32), torch.zeros(b, device="cuda"),
                           torch.zeros(b, dtype=torch.int64, device="cuda"), 1, 2)
    torch.cuda.synchronize()
    assert ref.device_status("refine", b) == X.XPRESS_OK
    exact = h.double() @ (W_in.double()[:, :r] @ W_h.double()).T
    assert float((out["z_final"].double() - exact).norm() / exact.norm()) < n * 2.0 ** -24


# More token chunks than a group of the LM head holds, and more than CTAs: 17
# (eight and nine) over 41 CTAs, 19 over four (five groups) and 300 over two.
@pytest.mark.parametrize("N,V,H", [(4100, 5128, 72), (4650, 392, 64), (76570, 136, 64)])
def test_lm_head_chunk_groups(X, N, V, H):
    test_lm_head_shapes(X, N, V, H)


# More blocks than a grid holds in y, and a ragged last row tile: the step is
# accepted and is the sum of the steps of its two halves (to the bound of
# test_train_row_tile_groups).
def test_train_many_short_blocks(X):
    cfg = W.Config("train_many", b=65520, B=2, H=64, V=64, r=256, dtype=W.BF16, K_max=2, logits="gauss4_spike", seed=93)
    ref, dt = _refiner(X, cfg, W.make_weights(cfg.H, cfg.V, cfg.r, cfg.B, cfg.dtype, 94, "paper"))
    inp = W.make_train_inputs(cfg)
    args = [X.to_device(inp[k], dt) for k in ("h", "s", "target")] + [torch.from_numpy(inp[k]).cuda()
                                                                     for k in ("ystar", "anchor")]
    loss, grads = ref.train_step(*args)
    n, halves = cfg.b // 2, ref.alloc_grads()
    parts = [ref.train_step(*(a[j].contiguous() for a in args), grads=halves)[0] for j in (slice(0, n), slice(n, cfg.b))]
    torch.cuda.synchronize()
    assert ref.device_status("train", cfg.b) == X.XPRESS_OK
    assert torch.allclose(loss, torch.cat(parts), rtol=1e-5, atol=1e-4)
    for k, g in grads.items():
        assert float((g - halves[k]).norm() / halves[k].norm()) < 6 * 2.0 ** -13, k


def _at_offset(t, n):
    """A copy of t whose first element lies n elements past an aligned address."""
    flat = torch.empty(t.numel() + n, dtype=t.dtype, device="cuda")
    flat[n:] = t.flatten()
    return flat[n:].view(t.shape)


# The acceptance reads the target's rows in 16-byte pieces: a target at another
# boundary is refused, with and without a workspace.
@pytest.mark.parametrize("dtype", [W.F32, W.BF16])
def test_accept_refuses_an_unaligned_target(X, dtype):
    cfg = W.tiny_config("acal", b=2, B=4, H=64, V=264, r=256, dtype=dtype, temps=(0.0, 1.0), seed=131)
    inp = W.make_inputs(cfg)
    ref, dt = _refiner(X, cfg, W.make_weights(cfg.H, cfg.V, cfg.r, cfg.B, cfg.dtype, 132, "paper"))
    d = device_inputs(dt, inp)
    o = ref.refine_block(d["h"], d["s"], d["draft"], d["anchor"], d["temperature"], d["seed"], inp["offset"], cfg.K_max)
    out = dict(accept_len=torch.empty(2, dtype=torch.int32, device="cuda"),
               out_tokens=torch.empty((2, 5), dtype=torch.int32, device="cuda"))
    target = _at_offset(d["target"], 2)
    with pytest.raises(X.XpressError) as err:
        ref.accept(target, d["s"], o["tokens"], o["lse"], o["logit_sel"], o["z_final"], d["temperature"], d["seed"],
                   inp["offset"], out=out)
    assert err.value.code == X.XPRESS_ERR_INVALID_ARG
    acc_in = X.XpressAcceptIn(2, *[t.data_ptr() for t in (target, d["s"], o["tokens"], o["lse"], o["logit_sel"],
                                                          o["z_final"], d["temperature"], d["seed"])], inp["offset"])
    with pytest.raises(X.XpressError) as err:
        X.xpress_accept_noalloc(ref.handle, acc_in, out["accept_len"].data_ptr(), out["out_tokens"].data_ptr(),
                                ref.stream.cuda_stream)
    assert err.value.code == X.XPRESS_ERR_INVALID_ARG


# z_final at a 4-byte boundary, on each path that writes it: fp32, the persistent
# kernel, and the token tiles of k_trans_tc.
@pytest.mark.parametrize("dtype,b,B", [(W.F32, 3, 5), (W.BF16, 2, 16), (W.BF16, 9, 15)])
def test_z_final_at_any_boundary(X, dtype, b, B):
    cfg = W.tiny_config("zal", b=b, B=B, H=64, V=2056, r=256, dtype=dtype, temps=(0.0, 1.0), seed=141)
    inp = W.make_inputs(cfg)
    ref, dt = _refiner(X, cfg, W.make_weights(cfg.H, cfg.V, cfg.r, cfg.B, cfg.dtype, 142, "strong"))
    d = device_inputs(dt, inp)
    args = (d["h"], d["s"], d["draft"], d["anchor"], d["temperature"], d["seed"], inp["offset"], cfg.K_max)
    want = ref.refine_block(*args)
    got = ref.alloc_outputs(b)
    got["z_final"] = _at_offset(torch.full_like(got["z_final"], float("nan")), 1)
    ref.refine_block(*args, out=got)
    torch.cuda.synchronize()
    assert ref.device_status("refine", b) == X.XPRESS_OK
    assert torch.equal(got["z_final"], want["z_final"]) and torch.equal(got["tokens"], want["tokens"])


# W_in of a bf16 refiner at a 2-byte boundary: the precompute that folds it in per
# call (at most 32 tokens, H not a multiple of 64), and those that take the
# refiner's folded copy.
@pytest.mark.parametrize("b,B,H", [(2, 8, 72), (2, 8, 128), (5, 16, 128)])
def test_bf16_W_in_at_any_boundary(X, b, B, H):
    cfg = W.tiny_config("wal", b=b, B=B, H=H, V=2056, r=256, dtype=W.BF16, temps=(0.0, 1.0), seed=151)
    inp = W.make_inputs(cfg)
    w = {k: X.to_device(v, X.XPRESS_BF16)
         for k, v in W.make_weights(cfg.H, cfg.V, cfg.r, cfg.B, cfg.dtype, 152, "strong").items()}
    d = device_inputs(X.XPRESS_BF16, inp)
    outs = []
    for weights in (w, {**w, "W_in": _at_offset(w["W_in"], 1)}):
        ref = X.Refiner(weights, cfg.H, cfg.V, cfg.r, cfg.B, X.XPRESS_BF16)
        outs.append(ref.refine_block(d["h"], d["s"], d["draft"], d["anchor"], d["temperature"], d["seed"],
                                     inp["offset"], cfg.K_max))
        torch.cuda.synchronize()
        assert ref.device_status("refine", b) == X.XPRESS_OK
    for k in ("tokens", "iters", "z_final", "logit_sel"):
        assert torch.equal(outs[0][k], outs[1][k]), k


# The fp32 residual draw with W_r at a 4-byte boundary.
def test_fp32_draw_with_W_r_at_any_boundary(X):
    cfg = W.tiny_config("wral", b=5, B=4, H=64, V=1032, r=256, dtype=W.F32, temps=(1.0, 0.7), seed=161,
                        logits="gauss4_spike", draft="sample")
    inp = W.make_inputs(cfg)
    w = {k: X.to_device(v, X.XPRESS_F32)
         for k, v in W.make_weights(cfg.H, cfg.V, cfg.r, cfg.B, cfg.dtype, 162, "strong").items()}
    d = device_inputs(X.XPRESS_F32, inp)
    outs = []
    for weights in (w, {**w, "W_r": _at_offset(w["W_r"], 1)}):
        ref = X.Refiner(weights, cfg.H, cfg.V, cfg.r, cfg.B, X.XPRESS_F32)
        o = ref.refine_block(d["h"], d["s"], d["draft"], d["anchor"], d["temperature"], d["seed"], inp["offset"], cfg.K_max)
        outs.append(ref.accept(d["target"], d["s"], o["tokens"], o["lse"], o["logit_sel"], o["z_final"],
                               d["temperature"], d["seed"], inp["offset"]))
        torch.cuda.synchronize()
        assert ref.device_status("accept", cfg.b) == X.XPRESS_OK
    assert int(outs[0]["accept_len"].min()) < cfg.B                # at least one residual draw
    for k in ("accept_len", "out_tokens"):
        assert torch.equal(outs[0][k], outs[1][k]), k


# Draws of more than two sweeps of the vocabulary: 87 in three of 32 (bf16), 40 in
# three of 16 (fp32).
@pytest.mark.parametrize("b,V,dtype", [(130, 264, W.BF16), (60, 296, W.F32)])
def test_accept_many_sweeps(X, b, V, dtype):
    test_accept_row_and_draw_edges(X, b, V, dtype, 0)
