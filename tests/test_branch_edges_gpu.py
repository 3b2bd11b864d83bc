"""GPU parity at the edges of the kernels' ranges that the shape sweeps do not reach: planes of 2^24 and 2^25 elements
(columns of 2048 and 4096 rows, shared by two and four tensor-memory lane quarters), and the block, the small planes and the log
gain gradients at theirs.  Bounds as in _checks.py."""
import numpy as np
import pytest
import torch

import oracle
from _checks import Guarded, bf16_round, check, check_grad, ref_inputs, to_dev
from paper_2607_25234_gb300 import inputs, whtmix

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2607_25234_gb300 import build
    build.build()
    oracle.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("B,n,N,C,dtype", [(1, 1 << 17, 1 << 17, 128, "f32"), (2, 70001, 1 << 17, 128, "bf16"),
                                           (1, 1 << 12, 1 << 12, 1 << 13, "bf16"), (1, 259200, 1 << 18, 128, "bf16"),
                                           (1, (1 << 18) - 3, 1 << 18, 128, "f32")])
def test_tall_columns_forward(B, n, N, C, dtype):
    d = inputs.make_inputs(B, N, C, dtype, seed=n, n_valid=n)
    x, g = to_dev(d["x"], dtype), to_dev(d["g"], "f32")
    y = Guarded((B, n, C), x.dtype)
    whtmix.forward_padded(x[:, :n].contiguous(), g, out=y.t)
    whtmix.sync()
    r = ref_inputs(d, dtype)
    check(y.t, oracle.forward(r["x"], r["g"])[:, :n], dtype, f"Y [{B},{n} of {N},{C}] {dtype}")
    y.assert_intact("Y")


@pytest.mark.parametrize("N,C,dtype", [(1 << 17, 128, "bf16"), (1 << 13, 1 << 11, "f32"), (1 << 18, 128, "f32")])
def test_tall_columns_log_gains(N, C, dtype):
    d = inputs.make_inputs(1, N, C, dtype, seed=N + C)
    g_t, g_c = inputs.make_log_gains(N, C, seed=3)
    x = to_dev(d["x"], dtype)
    y = Guarded(x.shape, x.dtype)
    whtmix.forward_separable(x, torch.from_numpy(g_t).cuda(), torch.from_numpy(g_c).cuda(), out=y.t)
    whtmix.sync()
    ref = oracle.forward_separable(ref_inputs(d, dtype)["x"], g_t.astype(np.float64), g_c.astype(np.float64))
    check(y.t, ref, dtype, f"separable Y [1,{N},{C}] {dtype}")
    y.assert_intact("Y")


# one and two channel blocks of 32 and a part of one; token counts below, at and past a warp's eight, a CTA's 32 and a chunk; the
# fourth to sixth and the last take 32 tokens a warp
@pytest.mark.parametrize("B,n,N,C,dtype", [(1, 2, 4, 32, "f32"), (2, 64, 64, 64, "bf16"), (1, 1 << 13, 1 << 13, 8, "f32"),
                                           (1, (1 << 17) - 4, 1 << 17, 32, "f32"), (1, 1 << 17, 1 << 17, 4, "bf16"),
                                           (1, 40000, 1 << 16, 64, "f32"), (3, 5, 8, 4, "f32"), (2, 17, 32, 64, "f32"), (2, 4000, 4096, 32, "f32"),
                                           (1, 1 << 14, 1 << 14, 2, "bf16"), (1, 2, 2, 1 << 13, "f32"), (2, 8192, 8192, 256, "bf16")])
def test_log_gain_gradients_in_one_pass(B, n, N, C, dtype):
    d = inputs.make_inputs(B, N, C, dtype, seed=n + C, n_valid=n, with_dy=True)
    g_t, g_c = inputs.make_log_gains(N, C, seed=5)
    x, dy = (to_dev(d[k], dtype)[:, :n].contiguous() for k in ("x", "dy"))
    out = [Guarded((B, n, C), x.dtype), Guarded((N,), torch.float32), Guarded((C,), torch.float32)]
    whtmix.backward_separable(x, torch.from_numpy(g_t).cuda(), torch.from_numpy(g_c).cuda(), dy, dx=out[0].t, dg_t=out[1].t,
                              dg_c=out[2].t)
    whtmix.sync()
    r = ref_inputs(d, dtype)
    dx, dgt, dgc = oracle.backward_separable(r["x"], g_t.astype(np.float64), g_c.astype(np.float64), r["dy"])
    check(out[0].t, dx[:, :n], dtype, "dX")
    check_grad(out[1].t, dgt, "f32", "dg_t")
    check_grad(out[2].t, dgc, "f32", "dg_c")
    for o, name in zip(out, ("dX", "dg_t", "dg_c")):
        o.assert_intact(name)


def bf16_dev(a):
    return torch.from_numpy(inputs.f32_to_bf16_bits(a).view(np.int16)).cuda().view(torch.bfloat16)


# the smallest and largest plane of the fused block for each channel count, one per kind of column pass between, and a
# batch of several plane groups
@pytest.mark.parametrize("B,N,C", [(1, 1024, 128), (3, 2048, 64), (2, 8192, 64), (5, 8192, 128), (1, 1 << 17, 64), (9, 1 << 15, 64)])
def test_fused_block(B, N, C):
    d = inputs.make_inputs(B, N, C, "bf16", seed=B + N + C)
    w_in, w_out = ((inputs.normal(s + C, C * C) / np.sqrt(C)).reshape(C, C).astype(np.float32) for s in (90, 91))
    x, g = to_dev(d["x"], "bf16"), to_dev(d["g"], "f32")
    y = Guarded(x.shape, torch.bfloat16)
    whtmix.block_forward(x, bf16_dev(w_in), g, bf16_dev(w_out), out=y.t)
    three = whtmix.project(whtmix.forward(whtmix.project(x, bf16_dev(w_in)), g), bf16_dev(w_out))
    whtmix.sync()
    y.assert_intact("block Y")
    assert torch.equal(y.t, three)  # the same sums in the same order, rounded at the same places
    x64, g64 = inputs.as_float64(d["x"], "bf16"), d["g"].astype(np.float64)
    wi, wo = (inputs.as_float64(inputs.f32_to_bf16_bits(w), "bf16") for w in (w_in, w_out))
    m = oracle.forward(bf16_round(x64 @ wi.T), g64)  # Z is rounded at each of these shapes
    ref, got = m @ wo.T, y.t.double().cpu().numpy()
    # M's and Y's roundings to bf16 (half an ulp, 2^-8 of a value) and the fp32 sums before them; a Z rounded to its other
    # neighbour moves M at its own place by 2^-7 |Z| mean(G), a hundredth of the sum over the channels that stands here
    bound = 2.0 ** -8 * np.abs(ref) + (2.0 ** -8 + 1e-5) * (np.abs(m) @ np.abs(wo).T) + 1e-5 * np.sqrt(np.mean(ref ** 2))
    assert (np.abs(got - ref) <= bound).all(), float(np.max(np.abs(got - ref) / bound))


# C = 256 to bf16, tiles of 64 tokens through three stages: one token, the edges of a tile, and two, three and four tiles a CTA
@pytest.mark.parametrize("T", [1, 63, 64, 65, 152 * 64 + 1, 2 * 152 * 64 + 77, 3 * 152 * 64 + 64])
def test_wide_projection(T):
    C = 256
    x, w = inputs.normal(60, T * C).reshape(T, C), (inputs.normal(61, C * C) / 16).reshape(C, C)
    xd, wd = bf16_dev(x.astype(np.float32)), bf16_dev(w.astype(np.float32))
    z = Guarded((T, C), torch.bfloat16)
    whtmix.project(xd, wd, out=z.t)
    own = xd.clone()
    whtmix.project(own, wd, out=own)
    whtmix.sync()
    z.assert_intact("Z")
    assert torch.equal(own, z.t)
    xe, we = xd.double().cpu().numpy(), wd.double().cpu().numpy()
    want, got = xe @ we.T, z.t.double().cpu().numpy()
    tol = np.abs(want) * 2.0 ** -8 + 1e-6 * (np.abs(xe) @ np.abs(we).T)  # half an ulp of bf16, and the fp32 sum
    assert (np.abs(got - want) <= tol).all(), float(np.max(np.abs(got - want) / tol))


# token counts about a chunk's tiles: a last chunk of one tile, a ragged last tile, more tiles than chunks
@pytest.mark.parametrize("B,N,C", [(1, 16, 256), (9, 32, 256), (1, 64, 64), (3, 32, 128), (77, 128, 256), (153, 64, 64), (160, 128, 128)])
def test_weight_gradient_chunks(B, N, C):
    """Bit for bit, so that no tile of tokens can be lost, doubled or taken from a neighbour: integer X and dY, projections that permute
    the channels and flip signs, unit gains.  Then Z, M = Z, dM and dZ = dM are small integers (the fp32 transforms are exact, their
    values integers below 2^24 over a power of two), and the weight gradients are sums of integers below 2^24."""
    x, dy = (inputs.small_ints(s + C, B * N * C, -2, 2).reshape(B, N, C).astype(np.float32) for s in (50, 51))
    w_in, w_out = (np.zeros((C, C), dtype=np.float32) for _ in range(2))
    for s, w in ((52, w_in), (53, w_out)):
        w[np.arange(C), np.argsort(inputs.normal(s + C, C))] = 2.0 * inputs.small_ints(s + 2 * C, C, 0, 1) - 1.0
    g = torch.ones(N, C, dtype=torch.float32, device="cuda")
    dx, dw_in, _, dw_out = whtmix.block_backward(bf16_dev(x), bf16_dev(w_in), g, bf16_dev(w_out), bf16_dev(dy))
    whtmix.sync()
    x64, dy64, wi, wo = (a.astype(np.float64).reshape(-1, C) for a in (x, dy, w_in, w_out))
    dz = dy64 @ wo
    for name, got, want in (("dX", dx, dz @ wi), ("dW_in", dw_in, dz.T @ x64), ("dW_out", dw_out, dy64.T @ (x64 @ wi.T))):
        got = got.double().cpu().numpy().reshape(want.shape)
        assert np.array_equal(got, want), f"{name}: {int((got != want).sum())} of {want.size} differ"


def run_padded(B, n, N, C, dtype, backward):
    d = inputs.make_inputs(B, N, C, dtype, seed=n + N, n_valid=n, with_dy=backward)
    x, g = to_dev(d["x"], dtype)[:, :n].contiguous(), to_dev(d["g"], "f32")
    r = ref_inputs(d, dtype)
    y = Guarded((B, n, C), x.dtype)
    whtmix.forward_padded(x, g, out=y.t)
    whtmix.sync()
    check(y.t, oracle.forward(r["x"], r["g"])[:, :n], dtype, f"Y [{B},{n} of {N},{C}] {dtype}")
    y.assert_intact("Y")
    if not backward:
        return
    dy = to_dev(d["dy"], dtype)[:, :n].contiguous()
    dx, dg = Guarded((B, n, C), x.dtype), Guarded((N, C), torch.float32)
    whtmix.backward_padded(x, g, dy, dx=dx.t, dg=dg.t)
    whtmix.sync()
    ref_dx, ref_dg = oracle.backward(r["x"], r["g"], r["dy"])
    check(dx.t, ref_dx[:, :n], dtype, f"dX [{B},{n} of {N},{C}] {dtype}")
    check_grad(dg.t, ref_dg, dtype, f"dG [{B},{n} of {N},{C}] {dtype}")
    dx.assert_intact("dX")
    dg.assert_intact("dG")


# the backward's dG sums: teams of one warp or group, teams with idle members, full teams over several sets of planes, and
# a second plane group, for every column height they cover
@pytest.mark.parametrize("B,n,N,C", [(1, 256, 256, 64), (6, 256, 256, 64), (40, 250, 256, 64), (515, 64, 256, 64), (17, 512, 512, 64),
                                     (20, 1024, 1024, 64), (33, 2047, 2048, 64), (1, 4096, 4096, 64), (3, 4096, 4096, 64),
                                     (35, 4000, 4096, 64), (2, 8192, 8192, 64), (9, 8192, 8192, 64), (12, 8191, 8192, 64), (17, 100, 8192, 64),
                                     (33, 60, 8192, 64), (5, 16384, 16384, 64),
                                     (9, 16384, 16384, 64), (1, 32768, 32768, 64), (7, 30000, 32768, 64), (1, 65536, 65536, 64),
                                     (3, 60000, 65536, 64), (1, 65536, 65536, 128), (2, 64800, 65536, 128)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_gain_gradient_sums(B, n, N, C, dtype):
    run_padded(B, n, N, C, dtype, backward=True)


# one plane a CTA (2^14, 2^15, and 2^16 from its smallest batch, 48 for bf16 and 64 for f32, and the three-phase kernel below): whole, cut inside a 16-byte chunk's row, one token stored;
# more planes than SMs
@pytest.mark.parametrize("B,n,N,C", [(1, 256, 256, 64), (3, 249, 256, 64), (2, 1, 512, 64), (3, 1023, 1024, 32), (48, 512, 512, 128),
                                     (49, 333, 512, 128),
                                     (63, 512, 512, 128), (64, 500, 512, 128), (310, 128, 128, 128), (160, 500, 512, 64)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_plane_in_tensor_memory(B, n, N, C, dtype):
    run_padded(B, n, N, C, dtype, False)


# tiles of 8, 4, 2 planes and one: a short last tile, padding in vectors of four elements and (one or two channels) not,
# more planes than a round of the dG sum
@pytest.mark.parametrize("B,n,N,C", [(1, 32, 32, 32), (9, 31, 32, 32), (5, 64, 64, 32), (130, 61, 64, 32), (257, 64, 64, 64), (3, 33, 64, 64),
                                     (2, 128, 128, 64), (5, 1, 128, 64), (3, 1021, 2048, 2), (4, 4093, 4096, 1), (2, 1, 1, 1 << 13)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_small_planes(B, n, N, C, dtype):
    run_padded(B, n, N, C, dtype, True)
