"""GPU parity of prefix key/value caching combined with truncation (Table 7's
composition): prefill of the prefix K/V, response-row gather, and the block
over response rows with cached prefix keys, through the C ABI, against the
oracle; and exactness against the uncached truncated layer on the same input."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.helpers import at_16, check_close, cuda, host, i32, to_dev

pytestmark = pytest.mark.gpu

S = pytest.importorskip("paper_2607_14557_gb300.seer")


@pytest.fixture(autouse=True)
def _device_clean():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield
    assert S.seer_check_device() == 0


def _workload(dtype):
    if dtype == "f32":
        return synth.workload(0)
    return synth.tiny_workload(dtype="bf16", seed=370, d=256, n_heads=2, head_dim=128, d_ff=768, batch=4, window=200,
                               boundary=("uniform", 8, 190), visual=("mult", 96, 1, 3))


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_cached_layer_matches_oracle_and_uncached_rows(dtype):
    from paper_2607_14557_gb300 import driver as D
    wl = _workload(dtype)
    lens = synth.lengths(wl)
    x, cu_full, resp = synth.hidden_full(wl, lens)
    w = synth.layer_weights(wl, 0)
    B, N, d, H = wl.batch, wl.window, wl.d, wl.n_heads
    dims = S.make_dims(d, H, wl.head_dim, wl.d_ff)
    W = D.LayerWeights.from_host(w, dtype)
    T_full = x.shape[0]
    path = D.SeerPath(dims, dtype, B, N, T_full, S.make_params(wl.act_eps))
    ctx = i32(lens.ctx)
    path.step(to_dev(x, dtype), i32(cu_full), i32(resp), ctx, W)         # detect, pack, uncached truncated layer
    it = torch.float32 if dtype == "f32" else torch.float16
    cache = torch.full((T_full, 2 * d), 7.0, dtype=it, device=cuda())
    S.seer_kv_prefill(W.struct(), dims, dtype, path.x_packed, path.cu, ctx, B, T_full, cache, path.cu, T_full, path.ws,
                      path.ws_bytes)
    xr = torch.zeros_like(path.x_packed)
    cu_r = torch.empty(B + 1, dtype=torch.int32, device=cuda())
    S.seer_gather_response(path.x_packed, dtype, path.cu, ctx, B, d, T_full, xr, cu_r)
    yr = torch.full_like(xr, 9.0)
    S.seer_layer_forward_cached(W.struct(), dims, dtype, xr, yr, cu_r, ctx, B, T_full, cache, path.cu, path.kv, T_full,
                                path.ws, path.ws_bytes)
    torch.cuda.synchronize()
    cu, kv, c = path.cu.cpu().numpy(), path.kv.cpu().numpy(), lens.ctx
    np.testing.assert_array_equal(path.L_star.cpu().numpy(), lens.boundary + 1)
    np.testing.assert_array_equal(cu_r.cpu().numpy(), cu - np.concatenate([[0], np.cumsum(c)]))
    cr = cu_r.cpu().numpy()
    xp, xrh, yrh, yfull, ch = host(path.x_packed), host(xr), host(yr), host(path.y), host(cache)
    for b in range(B):
        seg = xp[cu[b]:cu[b + 1]]
        np.testing.assert_array_equal(xrh[cr[b]:cr[b + 1]], seg[c[b]:])                 # gather is exact
        # the cached block reproduces the uncached truncated layer's response rows bit for bit
        np.testing.assert_array_equal(yrh[cr[b]:cr[b + 1]], yfull[cu[b] + c[b]:cu[b + 1]])
        k, v = oracle.kv_prefill(seg[:c[b]], w, H)
        check_close(ch[cu[b]:cu[b] + c[b]], np.concatenate([k, v], axis=1), dtype, f"prefix K/V {b}")
        ref = oracle.layer_forward_cached(seg[c[b]:], k, v, w, H, kv_valid=int(kv[b] - c[b]))
        check_close(yrh[cr[b]:cr[b + 1]], ref, dtype, f"cached block segment {b}")
    assert (yrh[cr[-1]:] == 9.0).all()                                                 # zero work past the rows


@pytest.mark.parametrize("d", [256, 4352])                           # norm from registers, and streaming
@pytest.mark.parametrize("ctx,bad", [([40], -1), ([1, 31, 0, 32, 33, 200, 65], -1), ([100, 64, 7], 1), ([0, 5], -1)])
def test_kv_prefill_stores_segments_where_the_offsets_say(d, ctx, bad):
    """16-bit prefill reads and writes rows in place: segments at odd offsets with gaps
    between them (slabs of 32 rows that straddle segments, empty prefixes) equal the
    norm and the projection of the gathered rows bit for bit, other cache rows stay,
    and a segment outside the cache is recorded and writes nothing."""
    B, H = len(ctx), d // 128
    g = torch.Generator(device="cuda").manual_seed(d + B)
    r = lambda *shape: torch.randn(shape, generator=g, device="cuda")
    starts_x = np.cumsum([3] + [c + 5 for c in ctx])                   # B + 1 offsets
    starts_kv = np.cumsum([1] + [c + 9 for c in ctx])
    T_x, T_kv = int(starts_x[-1]), int(starts_kv[-1])
    place = starts_kv.copy()
    if bad >= 0:
        place[bad] = T_kv - ctx[bad] + 1                               # one row past the end
    x = r(T_x, d).to(torch.bfloat16)
    w_qkv, gain = (0.02 * r(3 * d, d)).half(), (1 + 0.1 * r(d)).half()
    dims = S.make_dims(d, H, 128, 128)
    w = S.make_weights(w_qkv, 0, 0, 0, 0, gain, 0)
    n = S.seer_layer_workspace_size(dims, "bf16", T_x, B)
    ws = torch.empty(n, dtype=torch.uint8, device=cuda())
    cache = torch.full((T_kv, 2 * d), 7.0, dtype=torch.float16, device=cuda())
    S.seer_kv_prefill(w, dims, "bf16", x, i32(starts_x), i32(ctx), B, T_x, cache, i32(place), T_kv, ws, n)
    assert S.seer_check_device() == (2 if bad >= 0 else 0)
    rows = torch.cat([x[a:a + c] for a, c in zip(starts_x, ctx)])
    xn, kv = torch.empty_like(rows, dtype=torch.float16), torch.empty((len(rows), 2 * d), dtype=torch.float16, device=cuda())
    S.seer_rmsnorm(rows, "bf16", gain, xn, "f16", len(rows), None, d, 1e-5)
    S.seer_linear(xn, w_qkv[d:], "f16", None, "f16", kv, "f16", len(rows), None, 2 * d, d)
    want = torch.full_like(cache, 7.0)
    at = 0
    for b, c in enumerate(ctx):
        if b != bad:
            want[int(place[b]):int(place[b]) + c] = kv[at:at + c]
        at += c
    assert torch.equal(cache, want)


@pytest.mark.parametrize("ctx,resp", [([4200], [40]), ([5000, 4300], [200, 7]), ([9000], [300])])
def test_cached_layer_long_prefixes_few_rows(ctx, resp):
    """Few query tiles over long caches: each unit's keys are split over 8 or 4 CTAs."""
    wl = _workload("bf16")
    w = synth.layer_weights(wl, 0)
    d, H, B = wl.d, wl.n_heads, len(ctx)
    dims = S.make_dims(d, H, wl.head_dim, wl.d_ff)
    from paper_2607_14557_gb300 import driver as D
    W = D.LayerWeights.from_host(w, "bf16")
    rng = np.random.default_rng(sum(ctx))
    cu = np.concatenate([[0], np.cumsum([a + b for a, b in zip(ctx, resp)])])
    cr = np.concatenate([[0], np.cumsum(resp)])
    T, R = int(cu[-1]), int(cr[-1])
    x = synth.round_storage(rng.standard_normal((R, d)), "bf16")
    kv = torch.from_numpy(rng.standard_normal((T, 2 * d)).astype(np.float32)).half()
    cache = kv.to(cuda())
    y = torch.full((R, d), 9.0, dtype=torch.bfloat16, device=cuda())
    n = S.seer_layer_workspace_size(dims, "bf16", R, B)
    ws = torch.empty(n, dtype=torch.uint8, device=cuda())
    S.seer_layer_forward_cached(W.struct(), dims, "bf16", to_dev(x, "bf16"), y, i32(cr), i32(ctx), B, R, cache, i32(cu),
                                None, T, ws, n)
    assert S.seer_check_device() == 0
    k, got = kv.numpy().astype(np.float64), host(y)
    for b, c in enumerate(ctx):
        pre = k[cu[b]:cu[b] + c]
        ref = oracle.layer_forward_cached(x[cr[b]:cr[b + 1]], pre[:, :d], pre[:, d:], w, H)
        check_close(got[cr[b]:cr[b + 1]], ref, "bf16", f"cached block segment {b}")


@pytest.mark.parametrize("rope", [0.0, 1e4])
def test_layer_and_cache_buffers_on_16_byte_boundaries(rope):
    """A layer, a prefill and a cached layer whose activations, cache and workspace start
    on 16-byte boundaries, not 32-byte ones: segments of odd lengths, so rows reach the
    cache one by one; the same bits as from buffers on larger boundaries."""
    wl = _workload("bf16")
    from paper_2607_14557_gb300 import driver as D
    W = D.LayerWeights.from_host(synth.layer_weights(wl, 0), "bf16")
    d, ctx, resp = wl.d, [33, 7, 64], [21, 40, 5]
    B, cu, cr = len(ctx), np.concatenate([[0], np.cumsum(np.add(ctx, resp))]), np.concatenate([[0], np.cumsum(resp)])
    T, R = int(cu[-1]), int(cr[-1])
    dims = S.make_dims(d, wl.n_heads, wl.head_dim, wl.d_ff, rope_theta=rope)
    n = S.seer_layer_workspace_size(dims, "bf16", T, B)
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((T, d), generator=g, device="cuda").bfloat16()
    xr = torch.cat([x[int(a) + c:int(b)] for a, b, c in zip(cu[:-1], cu[1:], ctx)])
    out = []
    for place in (lambda t: t, at_16):
        ws = place(torch.zeros(n, dtype=torch.uint8, device="cuda"))
        y = place(torch.zeros((T, d), dtype=torch.bfloat16, device="cuda"))
        S.seer_layer_forward(W.struct(), dims, "bf16", place(x), y, i32(cu), None, B, T, None, 0, 0.0, None, ws, n)
        got = [y]
        if not rope:                                                   # the cache path has no rotary embedding
            cache = place(torch.zeros((T, 2 * d), dtype=torch.float16, device="cuda"))
            yr = place(torch.zeros((R, d), dtype=torch.bfloat16, device="cuda"))
            S.seer_kv_prefill(W.struct(), dims, "bf16", place(x), i32(cu), i32(ctx), B, T, cache, i32(cu), T, ws, n)
            S.seer_layer_forward_cached(W.struct(), dims, "bf16", place(xr), yr, i32(cr), i32(ctx), B, R, cache, i32(cu),
                                        None, T, ws, n)
            got += [cache, yr]
        out.append(got)
    assert all(torch.equal(p, q) for p, q in zip(*out))
    assert all(t.any() for t in out[0])


def test_cache_entry_points_reject_bad_arguments():
    x = torch.zeros((8, 256), dtype=torch.bfloat16, device=cuda())
    cu = i32([0, 8])
    with pytest.raises(RuntimeError):
        S.seer_gather_response(x, "bf16", cu, None, 1, 256, 8, x, cu)
    dims = S.make_dims(256, 2, 128, 768, rope_theta=1e4)
    w = S.seer_layer_weights()
    with pytest.raises(RuntimeError):
        S.seer_layer_forward_cached(w, dims, "bf16", x, x, cu, cu, 1, 8, x, cu, None, 8, x, 0)
