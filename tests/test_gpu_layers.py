"""Layers of one stream step (and frames of one chunk) that share their launches: the cache state of
every layer is that of the per-call entry points bit for bit, its output within the attention's
tolerance of theirs (the items are cut at other places, so partial results are merged elsewhere)."""
import numpy as np
import pytest

from paper_2601_01204_b200 import synth
from xkv_testlib import ATTN_MAXABS, ATTN_RELL2, attn_errors, bf16_tensor_to_f32, check_attention, compare_state, oracle_params, to_device_bf16

pytestmark = pytest.mark.gpu

H, D = 3, 64


@pytest.fixture(scope="module")
def xkv():
    import torch
    assert torch.cuda.is_available()
    import paper_2601_01204_b200.xkv as m
    return m


def frame(layer, t, n):
    return [to_device_bf16(b) for b in synth.gen_frame(70 + layer, layer, t, H, n, D)]


def per_call(cache, q, k, v, tail):
    cache.kv_append(k, v)
    cache.kv_score_evict(q)
    cache.kv_quant_pack()
    return cache.attn_packed_causal_tail(q, k, v) if tail else cache.attn_packed_causal(q)


@pytest.mark.parametrize("layers, n, budget, bits, once, tail", [
    (2, 130, 300, 4, 0, False),
    (29, 97, 260, 4, 0, False),          # one more than a launch takes
    (5, 257, 1200, 4, 0, True),
    (5, 140, 700, 4, 1, False),
    (3, 97, 300, 8, 1, False),
    (24, 257, 1030, 16, 0, False),
    (3, 1, 4, 4, 0, False),
])
def test_layers_of_one_step_match_the_calls(xkv, layers, n, budget, bits, once, tail):
    import torch
    p = xkv.Params(n_heads=H, budget=budget, max_frame_tokens=n, kv_bits=bits, key_mode=once)
    together, alone = ([xkv.Cache(p) for _ in range(layers)] for _ in range(2))
    for c in together:
        c.xkv_set_unquantised_tail(tail)
    for t in range(7):
        q, k, v = zip(*(frame(l, t, n) for l in range(layers)))
        out = [torch.empty_like(x) for x in q]
        xkv.xkv_stream_step(together, q, k, v, out)
        for l in range(layers):
            ref = per_call(alone[l], q[l], k[l], v[l], tail)
            check_attention(bf16_tensor_to_f32(out[l]), bf16_tensor_to_f32(ref), f"frame {t} layer {l}")
            compare_state(together[l].export(), alone[l].export(), f"frame {t} layer {l}")
    assert all(c.xkv_poll_status() == 0 for c in together)


def test_step_with_layers_of_different_forms_and_lengths(xkv):
    """Neighbours that cannot share a launch, and layers whose caches have different lengths."""
    import torch
    forms = [(300, 4, 0), (500, 4, 0), (500, 16, 0), (400, 16, 0), (300, 4, 1), (300, 8, 1), (260, 4, 0)]
    mk = lambda: [xkv.Cache(xkv.Params(n_heads=H, budget=b, max_frame_tokens=130, kv_bits=bits, key_mode=o)) for b, bits, o in forms]
    together, alone = mk(), mk()
    for t, n in enumerate([130, 64, 129, 130, 1, 130]):
        q, k, v = zip(*(frame(l, t, n) for l in range(len(forms))))
        out = [torch.empty_like(x) for x in q]
        xkv.xkv_stream_step(together, q, k, v, out)
        for l, c in enumerate(alone):
            ref = per_call(c, q[l], k[l], v[l], False)
            check_attention(bf16_tensor_to_f32(out[l]), bf16_tensor_to_f32(ref), f"frame {t} layer {l}")
            compare_state(together[l].export(), c.export(), f"frame {t} layer {l}")


def test_step_keeps_the_order_of_layers_that_share_memory(xkv):
    """A layer's output that is a later layer's input, one output buffer for all layers, and the same
    cache twice: the results are those of the layers one after the other."""
    import torch
    n = 130
    p = xkv.Params(n_heads=H, budget=300, max_frame_tokens=n, kv_bits=4)
    a, b = [xkv.Cache(p) for _ in range(2)], [xkv.Cache(p) for _ in range(2)]
    for t in range(5):
        (q0, k0, v0), (_, k1, v1), (q2, k2, v2) = (frame(l, t, n) for l in range(3))
        mid, last = torch.empty_like(q0), torch.empty_like(q0)
        xkv.xkv_stream_step([a[0], a[1], a[1]], [q0, mid, q2], [k0, k1, k2], [v0, v1, v2], [mid, last, last])
        m = per_call(b[0], q0, k0, v0, False)
        per_call(b[1], m, k1, v1, False)
        ref = per_call(b[1], q2, k2, v2, False)
        assert torch.equal(mid, m) and torch.equal(last, ref)
        for x, y in zip(a, b):
            compare_state(x.export(), y.export(), f"frame {t}")


def test_step_stops_at_the_first_bad_layer(xkv):
    import torch
    n = 64
    p = xkv.Params(n_heads=H, budget=300, max_frame_tokens=n, kv_bits=4)
    caches = [xkv.Cache(p) for _ in range(3)]
    q, k, v = zip(*(frame(l, 0, n) for l in range(3)))
    out = [torch.zeros_like(x) for x in q]
    caches[1].kv_append(k[1], v[1])                       # out of order for a step
    with pytest.raises(xkv.XkvError) as e:
        xkv.xkv_stream_step(caches, q, k, v, out)
    assert e.value.status == xkv.XKV_E_STATE
    assert [c.xkv_get_info().frames for c in caches] == [1, 0, 0]
    assert out[0].abs().max() > 0 and out[2].abs().max() == 0


def test_chunk_of_more_frames_than_a_launch_takes(xkv):
    from oracle import xkv_oracle as xo
    sizes = [9] * 27 + [1, 30, 7]
    n = sum(sizes)
    p = xkv.Params(n_heads=H, budget=700, max_frame_tokens=n, kv_bits=4)
    cache, ora = xkv.Cache(p), xo.OracleLayer(oracle_params(p))
    for t in range(4):
        bits = synth.gen_frame(5, 0, t, H, n, D)
        got = cache.xkv_prefill_chunk(*(to_device_bf16(b) for b in bits), sizes)
        cuts = np.cumsum(sizes)[:-1]
        ref = ora.step_chunk(*(np.split(synth.bf16_bits_to_f32(b), cuts, axis=1) for b in bits))
        check_attention(bf16_tensor_to_f32(got).transpose(1, 0, 2), np.concatenate(ref), f"chunk {t}")
        compare_state(cache.export(), ora.export(), f"chunk {t}")


@pytest.mark.parametrize("layers, n, budget, bits, once, tail", [
    (5, 1500, 10500, 4, 0, False),       # one layer, two, one, one
    (4, 1400, 10300, 16, 0, False),      # one, two, one
    (6, 1400, 10300, 4, 1, False),
    (4, 1400, 10300, 4, 0, True),        # the tail needs keys and values to the end: one at a time
    (5, 130, 300, 4, 0, False),          # short caches: one at a time
])
def test_host_buffer_step_in_pairs(xkv, layers, n, budget, bits, once, tail):
    """Caches long enough that the host-buffer step takes two layers at a time, with its outputs over
    the queries in the staging buffer, against the step on device tensors."""
    import torch
    p = xkv.Params(n_heads=H, budget=budget, max_frame_tokens=n, kv_bits=bits, key_mode=once)
    host, dev = ([xkv.Cache(p) for _ in range(layers)] for _ in range(2))
    for c in host + dev:
        c.xkv_set_unquantised_tail(tail)
    staging = torch.empty(xkv.xkv_stream_step_host_bytes(p, n), dtype=torch.uint8, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(9)
    for t in range(budget // n + 3):
        q, k, v = ([torch.randn(H, n, D, device="cuda", dtype=torch.bfloat16, generator=gen) for _ in range(layers)] for _ in range(3))
        out = [torch.empty_like(x) for x in q]
        xkv.xkv_stream_step(dev, q, k, v, out)
        hq, hk, hv = ([x.cpu().pin_memory() for x in xs] for xs in (q, k, v))
        ho = [torch.zeros(H, n, D, dtype=torch.bfloat16).pin_memory() for _ in range(layers)]
        xkv.xkv_stream_step_host(host, hq, hk, hv, ho, staging)
        for l in range(layers):
            # Both are within the tolerance of the exact result, so within twice of it of each other
            # (16-bit caches round P to bf16 against reference maxima that differ with the cuts).
            maxabs, rell2 = attn_errors(ho[l].float().numpy(), bf16_tensor_to_f32(out[l]))
            assert maxabs <= 2 * ATTN_MAXABS and rell2 <= 2 * ATTN_RELL2, (t, l, maxabs, rell2)
    for l in range(layers):
        compare_state(host[l].export(), dev[l].export(), f"layer {l}")
    assert all(c.xkv_poll_status() == 0 for c in host + dev)


@pytest.mark.parametrize("once", [0, 1])
def test_one_key_tile_inside_the_unquantised_frame(xkv, once):
    """The newest frame starts inside a key tile, covers the next one and ends inside the one after: only
    the outer two go through the producers' parameter tables.  Against the oracle, then the same launch
    again and again, bit for bit."""
    import torch
    from oracle import xkv_oracle as xo
    heads, n, budget = 16, 261, 1500                      # slots 1362 .. 1622: tiles 10 (from 1280), 11, 12
    p = xkv.Params(n_heads=heads, budget=budget, max_frame_tokens=n, kv_bits=4, key_mode=once)
    cache, ora = xkv.Cache(p), xo.OracleLayer(oracle_params(p))
    for t in range(budget // n + 3):
        bits = synth.gen_frame(17, 0, t, heads, n, D)
        q, k, v = (to_device_bf16(b) for b in bits)
        qf, kf, vf = (synth.bf16_bits_to_f32(b) for b in bits)
        got = per_call(cache, q, k, v, True)
        ora.append(kf, vf), ora.score_evict(qf), ora.quant_pack()
        ref = ora.attend(qf, full_precision_tail=True)
        check_attention(bf16_tensor_to_f32(got).transpose(1, 0, 2), ref, f"frame {t}")
    info = cache.xkv_get_info()
    assert (info.T_phys - n) % 128 and info.T_phys % 128 and info.T_phys // 128 - (info.T_phys - n) // 128 == 2
    first = got.clone()
    for rep in range(40):
        cache.xkv_debug_rewind_attention()
        assert torch.equal(cache.attn_packed_causal_tail(q, k, v, got).view(torch.int16), first.view(torch.int16)), rep
    assert cache.xkv_poll_status() == 0


@pytest.mark.parametrize("failed", [0, 2])
def test_a_failed_cache_does_not_touch_the_others_of_its_launch(xkv, failed):
    """A cache whose status word holds a time-out from before: the layers that share its launches keep
    their results and their status."""
    import torch
    layers, n, budget = 4, 200, 512
    p = xkv.Params(n_heads=H, budget=budget, max_frame_tokens=n, kv_bits=4)
    together, alone = ([xkv.Cache(p) for _ in range(layers)] for _ in range(2))
    together[failed].xkv_debug_timeout_probe()
    assert together[failed].xkv_poll_status() == xkv.XKV_E_TIMEOUT
    for t in range(4):
        q, k, v = zip(*(frame(l, t, n) for l in range(layers)))
        out = [torch.empty_like(x) for x in q]
        xkv.xkv_stream_step(together, q, k, v, out)
        for l in range(layers):
            ref = per_call(alone[l], q[l], k[l], v[l], False)
            check_attention(bf16_tensor_to_f32(out[l]), bf16_tensor_to_f32(ref), f"frame {t} layer {l}")
            compare_state(together[l].export(), alone[l].export(), f"frame {t} layer {l}")
    assert [c.xkv_poll_status() for c in together] == [xkv.XKV_E_TIMEOUT if l == failed else 0 for l in range(layers)]


def test_launches_of_a_step_count_for_every_layer(xkv):
    """A launch that serves several layers counts for each of them and is timed for the first one with
    profiling on, whichever that is."""
    import torch
    layers, n, budget = 4, 97, 300
    caches = [xkv.Cache(xkv.Params(n_heads=H, budget=budget, max_frame_tokens=n, kv_bits=4)) for _ in range(layers)]
    for t in range(5):
        q, k, v = zip(*(frame(l, t, n) for l in range(layers)))
        if t == 4:
            caches[2].xkv_profile_enable(True)
            caches[3].xkv_profile_enable(True)
            before = [c.xkv_get_info().launches for c in caches]
        xkv.xkv_stream_step(caches, q, k, v, [torch.empty_like(x) for x in q])
    # maintenance, regroup, attention, its merge, head means
    assert [c.xkv_get_info().launches - b for c, b in zip(caches, before)] == [5] * layers
    timed, rest = caches[2].xkv_profile_read(), caches[3].xkv_profile_read()
    assert all(timed[name][1] == 1 and timed[name][0] > 0 for name in ("maint", "pack", "attn", "attn_combine", "kbar"))
    assert all(count == 0 for _, count in rest.values())


def test_key_channels_that_are_not_numbers(xkv):
    """The extremes of a key group pass over what is not a number; a channel without any number has the
    empty extremes, in full and in ragged groups alike."""
    import torch
    n = 100                                               # one group of 64, one of 36
    k = to_device_bf16(synth.gen_frame(6, 0, 0, H, n, D)[1])
    some, none = k.clone(), k.clone()
    some[0, ::3, 5] = float("nan")
    none[0, ::3, 5] = k[0, 1, 5]                          # the same extremes in both groups ...
    none[0, 66::3, 5] = k[0, 67, 5]                       # ... from the numbers that are there
    some[:, :, 3] = float("nan")
    params = []
    for x in (some, none):
        cache = xkv.Cache(xkv.Params(n_heads=H, budget=300, max_frame_tokens=n, kv_bits=4))
        cache.kv_append(x, x)
        cache.kv_score_evict(x)
        cache.kv_quant_pack()
        e = cache.export()
        params.append((e["k_s_first"], e["k_z_first"]))
    (s, z), (s_ref, z_ref) = params
    rest = [c for c in range(D) if c != 3]
    assert np.array_equal(s[:, :, rest], s_ref[:, :, rest]) and np.array_equal(z[:, :, rest], z_ref[:, :, rest])
    assert np.all(s[:, :, 3] == -np.inf)                  # (-inf - inf) / 15


@pytest.mark.parametrize("layers", [1, 5])
def test_16bit_weights_are_normalised_as_they_are_multiplied(xkv, layers):
    """The softmax weights of a 16-bit cache are rounded to bf16.  With each rounding error d_i (relative
    variance r2) the output is off by sum w_i d_i (v_i - out) if the weights are divided by the sum of the
    rounded ones, by sum w_i d_i v_i if not: for rows that one key dominates next to nothing against as
    much as the rounding of the output itself.  The bound is the former and the output's rounding, plus
    10 % for the sample."""
    import torch
    heads, n, budget = 8, 211, 6007
    p = xkv.Params(n_heads=heads, budget=budget, max_frame_tokens=n, kv_bits=16)
    caches = [xkv.Cache(p) for _ in range(layers)]
    gen = torch.Generator(device="cuda").manual_seed(3)
    mk = lambda scale: [(scale * torch.randn(heads, n, D, device="cuda", generator=gen)).to(torch.bfloat16) for _ in range(layers)]
    for t in range(budget // n + 2):
        q, k, v = mk(6.0), mk(1.0), mk(1.0)
        out = [torch.empty_like(x) for x in q]
        xkv.xkv_stream_step(caches, q, k, v, out)
    r2 = (2.0 ** -7) ** 2 / 12 * 3 / (8 * np.log(2))      # mean of (ulp^2 / 12) / m^2 over mantissas m, log-uniform in [1, 2)
    for l in (0, layers - 1):
        e = caches[l].export()
        K, V = (torch.from_numpy(e[x]).cuda().double() for x in ("k_val", "v_val"))
        w = torch.softmax(q[l].double() @ K.transpose(1, 2) / 8.0, dim=-1)
        ref = w @ V
        # sum_i w_i^2 |v_i - out|^2 = sum_i w_i^2 (|v_i|^2 - 2 v_i out + |out|^2)
        w2 = w * w
        var = (w2 @ (V * V).sum(-1, keepdim=True)).sum() - 2 * ((w2 @ V) * ref).sum() + (w2.sum(-1) * (ref * ref).sum(-1)).sum()
        rounding = (ref.to(torch.bfloat16).double() - ref).norm() / ref.norm()
        bound = 1.1 * float(torch.sqrt(rounding ** 2 + r2 * var / ref.norm() ** 2))
        err = float((out[l].double() - ref).norm() / ref.norm())
        assert err <= bound, (l, err, bound)


@pytest.mark.parametrize("bits, once", [(4, 0), (4, 1), (16, 0)])
def test_steps_captured_into_graphs(xkv, bits, once):
    """Every step from the third on captured into a graph of its own and launched once: outputs and state of
    the plain steps bit for bit.  Afterwards the caches reset, and others are created, as ever."""
    import torch
    p = xkv.Params(n_heads=H, budget=700, max_frame_tokens=200, kv_bits=bits, key_mode=once)
    graphed, plain = ([xkv.Cache(p) for _ in range(3)] for _ in range(2))
    for t in range(7):
        q, k, v = zip(*(frame(l, t, 200) for l in range(3)))
        outs = [[torch.zeros_like(x) for x in q] for _ in range(2)]
        if t < 3:
            xkv.xkv_stream_step(graphed, q, k, v, outs[0])
        else:
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                xkv.xkv_stream_step(graphed, q, k, v, outs[0])
            graph.replay()
        xkv.xkv_stream_step(plain, q, k, v, outs[1])
        torch.cuda.synchronize()
        for l in range(3):
            assert torch.equal(outs[0][l].view(torch.int16), outs[1][l].view(torch.int16)), (t, l)
            compare_state(graphed[l].export(), plain[l].export(), f"frame {t} layer {l}")
    assert graphed[0].xkv_get_info().last_evicted > 0
    graphed[0].xkv_reset()
    for c in graphed[1:]:
        c.close()
    again = [graphed[0], xkv.Cache(p)]
    fresh = [xkv.Cache(p) for _ in range(2)]
    q, k, v = zip(*(frame(l, 0, 200) for l in range(2)))
    for caches in (again, fresh):
        xkv.xkv_stream_step(caches, q, k, v, [torch.empty_like(x) for x in q])
    for a, b in zip(again, fresh):
        compare_state(a.export(), b.export(), "after the graphs")
