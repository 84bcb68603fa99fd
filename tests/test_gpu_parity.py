"""CUDA path vs CPU oracle, element by element, through the C ABI (needs a B200)."""
import numpy as np
import pytest

from oracle import innerq_oracle as O
from paper_2602_23200_b200 import synth
from tests import _parity as P

pytestmark = pytest.mark.gpu


def _torch():
    import torch
    return torch


def gpu_cache(w, max_tokens=None, **opts):
    from paper_2602_23200_b200 import binding as B
    cfg = B.make_config(w, max_tokens=max_tokens or w.n_tokens + 300)
    return B.InnerQCache(cfg)


def dev(x):
    torch = _torch()
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def run_prefill_both(w, max_tokens=None):
    K, V = synth.kv_all(w)
    oc = O.from_workload(w, max_tokens=max_tokens or w.n_tokens + 300)
    oc.prefill(K, V)
    gc = gpu_cache(w, max_tokens)
    gc.innerq_quantize_prefill(dev(K), dev(V))
    return oc, gc, K, V


def check_decode(w, oc, gc, step=0, variants=(0,), splits=(0,)):
    q = synth.query(w, step)
    ref = oc.decode(q)
    worst = 0.0
    for variant in variants:
        for s in splits:
            gc.innerq_set_decode_options(s, variant)
            out = gc.innerq_decode_attention(dev(q)).cpu().numpy()
            worst = max(worst, P.assert_outputs_close(out, ref, f"{w.name} variant={variant} splits={s}"))
    gc.innerq_set_decode_options(0, 0)
    assert gc.innerq_read_device_error() == 0      # no bounded wait inside a kernel ever ran out
    return worst


CASES = [
    # bits, G, mode, sym_variant, N
    (2, 32, O.HYBRID, 0, 333),
    (2, 32, O.HYBRID, 1, 333),
    (2, 64, O.ASYM, 0, 420),
    (2, 128, O.HYBRID, 0, 700),
    (3, 32, O.HYBRID, 0, 333),
    (3, 64, O.SYM, 0, 300),
    (4, 64, O.HYBRID, 0, 420),
    (4, 32, O.SYM, 1, 333),
    (4, 128, O.ASYM, 0, 541),
]


# The merge of the splits: in a cluster (up to 16 CTAs a unit, 148 together, or pairs; eight parts a round) and through tickets.
@pytest.mark.parametrize("heads,r,kb,vb,G,N,splits", [
    (1, 4, 2, 2, 32, 4700, (1, 2, 7, 8, 9, 15, 16, 17)), (1, 1, 2, 2, 32, 4700, (2, 8, 9, 16, 17)),
    (2, 8, 3, 4, 64, 2400, (1, 3, 8)), (37, 1, 4, 4, 32, 1500, (4, 5)), (37, 2, 4, 2, 32, 1500, (4, 5)),
    (100, 1, 2, 2, 64, 1400, (2, 3)),      # pairs of CTAs that fill the GPU
])
def test_merge_of_splits(heads, r, kb, vb, G, N, splits):
    w = synth.tiny(n_tokens=N, group=G, k_bits=kb, v_bits=vb, batch=1, n_kv_heads=heads, n_q_heads=heads * r)
    oc, gc, _, _ = run_prefill_both(w)
    check_decode(w, oc, gc, splits=(0,) + splits)


# What the extension module does not take goes to the binding's general forms: a subclass, a stream that is given, tensors
# that are refused, a cache that has been closed.
def test_step_calls_outside_the_extension():
    torch = _torch()
    w = synth.tiny(n_tokens=200)
    _, gc, _, _ = run_prefill_both(w)
    q = dev(synth.query(w, 0))
    ref = gc.innerq_decode_attention(q)
    assert torch.equal(gc.innerq_decode_attention(torch.nn.Parameter(q, requires_grad=False)), ref)
    assert torch.equal(gc.innerq_decode_attention(q, stream=torch.cuda.current_stream()), ref)
    out = torch.empty_like(ref)
    assert gc.innerq_decode_attention(q, out) is out and torch.equal(out, ref)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        other = gc.innerq_decode_attention(q)
    torch.cuda.synchronize()
    assert torch.equal(other, ref)
    k = torch.zeros((w.batch, w.n_kv_heads, 128), dtype=torch.float16, device="cuda")
    for bad, err in ((q.float(), TypeError), (q.cpu(), TypeError), (q[:, :, ::2], TypeError), (q[:1], ValueError), (None, TypeError)):
        with pytest.raises(err):
            gc.innerq_decode_attention(bad)
    for bad, err in ((k.float(), TypeError), (k[:, :1], (TypeError, ValueError)), (3, TypeError)):
        with pytest.raises(err):
            gc.innerq_append_token(k, bad)
    with pytest.raises(ValueError):
        gc.innerq_quantize_prefill(torch.zeros((w.batch, w.n_kv_heads + 1, 8, 128), dtype=torch.float16, device="cuda"), k)
    gc.close()
    with pytest.raises(Exception):
        gc.innerq_decode_attention(q)
    with pytest.raises(Exception):
        gc.innerq_append_token(k, k)


# The same for the outer-grouped cache: clusters of up to 16 CTAs, tickets with 17, pairs that fill the GPU.
@pytest.mark.parametrize("heads,r,bits,G,N,splits", [(2, 4, 2, 32, 4200, (0, 1, 2, 9, 15, 16, 17)), (1, 4, 4, 64, 2400, (0, 3, 4)),
                                                     (100, 4, 4, 32, 700, (0, 2, 3))])
def test_merge_of_splits_outer(heads, r, bits, G, N, splits):
    w = synth.tiny(n_tokens=N, group=G, k_bits=bits, v_bits=bits, batch=1, n_kv_heads=heads, n_q_heads=heads * r, grouping=O.OUTER,
                   k_normalize=0, k_mode=O.ASYM, v_mode=O.ASYM)
    oc, gc, _, _ = run_prefill_both(w)
    check_decode(w, oc, gc, splits=splits)


# Batched launches that merge in clusters, where the short sequences' CTAs leave before the long ones' have worked.
@pytest.mark.parametrize("kw", [dict(), dict(k_bits=4, v_bits=4, group=64), dict(n_q_heads=2),
                                dict(grouping=O.OUTER, k_normalize=0, k_mode=O.ASYM, v_mode=O.ASYM)], ids=["2bit", "4bit_g64", "one_row", "outer"])
def test_batched_clusters_with_sequences_of_few_rows(kw):
    from paper_2602_23200_b200 import binding as B
    base = synth.tiny(**dict(dict(batch=1, n_q_heads=8, n_kv_heads=2), **kw))
    ws, ocs, gcs = [], [], []
    for i, n in enumerate([30, 2080, 300, 900]):
        w = base.with_(n_tokens=n, wid=base.wid + 900 + i)
        oc, gc, _, _ = run_prefill_both(w, max_tokens=2400)
        ws.append(w); ocs.append(oc); gcs.append(gc)
    for order in ([0, 1, 2, 3], [1, 3, 0], [2, 0], [0, 2, 3, 1]):
        q = np.stack([synth.query(ws[i], 5 + i) for i in order])
        q_d = dev(q)
        outs = [B.innerq_decode_attention_batched([gcs[i] for i in order], q_d) for _ in range(3)]
        for out in outs:
            for row, i in enumerate(order):
                P.assert_outputs_close(out[row].cpu().numpy(), ocs[i].decode(q[row]), f"sequence {i} of {order}")
    assert all(gc.innerq_read_device_error() == 0 for gc in gcs)


@pytest.mark.parametrize("bits,G,mode,variant,N", CASES)
def test_prefill_and_decode_inner(bits, G, mode, variant, N):
    w = synth.tiny(n_tokens=N, group=G, k_bits=bits, v_bits=bits, k_mode=mode, v_mode=mode, sym_variant=variant)
    oc, gc, _, _ = run_prefill_both(w)
    P.assert_export_equal(gc.innerq_cache_export(), oc.export(), O.INNER, G, mode == O.HYBRID, mode == O.HYBRID)
    check_decode(w, oc, gc, variants=(0, 1, 3, 4), splits=(0, 1, 3, 7))


# Edges of the prefill quantisers: nothing / one row / one batch of 8 rows more or less quantised, one group more or
# less, numbers of (unit, group) items that the CTAs do not divide evenly, caches without key norms, and values far from
# zero in narrow groups (shift), whose rounded zero-point pushes codes out of range so that the clamping paths run.
@pytest.mark.parametrize("kb,vb,G,N,batch,heads,norm,variant,shift", [
    (2, 2, 32, 20, 1, 1, 1, 0, 0.0), (2, 2, 32, 21, 1, 3, 1, 0, 0.0), (3, 3, 32, 28, 1, 1, 1, 0, 0.0),
    (4, 4, 32, 29, 5, 1, 1, 0, 0.0), (2, 3, 32, 52, 1, 37, 1, 0, 0.0), (3, 2, 64, 83, 1, 5, 1, 0, 0.0),
    (4, 2, 64, 84, 3, 3, 1, 0, 0.0), (2, 4, 128, 148, 1, 7, 1, 0, 0.0), (3, 4, 128, 275, 1, 1, 1, 0, 0.0),
    (2, 2, 32, 333, 1, 2, 0, 0, 0.0), (4, 3, 128, 2117, 1, 1, 0, 0, 0.0),
    (2, 2, 32, 333, 1, 2, 1, 0, 700.0), (3, 3, 64, 333, 1, 2, 1, 1, -700.0), (4, 4, 128, 333, 1, 2, 0, 0, 700.0),
    (2, 4, 32, 333, 1, 2, 0, 1, 3.0), (4, 2, 64, 9001, 1, 1, 1, 0, 0.0),
])
def test_prefill_edges(kb, vb, G, N, batch, heads, norm, variant, shift):
    w = synth.tiny(n_tokens=N, group=G, k_bits=kb, v_bits=vb, batch=batch, n_kv_heads=heads, n_q_heads=heads, k_normalize=norm,
                   sym_variant=variant)
    K, V = synth.kv_all(w)
    if shift:
        K, V = (K * np.float16(0.1) + np.float16(shift)), (V * np.float16(0.1) + np.float16(shift))
    oc = O.from_workload(w, max_tokens=N + 300)
    gc = gpu_cache(w)
    for _ in range(2):                     # the second prefill runs over the first one's workspace and cache
        oc.prefill(K, V)
        gc.innerq_quantize_prefill(dev(K), dev(V))
        P.assert_export_equal(gc.innerq_cache_export(), oc.export(), O.INNER, G, True, True)
        K, V = np.ascontiguousarray(K[..., ::-1, :]), np.ascontiguousarray(V[..., ::-1, :])


# Groups whose mode the quantisers' quick error sums cannot tell (both errors zero or equal: zero and constant runs, two
# levels) among ordinary ones, with values from a pointer that is only 4-byte aligned (no windows, whose copies need 16).
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("G", [32, 64, 128])
def test_prefill_groups_with_equal_errors(bits, G):
    torch = _torch()
    N, heads = 5 * 128, 3      # (no remainder: nothing of V in a window)
    w = synth.tiny(n_tokens=N, group=G, k_bits=bits, v_bits=bits, batch=1, n_kv_heads=heads, n_q_heads=heads, w_sink=0, w_recent=0)
    K, V = synth.kv_all(w)
    for X in (K, V):
        X[:, 0, 100:300] = 0
        X[:, 1, :, 40:72] = 0
        X[:, 2, 256:] = np.where(X[:, 2, 256:] > 0, np.float16(2), np.float16(-2))
    V[:, 1, :, 5] = 1.5
    oc = O.from_workload(w, max_tokens=N + 300)
    oc.prefill(K, V)
    gc = gpu_cache(w)
    shifted = torch.empty(V.size + 8, dtype=torch.float16, device="cuda")
    shifted[2:2 + V.size] = dev(V).reshape(-1)
    for v in (dev(V), shifted[2:2 + V.size].view(V.shape)):
        gc.innerq_quantize_prefill(dev(K), v)
        P.assert_export_equal(gc.innerq_cache_export(), oc.export(), O.INNER, G, True, True)


# A group with a NaN or an infinity among values of one sign (which alone would be asymmetric): no sum tells its mode, it is
# symmetric, whether a prompt or an append packs it.
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("G", [32, 64, 128])
def test_prefill_and_append_agree_on_groups_that_are_not_finite(bits, G):
    N = 4 * 128
    w = synth.tiny(n_tokens=N + 16, group=G, k_bits=bits, v_bits=bits, batch=1, n_kv_heads=2, n_q_heads=2, w_sink=0, w_recent=16,
                   k_normalize=0)
    rng = np.random.default_rng(bits * G)
    K, V = (rng.uniform(5, 7, (1, 2, N + 16, 128)).astype(np.float16) for _ in range(2))
    special = [(x, t, c) for x, t in ((np.nan, 3), (-np.nan, 70), (np.inf, 200), (-np.inf, 331)) for c in (0, 37, 65, 126)]
    for x, t, c in special:
        K[0, 0, t, c] = V[0, 1, t + c // 2, c] = x
    K[0, 1, 400, 96:] = np.nan                 # nothing but NaN
    a, b = gpu_cache(w), gpu_cache(w)
    a.innerq_quantize_prefill(dev(K), dev(V))
    b.innerq_quantize_prefill(dev(K[:, :, :0]), dev(V[:, :, :0]))
    k, v = dev(K.transpose(2, 0, 1, 3)), dev(V.transpose(2, 0, 1, 3))
    for t in range(N + 16):
        b.innerq_append_token(k[t], v[t])
    a, b = a.innerq_cache_export(), b.innerq_cache_export()
    for name, X in (("k", K[0, :, :N].reshape(2, N, 128 // G, G)), ("v", V[0, :, :N].reshape(2, N // G, G, 128).swapaxes(2, 3))):
        symmetric = (a[f"{name}_scale"] & 0x8000) == 0
        assert np.array_equal(symmetric, ~np.isfinite(X).all(-1)), name
        assert np.array_equal(symmetric, (b[f"{name}_scale"] & 0x8000) == 0), name
        keep = np.isfinite(X).all(-1)
        assert np.array_equal(a[f"{name}_scale"][keep], b[f"{name}_scale"][keep]), name


# The same in the modes without a choice, and the literal symmetric formula: a NaN leaves the scale to the group's numbers.
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("mode,variant", [(O.SYM, 0), (O.ASYM, 0), (O.HYBRID, 1)])
@pytest.mark.parametrize("G", [32, 128])
def test_prefill_and_append_agree_on_scales_of_groups_with_a_nan(bits, mode, variant, G):
    N = 3 * 128
    w = synth.tiny(n_tokens=N + 16, group=G, k_bits=bits, v_bits=bits, batch=1, n_kv_heads=2, n_q_heads=2, w_sink=0, w_recent=16,
                   k_normalize=0, k_mode=mode, v_mode=mode, sym_variant=variant)
    rng = np.random.default_rng(bits + G)
    K, V = (rng.normal(0, 3, (1, 2, N + 16, 128)).astype(np.float16) for _ in range(2))
    for t, c in ((3, 0), (70, 37), (70, 38), (200, 65), (383, 127)):
        K[0, t & 1, t, c] = V[0, t & 1, t, c] = np.nan
    V[0, 0, 128:256, 9] = np.nan               # nothing but NaN
    a, b = gpu_cache(w), gpu_cache(w)
    a.innerq_quantize_prefill(dev(K), dev(V))
    b.innerq_quantize_prefill(dev(K[:, :, :0]), dev(V[:, :, :0]))
    k, v = dev(K.transpose(2, 0, 1, 3)), dev(V.transpose(2, 0, 1, 3))
    for t in range(N + 16):
        b.innerq_append_token(k[t], v[t])
    a, b = a.innerq_cache_export(), b.innerq_cache_export()
    for name, X in (("k", K[0, :, :N].reshape(2, N, 128 // G, G)), ("v", V[0, :, :N].reshape(2, N // G, G, 128).swapaxes(2, 3))):
        nan = np.isnan(X)
        groups = ~nan.all(-1)
        if mode == O.HYBRID:                   # (of the others, ones with nearly equal errors may go either way)
            groups &= nan.any(-1)
        assert groups.any()
        for part in ("scale", "zero"):
            assert np.array_equal(a[f"{name}_{part}"][groups], b[f"{name}_{part}"][groups]), (name, part)


# The fp16 windows: fewer tokens than the sink holds, nothing but windows, windows of no, one and many tokens, and unit
# counts at which a thread's next piece is units further on or less than a unit's pieces away.
@pytest.mark.parametrize("grouping", [O.INNER, O.OUTER, O.FP16])
@pytest.mark.parametrize("batch,heads,N,w_sink,w_recent", [(1, 2, 3, 4, 16), (1, 1, 4, 4, 0), (37, 8, 1, 4, 16), (41, 8, 150, 4, 130),
                                                           (1, 2, 700, 5, 300), (2, 3, 900, 0, 1), (1, 1, 2500, 4, 2048)])
def test_prefill_windows(grouping, batch, heads, N, w_sink, w_recent):
    inner = grouping == O.INNER
    w = synth.tiny(n_tokens=N, batch=batch, n_kv_heads=heads, n_q_heads=heads, w_sink=w_sink, w_recent=w_recent, grouping=grouping,
                   k_normalize=int(inner), **({} if inner else dict(k_mode=O.ASYM, v_mode=O.ASYM)))
    oc, gc, K, V = run_prefill_both(w, max_tokens=N + 40)
    for _ in range(2):                     # the second prefill runs over the first one's windows
        e = gc.innerq_cache_export()
        if grouping == O.FP16:
            for name, x in (("k_sink", K), ("v_sink", V)):
                np.testing.assert_array_equal(np.asarray(e[name])[:, :N].view(np.float16), x.reshape(-1, N, 128))
        else:
            P.assert_export_equal(e, oc.export(), grouping, w.group, k_hybrid=inner, v_hybrid=inner)
        K, V = K[..., ::-1, :].copy(), V[..., ::-1, :].copy()
        oc.prefill(K, V)
        gc.innerq_quantize_prefill(dev(K), dev(V))


@pytest.mark.parametrize("bits,G,N", [(2, 32, 333), (3, 64, 420), (4, 128, 541)])
def test_prefill_and_decode_outer(bits, G, N):
    w = synth.tiny(n_tokens=N, group=G, k_bits=bits, v_bits=bits, grouping=O.OUTER, k_normalize=0,
                   k_mode=O.ASYM, v_mode=O.ASYM)
    oc, gc, _, _ = run_prefill_both(w)
    P.assert_export_equal(gc.innerq_cache_export(), oc.export(), O.OUTER, G, False, False)
    check_decode(w, oc, gc, splits=(0, 2))


@pytest.mark.parametrize("bits,G,r,N", [(2, 32, 1, 700), (2, 64, 4, 600), (2, 128, 2, 900), (4, 32, 4, 500),
                                        (4, 64, 8, 555), (4, 128, 1, 1300)])
def test_outer_grouped_fused_kernel(bits, G, r, N):
    # the outer-grouped comparison cache on the fused kernel (variant 3 refuses to fall back), against the generic
    # kernel (variant 1) and the oracle; then appends through the reversed skew zone (packed values, fp16 keys)
    w = synth.tiny(n_tokens=N, group=G, k_bits=bits, v_bits=bits, grouping=O.OUTER, k_normalize=0, k_mode=O.ASYM,
                   v_mode=O.ASYM, n_q_heads=2 * r)
    oc, gc, _, _ = run_prefill_both(w)
    P.assert_export_equal(gc.innerq_cache_export(), oc.export(), O.OUTER, G, False, False)
    check_decode(w, oc, gc, variants=(3, 1), splits=(0, 2, 5))
    for step in range(G + 5):
        k1, v1 = synth.new_token(w, step)
        oc.append(k1, v1)
        gc.innerq_append_token(dev(k1), dev(v1))
        if step in (0, 1, 15, 16, 17, G - 1, G, G + 4):
            check_decode(w, oc, gc, step=step, variants=(3,), splits=(0, 3))
    P.assert_export_equal(gc.innerq_cache_export(), oc.export(), O.OUTER, G, False, False)


@pytest.mark.parametrize("N,mode", [(700, O.HYBRID), (1333, O.ASYM), (164, O.HYBRID), (37, O.HYBRID)])
def test_one_query_head_per_kv_head_kernel_instance(N, mode):
    # 2-bit, G = 32, one query head per KV head: the instance of the fused kernel whose tensor-core columns are
    # (channel group, digit), against the oracle and the generic kernel, for several split counts, one and two chunks
    # per loop iteration, and through appends that cross a value-group eviction
    w = synth.tiny(n_tokens=N, group=32, n_q_heads=2, k_mode=mode, v_mode=mode)
    oc, gc, _, _ = run_prefill_both(w)
    check_decode(w, oc, gc, variants=(2, 3, 4, 1), splits=(0, 1, 3))
    for step in range(40):
        k1, v1 = synth.new_token(w, step)
        oc.append(k1, v1)
        gc.innerq_append_token(dev(k1), dev(v1))
        if step in (0, 7, 31, 32, 39):
            check_decode(w, oc, gc, step=step, variants=(3, 4), splits=(0, 2))



def test_fp16_cache_decode():
    w = synth.tiny(n_tokens=500, grouping=O.FP16, k_normalize=0)
    oc, gc, K, V = run_prefill_both(w)
    e = gc.innerq_cache_export()
    assert e["n_tokens"] == 500 and np.array_equal(e["k_sink"].reshape(K.shape), K)
    check_decode(w, oc, gc, splits=(0, 1, 5))
    for step in range(3):
        k1, v1 = synth.new_token(w, step)
        oc.append(k1, v1)
        gc.innerq_append_token(dev(k1), dev(v1))
    check_decode(w, oc, gc, step=1)


def test_mixed_bits_and_modes():
    w = synth.tiny(n_tokens=400, group=32, k_bits=3, v_bits=2, k_mode=O.SYM, v_mode=O.HYBRID)
    oc, gc, _, _ = run_prefill_both(w)
    P.assert_export_equal(gc.innerq_cache_export(), oc.export(), O.INNER, 32, False, True)
    check_decode(w, oc, gc, variants=(0, 1, 3))


# key bits, value bits, key mode, value mode, G, query heads per KV head, N: packed formats of the fused kernel
# beyond equal-width hybrid ones (3-bit planes, symmetric-only 2-byte metadata, keys and values of different widths
# or metadata forms), with one query head per KV head (group-per-column kernel), several, and two passes of four
FORMATS = [
    (3, 3, O.HYBRID, O.HYBRID, 32, 1, 700),
    (3, 3, O.SYM, O.SYM, 32, 1, 700),
    (3, 2, O.SYM, O.SYM, 32, 1, 600),
    (3, 2, O.SYM, O.HYBRID, 32, 1, 1500),
    (3, 2, O.SYM, O.HYBRID, 64, 4, 600),
    (3, 2, O.SYM, O.SYM, 128, 2, 900),
    (2, 2, O.SYM, O.SYM, 128, 2, 900),
    (4, 4, O.SYM, O.SYM, 32, 1, 500),
    (3, 3, O.ASYM, O.ASYM, 128, 8, 900),
    (3, 3, O.SYM, O.SYM, 64, 8, 555),
    # keys and values of different widths, and 2-bit caches whose two tensors differ in metadata form
    (2, 4, O.HYBRID, O.HYBRID, 32, 1, 700),
    (4, 2, O.HYBRID, O.ASYM, 64, 4, 600),
    (2, 3, O.SYM, O.HYBRID, 32, 2, 500),
    (4, 3, O.HYBRID, O.SYM, 128, 4, 900),
    (3, 4, O.SYM, O.SYM, 64, 1, 450),
    (2, 2, O.SYM, O.HYBRID, 32, 1, 1200),
    (2, 2, O.HYBRID, O.SYM, 64, 4, 640),
]


@pytest.mark.parametrize("kb,vb,km,vm,G,r,N", FORMATS)
def test_fused_kernel_formats(kb, vb, km, vm, G, r, N):
    w = synth.tiny(n_tokens=N, group=G, k_bits=kb, v_bits=vb, k_mode=km, v_mode=vm, n_q_heads=2 * r)
    oc, gc, _, _ = run_prefill_both(w)
    P.assert_export_equal(gc.innerq_cache_export(), oc.export(), O.INNER, G, km == O.HYBRID, vm == O.HYBRID)
    check_decode(w, oc, gc, variants=(3, 1), splits=(0, 2, 5))       # 3: the fused kernel or an error, 1: generic kernel
    for step in range(G + 3):                                          # across a value-group eviction
        k1, v1 = synth.new_token(w, step)
        oc.append(k1, v1)
        gc.innerq_append_token(dev(k1), dev(v1))
    check_decode(w, oc, gc, step=7, variants=(3,), splits=(0, 3))
    # what the appends packed (one row per step, one value group on the way), bit for bit
    P.assert_export_equal(gc.innerq_cache_export(), oc.export(), O.INNER, G, km == O.HYBRID, vm == O.HYBRID)


def test_a_bounded_wait_that_runs_out_is_reported_and_leaves_the_context_usable():
    # The decode kernels wait for their asynchronous copies a bounded number of times and, if a wait runs out, set
    # the cache's device error word and return.  The self-test kernel takes that road on purpose: the kernels' own
    # wait routine, on a barrier nothing ever arrives on.  No fault, no hang: the kernel gives up after 256 polls.
    w = synth.tiny(n_tokens=300)
    oc, gc, _, _ = run_prefill_both(w)
    check_decode(w, oc, gc)                                   # error word still 0 (asserted there)
    gc.innerq_selftest_wait_expiry()
    assert gc.innerq_read_device_error() == 1                 # the expiry is reported ...
    assert gc.innerq_read_device_error() == 1                 # ... for good: the word is sticky
    q = synth.query(w, 3)
    out = gc.innerq_decode_attention(dev(q)).cpu().numpy()    # ... and the context and the cache still work
    P.assert_outputs_close(out, oc.decode(q), "after a wait that ran out")
    # another cache has its own error word
    _, g2, _, _ = run_prefill_both(w)
    assert g2.innerq_read_device_error() == 0


@pytest.mark.parametrize("N", [1, 3, 4, 5, 19, 20, 21, 52, 53])
def test_short_contexts_and_window_edges(N):
    # N <= w_sink, N <= w_sink + w_recent (nothing quantised), first quantised key token, first value group
    w = synth.tiny(n_tokens=N)
    oc, gc, K, V = run_prefill_both(w)
    e, eo = gc.innerq_cache_export(), oc.export()
    P.assert_export_equal(e, eo, O.INNER, w.group)
    check_decode(w, oc, gc, variants=(0, 1))
    if N <= w.w_sink + w.w_recent:
        # every token is in a window: the result is plain attention on the fp16 inputs
        q = synth.query(w)
        out = gc.innerq_decode_attention(dev(q)).cpu().numpy()
        for b in range(w.batch):
            for j in range(w.n_q_heads):
                h = j // w.q_per_kv
                ref = O.dense_attention(q[b, j], K[b, h], V[b, h])
                P.assert_outputs_close(out[b, j][None], ref[None], "all-window")


def test_empty_prefill_then_appends_through_every_phase():
    # start from an empty cache; append through sink fill, recent fill, first key eviction, value evictions
    w = synth.tiny(n_tokens=0, w_sink=4, w_recent=16, group=32)
    oc = O.from_workload(w, max_tokens=200)
    gc = gpu_cache(w, max_tokens=200)
    torch = _torch()
    gc.innerq_quantize_prefill(torch.empty((w.batch, w.n_kv_heads, 0, 128), dtype=torch.float16, device="cuda"),
                               torch.empty((w.batch, w.n_kv_heads, 0, 128), dtype=torch.float16, device="cuda"))
    for step in range(120):
        k1, v1 = synth.new_token(w, step)
        oc.append(k1, v1)
        gc.innerq_append_token(dev(k1), dev(v1))
        if step in (0, 3, 4, 19, 20, 21, 51, 52, 83, 84, 119):
            P.assert_export_equal(gc.innerq_cache_export(), oc.export(), O.INNER, w.group)
            check_decode(w, oc, gc, step=step, variants=(0, 1))


@pytest.mark.parametrize("grouping", [O.INNER, O.OUTER])
def test_prefill_then_appends_matches_oracle(grouping):
    w = synth.tiny(n_tokens=150, grouping=grouping, k_normalize=int(grouping == O.INNER), append_scale=0.5,
                   k_mode=O.HYBRID if grouping == O.INNER else O.ASYM,
                   v_mode=O.HYBRID if grouping == O.INNER else O.ASYM)
    oc, gc, _, _ = run_prefill_both(w)
    for step in range(100):
        k1, v1 = synth.new_token(w, step)
        oc.append(k1, v1)
        gc.innerq_append_token(dev(k1), dev(v1))
        if step % 33 == 32:
            check_decode(w, oc, gc, step=step)
    P.assert_export_equal(gc.innerq_cache_export(), oc.export(), grouping, w.group,
                          grouping == O.INNER, grouping == O.INNER)
    check_decode(w, oc, gc, step=1000, variants=(0, 1) if grouping == O.INNER else (0,))


def test_step_from_host_buffers_matches_separate_calls_and_oracle():
    # innerq_decode_step_host = copies in + append + decode + copy out; across a value-group eviction
    torch = _torch()
    w = synth.tiny(n_tokens=300, k_bits=3, v_bits=2, k_mode=O.SYM, v_mode=O.HYBRID)
    oc, gc, K, V = run_prefill_both(w)
    gc2 = gpu_cache(w)
    gc2.innerq_quantize_prefill(dev(K), dev(V))
    out_h = torch.empty((w.batch, w.n_q_heads, 128), dtype=torch.float16).pin_memory()
    for step in range(40):
        k1, v1 = synth.new_token(w, step)
        q = synth.query(w, step)
        oc.append(k1, v1)
        pin = (lambda t: t.pin_memory()) if step % 2 == 0 else (lambda t: t)    # in-place over the bus / staged copies
        gc.innerq_decode_step_host(pin(torch.from_numpy(k1)), pin(torch.from_numpy(v1)), pin(torch.from_numpy(q)), out_h)
        torch.cuda.synchronize()
        gc2.innerq_append_token(dev(k1), dev(v1))
        ref2 = gc2.innerq_decode_attention(dev(q)).cpu()
        assert torch.equal(out_h, ref2)                       # same kernels, same inputs: identical bits
        if step % 13 == 0 or step == 39:
            P.assert_outputs_close(out_h.numpy(), oc.decode(q), f"host step {step}")
    P.assert_export_equal(gc.innerq_cache_export(), oc.export(), O.INNER, w.group, False, True)
    assert gc.n_tokens == 340


@pytest.mark.parametrize("r,G,bits", [(3, 64, 2), (6, 32, 4), (5, 128, 3), (16, 64, 2)])
def test_query_heads_per_kv_head_not_a_multiple_of_four(r, G, bits):
    # the fused kernel takes up to four query heads of a KV head per pass: partial and multiple passes
    w = synth.tiny(n_tokens=450, group=G, k_bits=bits, v_bits=bits, n_q_heads=2 * r)
    oc, gc, _, _ = run_prefill_both(w)
    check_decode(w, oc, gc, variants=(3, 4, 1), splits=(0, 2))


@pytest.mark.parametrize("w_sink,w_recent", [(0, 0), (0, 7), (5, 0)])
def test_degenerate_windows(w_sink, w_recent):
    # no sink and / or no recent window: every token (w_recent = 0: even the newest) is quantised
    w = synth.tiny(n_tokens=230, w_sink=w_sink, w_recent=w_recent)
    oc, gc, _, _ = run_prefill_both(w)
    P.assert_export_equal(gc.innerq_cache_export(), oc.export(), O.INNER, w.group)
    check_decode(w, oc, gc, variants=(0, 1))
    for step in range(40):
        k1, v1 = synth.new_token(w, step)
        oc.append(k1, v1)
        gc.innerq_append_token(dev(k1), dev(v1))
        if step in (0, 1, 25, 26, 39):
            check_decode(w, oc, gc, step=step, variants=(0, 1))
    P.assert_export_equal(gc.innerq_cache_export(), oc.export(), O.INNER, w.group)


@pytest.mark.parametrize("grouping,r,G,bits,n_q", [(O.INNER, 1, 32, 2, 4), (O.INNER, 1, 32, 2, 7), (O.INNER, 4, 64, 2, 3),
                                                    (O.INNER, 2, 128, 4, 5), (O.INNER, 1, 64, 3, 9), (O.OUTER, 1, 32, 2, 6),
                                                    (O.OUTER, 4, 64, 4, 2)])
def test_multi_query_decode(grouping, r, G, bits, n_q):
    # n_q query tokens per sequence against one cache state, causal among the newest n_q tokens; rows of a KV
    # head share passes over the packed cache four at a time
    inner = grouping == O.INNER
    w = synth.tiny(batch=2, n_q_heads=2 * r, n_kv_heads=2, n_tokens=4 + 20 * 32 + 77, group=G, k_bits=bits, v_bits=bits,
                   w_sink=4, w_recent=24, grouping=grouping, k_normalize=int(inner),
                   **({} if inner else dict(k_mode=O.ASYM, v_mode=O.ASYM)))
    oc, gc, _, _ = run_prefill_both(w)
    for step in range(3):                 # a few appended tokens, so the ring buffers are rotated
        k1, v1 = synth.new_token(w, step)
        oc.append(k1, v1)
        gc.innerq_append_token(dev(k1), dev(v1))
    q = np.stack([synth.query(w, 10 + i) for i in range(n_q)], axis=1)           # [B, n_q, Hq, D]
    ref = oc.decode_multi(q)
    for splits in (0, 1, 3):
        gc.innerq_set_decode_options(splits, 0)
        out = gc.innerq_decode_attention_multi(dev(q)).cpu().numpy()
        P.assert_outputs_close(out, ref, f"multi-query n_q={n_q} splits={splits}")
    gc.innerq_set_decode_options(0, 0)
    # the newest query row is the plain decode of the same cache
    one = gc.innerq_decode_attention(dev(q[:, n_q - 1])).cpu().numpy()
    P.assert_outputs_close(one, ref[:, n_q - 1], "newest query = single-token decode")
    assert gc.innerq_read_device_error() == 0


# Several groups of four query rows in one launch (and, beyond eight groups, in several): query heads and query tokens, key
# rows whose length falls and rises by 2^+-10 along the context: peaked and flat parts of the context in one range, scores
# far above and below the range's soft-max reference.  (Renewed references: test_rows_that_share_a_launch_lose_no_precision.)
@pytest.mark.parametrize("r,n_q,G,kb,vb,N", [(8, 1, 32, 2, 2, 3001), (9, 1, 64, 3, 3, 2900), (16, 1, 128, 4, 4, 3001),
                                             (4, 5, 32, 4, 2, 3001), (4, 9, 64, 2, 2, 2500), (1, 33, 128, 2, 2, 3001),
                                             (5, 3, 32, 3, 2, 700), (8, 2, 64, 4, 3, 150)])
@pytest.mark.parametrize("grouping", [O.INNER, O.OUTER])
def test_many_query_rows_in_one_launch(grouping, r, n_q, G, kb, vb, N):
    if grouping == O.OUTER:
        kb = vb = 2 if kb < 4 else 4
    w = synth.tiny(n_tokens=N, group=G, k_bits=kb, v_bits=vb, batch=1, n_kv_heads=2, n_q_heads=2 * r, w_recent=64, grouping=grouping,
                   k_normalize=int(grouping == O.INNER), **({} if grouping == O.INNER else dict(k_mode=O.ASYM, v_mode=O.ASYM)))
    K, V = synth.kv_all(w)
    K = (K * np.exp2(10.0 * np.cos(np.arange(N) / 300.0) - 8.0)[None, None, :, None]).astype(np.float16)
    oc, gc = O.from_workload(w, max_tokens=N + 300), gpu_cache(w)
    oc.prefill(K, V)
    gc.innerq_quantize_prefill(dev(K), dev(V))
    q = np.stack([synth.query(w, i) for i in range(n_q)], axis=1)
    ref = oc.decode_multi(q)
    for _ in range(2):
        out = gc.innerq_decode_attention_multi(dev(q)) if n_q > 1 else gc.innerq_decode_attention(dev(q[:, 0]))[:, None]
        P.assert_outputs_close(out.cpu().numpy(), ref, f"r={r} n_q={n_q}")
    assert gc.innerq_read_device_error() == 0


@pytest.fixture(scope="module")
def split_plan(tmp_path_factory):
    """(passes, splits, splits of one group alone, iterations between two references with one / two chunks each) of a call
    with automatic splits, from the library's own arithmetic."""
    import os
    import subprocess
    here = os.path.dirname(os.path.abspath(__file__))
    exe = str(tmp_path_factory.mktemp("split") / "host_split_check")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(here, "..", "paper_2602_23200_b200", "csrc"), "-o", exe,
                    os.path.join(here, "host_split_check.cpp")], check=True)

    def plan(w, n_q):
        args = (w.batch * w.n_kv_heads, w.n_q_heads // w.n_kv_heads, n_q, w.w_sink, w.w_recent, w.group, w.n_tokens,
                int(w.grouping == O.OUTER))
        out = subprocess.run([exe, *map(str, args)], check=True, capture_output=True, text=True).stdout
        return tuple(int(x) for x in out.split())
    return plan


# Groups of query rows that share a launch have longer ranges per warp than a launch of one group, whose 16 bits of p are
# relative to the range's soft-max reference: the references are renewed, and the error against the oracle's 64 bits is no
# larger than with one launch per group (which the split count of one group asks for).  Key rows whose length rises and
# falls by 2^+-3 along the context move the references both ways.  2 %: over n outputs (8192 and more) the norm of a random
# error varies by 1 / sqrt(2 n), 0.8 % or less.
RENEWED = [  # grouping, bits, G, batch, KV heads, r, n_q, N, paged
    (O.OUTER, 4, 128, 1, 2, 4, 8, 65536, False), (O.OUTER, 2, 32, 1, 4, 4, 8, 20000, False), (O.OUTER, 4, 64, 1, 2, 4, 8, 40000, True),
    # G = 32 with one chunk per iteration (as one group alone takes there) and with two, then three value group sizes
    (O.INNER, 2, 32, 2, 8, 4, 8, 8192, False), (O.INNER, 2, 32, 5, 8, 16, 1, 8000, False), (O.INNER, 2, 64, 2, 8, 4, 5, 16384, True),
    (O.INNER, 4, 64, 1, 8, 4, 5, 16384, False), (O.INNER, 3, 128, 1, 8, 4, 5, 16384, False), (O.INNER, 2, 128, 3, 8, 8, 1, 16384, False),
]


@pytest.mark.parametrize("grouping,bits,G,batch,hkv,r,n_q,N,paged", RENEWED)
def test_rows_that_share_a_launch_lose_no_precision(split_plan, grouping, bits, G, batch, hkv, r, n_q, N, paged):
    from paper_2602_23200_b200 import binding as B
    inner = grouping == O.INNER
    w = synth.tiny(batch=batch, n_q_heads=hkv * r, n_kv_heads=hkv, n_tokens=N, group=G, k_bits=bits, v_bits=bits, w_recent=128,
                   grouping=grouping, k_normalize=int(inner), **({} if inner else dict(k_mode=O.ASYM, v_mode=O.ASYM)))
    passes, splits, alone, reset, _ = split_plan(w, n_q)
    assert passes > 1 and splits < alone and reset > 0, "the case has to reach the renewed references"
    K, V = synth.kv_all(w)
    K = (K * np.exp2(3.0 * np.cos(np.arange(N) / 300.0) - 3.0)[None, None, :, None]).astype(np.float16)
    oc = O.from_workload(w)
    oc.prefill(K, V)
    cfg = B.make_config(w, max_tokens=N)
    gc = B.InnerQCache(cfg, pool=B.PagePool(cfg, 512, N // 512 + 1)) if paged else B.InnerQCache(cfg)
    gc.ensure_pages(N)
    gc.innerq_quantize_prefill(dev(K), dev(V))
    q = np.stack([synth.query(w, i) for i in range(n_q)], axis=1)
    ref = oc.decode_multi(q)
    err = []
    for n_splits in (alone, 0):
        gc.innerq_set_decode_options(n_splits, 0)
        out = (gc.innerq_decode_attention_multi(dev(q)) if n_q > 1 else gc.innerq_decode_attention(dev(q[:, 0]))[:, None]).cpu().numpy()
        P.assert_outputs_close(out, ref, f"n_splits={n_splits}")
        err.append(float(np.linalg.norm(out.astype(np.float64) - ref) / np.linalg.norm(ref)))
    print(f"error alone {err[0]:.3e}, together {err[1]:.3e}")
    assert err[1] <= 1.02 * err[0], err
    assert gc.innerq_read_device_error() == 0


# Many units with short windows: a unit has fewer split partials (7) than the call has groups of query rows (8).
@pytest.mark.parametrize("grouping", [O.INNER, O.OUTER])
def test_multi_query_over_many_units(grouping):
    inner = grouping == O.INNER
    w = synth.tiny(batch=128, n_q_heads=16, n_kv_heads=4, n_tokens=230, group=32, w_sink=4, w_recent=64, grouping=grouping,
                   k_normalize=int(inner), **({} if inner else dict(k_mode=O.ASYM, v_mode=O.ASYM)))
    oc, gc, _, _ = run_prefill_both(w)
    q = np.stack([synth.query(w, i) for i in range(8)], axis=1)
    ref = oc.decode_multi(q)
    for splits in (0, 1):
        gc.innerq_set_decode_options(splits, 0)
        P.assert_outputs_close(gc.innerq_decode_attention_multi(dev(q)).cpu().numpy(), ref, f"512 units, splits={splits}")
    assert gc.innerq_read_device_error() == 0


def test_multi_query_short_contexts_and_limits():
    from paper_2602_23200_b200 import binding as B
    # everything in the windows: even sink tokens are masked by position
    w = synth.tiny(n_tokens=11, w_sink=4, w_recent=16)
    oc, gc, _, _ = run_prefill_both(w)
    for n_q in (1, 2, 6, 11):
        q = np.stack([synth.query(w, i) for i in range(n_q)], axis=1)
        out = gc.innerq_decode_attention_multi(dev(q)).cpu().numpy()
        P.assert_outputs_close(out, oc.decode_multi(q), f"windows only, n_q={n_q}")
    q12 = np.stack([synth.query(w, i) for i in range(12)], axis=1)
    with pytest.raises(B.InnerQError) as ei:              # more query tokens than cached tokens
        gc.innerq_decode_attention_multi(dev(q12))
    assert ei.value.status == -1
    # hidden tokens would reach into the chunks where keys and values are both packed: refused, nothing launched
    w = synth.tiny(n_tokens=4 + 64 + 8, w_sink=4, w_recent=8)
    oc, gc, _, _ = run_prefill_both(w)
    e = oc.export()
    room = w.n_tokens - e["n_sink"] - min(e["n_qk"], e["n_qv"])       # tokens that can be hidden
    q_ok = np.stack([synth.query(w, i) for i in range(room + 1)], axis=1)
    P.assert_outputs_close(gc.innerq_decode_attention_multi(dev(q_ok)).cpu().numpy(), oc.decode_multi(q_ok), "at the limit")
    q_bad = np.stack([synth.query(w, i) for i in range(room + 2)], axis=1)
    with pytest.raises(B.InnerQError) as ei:
        gc.innerq_decode_attention_multi(dev(q_bad))
    assert ei.value.status == -2
    # an unquantised cache has no fused kernel: refused as well
    wf = synth.tiny(n_tokens=40, grouping=O.FP16, k_normalize=0)
    _, gf, _, _ = run_prefill_both(wf)
    with pytest.raises(B.InnerQError) as ei:
        gf.innerq_decode_attention_multi(dev(np.stack([synth.query(wf, i) for i in range(2)], axis=1)))
    assert ei.value.status == -2


@pytest.mark.parametrize("grouping,r,G,bits", [(O.INNER, 1, 32, 2), (O.INNER, 4, 64, 2), (O.INNER, 2, 128, 4), (O.INNER, 1, 32, 3),
                                               (O.OUTER, 2, 32, 2)])
def test_batched_calls_over_sequences_of_different_lengths(grouping, r, G, bits):
    # every sequence has its own cache object and length; one launch appends to / decodes all of them
    from paper_2602_23200_b200 import binding as B
    inner = grouping == O.INNER
    lengths = [1, 37, 164, 700, 333, 4 + 16 + G]
    base = synth.tiny(batch=1, n_q_heads=2 * r, n_kv_heads=2, group=G, k_bits=bits, v_bits=bits, grouping=grouping,
                      k_normalize=int(inner), **({} if inner else dict(k_mode=O.ASYM, v_mode=O.ASYM)))
    ws, ocs, gcs = [], [], []
    for i, n in enumerate(lengths):
        w = base.with_(n_tokens=n, wid=base.wid + 100 + i)
        oc, gc, _, _ = run_prefill_both(w, max_tokens=1000)
        ws.append(w); ocs.append(oc); gcs.append(gc)

    def decode_all(step, who=None):
        who = list(range(len(gcs))) if who is None else who
        q = np.stack([synth.query(ws[i], step) for i in who])                      # [n, 1, Hq, D]
        out = B.innerq_decode_attention_batched([gcs[i] for i in who], dev(q)).cpu().numpy()
        for row, i in enumerate(who):
            P.assert_outputs_close(out[row], ocs[i].decode(q[row]), f"sequence {i} (N={ocs[i].N}) step {step}")

    decode_all(0)
    for step in range(2 * G + 3):                   # every sequence crosses group evictions at its own steps
        who = [i for i in range(len(gcs)) if not (i == 2 and step % 3 == 0)]       # sequence 2 skips some steps
        toks = [synth.new_token(ws[i], step) for i in who]
        for (k1, v1), i in zip(toks, who):
            ocs[i].append(k1, v1)
        B.innerq_append_token_batched([gcs[i] for i in who], dev(np.stack([t[0] for t in toks])),
                                      dev(np.stack([t[1] for t in toks])))
        if step in (0, 1, G - 1, G, 2 * G + 2):
            decode_all(step + 1)
            decode_all(step + 1, who=[3, 0])                                        # any subset, any order
    for i, (oc, gc) in enumerate(zip(ocs, gcs)):
        assert gc.n_tokens == oc.N
        P.assert_export_equal(gc.innerq_cache_export(), oc.export(), grouping, G, k_hybrid=inner, v_hybrid=inner)
        assert gc.innerq_read_device_error() == 0
    # a single-cache call on one of them still agrees
    q = synth.query(ws[4], 99)
    P.assert_outputs_close(gcs[4].innerq_decode_attention(dev(q)).cpu().numpy(), ocs[4].decode(q), "single after batched")


def test_batched_calls_with_caches_that_hold_a_batch_themselves():
    # every cache object may itself hold several sequences of one length: rows of k_new / q are [cache][batch, ...]
    from paper_2602_23200_b200 import binding as B
    base = synth.tiny(batch=3, n_q_heads=4, n_kv_heads=2, group=64)
    ws, ocs, gcs = [], [], []
    for i, n in enumerate([90, 333, 200]):
        w = base.with_(n_tokens=n, wid=base.wid + 700 + i)
        oc, gc, _, _ = run_prefill_both(w, max_tokens=500)
        ws.append(w); ocs.append(oc); gcs.append(gc)
    for step in range(70):
        toks = [synth.new_token(w, step) for w in ws]
        for (k1, v1), oc in zip(toks, ocs):
            oc.append(k1, v1)
        B.innerq_append_token_batched(gcs, dev(np.stack([t[0] for t in toks])), dev(np.stack([t[1] for t in toks])))
        if step in (0, 63, 64, 69):
            q = np.stack([synth.query(w, step) for w in ws])                     # [3, batch, Hq, D]
            out = B.innerq_decode_attention_batched(gcs, dev(q)).cpu().numpy()
            for i in range(3):
                P.assert_outputs_close(out[i], ocs[i].decode(q[i]), f"cache {i} step {step}")
    for w, oc, gc in zip(ws, ocs, gcs):
        P.assert_export_equal(gc.innerq_cache_export(), oc.export(), O.INNER, w.group)


def test_result_is_a_plain_contiguous_tensor_whatever_the_query_is():
    # a query may be a tensor subclass, or carry any stride on a dimension of one element; the result does not inherit it
    import torch
    from paper_2602_23200_b200 import binding as B

    class Sub(torch.Tensor):
        pass

    w = synth.tiny(batch=1, n_q_heads=4, n_kv_heads=2, n_tokens=60)
    oc, gc, _, _ = run_prefill_both(w)
    q0 = dev(synth.query(w, 0))
    want = gc.innerq_decode_attention(q0)
    for q in (q0.as_subclass(Sub), torch.nn.Parameter(q0, requires_grad=False), torch.as_strided(q0, q0.shape, (0, 128, 1)),
              torch.stack([q0, q0], 1)[:, 0]):
        for out in (gc.innerq_decode_attention(q), B.innerq_decode_attention_batched([gc], q.unsqueeze(0))[0]):
            assert type(out) is torch.Tensor and out.stride() == (4 * 128, 128, 1) and not out.requires_grad
            assert torch.equal(out, want)


def test_general_forms_give_what_the_extension_module_gives():
    import torch
    w = synth.tiny(batch=2, n_q_heads=4, n_kv_heads=2, n_tokens=400)
    K, V = (dev(x) for x in synth.kv_all(w))
    a, b = gpu_cache(w), gpu_cache(w)
    assert a._steps is not None
    b._steps = None
    host = [torch.empty((2, 4, 128), dtype=torch.float16).pin_memory() for _ in range(2)]
    for c in (a, b):
        c.innerq_quantize_prefill(K, V)
    for step in range(40):
        k1, v1, q = (torch.from_numpy(x).pin_memory() for x in (*synth.new_token(w, step), synth.query(w, step)))
        if step % 3 == 2:
            for c, out in zip((a, b), host):
                c.innerq_decode_step_host(k1, v1, q, out)
            torch.cuda.synchronize()
            assert torch.equal(*host), step
        else:
            for c in (a, b):
                c.innerq_append_token(k1.cuda(), v1.cuda())
            given = torch.empty((2, 4, 128), dtype=torch.float16, device="cuda")
            out = a.innerq_decode_attention(q.cuda())
            assert b.innerq_decode_attention(q.cuda(), given) is given and torch.equal(out, given), step
            assert torch.equal(a.innerq_decode_attention(q.cuda(), given), b.innerq_decode_attention(q.cuda())), step
    a, b = a.innerq_cache_export(), b.innerq_cache_export()
    assert all(np.array_equal(a[key], b[key]) for key in a)


def test_exception_behind_the_extension_module_leaves_the_interpreter_whole(tmp_path):
    # an entry point that throws: the call is left to the general forms, with the interpreter's lock held again
    import subprocess
    import sys
    (tmp_path / "boom.cpp").write_text('#include <stdexcept>\nextern "C" int boom() { throw std::runtime_error("boom"); }\n')
    so = str(tmp_path / "boom.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-o", so, str(tmp_path / "boom.cpp")], check=True)
    code = f"""
import ctypes, torch
from paper_2602_23200_b200 import binding as B
boom = ctypes.cast(ctypes.CDLL({so!r}).boom, ctypes.c_void_p).value
kv, q = (1, 2, 128), (1, 4, 128)
steps = B._load_steps()(0, torch.cuda.current_device(), kv, q, boom, boom, boom, boom)
k, query = (torch.zeros(s, dtype=torch.float16, device="cuda") for s in (kv, q))
for _ in range(3):
    got = [steps.append(k, k), steps.decode(query, None), steps.decode(query, query), steps.prefill(k[:, :, None], k[:, :, None]),
           steps.step_host(k.cpu(), k.cpu(), query.cpu(), query.cpu(), 4096)]
    assert got == [1] * 5, got
print("whole")
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "whole", r.stderr


def test_batched_calls_argument_checks():
    from paper_2602_23200_b200 import binding as B
    w = synth.tiny(batch=1, n_q_heads=2, n_kv_heads=2, n_tokens=50)
    _, a, _, _ = run_prefill_both(w, max_tokens=51)
    _, b, _, _ = run_prefill_both(w, max_tokens=51)
    _, other, _, _ = run_prefill_both(w.with_(group=64), max_tokens=51)
    q2 = dev(np.stack([synth.query(w, 0), synth.query(w, 1)]))
    k1, v1 = synth.new_token(w, 0)
    kv2 = dev(np.stack([k1, k1])), dev(np.stack([v1, v1]))
    for bad in ([a, a], [a, other]):                       # the same cache twice; different configurations
        with pytest.raises(B.InnerQError) as ei:
            B.innerq_decode_attention_batched(bad, q2)
        assert ei.value.status == -1
        with pytest.raises(B.InnerQError) as ei:
            B.innerq_append_token_batched(bad, *kv2)
        assert ei.value.status == -1
    B.innerq_append_token_batched([a], dev(k1[None]), dev(v1[None]))           # a is full now (51 of 51)
    with pytest.raises(B.InnerQError) as ei:
        B.innerq_append_token_batched([b, a], *kv2)
    assert ei.value.status == -3 and b.n_tokens == 50 and a.n_tokens == 51      # nothing was appended to b either
    wf = w.with_(grouping=O.FP16, k_normalize=0)
    _, f, _, _ = run_prefill_both(wf, max_tokens=51)
    with pytest.raises(B.InnerQError) as ei:
        B.innerq_decode_attention_batched([f], dev(synth.query(wf, 0)[None]))
    assert ei.value.status == -2
    out = B.innerq_decode_attention_batched([b, a], q2)
    assert _torch().isfinite(out.float()).all()


def test_batched_calls_with_more_caches_than_one_launch_takes():
    from paper_2602_23200_b200 import binding as B
    n = 37                                                  # a launch takes 32: two launches
    base = synth.tiny(batch=1, n_q_heads=2, n_kv_heads=1)
    ws, ocs, gcs = [], [], []
    for i in range(n):
        w = base.with_(n_tokens=20 + 13 * i, wid=base.wid + 300 + i)
        oc, gc, _, _ = run_prefill_both(w, max_tokens=600)
        ws.append(w); ocs.append(oc); gcs.append(gc)
    toks = [synth.new_token(ws[i], 0) for i in range(n)]
    for (k1, v1), oc in zip(toks, ocs):
        oc.append(k1, v1)
    B.innerq_append_token_batched(gcs, dev(np.stack([t[0] for t in toks])), dev(np.stack([t[1] for t in toks])))
    assert gcs[0].innerq_last_launch_count(1) == 2
    q = np.stack([synth.query(ws[i], 1) for i in range(n)])
    out = B.innerq_decode_attention_batched(gcs, dev(q)).cpu().numpy()
    for i in range(n):
        assert gcs[i].n_tokens == ocs[i].N
        P.assert_outputs_close(out[i], ocs[i].decode(q[i]), f"sequence {i} of {n}")


@pytest.mark.parametrize("grouping,r,G", [(O.INNER, 1, 32), (O.INNER, 4, 64), (O.OUTER, 2, 32)])
def test_steps_enqueued_back_to_back_without_host_synchronisation(grouping, r, G):
    # The kernels of consecutive steps overlap on the GPU (each is a programmatic dependent of the one before it and
    # the decode streams the settled part of the cache before it waits): enqueue many steps with no host
    # synchronisation in between, then check every step's output and the final cache against the oracle.
    torch = _torch()
    inner = grouping == O.INNER
    w = synth.tiny(batch=2, n_q_heads=4 * r, n_kv_heads=4, n_tokens=4 + 16 + 40 * 32 + 11, group=G, grouping=grouping,
                   k_normalize=int(inner), **({} if inner else dict(k_mode=O.ASYM, v_mode=O.ASYM)))
    n_steps = 2 * G + 9
    oc, gc, _, _ = run_prefill_both(w, max_tokens=w.n_tokens + n_steps + 4)
    toks = [synth.new_token(w, s) for s in range(n_steps)]
    qs = [synth.query(w, s) for s in range(n_steps)]
    k_all, v_all = dev(np.stack([t[0] for t in toks])), dev(np.stack([t[1] for t in toks]))
    q_all = dev(np.stack(qs))
    outs = torch.empty_like(q_all)
    torch.cuda.synchronize()
    for s in range(n_steps):                       # nothing here waits for the GPU
        gc.innerq_append_token(k_all[s], v_all[s])
        gc.innerq_decode_attention(q_all[s], outs[s])
        if s % 7 == 3:                             # some steps decode twice, some append twice in a row
            gc.innerq_decode_attention(q_all[s], outs[s])
    torch.cuda.synchronize()
    got = outs.cpu().numpy()
    for s in range(n_steps):
        oc.append(*toks[s])
        P.assert_outputs_close(got[s], oc.decode(qs[s]), f"step {s}")
    P.assert_export_equal(gc.innerq_cache_export(), oc.export(), grouping, G, k_hybrid=inner, v_hybrid=inner)
    assert gc.innerq_read_device_error() == 0


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_random_interleaving_of_calls_on_one_stream(seed):
    # Three caches of different formats share one stream; appends, decodes (fused and plain kernels), multi-query
    # decodes and exports are enqueued in random order with no host synchronisation except at exports.  Every output is
    # checked afterwards: the overlap of consecutive kernels must never let a decode miss an append.
    torch = _torch()
    rng = np.random.default_rng(seed)
    specs = [dict(n_q_heads=4, n_kv_heads=4, group=32, k_bits=2, v_bits=2, w_recent=16),
             dict(n_q_heads=8, n_kv_heads=2, group=64, k_bits=4, v_bits=4, w_recent=24),
             dict(n_q_heads=4, n_kv_heads=2, group=32, k_bits=2, v_bits=2, w_recent=16, grouping=O.OUTER, k_normalize=0,
                  k_mode=O.ASYM, v_mode=O.ASYM)]
    ws, ocs, gcs, steps = [], [], [], []
    pool = 160                                     # inputs are put on the device up front: no copy between the calls
    toks, qs, toks_d, qs_d = [], [], [], []
    for i, kw in enumerate(specs):
        w = synth.tiny(batch=1, n_tokens=4 + kw["w_recent"] + 60 * 32 + 5 * i, wid=500 + 10 * seed + i, **kw)
        oc, gc, _, _ = run_prefill_both(w, max_tokens=w.n_tokens + pool + 8)
        ws.append(w); ocs.append(oc); gcs.append(gc); steps.append(0)
        toks.append([synth.new_token(w, s_) for s_ in range(pool)])
        qs.append([synth.query(w, 1000 + s_) for s_ in range(pool)])
        toks_d.append((dev(np.stack([t[0] for t in toks[i]])), dev(np.stack([t[1] for t in toks[i]]))))
        qs_d.append(dev(np.stack(qs[i])))
    torch.cuda.synchronize()
    # 1. the sequence of calls (multi-query is always possible here: the recent window holds at least 16 tokens)
    ops = []
    n_queries = [0] * len(gcs)
    for it in range(300):
        i = int(rng.integers(len(gcs)))
        op = str(rng.choice(["append", "append", "decode", "decode", "plain", "multi"], p=[.3, .2, .25, .1, .05, .1]))
        if op == "append":
            if steps[i] >= pool:
                continue
            ops.append((op, i, steps[i], 0)); steps[i] += 1
        elif op == "multi":
            n_q = int(rng.integers(2, 5))
            ops.append((op, i, n_queries[i] % (pool - 4), n_q)); n_queries[i] += n_q
        else:
            ops.append((op, i, n_queries[i] % pool, 0)); n_queries[i] += 1
    # 2. everything is enqueued without the host ever waiting for the GPU
    outs = []
    for op, i, j, n_q in ops:
        gc = gcs[i]
        if op == "append":
            gc.innerq_append_token(toks_d[i][0][j], toks_d[i][1][j])
            outs.append(None)
        elif op == "multi":
            outs.append(gc.innerq_decode_attention_multi(qs_d[i][j:j + n_q].transpose(0, 1).contiguous()))
        else:
            gc.innerq_set_decode_options(0, 1 if op == "plain" else 0)
            outs.append(gc.innerq_decode_attention(qs_d[i][j]))
            gc.innerq_set_decode_options(0, 0)
    torch.cuda.synchronize()
    # 3. the oracle goes through the same sequence
    for (op, i, j, n_q), out in zip(ops, outs):
        oc = ocs[i]
        if op == "append":
            oc.append(*toks[i][j])
        elif op == "multi":
            P.assert_outputs_close(out.cpu().numpy(), oc.decode_multi(np.stack(qs[i][j:j + n_q], axis=1)), f"multi, cache {i}")
        else:
            P.assert_outputs_close(out.cpu().numpy(), oc.decode(qs[i][j]), f"{op}, cache {i}")
    for i, gc in enumerate(gcs):
        w = ws[i]
        assert gc.n_tokens == ocs[i].N and gc.innerq_read_device_error() == 0
        P.assert_export_equal(gc.innerq_cache_export(), ocs[i].export(), w.grouping, w.group,
                              k_hybrid=w.k_mode == O.HYBRID, v_hybrid=w.v_mode == O.HYBRID)


@pytest.mark.parametrize("seed", [1, 2, 3, 4])
def test_prefills_between_steps_on_one_stream(seed):
    # A prefill's kernels overlap their neighbours (the first is a programmatic dependent of whatever runs before it, the second
    # lets its dependents start at once): prefills of two prompts each, appends and decodes of three caches in random order and
    # in the orders where little lies between two calls of a cache, nothing of it synchronised with the host.
    torch = _torch()
    rng = np.random.default_rng(100 + seed)
    specs = [dict(n_q_heads=4, n_kv_heads=4, group=32, k_bits=2, v_bits=2, w_recent=16),
             dict(n_q_heads=8, n_kv_heads=2, group=64, k_bits=4, v_bits=3, w_recent=24),
             dict(n_q_heads=4, n_kv_heads=2, group=32, k_bits=2, v_bits=2, w_recent=16, grouping=O.OUTER, k_normalize=0,
                  k_mode=O.ASYM, v_mode=O.ASYM)]
    pool, n_prompts = 60, 3
    ws, ocs, gcs, prompts, toks, qs, on_gpu = [], [], [], [], [], [], []
    for i, kw in enumerate(specs):
        lengths = [int(n) for n in rng.integers(30, 2500, n_prompts - 1)] + [4 + kw["w_recent"] + 20 * 32 + 5 * i]
        w = synth.tiny(batch=1, n_tokens=max(lengths), wid=700 + 10 * seed + i, **kw)
        K, V = synth.kv_all(w)
        ws.append(w)
        ocs.append(O.from_workload(w, max_tokens=w.n_tokens + 300))
        gcs.append(gpu_cache(w))
        prompts.append([(np.ascontiguousarray(K[:, :, -n:]), np.ascontiguousarray(V[:, :, -n:])) for n in lengths])
        toks.append([synth.new_token(w, s) for s in range(pool)])
        qs.append([synth.query(w, s) for s in range(pool)])
        on_gpu.append(([(dev(k), dev(v)) for k, v in prompts[i]], dev(np.stack([t[0] for t in toks[i]])),
                       dev(np.stack([t[1] for t in toks[i]])), dev(np.stack(qs[i]))))
    ops = [("prefill", i, int(rng.integers(n_prompts))) for i in range(3)]
    close = ["PA PB aB dB dA", "dA PB aA dA", "PA PA aA dA", "aA dA PA dA aA", "PA aB dB aA dA", "PA PB PC dC dB dA", "dB dA PA aB dB"]
    for it in range(24):
        names = dict(zip("ABC", rng.permutation(3)))
        ops += [({"P": "prefill", "a": "append", "d": "decode"}[c[0]], int(names[c[1]]), int(rng.integers(n_prompts)))
                for c in str(rng.choice(close)).split()]
        for _ in range(int(rng.integers(6))):
            ops.append((str(rng.choice(["append", "append", "decode", "decode", "prefill"])), int(rng.integers(3)),
                        int(rng.integers(n_prompts))))
    count = [0, 0, 0]
    ops = [(op, i, j if op == "prefill" else (count.__setitem__(i, count[i] + 1) or count[i] % pool)) for op, i, j in ops]
    torch.cuda.synchronize()
    outs = []
    for op, i, j in ops:
        prompt, k, v, q = on_gpu[i]
        if op == "prefill":
            gcs[i].innerq_quantize_prefill(*prompt[j])
        elif op == "append":
            gcs[i].innerq_append_token(k[j], v[j])
        outs.append(gcs[i].innerq_decode_attention(q[j]) if op == "decode" else None)
    torch.cuda.synchronize()
    for n, ((op, i, j), out) in enumerate(zip(ops, outs)):
        if op == "prefill":
            ocs[i].prefill(*prompts[i][j])
        elif op == "append":
            ocs[i].append(*toks[i][j])
        else:
            P.assert_outputs_close(out.cpu().numpy(), ocs[i].decode(qs[i][j]), f"call {n}, cache {i}")
    for w, oc, gc in zip(ws, ocs, gcs):
        assert gc.n_tokens == oc.N and gc.innerq_read_device_error() == 0
        P.assert_export_equal(gc.innerq_cache_export(), oc.export(), w.grouping, w.group,
                              k_hybrid=w.k_mode == O.HYBRID, v_hybrid=w.v_mode == O.HYBRID)


def test_capacity_and_argument_errors():
    from paper_2602_23200_b200 import binding as B
    torch = _torch()
    w = synth.tiny(n_tokens=40)
    gc = gpu_cache(w, max_tokens=41)
    K, V = synth.kv_all(w)
    gc.innerq_quantize_prefill(dev(K), dev(V))
    k1, v1 = synth.new_token(w, 0)
    gc.innerq_append_token(dev(k1), dev(v1))
    with pytest.raises(B.InnerQError) as ei:
        gc.innerq_append_token(dev(k1), dev(v1))
    assert ei.value.status == -3 and gc.n_tokens == 41
    K2, V2 = synth.kv_all(w.with_(n_tokens=42))
    with pytest.raises(B.InnerQError) as ei:
        gc.innerq_quantize_prefill(dev(K2), dev(V2))
    assert ei.value.status == -3 and gc.n_tokens == 41
    empty = gpu_cache(w, max_tokens=41)
    q = dev(synth.query(w))
    with pytest.raises(B.InnerQError) as ei:
        empty.innerq_decode_attention(q)
    assert ei.value.status == -1
    # the context is still healthy
    out = gc.innerq_decode_attention(q)
    assert torch.isfinite(out.float()).all()


def test_config1_full_parity():
    w = synth.config1()
    oc, gc, _, _ = run_prefill_both(w)
    flips = P.assert_export_equal(gc.innerq_cache_export(), oc.export(), O.INNER, w.group)
    worst = check_decode(w, oc, gc, variants=(0, 1, 3, 4), splits=(0, 1, 4, 13))
    print(f"config1: contested flips {flips}, worst err/tol {worst:.3f}")


@pytest.mark.parametrize("kw", [dict(), dict(group=64, k_bits=3, v_bits=3, n_q_heads=8), dict(k_bits=4, v_bits=2, k_mode=O.SYM),
                                dict(grouping=O.OUTER, k_normalize=0, k_mode=O.ASYM, v_mode=O.ASYM, group=64),
                                dict(grouping=O.FP16, k_normalize=0)],
                         ids=["2bit", "3bit_g64", "k4sym_v2", "outer", "fp16"])
def test_import_restores_an_exported_cache(kw):
    # checkpoint / resume: export a cache that has been prefilled and stepped, import the arrays into a fresh cache of
    # the same configuration: identical export, identical decode output (same bits), and both caches continue alike
    import torch
    w = synth.tiny(n_tokens=500, **kw)
    oc, gc, _, _ = run_prefill_both(w)
    for step in range(w.group + 5):
        k1, v1 = synth.new_token(w, step)
        oc.append(k1, v1)
        gc.innerq_append_token(dev(k1), dev(v1))
    saved = gc.innerq_cache_export()
    g2 = gpu_cache(w)
    g2.innerq_cache_import(saved)
    assert g2.n_tokens == gc.n_tokens
    again = g2.innerq_cache_export()
    for key, val in saved.items():
        assert np.array_equal(np.asarray(val), np.asarray(again[key])), key
    q = dev(synth.query(w, 3))
    assert torch.equal(gc.innerq_decode_attention(q), g2.innerq_decode_attention(q))
    check_decode(w, oc, g2, step=3)
    for step in range(100, 100 + w.group + 2):                 # both continue through another group eviction
        k1, v1 = synth.new_token(w, step)
        oc.append(k1, v1)
        for c in (gc, g2):
            c.innerq_append_token(dev(k1), dev(v1))
    a, b = gc.innerq_cache_export(), g2.innerq_cache_export()
    for key, val in a.items():
        assert np.array_equal(np.asarray(val), np.asarray(b[key])), key
    check_decode(w, oc, g2, step=9)
