"""GPU: pa_prefill_backward (dQ, dK, dV) against the fp64 oracle's gradients of Eq. (1), element by
element.  The forward pass that feeds it (O, LSE) is the library's own."""
import numpy as np
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu

# bf16 operands (P and dS are rounded to bf16 before their second product), fp32 accumulation and
# fp32 outputs: the same bounds as for the forward output, relative to the largest gradient entry
# when that exceeds one.
G_MAX_ABS = 2e-2
G_MEAN_ABS = 2e-3


@pytest.fixture(scope="module")
def pa():
    import paper_2503_03588_b200 as pa_

    return pa_


def _compare(got, ref, what):
    got = got.double().cpu().numpy()
    assert got.shape == ref.shape and np.isfinite(got).all(), what
    unit = max(1.0, float(np.abs(ref).max()))
    err = np.abs(got - ref)
    assert err.max() <= G_MAX_ABS * unit, (what, float(err.max()), unit)
    assert err.mean() <= G_MEAN_ABS * unit, (what, float(err.mean()), unit)
    return float(err.max()), float(err.mean())


def _run(pa, oracle, N, Hq, Hkv, D, W, S, batch=1, use_power=True, k_scale=1.0, scale=0.0, seed=0):
    Q = si.bf16_randn((batch, N, Hq, D), 1000 + seed)
    K = si.bf16_randn((batch, N, Hkv, D), 1001 + seed, k_scale)
    V = si.bf16_randn((batch, N, Hkv, D), 1002 + seed)
    dO = si.bf16_randn((batch, N, Hq, D), 1003 + seed)
    rp, ci = oracle.block_layout(N, 64, W, S, use_power=use_power)
    rp, ci = torch.as_tensor(rp).cuda(), torch.as_tensor(ci).cuda()
    Qd, Kd, Vd, dOd = Q.cuda(), K.cuda(), V.cuda(), dO.cuda()
    o, lse, ws = pa.pa_prefill(Qd, Kd, Vd, rp, ci, softmax_scale=scale)
    pa.pa_prefill_status(ws)
    dq, dk, dv, wsb = pa.pa_prefill_backward(Qd, Kd, Vd, o, lse, dOd, rp, ci, softmax_scale=scale)
    pa.pa_prefill_status(wsb)   # the backward workspace starts with the same status block; synchronises
    rq, rk, rv = oracle.backward(Q, K, V, dO, 64, W, S, scale=scale if scale else None, use_power=use_power)
    what = f"N={N} Hq={Hq} Hkv={Hkv} D={D} W={W} S={S}"
    return [_compare(g, r, f"{n} {what}") for g, r, n in ((dq, rq, "dQ"), (dk, rk, "dK"), (dv, rv, "dV"))]


@pytest.mark.parametrize("N,Hq,Hkv,D,W,S", [
    (64, 2, 2, 64, 5, 1),        # one block
    (1, 2, 1, 128, 5, 1),        # one token
    (200, 4, 2, 128, 5, 1),      # ragged tail
    (1000, 7, 1, 128, 5, 1),     # a 7-head group
    (1536, 28, 4, 128, 5, 1),    # the 7B-like head shape
    (777, 8, 2, 64, 0, 0),       # pure power-of-two pattern
    (900, 6, 2, 128, 30, 2),     # window covers everything: dense causal
    (130, 5, 1, 128, 2, 1),      # a 5-head group: three head pairs, the last with a padding head
    (4097, 6, 3, 128, 7, 2),     # pairs only, one token in the last block
])
def test_backward_small_shapes(pa, oracle, N, Hq, Hkv, D, W, S):
    _run(pa, oracle, N, Hq, Hkv, D, W, S, batch=2, seed=N)


def test_backward_sink_column_spread_over_many_ctas(pa, oracle):
    """4200 tokens = 66 blocks: the sink block is listed by every row, so its column is cut into
    three chunks whose parts meet through atomics; peaky logits and a custom scale on top."""
    stats = _run(pa, oracle, 4200, 8, 2, 128, 5, 1, k_scale=2.0, scale=0.07, seed=5)
    print("backward error stats (max, mean) for dQ, dK, dV:", stats)


def test_backward_sliding_window_layout(pa, oracle):
    _run(pa, oracle, 1100, 8, 2, 128, 4, 1, use_power=False, seed=6)


@pytest.mark.parametrize("N,Hq,Hkv,W,S", [
    (1000, 7, 1, 5, 1),      # a 7-head group: four head pairs, the last with a padding head
    (2100, 3, 3, 2, 0),      # one query head per KV head: every pair has a padding head
    (4200, 8, 2, 5, 1),      # the sink column in three chunks
])
def test_backward_head_dim_128_on_the_warp_level_kernels(pa, pa_env, oracle, N, Hq, Hkv, W, S):
    """The tcgen05 kernels run by default; PA_BACKWARD_PATH=mma asks for the warp-level MMA kernels.  Both meet
    the oracle."""
    _run(pa, oracle, N, Hq, Hkv, 128, W, S, seed=N)
    pa_env(PA_BACKWARD_PATH="mma")
    _run(pa, oracle, N, Hq, Hkv, 128, W, S, seed=N)


@pytest.mark.parametrize("N,Hq,Hkv,W,S", [
    (1000, 5, 1, 5, 1),      # an odd group
    (777, 8, 2, 0, 0),       # pure power-of-two pattern, ragged
    (4200, 4, 2, 5, 1),      # the sink column in several chunks
])
def test_backward_head_dim_64_on_the_warp_level_kernels(pa, pa_env, oracle, N, Hq, Hkv, W, S):
    pa_env(PA_BACKWARD_PATH="mma")
    _run(pa, oracle, N, Hq, Hkv, 64, W, S, batch=2, seed=N + 1)


def test_backward_many_items_per_cta(pa, oracle):
    """12K tokens x 8 heads x batch 2: 1500 (query block, head pair) items for the persistent dQ
    kernel, several per CTA with rows of every length, and dK / dV columns in one to six chunks;
    dK and dV are checked on sampled keys."""
    N, Hq, Hkv, D, W, S = 12000, 8, 2, 128, 3, 1
    Q, K, V = (si.bf16_randn((2, N, h, D), 1200 + i) for i, h in enumerate((Hq, Hkv, Hkv)))
    dO = si.bf16_randn((2, N, Hq, D), 1204)
    rp, ci = pa.pa_build_layout(N, 64, W, S)
    Qd, Kd, Vd, dOd = Q.cuda(), K.cuda(), V.cuda(), dO.cuda()
    o, lse, ws = pa.pa_prefill(Qd, Kd, Vd, rp, ci)
    pa.pa_prefill_status(ws)
    dq, dk, dv, wsb = pa.pa_prefill_backward(Qd, Kd, Vd, o, lse, dOd, rp, ci)
    pa.pa_prefill_status(wsb)
    keys = sorted({0, 63, 64, N - 1, 4095, 4096} | {int(x) for x in np.random.default_rng(1205).integers(0, N, 20)})
    rq, rk, rv = oracle.backward(Q, K, V, dO, 64, W, S, key_rows=keys)
    kidx = torch.as_tensor(keys).cuda()
    _compare(dq, rq, "dQ 12K")
    _compare(dk[:, kidx], rk[:, keys], "dK 12K")
    _compare(dv[:, kidx], rv[:, keys], "dV 12K")


def test_backward_wait_that_runs_out_ends_the_kernels_with_a_status(pa, oracle):
    """The tcgen05 backward kernels bound every barrier wait like the prefill kernel.  With the limit
    at one cycle an ordinary wait that is not over at its first try (the first tiles take microseconds
    to arrive) runs out: the call returns, the status block at the head of the backward workspace
    reports PA_ERR_TIMEOUT, and the next call, back at the default limit, is correct."""
    N, Hq, Hkv, D, W, S = 3000, 8, 2, 128, 5, 1
    Q, K, V = (si.bf16_randn((1, N, h, D), 1300 + i) for i, h in enumerate((Hq, Hkv, Hkv)))
    dO = si.bf16_randn((1, N, Hq, D), 1304)
    rp, ci = pa.pa_build_layout(N, 64, W, S)
    Qd, Kd, Vd, dOd = Q.cuda(), K.cuda(), V.cuda(), dO.cuda()
    o, lse, ws = pa.pa_prefill(Qd, Kd, Vd, rp, ci)
    pa.pa_prefill_status(ws)
    try:
        pa.pa_set_wait_limit_cycles(1)
        dq, dk, dv, wsb = pa.pa_prefill_backward(Qd, Kd, Vd, o, lse, dOd, rp, ci)
        with pytest.raises(pa.PaError, match="PA_ERR_TIMEOUT"):
            pa.pa_prefill_status(wsb)
    finally:
        pa.pa_set_wait_limit_cycles(0)
    dq, dk, dv, wsb = pa.pa_prefill_backward(Qd, Kd, Vd, o, lse, dOd, rp, ci)
    assert pa.pa_prefill_status(wsb) == 0
    rq, rk, rv = oracle.backward(Q, K, V, dO, 64, W, S)
    for g, r, n in ((dq, rq, "dQ"), (dk, rk, "dK"), (dv, rv, "dV")):
        _compare(g, r, n + " after a timed-out call")


def test_backward_at_16k_on_sampled_keys(pa, oracle):
    """A sweep-sized case: 16K tokens with the 7B-like heads.  The oracle evaluates dQ on every row
    (its first pass covers them all anyway) and dK, dV on sampled key positions: the sink block (its
    column is spread over eight CTAs), block boundaries, power-of-two distances and a random draw."""
    N, Hq, Hkv, D, W, S = 16384, 28, 4, 128, 5, 1
    Q, K, V = si.bf16_randn((1, N, Hq, D), 1101), si.bf16_randn((1, N, Hkv, D), 1102), si.bf16_randn((1, N, Hkv, D), 1103)
    dO = si.bf16_randn((1, N, Hq, D), 1104)
    rp, ci = pa.pa_build_layout(N, 64, W, S)
    Qd, Kd, Vd, dOd = Q.cuda(), K.cuda(), V.cuda(), dO.cuda()
    o, lse, ws = pa.pa_prefill(Qd, Kd, Vd, rp, ci)
    pa.pa_prefill_status(ws)
    dq, dk, dv, wsb = pa.pa_prefill_backward(Qd, Kd, Vd, o, lse, dOd, rp, ci)
    pa.pa_prefill_status(wsb)
    keys = sorted({0, 1, 63, 64, 65, N - 1, N - 64, N - 65, 8191, 8192, 12288 + 17}
                  | {int(x) for x in np.random.default_rng(1105).integers(0, N, 24)})
    rq, rk, rv = oracle.backward(Q, K, V, dO, 64, W, S, key_rows=keys)
    kidx = torch.as_tensor(keys).cuda()
    print("16K backward (max, mean):", _compare(dq, rq, "dQ 16K"), _compare(dk[:, kidx], rk[:, keys], "dK 16K"),
          _compare(dv[:, kidx], rv[:, keys], "dV 16K"))


def test_backward_on_views_of_a_packed_qkv_tensor(pa, oracle):
    """Q, K and V as head slices of one [batch, seq, Hq + 2 Hkv, D] tensor: the kernels take the
    strides as given (the tensor maps of the tcgen05 kernels are built from them)."""
    N, Hq, Hkv, D, W, S = 1300, 8, 2, 128, 3, 1
    qkv = si.bf16_randn((2, N, Hq + 2 * Hkv, D), 1400).cuda()
    q, k, v = qkv[:, :, :Hq], qkv[:, :, Hq:Hq + Hkv], qkv[:, :, Hq + Hkv:]
    dO = si.bf16_randn((2, N, Hq, D), 1401)
    rp, ci = pa.pa_build_layout(N, 64, W, S)
    o, lse, ws = pa.pa_prefill(q, k, v, rp, ci)
    pa.pa_prefill_status(ws)
    dq, dk, dv, wsb = pa.pa_prefill_backward(q, k, v, o, lse, dO.cuda(), rp, ci)
    pa.pa_prefill_status(wsb)
    rq, rk, rv = oracle.backward(q.cpu().contiguous(), k.cpu().contiguous(), v.cpu().contiguous(), dO, 64, W, S)
    for g, r, n in ((dq, rq, "dQ"), (dk, rk, "dK"), (dv, rv, "dV")):
        _compare(g, r, n + " packed qkv")


def test_backward_on_kv_head_shards_reproduces_the_whole_call(pa):
    """Head sharding needs no exchange in the backward pass either: dQ belongs to the query heads and
    dK, dV to the KV heads a rank holds.  The ranks' calls on head slices (run here one after the other
    on the one GPU) give dQ bit for bit and dK, dV up to the order of their fp32 additions."""
    from paper_2503_03588_b200.sharding import kv_head_shard, shard_prefill_tensors

    N, Hq, Hkv, D = 3000, 28, 4, 128
    Q, K, V = (si.bf16_randn((1, N, h, D), 1500 + i).cuda() for i, h in enumerate((Hq, Hkv, Hkv)))
    dO = si.bf16_randn((1, N, Hq, D), 1504).cuda()
    rp, ci = pa.pa_build_layout(N, 64, 5, 1)
    o, lse, ws = pa.pa_prefill(Q, K, V, rp, ci)
    pa.pa_prefill_status(ws)
    dq_full, dk_full, dv_full, wsb = pa.pa_prefill_backward(Q, K, V, o, lse, dO, rp, ci)
    pa.pa_prefill_status(wsb)
    for world in (2, 4):
        for rank in range(world):
            qs_, ks_, vs_, heads = shard_prefill_tensors(Q, K, V, world, rank)
            _, kv_heads = kv_head_shard(Hq, Hkv, world, rank)
            dq, dk, dv, wsr = pa.pa_prefill_backward(qs_, ks_, vs_, o[:, :, heads], lse[:, heads].contiguous(), dO[:, :, heads], rp, ci)
            pa.pa_prefill_status(wsr)
            assert torch.equal(dq, dq_full[:, :, heads]), (world, rank)
            assert torch.allclose(dk, dk_full[:, :, kv_heads], rtol=1e-4, atol=1e-5), (world, rank)
            assert torch.allclose(dv, dv_full[:, :, kv_heads], rtol=1e-4, atol=1e-5), (world, rank)


def _random_causal_csr(nqb, rng):
    """Rows of 0 to nqb ascending blocks, some rows and some columns empty, some columns listed by all."""
    allowed = rng.random(nqb) < 0.8
    allowed[: max(1, nqb // 20)] = True
    rows = []
    for i in range(nqb):
        density = rng.choice([0.0, 0.05, 0.5, 1.0], p=[0.1, 0.5, 0.2, 0.2])
        rows.append([j for j in range(i + 1) if allowed[j] and rng.random() < density])
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    return rp, np.asarray([j for r in rows for j in r], dtype=np.int32), rows


@pytest.mark.parametrize("N,Hq,Hkv,D", [
    (64 * 32 + 1, 2, 1, 128),    # 33 columns: one word and one bit of rows
    (64 * 65, 4, 2, 64),         # 65 columns: one beyond what a block transposes
    (64 * 40 - 9, 66, 33, 64),   # more heads than one pass over a token's rows takes; ragged tokens
    (64 * 70 + 3, 3, 3, 128),    # rows of up to 71 entries; one head per group
])
def test_backward_on_arbitrary_causal_layouts(pa, oracle, N, Hq, Hkv, D):
    """The transposed lists of layouts with empty rows, empty columns, columns listed by every row and rows
    of more than 32 entries; the oracle takes the dense mask that the CSR stands for."""
    nqb = (N + 63) // 64
    rp, ci, rows = _random_causal_csr(nqb, np.random.default_rng(N))
    dense = np.zeros((N, N), dtype=bool)
    for i, r in enumerate(rows):
        for j in r:
            dense[i * 64:(i + 1) * 64, j * 64:(j + 1) * 64] = True
    dense &= np.tril(np.ones((N, N), dtype=bool))
    Q, K, V = (si.bf16_randn((1, N, h, D), 1600 + N + x) for x, h in enumerate((Hq, Hkv, Hkv)))
    dO = si.bf16_randn((1, N, Hq, D), 1604 + N)
    Qd, Kd, Vd, dOd, rpd, cid = (t.cuda() for t in (Q, K, V, dO, torch.as_tensor(rp), torch.as_tensor(ci)))
    o, lse, ws = pa.pa_prefill(Qd, Kd, Vd, rpd, cid)
    pa.pa_prefill_status(ws)
    dq, dk, dv, wsb = pa.pa_prefill_backward(Qd, Kd, Vd, o, lse, dOd, rpd, cid,
                                             dk=torch.full((1, N, Hkv, D), 7.0, device="cuda"),
                                             dv=torch.full((1, N, Hkv, D), 7.0, device="cuda"))
    pa.pa_prefill_status(wsb)
    for g, r, n in zip((dq, dk, dv), oracle.backward(Q, K, V, dO, 64, 5, 1, dense=dense), ("dQ", "dK", "dV")):
        _compare(g, r, n + " random layout")


@pytest.mark.parametrize("D", [64, 128])
def test_backward_of_many_short_lists(pa, oracle, D):
    """Key blocks listed by one or two rows, one head pair per group: work items of one and two steps, several per
    CTA, so that a warp's next step lies one, two or three items ahead."""
    nqb, Hkv = 12, 40
    N, Hq = 64 * nqb - 5, 2 * Hkv
    rows = [[i - 1, i] if i % 3 == 2 else [i] for i in range(nqb)]
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    ci = np.asarray([j for r in rows for j in r], dtype=np.int32)
    dense = np.zeros((N, N), dtype=bool)
    for i, r in enumerate(rows):
        for j in r:
            dense[i * 64:(i + 1) * 64, j * 64:(j + 1) * 64] = True
    dense &= np.tril(np.ones((N, N), dtype=bool))
    Q, K, V = (si.bf16_randn((1, N, h, D), 1700 + D + x) for x, h in enumerate((Hq, Hkv, Hkv)))
    dO = si.bf16_randn((1, N, Hq, D), 1704 + D)
    Qd, Kd, Vd, dOd, rpd, cid = (t.cuda() for t in (Q, K, V, dO, torch.as_tensor(rp), torch.as_tensor(ci)))
    o, lse, _ = pa.pa_prefill(Qd, Kd, Vd, rpd, cid)
    dq, dk, dv, wsb = pa.pa_prefill_backward(Qd, Kd, Vd, o, lse, dOd, rpd, cid)
    pa.pa_prefill_status(wsb)
    for g, r, n in zip((dq, dk, dv), oracle.backward(Q, K, V, dO, 64, 5, 1, dense=dense), ("dQ", "dK", "dV")):
        _compare(g, r, n + " short lists")


@pytest.mark.parametrize("D", [64, 128])
def test_backward_of_keys_and_values_shared_by_the_batch(pa, D):
    """Q, K and V expanded over the batch (stride 0): the gradients of their copies, per batch entry (dQ bit for bit,
    dK and dV up to the order of their fp32 additions)."""
    batch, N, Hq, Hkv = 3, 1000, 6, 2
    q, k, v = (si.bf16_randn((1, N, h, D), 1820 + x).cuda().expand(batch, -1, -1, -1) for x, h in enumerate((Hq, Hkv, Hkv)))
    d_o = si.bf16_randn((batch, N, Hq, D), 1823).cuda()
    copies = [x.contiguous() for x in (q, k, v)]
    rp, ci = pa.pa_build_layout(N, 64, 5, 1)
    o, lse, _ = pa.pa_prefill(*copies, rp, ci)
    dq, dk, dv, ws = pa.pa_prefill_backward(q, k, v, o, lse, d_o, rp, ci)
    pa.pa_prefill_status(ws)
    rq, rk, rv, _ = pa.pa_prefill_backward(*copies, o, lse, d_o, rp, ci)
    assert torch.equal(dq, rq)
    assert torch.allclose(dk, rk, rtol=1e-4, atol=1e-5) and torch.allclose(dv, rv, rtol=1e-4, atol=1e-5)


@pytest.mark.parametrize("D", [64, 128])
def test_backward_with_chunks_of_full_size(pa, oracle, D):
    """Enough work that chunks have their full 32 query blocks: only the columns of several chunks, and those that
    nobody lists, are cleared beforehand, and the KV heads are walked one after the other (Q and dO exceed 64 MB).
    Columns nobody lists, of one chunk and of two; ragged length, batch 3.  The same gradients come out of calls on
    eight KV heads of one batch entry each, which clear everything and deal a slot's heads together; two heads are
    compared with the oracle."""
    nqb, batch, H = 41, 3, 64
    N = 64 * nqb - 20
    rng = np.random.default_rng(1900)
    rows = [[j for j in range(i + 1) if j < 2 or j == i or (j % 4 and rng.random() < 0.25)] for i in range(nqb)]
    rows[12] = [j for j in rows[12] if j != 12]
    rows = [r if i < 12 else [j for j in r if j != 12] for i, r in enumerate(rows)]   # nobody lists block 12
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    ci = np.asarray([j for r in rows for j in r], dtype=np.int32)
    listers = np.bincount(ci, minlength=nqb)
    assert listers[12] == 0 and listers[0] > 32 and 0 < listers[nqb - 1] <= 32
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert len(ci) * H * batch >= 32 * 8 * sms and batch * N * H * D * 4 > 64 << 20
    Q, K, V, dO = (si.bf16_randn((batch, N, H, D), 1901 + x).cuda() for x in range(4))
    rpd, cid = torch.as_tensor(rp).cuda(), torch.as_tensor(ci).cuda()
    o, lse, ws = pa.pa_prefill(Q, K, V, rpd, cid)
    pa.pa_prefill_status(ws)
    dq, dk, dv, ws = pa.pa_prefill_backward(Q, K, V, o, lse, dO, rpd, cid, *(torch.full((batch, N, H, D), 7.0, device="cuda")
                                                                             for _ in range(3)))
    pa.pa_prefill_status(ws)
    assert not dk[:, 64 * 12:64 * 13].any() and not dv[:, 64 * 12:64 * 13].any()
    for b in range(batch):
        for h in range(0, H, 8):
            part = [x[b:b + 1, :, h:h + 8] for x in (Q, K, V, o, dO)]
            pq, pk, pv, _ = pa.pa_prefill_backward(*part[:4], lse[b:b + 1, h:h + 8].contiguous(), part[4], rpd, cid)
            assert torch.equal(dq[b:b + 1, :, h:h + 8], pq), (b, h)
            for got, ref in ((dk, pk), (dv, pv)):
                assert torch.allclose(got[b:b + 1, :, h:h + 8], ref, rtol=1e-4, atol=1e-5), (b, h)
    dense = np.zeros((N, N), dtype=bool)
    for i, r in enumerate(rows):
        for j in r:
            dense[i * 64:(i + 1) * 64, j * 64:(j + 1) * 64] = True
    dense &= np.tril(np.ones((N, N), dtype=bool))
    two = [x[1:2, :, 30:32].cpu().contiguous() for x in (Q, K, V, dO)]
    for g, r, n in zip((dq, dk, dv), oracle.backward(*two, 64, 5, 1, dense=dense), ("dQ", "dK", "dV")):
        _compare(g[1:2, :, 30:32], r, n + " full chunks")


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_backward_of_a_group_beside_one_that_is_not_finite(pa, D, bad):
    """Groups of three heads: the second tile of a group has room for a head that is not there, next to which the
    next group's first head lies in memory.  What that one holds changes nothing in this group's gradients."""
    N, Hq, Hkv = 500, 6, 2
    Q, K, V, dO = (si.bf16_randn((1, N, h, D), 1950 + x).cuda() for x, h in enumerate((Hq, Hkv, Hkv, Hq)))
    rp, ci = pa.pa_build_layout(N, 64, 5, 1)
    o, lse, _ = pa.pa_prefill(Q, K, V, rp, ci)
    clean = pa.pa_prefill_backward(Q, K, V, o, lse, dO, rp, ci)[:3]
    Q[:, :, 3:], dO[:, :, 3:] = bad, bad
    dq, dk, dv, ws = pa.pa_prefill_backward(Q, K, V, o, lse, dO, rp, ci)
    pa.pa_prefill_status(ws)
    assert torch.equal(dq[:, :, :3], clean[0][:, :, :3])
    for got, ref in ((dk, clean[1]), (dv, clean[2])):
        assert torch.allclose(got[:, :, 0], ref[:, :, 0], rtol=1e-4, atol=1e-5)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("N,Hq,Hkv,D,batch", [(100, 2, 2, 64, 1), (1000, 7, 1, 128, 1), (3000, 8, 2, 64, 2), (9000, 16, 16, 64, 2)])
def test_backward_calls_back_to_back_on_one_workspace(pa, N, Hq, Hkv, D, batch, graph):
    """The dQ kernel runs beside the dK / dV kernel, and the preparation of the next call, which may start beside both (the
    first two sizes: one round of items), may not touch what either reads: two problems in turn on the same workspace
    with nothing in between, issued one by one and from a graph, where no launch lets a gap open, from fewer items
    than SMs to chunks of full size, whose dK and dV are cleared by a kernel of their own."""
    turns = 8
    rp, ci = pa.pa_build_layout(N, 64, 5, 1)
    problems = []
    for seed in (2100, 2200):
        Q, K, V, dO = (si.bf16_randn((batch, N, h, D), seed + i).cuda() for i, h in enumerate((Hq, Hkv, Hkv, Hq)))
        o, lse, _ = pa.pa_prefill(Q, K, V, rp, ci)
        *alone, ws = pa.pa_prefill_backward(Q, K, V, o, lse, dO, rp, ci)
        torch.cuda.synchronize()
        problems.append((Q, K, V, o, lse, dO, alone))
    outs = [[torch.full_like(x, float("nan")) for x in problems[0][6]] for _ in range(turns)]

    def issue():
        for turn, (dq, dk, dv) in enumerate(outs):
            Q, K, V, o, lse, dO, _ = problems[turn % 2]
            pa.pa_prefill_backward(Q, K, V, o, lse, dO, rp, ci, dq=dq, dk=dk, dv=dv, workspace=ws)

    torch.cuda.synchronize()
    if graph:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            issue()
        g.replay()
    else:
        issue()
    pa.pa_prefill_status(ws)
    for turn, got in enumerate(outs):
        for x, ref in zip(got, problems[turn % 2][6]):
            # (parts of dK and dV are added up in no fixed order: fp32 sums of at most some thousand terms)
            assert (x - ref).abs().max() <= 1e-5 * ref.abs().max()
