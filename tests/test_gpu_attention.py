"""Bank-reading attention (Sec. 3.2) on grids that take the two-query-tile kernel.

The tensor-core attention has two schedules: one CTA per 128 queries with the key
range split between its two softmax groups (small grids), and one CTA per 256 queries
whose two query tiles share every key tile (grids of at least two CTAs per SM).  These
cases have enough heads to take the second one.  They use ragged bank occupancies and
window lengths, query counts that leave a partial second tile or none, and heads with
no keys.  Every output is compared with the oracle's softmax attention over
[bank | window] in float64, within 2e-2 absolute.
"""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import load_state, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dkv():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2608_27922_gb300 import dkv as d
    return d


def _bf16(rng, shape, scale):
    return synth.round_to_bf16((rng.standard_normal(shape) * scale).astype(np.float32))


def _bank_with(dkv, occ, M, d=128, seed=0):
    """A bank whose head h holds occ[h] random bf16 states (the oracle's copy alongside)."""
    rng = np.random.default_rng(seed)
    H = len(occ)
    ob = oracle.LayerBank.empty([M] * H, d)
    for h, m in enumerate(occ):
        hb = ob.heads[h]
        hb.K = _bf16(rng, (m, d), 1.5).astype(np.float64)
        hb.V = _bf16(rng, (m, d), 1.0).astype(np.float64)
        hb.rho = np.ones(m, np.float32)
        hb.base = np.ones(m, np.float32)
        hb.step = np.zeros(m, np.int64)
        hb.src = np.arange(m, dtype=np.int64)
    bank = dkv.BankLayer(H, d, [M] * H, 64, torch.bfloat16, score_mode=dkv.DKV_SCORE_TENSOR)
    load_state(bank, ob)
    return bank, ob


@pytest.mark.parametrize("Nq,W", [(300, 200), (256, 0), (129, 77), (520, 128)])
def test_two_tile_attention_matches_oracle(dkv, Nq, W):
    H, M, d = 320, 400, 128   # >= 2 CTAs per SM in every case
    occ = [(37 * h) % (M + 1) for h in range(H)]   # 0 .. 400, ragged
    occ[5] = 0
    bank, ob = _bank_with(dkv, occ, M, seed=Nq + W)
    rng = np.random.default_rng(Nq)
    Q = _bf16(rng, (H, Nq, d), 1.5)
    Kw = _bf16(rng, (H, W, d), 1.5) if W else None
    Vw = _bf16(rng, (H, W, d), 1.0) if W else None
    O = bank.attend(to_dev(Q, torch.bfloat16), None if Kw is None else to_dev(Kw, torch.bfloat16),
                    None if Vw is None else to_dev(Vw, torch.bfloat16)).float().cpu().numpy()
    bank.sync()
    err = 0.0
    for h in range(H):
        kw = np.zeros((0, d)) if Kw is None else Kw[h]
        vw = np.zeros((0, d)) if Vw is None else Vw[h]
        if occ[h] + kw.shape[0] == 0:
            assert np.all(O[h] == 0), h            # no keys at all: zero output
            continue
        ref = oracle.attend(ob.heads[h], Q[h], kw, vw)
        err = max(err, float(np.abs(O[h] - ref).max()))
    assert err < 2e-2, err
    bank.close()


def test_two_tile_attention_reads_a_long_bank(dkv):
    """Many key tiles (bank 4,000 states + window 700) on the two-tile grid: the key and
    value slots are reused many times over."""
    H, M, d, Nq, W = 152, 4000, 128, 300, 700
    occ = [M - (h % 3) * 61 for h in range(H)]
    bank, ob = _bank_with(dkv, occ, M, seed=7)
    rng = np.random.default_rng(8)
    Q = _bf16(rng, (H, Nq, d), 1.5)
    Kw, Vw = _bf16(rng, (H, W, d), 1.5), _bf16(rng, (H, W, d), 1.0)
    O = bank.attend(to_dev(Q, torch.bfloat16), to_dev(Kw, torch.bfloat16), to_dev(Vw, torch.bfloat16))
    O = O.float().cpu().numpy()
    bank.sync()
    err = 0.0
    for h in range(0, H, 7):
        err = max(err, float(np.abs(O[h] - oracle.attend(ob.heads[h], Q[h], Kw[h], Vw[h])).max()))
    assert err < 2e-2, err
    bank.close()


@pytest.mark.parametrize("occ,M,Nq,W", [
    ([5000], 5000, 16, 700),                  # one unit, cut into many parts
    ([0], 300, 1, 0),                         # no key at all
    ([1], 300, 130, 0),                       # one key, two query tiles
    ([0, 900, 0, 128, 1, 77], 900, 200, 0),   # heads without keys between cut units
    ([3000, 129], 3000, 128, 1),              # a window of one key after a bank that ends inside a tile
    ([2000] * 13, 2000, 1560, 333),           # more query tiles than SMs: shares over unit boundaries
])
def test_shared_key_tiles_match_oracle(dkv, occ, M, Nq, W):
    """Grids below two CTAs per SM: the key tiles of all (head, query tile) units in equal
    shares, units cut by share boundaries merged from fp32 parts.  The same call on a handle
    whose workspace lacks the parts' scratch takes whole units; both match the oracle."""
    H, d = len(occ), 128
    bank, ob = _bank_with(dkv, occ, M, seed=Nq + W)
    rng = np.random.default_rng(Nq)
    Q = _bf16(rng, (H, Nq, d), 1.5)
    Kw = _bf16(rng, (H, W, d), 1.5) if W else None
    Vw = _bf16(rng, (H, W, d), 1.0) if W else None
    Qd = to_dev(Q, torch.bfloat16)
    Kd, Vd = (to_dev(Kw, torch.bfloat16), to_dev(Vw, torch.bfloat16)) if W else (None, None)
    p = dkv.dkv_params_default(d)
    p.score_mode = dkv.DKV_SCORE_FP32
    small = dkv.dkv_bank_workspace_size(H, d, [M] * H, 64, dkv.DKV_DTYPE_BF16, p)
    assert small < bank.workspace.numel()
    spare = torch.empty(small, dtype=torch.uint8, device="cuda")
    bufs = dkv.dkv_buffers_t(bank.k.data_ptr(), bank.v.data_ptr(), bank.rho.data_ptr(), bank.base.data_ptr(),
                             bank.knorm.data_ptr(), bank.prov_step.data_ptr(), bank.prov_src.data_ptr(),
                             bank.occupancy.data_ptr(), spare.data_ptr(), small)
    O = bank.attend(Qd, Kd, Vd)
    whole = torch.full_like(O, 7.0)
    other = dkv.dkv_bank_create(H, d, [M] * H, 64, dkv.DKV_DTYPE_BF16, bank.params, bufs)
    dkv.dkv_bank_attend(other, Qd, Nq, Kd, Vd, W, whole)
    bank.sync()
    dkv.dkv_bank_sync(other)
    dkv.dkv_bank_destroy(other)
    O, whole = O.float().cpu().numpy(), whole.float().cpu().numpy()
    for h in range(H):
        if occ[h] + W == 0:
            assert np.all(O[h] == 0) and np.all(whole[h] == 0), h
            continue
        kw = np.zeros((0, d)) if Kw is None else Kw[h]
        vw = np.zeros((0, d)) if Vw is None else Vw[h]
        ref = oracle.attend(ob.heads[h], Q[h], kw, vw)
        assert np.abs(O[h] - ref).max() < 2e-2 and np.abs(whole[h] - ref).max() < 2e-2, h
    bank.close()


@pytest.mark.parametrize("occ", [2200, 9000])
def test_attention_bits_follow_the_bank_alone(dkv, occ):
    """156 units on the SMs, 9,360 states of budget: whole units pay with 2,200 states (18 key
    tiles), equal shares with 9,000.  The same bank and queries give the same bits on the handle
    that imported the bank, on one that was only handed its buffers, in a replayed graph, and on
    a handle that held another bank before."""
    H, M, d, Nq = 12, 9360, 128, 1560
    g = torch.Generator(device="cuda")
    g.manual_seed(occ)
    bank = dkv.BankLayer(H, d, [M] * H, 64, torch.bfloat16)
    bank.k.normal_(generator=g)
    bank.v.normal_(generator=g)
    bank.base.fill_(1.0)
    bank.import_state([occ] * H)
    Q = torch.randn(H, Nq, d, device="cuda", generator=g).bfloat16()
    want = bank.attend(Q, None, None)
    bufs = dkv.dkv_buffers_t(bank.k.data_ptr(), bank.v.data_ptr(), bank.rho.data_ptr(), bank.base.data_ptr(),
                             bank.knorm.data_ptr(), bank.prov_step.data_ptr(), bank.prov_src.data_ptr(),
                             bank.occupancy.data_ptr(), bank.workspace.data_ptr(), bank.workspace.numel())
    bank.sync()
    other = dkv.dkv_bank_create(H, d, [M] * H, 64, dkv.DKV_DTYPE_BF16, bank.params, bufs)
    handed = torch.zeros_like(want)
    dkv.dkv_bank_attend(other, Q, Nq, None, None, 0, handed)
    dkv.dkv_bank_sync(other)
    dkv.dkv_bank_destroy(other)
    assert torch.equal(want, handed)

    captured = torch.zeros_like(want)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        bank.attend(Q, None, None, captured)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(want, captured)

    again = dkv.BankLayer(H, d, [M] * H, 64, torch.bfloat16)
    again.k.copy_(bank.k)
    again.v.copy_(bank.v)
    again.base.fill_(1.0)
    again.import_state([M] * H)
    again.attend(Q, None, None)
    again.import_state([occ] * H)
    assert torch.equal(want, again.attend(Q, None, None))
    bank.sync()
    again.sync()
    bank.close()
    again.close()


@pytest.mark.parametrize("captured", [False, True])
def test_attention_on_two_streams_shares_the_scratch_in_turn(dkv, captured):
    """Attends of one handle on two streams, without events between them, whose units are cut
    (the handle's scratch holds the parts): each gives the bits that it gives alone."""
    H, M, d, Nq, W, reps = 2, 9000, 128, 200, 300, 6
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    bank = dkv.BankLayer(H, d, [M] * H, 64, torch.bfloat16)
    bank.k.normal_(generator=g)
    bank.v.normal_(generator=g)
    bank.base.fill_(1.0)
    bank.import_state([M, M - 700])
    Qs = [torch.randn(H, Nq, d, device="cuda", generator=g).bfloat16() for _ in range(2 * reps)]
    Kw, Vw = (torch.randn(H, W, d, device="cuda", generator=g).bfloat16() for _ in range(2))
    want = [bank.attend(q, Kw, Vw) for q in Qs]
    out = [torch.zeros_like(q) for q in Qs]
    torch.cuda.synchronize()
    side = torch.cuda.Stream()

    def both(main):
        side.wait_stream(main)
        for i in range(reps):
            bank.attend(Qs[2 * i], Kw, Vw, out[2 * i], stream=main.cuda_stream)
            bank.attend(Qs[2 * i + 1], Kw, Vw, out[2 * i + 1], stream=side.cuda_stream)
        main.wait_stream(side)

    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            both(torch.cuda.current_stream())
        graph.replay()
    else:
        both(torch.cuda.current_stream())
    torch.cuda.synchronize()
    bank.sync()
    for i, (a, b) in enumerate(zip(want, out)):
        assert torch.equal(a, b), i
    bank.close()
