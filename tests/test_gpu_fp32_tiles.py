"""The tiled fp32 kernels at the edges of their tiles.

Pair passes: a block takes 16, 32 or 64 rows against tiles of 128 columns, chosen by how many
rows the call has; every choice adds a row's terms in the same order, so a head updated alone
(16 rows a block, a cluster of blocks) and among many (32 or 64) ends with the same bits.  Attention: 16, 32 or 64
queries a block, and with few blocks a cluster splits the key range; compared with float64.
Allocation-free order: key arrays without 16-byte alignment take element loads and must give
what aligned ones do.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dkv():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2608_27922_gb300 import dkv as d
    return d


@pytest.mark.parametrize("H,N,M,d,dtype,desc", [
    (40, 129, 257, 64, torch.float32, 0),
    (48, 127, 400, 128, torch.bfloat16, 0),
    (160, 65, 130, 128, torch.float32, 0),
    (40, 128, 256, 64, torch.bfloat16, 1),
    (30, 200, 383, 128, torch.float32, 1),
])
def test_rows_per_block_do_not_change_a_bit(dkv, H, N, M, d, dtype, desc):
    g = torch.Generator(device="cuda").manual_seed(N)
    K = torch.randn(4, H, N, d, generator=g, device="cuda").to(dtype)
    V = torch.randn(4, H, N, d, generator=g, device="cuda").to(dtype)
    kw = dict(score_mode=dkv.DKV_SCORE_FP32, sync_heads=0, descriptor=desc)
    many = dkv.BankLayer(H, d, [M] * H, N, dtype, **kw)
    for t in range(4):
        many.update(K[t], V[t], t)
    many.sync()
    for h in (0, H - 1):
        one = dkv.BankLayer(1, d, [M], N, dtype, **kw)
        for t in range(4):
            one.update(K[t, h:h + 1].contiguous(), V[t, h:h + 1].contiguous(), t)
        one.sync()
        m = one.occupancy_host()[0]
        assert m == many.occupancy_host()[h] and m > 0
        for name in ("k", "v", "rho", "base", "prov_step", "prov_src"):
            assert torch.equal(getattr(one, name)[0, :m], getattr(many, name)[h, :m]), (h, name)
        one.close()
    many.close()


@pytest.mark.parametrize("N,m,M,d,dtype,desc", [
    (16, 129, 129, 64, torch.float32, 0),      # a second tile of one column
    (1, 1025, 4000, 128, torch.bfloat16, 0),   # nine tiles over eight blocks
    (65, 40, 3000, 128, torch.bfloat16, 0),    # blocks of the cluster without a tile
    (300, 1152, 1300, 64, torch.float32, 1),   # whole tiles, [K; V]
    (1000, 640, 1500, 128, torch.float32, 0),  # crossings and new baselines over clusters too
])
def test_clusters_hand_the_sums_on(dkv, N, m, M, d, dtype, desc):
    """One head alone spreads its column tiles over a cluster of blocks; the same head among 200
    fills the GPU without.  Scores, crossings and the updated bank have the same bits."""
    g = torch.Generator(device="cuda").manual_seed(N + m)
    k, v = (torch.randn(1, M, d, generator=g, device="cuda").to(dtype) for _ in range(2))
    K, V = (torch.randn(1, N, d, generator=g, device="cuda").to(dtype) for _ in range(2))
    rho = torch.rand(1, M, generator=g, device="cuda") + 1
    got = []
    for H in (1, 200):
        bank = dkv.BankLayer(H, d, [M] * H, N, dtype, score_mode=dkv.DKV_SCORE_FP32, sync_heads=0, descriptor=desc)
        bank.k.copy_(k.expand(H, -1, -1))
        bank.v.copy_(v.expand(H, -1, -1))
        bank.rho.copy_(rho.expand(H, -1))
        bank.base.copy_(bank.rho / 1.2)
        bank.import_state([m] * H)
        bank.admit(K.expand(H, -1, -1).contiguous(), V.expand(H, -1, -1).contiguous(), 1)
        bank.sync()
        mid = bank.intermediates()
        res = [mid["score"][H - 1].clone(), mid["cross"][H - 1, :m].clone()]
        bank.compress()
        bank.sync()
        n = bank.occupancy_host()[H - 1]
        got.append(res + [getattr(bank, x)[H - 1, :n].clone() for x in ("k", "rho", "base", "prov_src")])
        bank.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)
    if not desc:
        scores, perm = torch.empty(N, device="cuda"), torch.empty(N, dtype=torch.int32, device="cuda")
        dkv.dkv_candidate_order_noalloc(k[0], (rho / 1.2)[0], m, K[0], N, d, dkv.DKV_DTYPE_FP32
                                        if dtype == torch.float32 else dkv.DKV_DTYPE_BF16,
                                        dkv.dkv_params_default(d), scores, perm)
        assert torch.equal(scores, got[0][0])


@pytest.mark.parametrize("H,Nq,occ,M,W,d,dtype", [
    (1, 17, 900, 1000, 130, 64, torch.float32),      # cluster of 2, one query in the last block
    (1, 16, 4000, 4000, 1, 128, torch.bfloat16),     # cluster of 8, a window of one key
    (2, 5, 40, 2000, 0, 128, torch.float32),         # parts of the cluster without any key
    (12, 300, 127, 127, 2, 64, torch.bfloat16),      # 32 queries a block, tile ends in the window
    (60, 321, 129, 129, 0, 128, torch.float32),      # 64 queries a block
    (60, 320, 128, 128, 128, 64, torch.float32),     # whole tiles only
    (3, 33, 0, 64, 0, 64, torch.float32),            # no key at all
])
def test_attention_tiles_and_parts(dkv, H, Nq, occ, M, W, d, dtype):
    g = torch.Generator(device="cuda").manual_seed(Nq + W)
    bank = dkv.BankLayer(H, d, [M] * H, 16, dtype, score_mode=dkv.DKV_SCORE_FP32)
    bank.k.normal_(generator=g)
    bank.v.normal_(generator=g)
    bank.base.fill_(1)
    bank.import_state([occ] * H)
    Q = torch.randn(H, Nq, d, generator=g, device="cuda").to(dtype)
    Kw = torch.randn(H, max(W, 1), d, generator=g, device="cuda").to(dtype)
    Vw = torch.randn(H, max(W, 1), d, generator=g, device="cuda").to(dtype)
    O = bank.attend(Q, Kw if W else None, Vw if W else None).double()
    bank.sync()
    if occ + W == 0:
        assert not O.any()
        return
    k = torch.cat([bank.k[:, :occ], Kw[:, :W]], 1).double()
    v = torch.cat([bank.v[:, :occ], Vw[:, :W]], 1).double()
    ref = torch.softmax(Q.double() @ k.transpose(1, 2) / d ** 0.5, -1) @ v
    # fp32: scores up to |s| = 12 within 2^-24 * 12 * sqrt(d), weights and sums of n terms of
    # order 1 within sqrt(n) 2^-24 each: below 2e-5 of the largest value; bf16 results round to
    # 2^-9 of themselves (|O| < 4)
    tol = 2e-5 * 4 if dtype == torch.float32 else 4 * 2.0 ** -9
    assert (O - ref).abs().max().item() < tol
    bank.close()


@pytest.mark.parametrize("N,m,d,dtype", [(1, 1, 64, torch.bfloat16), (15, 127, 128, torch.float32),
                                         (17, 129, 64, torch.float32), (257, 128, 128, torch.bfloat16),
                                         (9800, 130, 64, torch.bfloat16)])
def test_order_of_unaligned_keys(dkv, N, m, d, dtype):
    g = torch.Generator(device="cuda").manual_seed(N)
    code = dkv.DKV_DTYPE_BF16 if dtype == torch.bfloat16 else dkv.DKV_DTYPE_FP32
    base = torch.rand(m, generator=g, device="cuda") + 0.5
    p = dkv.dkv_params_default(d)
    got = []
    kb = torch.randn(m * d, generator=g, device="cuda").to(dtype)
    kc = torch.randn(N * d, generator=g, device="cuda").to(dtype)
    for off in (0, 1):   # one element past a 16-byte boundary
        b1 = torch.zeros(m * d + 8, dtype=dtype, device="cuda")[off:off + m * d].copy_(kb)
        c1 = torch.zeros(N * d + 8, dtype=dtype, device="cuda")[off:off + N * d].copy_(kc)
        s = torch.full((N,), float("nan"), device="cuda")
        perm = torch.full((N,), -1, dtype=torch.int32, device="cuda")
        dkv.dkv_candidate_order_noalloc(b1, base, m, c1, N, d, code, p, s, perm)
        torch.cuda.synchronize()
        got.append((s.cpu().numpy(), perm.cpu().numpy()))
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
    assert np.array_equal(got[0][1], np.argsort(got[0][0], kind="stable"))
