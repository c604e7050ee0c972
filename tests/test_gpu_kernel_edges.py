"""GPU parity at the sizes where the kernels' work splits change: blocks and tiles of the attention kernels, streams
per CTA of the encoders, remainders of the export kernels, 8 and 16 query rows."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_19880_b200 as dq
from paper_2609_19880_b200 import _build, workloads

import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    assert torch.cuda.is_available()
    dq.lib()


def _np(t):
    return t.cpu().numpy()


def _cfg(lens, hq=32, hkv=8, **over):
    cfg = workloads.make_config(2, scale=1 / 16)
    for k, v in dict(over, batch=len(lens), seq_lens=list(lens), hq=hq, hkv=hkv).items():
        setattr(cfg, k, v)
    return cfg


def _setup(cfg, hs=0, pair=False, sigma=32):
    w = workloads.generate(cfg, device="cuda")
    if hs:
        tk, tv, ok, ov = gc.wide_tables(cfg, hs, pair=pair, k_rec=335 * hs // 8 + 2, v_rec=235 * hs // 8 + 2)
        return w, tk, tv, ok, ov, gc.WideGpuCache(w, tk, tv, hs)
    tk, tv, ok, ov = gc.tables(cfg, pair=pair, sigma=sigma)
    return w, tk, tv, ok, ov, gc.GpuCache(w, ok.rec, ov.rec)


def _containers(cache, ok, ov, hs):
    k, v = _np(cache.k_cont), _np(cache.v_cont)
    return (gc.from_interleaved(k, ok.rec), gc.from_interleaved(v, ov.rec)) if hs else (k, v)


# One block of the single-wave kernels is 4, 8, .. warps of 32 tokens (every count from 4 for token-wide streams); the
# last lists are the first ones whose blocks no longer fit the GPU once.
@pytest.mark.parametrize("hs,pair", [(0, False), (0, True), (8, False), (8, True)])
@pytest.mark.parametrize("lens", [[1], [32], [33], [127], [128], [129], [255], [257, 1], [511, 0, 513], [1025], [2304],
                                  [2305], [4700], [148 * 4 * 32 - 5], [100] * 40])
def test_attention_block_edges(lens, hs, pair):
    cfg = _cfg(lens)
    w, tk, tv, ok, ov, cache = _setup(cfg, hs, pair)
    gc.gpu_encode(w, tk, tv, cache)
    out, out32 = gc.gpu_attention(w, tk, tv, cache)
    kc, vc = _containers(cache, ok, ov, hs)
    ref = oracle.attention(ok, ov, workloads.bf16_bits(w.q), kc, vc, _np(cache.mean_q), _np(cache.mean_scale),
                           _np(w.page_table), _np(w.seq_lens), cfg.hkv, gc.SM_SCALE)
    assert gc.check_attention(out, out32, ref) < 3e-4


@pytest.mark.parametrize("lens,hq,hkv", [([1], 32, 8), ([33, 128], 28, 4), ([129, 257, 512], 8, 8), ([600] * 3, 16, 2),
                                         ([2304], 32, 8), ([4641], 40, 8)])
def test_decode_step_block_edges(lens, hq, hkv):
    """The step against the two calls that it stands for, bit for bit in the cache, in tolerance against the oracle."""
    cfg = _cfg(lens, hq, hkv)
    w, tk, tv, ok, ov, cache = _setup(cfg)
    gc.gpu_encode(w, tk, tv, cache)
    kc, vc, mq, ms, _, _ = gc.oracle_encode(w, ok, ov)
    last = torch.tensor(np.cumsum(lens) - 1)
    k, v, slot = w.k[last.cuda()].contiguous(), w.v[last.cuda()].contiguous(), w.slot[last.cuda()].contiguous()
    cache.k_cont.view(-1, cfg.hkv, 16, ok.rec)[(slot // 16).long(), :, (slot % 16).long()] = 0   # the step writes them anew
    cache.v_cont.view(-1, cfg.hkv, 16, ov.rec)[(slot // 16).long(), :, (slot % 16).long()] = 0
    out = torch.empty((cfg.batch, cfg.hq, 128), dtype=torch.bfloat16, device="cuda")
    out32 = torch.empty((cfg.batch, cfg.hq, 128), dtype=torch.float32, device="cuda")
    ws = torch.full((dq.dq_decode_workspace_bytes(cfg.batch, cfg.hq, w.page_table.shape[1]),), 0xA5, dtype=torch.uint8,
                    device="cuda")
    dq.dq_decode_step(tk, tv, k, v, slot, w.q, cache.k_cont, cache.v_cont, cache.mean_q, cache.mean_scale, w.page_table,
                      w.seq_lens, cfg.hkv, gc.SM_SCALE, out, ws, out32, cache.status)
    torch.cuda.synchronize()
    pos = torch.tensor([n - 1 for n in lens], dtype=torch.int32)
    oracle.window_means(workloads.bf16_bits(k), np.arange(len(lens), dtype=np.int32), _np(pos), mq, ms, 1)
    oracle.encode_tokens(ok, workloads.bf16_bits(k), np.arange(len(lens), dtype=np.int32), _np(pos), _np(slot), kc, mq, ms)
    oracle.encode_tokens(ov, workloads.bf16_bits(v), np.arange(len(lens), dtype=np.int32), _np(pos), _np(slot), vc)
    assert np.array_equal(_np(cache.k_cont), kc) and np.array_equal(_np(cache.v_cont), vc)
    ref = oracle.attention(ok, ov, workloads.bf16_bits(w.q), kc, vc, mq, ms, _np(w.page_table), _np(w.seq_lens), cfg.hkv,
                           gc.SM_SCALE)
    assert gc.check_attention(out, out32, ref) < 3e-4


# q_len * (hq / hkv) rows: 9, 15, 16 in one 16-row pass; 20 and 24 in a 16-row and an 8- or 16-row pass.
@pytest.mark.parametrize("q_len,hq,hkv,kw", [(3, 12, 4, {}), (3, 40, 8, {}), (4, 32, 8, dict(pair=True)), (2, 64, 8, dict(sigma=24)),
                                             (5, 32, 8, dict(pair=True, sigma=24)), (6, 32, 8, {}), (9, 2, 2, {}), (16, 2, 2, {})])
@pytest.mark.parametrize("resid", [None, [128, 1, 0, 5]])
def test_sixteen_query_rows(q_len, hq, hkv, kw, resid):
    cfg = _cfg([5, 300, 1023, 700], hq, hkv)
    w, tk, tv, ok, ov, cache = _setup(cfg, **kw)
    gc.gpu_encode(w, tk, tv, cache)
    B = cfg.batch
    gen = torch.Generator(device="cuda").manual_seed(q_len)
    q = torch.randn((B, q_len, hq, 128), generator=gen, device="cuda").to(torch.bfloat16)
    rk = rv = rl = None
    if resid is not None:
        rk, rv = (x.view(B, 128, hkv, 128).contiguous()
                  for x in workloads.make_kv(cfg, B * 128, gen, torch.device("cuda"), w.k_offsets, w.k_gain))
        rl = torch.tensor(resid, dtype=torch.int32, device="cuda")
    out = torch.empty((B, q_len, hq, 128), dtype=torch.bfloat16, device="cuda")
    out32 = torch.empty((B, q_len, hq, 128), dtype=torch.float32, device="cuda")
    need = dq.dq_decode_workspace_bytes(B, hq * min(q_len, 8 // (hq // hkv)), w.page_table.shape[1])   # the least allowed
    ws = torch.full((need + 4096,), 0x5A, dtype=torch.uint8, device="cuda")
    dq.dq_decode_attention_multi(tk, tv, q, cache.k_cont, cache.v_cont, cache.mean_q, cache.mean_scale, w.page_table,
                                 w.seq_lens, hkv, gc.SM_SCALE, out, ws[:need], out32, rk, rv, rl)
    torch.cuda.synchronize()
    assert bool((ws[need:] == 0x5A).all())
    lens, rlens = np.array(cfg.seq_lens, np.int64), np.array(resid or [0] * B, np.int64)
    for i in range(q_len):
        off = q_len - 1 - i
        more = {} if resid is None else dict(resid_k=workloads.bf16_bits(rk), resid_v=workloads.bf16_bits(rv),
                                             resid_lens=np.maximum(0, rlens - off).astype(np.int32))
        vis = np.maximum(0, lens - np.maximum(0, off - rlens)).astype(np.int32)
        ref = oracle.attention(ok, ov, workloads.bf16_bits(q[:, i]), _np(cache.k_cont), _np(cache.v_cont), _np(cache.mean_q),
                               _np(cache.mean_scale), _np(w.page_table), vis, hkv, gc.SM_SCALE, **more)
        assert gc.check_attention(out[:, i].contiguous(), out32[:, i].contiguous(), ref) < 3e-4


# Streams of a kind = 8 n (n / hs token-wide): from the few-stream kernel to 4, 8, .. 32 streams per CTA of the batch
# kernels, with incomplete last CTAs.
@pytest.mark.parametrize("hs,pair", [(0, False), (0, True), (8, False), (8, True), (2, False)])
@pytest.mark.parametrize("n", [1, 9, 148, 149, 300, 1001, 2003, 4111])
def test_encoder_split_edges(n, hs, pair):
    cfg = _cfg([n])
    w, tk, tv, ok, ov, cache = _setup(cfg, hs, pair)
    gc.gpu_encode(w, tk, tv, cache)
    torch.cuda.synchronize()
    kc, vc, mq, ms, sk, sv = gc.oracle_encode_wide(w, ok, ov, hs) if hs else gc.oracle_encode(w, ok, ov)
    assert np.array_equal(_np(cache.mean_q), mq) and np.array_equal(_np(cache.mean_scale), ms)
    got_k, got_v = _containers(cache, ok, ov, hs)
    assert np.array_equal(got_k, kc) and np.array_equal(got_v, vc)
    st = _np(cache.status)
    assert list(st[:3]) == [a + b for a, b in zip(sk[:3], sv[:3])] and st[3] == max(sk[3], sv[3])


@pytest.mark.parametrize("hs,pair", [(0, False), (0, True), (8, False), (2, True)])
@pytest.mark.parametrize("n", [1, 3, 16, 31, 33, 130])
def test_export_remainders(n, hs, pair):
    cfg = _cfg([150], hkv=8)
    w, tk, tv, ok, ov, _ = _setup(cfg, hs, pair)
    kc, vc, mq, ms, _, _ = gc.oracle_encode_wide(w, ok, ov, hs) if hs else gc.oracle_encode(w, ok, ov)
    pick = torch.randperm(150, generator=torch.Generator().manual_seed(n))[:n].cuda()
    seq_id, pos, slot = (x[pick].contiguous() for x in (w.seq_id, w.pos, w.slot))
    for t_lib, t_or, cont, m in ((tk, ok, kc, (mq, ms)), (tv, ov, vc, (None, None))):
        sym_ref, deq_ref = oracle.decode_tokens(t_or, cont, _np(seq_id), _np(pos), _np(slot), cfg.hkv, *m)
        sym = torch.zeros(sym_ref.shape, dtype=torch.uint8, device="cuda")
        deq = torch.zeros(deq_ref.shape, dtype=torch.float32, device="cuda")
        dev = torch.from_numpy(gc.to_interleaved(cont) if hs else cont).cuda()
        mean = [None if x is None else torch.from_numpy(x).cuda() for x in m]
        dq.dq_decode_tokens(t_lib, dev, slot, cfg.hkv, sym, deq, *mean, seq_id, pos)
        torch.cuda.synchronize()
        assert np.array_equal(_np(sym), sym_ref) and np.array_equal(_np(deq).view(np.uint32), deq_ref.view(np.uint32))
