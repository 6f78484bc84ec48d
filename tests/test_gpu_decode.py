"""GPU parity of the decoding-stage attention over the packed (shortened) KV cache against the CPU oracle, and of the
KV-cache rows a block step emits."""
import numpy as np
import pytest
import torch

from oracle import dash_oracle as oc
from paper_2604_18103_b200 import dash
from paper_2604_18103_b200 import workloads as wl
from test_gpu_kernels import assert_close_rms

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(autouse=True)
def _status_clean():
    yield
    assert dash.dash_check_status() == dash.OK


def _decode_case(lengths, Hq, Hkv, D, seed, pad=0):
    cu = wl.cu_from_lengths(lengths)
    n, S = int(cu[-1]), len(lengths)
    g = torch.Generator().manual_seed(seed)
    q = torch.randn(S, Hq, D, generator=g).to(torch.bfloat16)
    K = torch.randn(n + pad, Hkv, D, generator=g).to(torch.bfloat16)
    V = torch.randn(n + pad, Hkv, D, generator=g).to(torch.bfloat16)
    if pad:                      # rows past the packed end hold poison that must never reach an output
        K[n:], V[n:] = float("inf"), float("nan")
    out, lse = dash.dash_decode_attention(q.to(DEV), K.to(DEV), V.to(DEV), cu.to(DEV), want_lse=True)
    torch.cuda.synchronize()
    Oref, lref = oc.decode_attention(q, K[:n], V[:n], cu)
    assert_close_rms(out.float().cpu().numpy(), Oref, f"decode O {lengths[:6]} Hq{Hq} D{D}")
    got = lse.cpu().numpy()
    live = np.isfinite(lref)
    assert np.allclose(got[live], lref[live], atol=2e-2) and np.all(np.isinf(got[~live]) & (got[~live] < 0))


def test_decode_single_sequence_ragged_blocks():
    _decode_case([300], 4, 2, 128, 1)


def test_decode_batch_with_empty_short_and_long_caches_and_poisoned_tail():
    _decode_case([129, 0, 1, 5000, 64, 128], 14, 2, 128, 2, pad=130)


def test_decode_qwen_heads_long_cache_split_over_many_ctas():
    _decode_case([100000], 28, 4, 128, 3)


def test_decode_one_kv_head_more_key_splits_than_one_merge_round_takes():
    # a single KV head: all CTAs split the same head group's keys (261 splits), more than the 256 the merge fetches in its first round
    _decode_case([100000], 8, 1, 128, 8)


def test_decode_few_long_sequences_one_item_per_cta():
    # unequal long caches whose keys are cut into one item per CTA (the last chunk of every sequence and head is shorter)
    _decode_case([40000, 30001, 20000, 9000], 28, 4, 128, 7, pad=3)


def _large_batch(S, seed, long_at=10):
    """Lengths of S caches up to 700 rows, one of 9000; empty where the self-planning warp's lanes begin and end their groups of 32 sequences."""
    lengths = torch.randint(1, 700, (S,), generator=torch.Generator().manual_seed(seed)).tolist()
    for s in (3, 31, 32, 63, 64, 95, 96, 127, S - 1):
        if s < S:
            lengths[s] = 0
    lengths[long_at] = 9000
    return lengths


@pytest.mark.parametrize("S", [33, 45, 64, 65, 96, 97, 127, 128])
def test_decode_batch_that_the_ctas_plan_for_themselves(S):
    # one to four sequences per lane of the planning warp; the last boundary is the warp's 129th at S = 128
    _decode_case(_large_batch(S, S), 14, 2, 128, S, pad=7)
    _decode_case(_large_batch(S, S + 1, long_at=S - 2), 8, 8, 64, S + 1)


@pytest.mark.parametrize("S", [129, 200, 300])
def test_decode_large_batch_takes_the_planned_path(S):
    # more sequences than the CTAs plan for themselves (128): items come from the plan kernel, by ticket, and the merge finds them in its list
    _decode_case(_large_batch(S, 6), 14, 2, 128, 6, pad=7)
    _decode_case(_large_batch(S, 7, long_at=S - 2), 4, 4, 64, 7)


def test_decode_random_batches_match_oracle():
    """Seeded sweep over batch sizes on both sides of the self-planning limit (128), length mixes (many short, one long, equal,
    block-aligned), head groupings and head dims."""
    g = torch.Generator().manual_seed(2024)
    for trial in range(24):
        S = int(torch.randint(1, 41, (1,), generator=g)) if trial < 16 else int(torch.randint(41, 260, (1,), generator=g))
        kind = trial % 4
        if kind == 0:
            lens = torch.randint(0, 3000 if S <= 40 else 500, (S,), generator=g).tolist()
        elif kind == 1:
            lens = [int(torch.randint(1, 60000, (1,), generator=g))] + torch.randint(0, 300, (S - 1,), generator=g).tolist()
        elif kind == 2:
            lens = [int(torch.randint(100, 9000 if S <= 40 else 900, (1,), generator=g))] * S
        else:
            lens = (torch.randint(0, 40 if S <= 40 else 6, (S,), generator=g) * 128).tolist()
        Hkv, G, D = [1, 2, 4][trial % 3], [1, 4, 7, 8][trial % 4], [64, 128][trial % 2]
        _decode_case(lens, Hkv * G, Hkv, D, 100 + trial)


@pytest.mark.parametrize("lens", [[37888], [37889], [20000], [2500, 1700, 3300, 2900, 2100, 2600, 1900, 3000], [128 * 37] * 8, [128 * 37] * 7 + [128 * 38],
                                  [485 + 31 * (i % 7) for i in range(33)], [128 * 9] * 74, [1250 + 11 * i for i in range(96)]], ids=lambda x: f"{len(x)}x{x[0]}")
def test_decode_chunk_lengths_on_both_sides_of_the_plans_rule(lens):
    """One KV head per sequence: as many items as CTAs at an even share, one more than that, and batches in which the plan takes a longer chunk or two
    items per CTA."""
    _decode_case(lens, 4, 1, 64, len(lens))


@pytest.mark.parametrize("S", [1, 5, 40, 128])
def test_decode_over_boundaries_that_the_call_in_front_writes(S):
    """Decoding directly behind the compaction that shortens its caches: the decode kernel plans from the boundaries as they stand, while the
    kernels that write them may still run, and has to make the plan again where they change.  Here they change in every round (other
    masks into the same buffers), with rounds enqueued back to back; each result is the bits of a call made later on the same caches."""
    Hq, Hkv, D, L = 8, 2, 128, 20000 // S
    n = S * L
    cu = wl.cu_from_lengths([L] * S).to(DEV)
    g = torch.Generator(device=DEV).manual_seed(S)
    K, V = (torch.randn(n, Hkv * D, generator=g, device=DEV).to(torch.bfloat16) for _ in range(2))
    q = torch.randn(S, Hq, D, generator=g, device=DEV).to(torch.bfloat16)
    masks = [(torch.rand(n, generator=g, device=DEV) < keep).to(torch.uint8) for keep in (0.9, 0.02, 0.5, 0.0, 1.0, 0.3)]
    masks[2][:L] = 0                                       # the first sequence's cache is empty
    Kc, Vc = torch.zeros_like(K), torch.zeros_like(V)
    lists = {"idx": torch.zeros(n, dtype=torch.int32, device=DEV), "cu_out": torch.zeros(S + 1, dtype=torch.int32, device=DEV),
             "n_out": torch.zeros(1, dtype=torch.int32, device=DEV)}
    ws_c, ws_d = dash.workspace(dash.dash_workspace_bytes(dash.WS_COMPACT, n, S), DEV), dash.workspace(dash.dash_workspace_bytes(dash.WS_DECODE, n, S, Hq, Hkv, D), DEV)

    def compact(m):
        dash.dash_compact(m, cu, rows=[K, V], rows_out=[Kc, Vc], outputs=lists, ws=ws_c)

    def decode(out):
        return dash.dash_decode_attention(q, Kc.view(n, Hkv, D), Vc.view(n, Hkv, D), lists["cu_out"], out=out, ws=ws_d)

    outs = [torch.empty_like(q) for _ in range(4 * len(masks))]
    torch.cuda.synchronize()
    for i, out in enumerate(outs):
        compact(masks[i % len(masks)])
        decode(out)
    torch.cuda.synchronize()
    for i, m in enumerate(masks):
        compact(m)
        torch.cuda.synchronize()
        ref = decode(None)
        torch.cuda.synchronize()
        cu_m, k = lists["cu_out"].cpu(), int(lists["n_out"].item())
        Oref, _ = oc.decode_attention(q.cpu(), Kc[:k].view(k, Hkv, D).cpu(), Vc[:k].view(k, Hkv, D).cpu(), cu_m)
        assert_close_rms(ref.float().cpu().numpy(), Oref, f"mask {i}")
        for out in outs[i::len(masks)]:
            assert torch.equal(out, ref), i


def test_decode_head_dim_64_no_grouping_and_wide_grouping():
    _decode_case([777, 2000], 4, 4, 64, 4)
    _decode_case([1500], 8, 1, 64, 5, pad=3)


@pytest.mark.parametrize("D", [64, 128])
def test_decode_right_behind_prefill_attention(D):
    """Decoding enqueued directly behind a prefill attention on the same caches, several times over without a pause (the decode kernel
    is let in while the last CTAs of the attention kernel drain): both results are the bits of calls made one at a time."""
    Hq, Hkv, S, L = 8, 8, 12, 700
    cu = wl.cu_from_lengths([L] * S)
    g = torch.Generator().manual_seed(17)
    Q, K, V = (torch.randn(S * L, h, D, generator=g).to(torch.bfloat16).to(DEV) for h in (Hq, Hkv, Hkv))
    q, cu = Q[L - 1::L].contiguous(), cu.to(DEV)
    ws_a = dash.workspace(dash.dash_workspace_bytes(dash.WS_ATTENTION, S * L, S, Hq, Hkv, D), DEV)
    ws_d = dash.workspace(dash.dash_workspace_bytes(dash.WS_DECODE, S * L, S, Hq, Hkv, D), DEV)
    O = dash.dash_varlen_attention(Q, K, V, cu, L, ws=ws_a)
    torch.cuda.synchronize()
    out = dash.dash_decode_attention(q, K, V, cu, ws=ws_d)
    torch.cuda.synchronize()
    assert_close_rms(out.float().cpu().numpy(), O[L - 1::L].float().cpu().numpy(), "the last row of every sequence")
    runs = [(torch.empty_like(O), torch.empty_like(out)) for _ in range(8)]
    for a, d in runs:
        dash.dash_varlen_attention(Q, K, V, cu, L, O=a, ws=ws_a)
        dash.dash_decode_attention(q, K, V, cu, out=d, ws=ws_d)
    torch.cuda.synchronize()
    for a, d in runs:
        assert torch.equal(a, O) and torch.equal(d, out)


def test_block_step_emits_the_kv_cache_rows_a_decode_step_reads():
    w = wl.config2(T=600, seed=41, shape=wl.MINI)
    w.cu = wl.cu_from_lengths([250, 350])
    sh, T, S = w.shape, w.T, w.S
    H = w.tensors["H"]
    W = dict(w.weights[0]); W.update(wl.ffn_weights(sh, 41))
    pos = wl.positions(w.cu)
    ref = oc.block_step(H, W, w.cu, pos, sh, tau=0.0)
    block = dash.Block(sh, W, DEV, tau=0.0)
    Kc = torch.zeros(T, sh.Hkv, sh.D, dtype=sh.dtype, device=DEV)
    Vc = torch.zeros_like(Kc)
    block.set_kv_cache(Kc, Vc)
    lay = dash.dash_block_workspace(block, T, S)
    ws = dash.workspace(lay.total, DEV)
    outs = dict(H=torch.zeros(T, sh.d, dtype=sh.dtype, device=DEV), tok=torch.zeros(T, dtype=torch.int32, device=DEV),
                pos=torch.zeros(T, dtype=torch.int32, device=DEV), cu=torch.zeros(S + 1, dtype=torch.int32, device=DEV))
    x_full = torch.zeros(T, sh.d, dtype=sh.dtype, device=DEV)
    n_next, r, mask = torch.zeros(1, dtype=torch.int32, device=DEV), torch.zeros(T, device=DEV), torch.zeros(T, dtype=torch.uint8, device=DEV)
    cu_d = w.cu.to(DEV)
    dash.dash_block_step(block, H.to(DEV), torch.arange(T, dtype=torch.int32, device=DEV), pos.to(DEV), cu_d, 350, x_full, outs["H"],
                         outs["tok"], outs["pos"], outs["cu"], n_next, r, mask, ws)
    torch.cuda.synchronize()
    # the cache holds the rotary-applied keys and the values of every entering token
    assert_close_rms(Kc.float().cpu().numpy().reshape(T, -1), ref["K"].reshape(T, -1), "K cache")
    assert_close_rms(Vc.float().cpu().numpy().reshape(T, -1), ref["V"].reshape(T, -1), "V cache")
    nq = (sh.Hq + 2 * sh.Hkv) * sh.D
    QKV = ws[lay.attn.QKV:lay.attn.QKV + T * nq * 2].view(sh.dtype).view(T, nq)
    assert torch.equal(Kc.view(T, -1), QKV[:, sh.Hq * sh.D:(sh.Hq + sh.Hkv) * sh.D])
    # the last prompt token of each sequence, decoded over the emitted cache, reproduces its prefill attention output
    last = (w.cu[1:] - 1).long().to(DEV)
    q = QKV[last][:, :sh.Hq * sh.D].reshape(S, sh.Hq, sh.D).contiguous()
    out = dash.dash_decode_attention(q, Kc, Vc, cu_d)
    O = ws[lay.attn.O:lay.attn.O + T * sh.Hq * sh.D * 2].view(sh.dtype).view(T, sh.Hq, sh.D)[last]
    assert_close_rms(out.float().cpu().numpy(), O.float().cpu().numpy(), "decode over the emitted cache vs prefill row")
    assert_close_rms(out.float().cpu().numpy(), ref["O"][last.cpu().numpy()], "decode over the emitted cache vs oracle", atol=2.0 ** -8)


def test_decode_through_ctypes_is_the_same_call(monkeypatch):
    """Where the binding's C part is not built: with and without the caller's buffers, strided caches, an empty one, the caller's scale."""
    cu = wl.cu_from_lengths([129, 0, 700]).to(DEV)
    g = torch.Generator(device=DEV).manual_seed(5)
    q = torch.randn(3, 14, 128, generator=g, device=DEV).to(torch.bfloat16)
    K, V = torch.randn(2, 829, 4, 128, generator=g, device=DEV).to(torch.bfloat16)[:, :, :2]
    ws = dash.workspace(dash.dash_workspace_bytes(dash.WS_DECODE, 829, 3, 14, 2, 128), DEV)

    def both(scale):
        out = torch.zeros_like(q)
        return [dash.dash_decode_attention(q, K, V, cu, scale=scale, out=out, ws=ws), *dash.dash_decode_attention(q, K, V, cu, scale=scale, want_lse=True)]

    assert dash._pycall
    want = both(None) + both(0.05)
    monkeypatch.setattr(dash, "_pycall", False)
    got = both(None) + both(0.05)
    assert all(torch.equal(a, b) for a, b in zip(got, want)) and not torch.equal(want[0], want[3])
    empty = dash.dash_decode_attention(q[:1], K[:0], V[:0], torch.zeros(2, dtype=torch.int32, device=DEV))
    assert (empty == 0).all()
