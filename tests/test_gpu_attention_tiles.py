"""Prefill attention where its tiles begin and end: query tiles of 128 rows that go through the key blocks in pairs or alone, item lists from one
item to several per SM, sequences on both sides of every tile boundary, rescaling in either tile of a pair."""
import math

import pytest
import torch

from paper_2604_18103_b200 import dash
from paper_2604_18103_b200 import workloads as wl
from test_gpu_kernels import _attention_case, _indexed_attention_case
from test_gpu_layer import StepBuffers, run_step

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# few items: tiles alone; the last list is long enough for pairs, with odd and even numbers of tiles and empty sequences
EDGES = [[1], [127], [128], [129], [255, 256, 257], [385, 0, 1, 512, 640, 641], [1, 128, 129, 256, 0, 257, 300, 383, 384, 385, 511, 513, 900] * 4]


@pytest.mark.parametrize("lengths", EDGES, ids=lambda x: f"{len(x)}x{max(x)}")
@pytest.mark.parametrize("D", [64, 128])
def test_attention_at_the_edges_of_tiles(lengths, D):
    pairs, tiles = len(lengths) > 6, [(x + 127) // 128 for x in lengths]
    assert all(_entries(lengths, h, g, D) == sum((t + pairs) // (1 + pairs) for t in tiles) for h, g in ((4, 2), (7, 1)))
    _attention_case(lengths, 4, 2, D, torch.bfloat16, 31, pad=7)
    _attention_case(lengths, 7, 1, D, torch.bfloat16, 32)


PAIRED = [900, 640, 513, 385] * 5                       # enough for pairs with 14 heads and up


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("at", [100, 128, 255, 256, 700])
def test_attention_rescales_in_either_tile_of_a_pair(at, D):
    # scores grow at a key, the call has its tiles in pairs: the jump lies inside the first block, on block boundaries,
    # in the diagonal block of a pair's lower and of its upper tile.  One or two keys take all the weight of a row then, and the rounding of P and of
    # O to bf16 is off by up to 2^-9 (sum p |v| + |o|) <= 2^-8 max |v|: 0.0207 for the largest of these 3e6 normal values, 5.3; the smallest
    # root mean square that a row is held against is 0.9, hence the 0.025.
    _attention_case(PAIRED, 14, 2, D, torch.bfloat16, 33, pad=5, tol=2.5e-2, key_gain=[(at, 30.0), (at + 130, 3.0)])


@pytest.mark.parametrize("D", [64, 128])
def test_fp32_attention_in_pairs(D):
    """fp32 results have a store path of their own.  Of values that bf16 holds exactly the two calls have the same operands, so the fp32 result rounded to
    bf16 is the bf16 result, to the bit; that one is held against the oracle."""
    assert _entries(PAIRED, 14, 2, D, dtype=torch.float32) == sum((x + 255) // 256 for x in PAIRED)
    g = torch.Generator().manual_seed(38)
    cu, n = wl.cu_from_lengths(PAIRED).to(DEV), sum(PAIRED)
    Q, K, V = (torch.randn(n, h, D, generator=g).to(torch.bfloat16).to(DEV) for h in (14, 2, 2))
    O, lse = dash.dash_varlen_attention(Q, K, V, cu, max(PAIRED), want_lse=True)
    O32, lse32 = dash.dash_varlen_attention(Q.float(), K.float(), V.float(), cu, max(PAIRED), want_lse=True)
    assert torch.equal(O32.to(torch.bfloat16), O) and torch.equal(lse32, lse)
    _attention_case(PAIRED, 14, 2, D, torch.bfloat16, 38)


@pytest.mark.parametrize("D", [64, 128])
def test_fp32_step_multiplies_the_bf16_copy_of_its_attention_in_pairs(D):
    """A step's attention leaves O in fp32 and, for the output projection, in bf16: O is what the plain call gives for the step's Q, K and V, to the bit,
    and U is bf16(O) Wo up to fp32 sums of Hq D products, each sum off by at most Hq D 2^-24 of the sum of their absolute values."""
    shape = wl.LayerShape(d=256, Hq=16, Hkv=4, D=D, rope_base=1.0e4, dtype=torch.float32)
    cu = wl.cu_from_lengths(PAIRED)
    n, nq, hd = int(cu[-1]), (shape.Hq + 2 * shape.Hkv) * D, shape.Hq * D
    W = wl.layer_weights(shape, 39)
    layer = dash.Layer(shape, W, DEV, sel_mode=dash.SEL_KEEP_COUNT, keep_counts=torch.tensor([x // 2 for x in PAIRED], dtype=torch.int32, device=DEV))
    bufs = StepBuffers(layer, n, len(PAIRED), n, shape.dtype)
    H, tok = wl.hidden_states(n, shape.d, 39, shape.dtype).to(DEV), torch.arange(n, dtype=torch.int32, device=DEV)
    run_step(layer, H, tok, wl.positions(cu).to(DEV), cu.to(DEV), max(PAIRED), torch.zeros_like(H), bufs)
    QKV, O = bufs.view(bufs.lay.QKV, n, nq, torch.float32), bufs.view(bufs.lay.O, n, hd, torch.float32)
    q, k, v = (x.view(n, -1, D) for x in QKV.split([hd, shape.Hkv * D, shape.Hkv * D], dim=1))
    assert torch.equal(O, dash.dash_varlen_attention(q, k, v, cu.to(DEV), max(PAIRED)).view(n, hd))
    U, O16, Wo = bufs.view(bufs.lay.U, n, shape.d, torch.float32).double(), O.to(torch.bfloat16).double(), W["Wo"].to(DEV).to(torch.bfloat16).double()
    assert bool(((U - O16 @ Wo).abs() <= hd * 2.0 ** -24 * (O16.abs() @ Wo.abs())).all())


def test_attention_of_a_sequence_is_the_same_alone_and_in_a_batch():
    """A row's arithmetic does not hang on whether its tile goes alone or in a pair, nor on what else is in the call: bit for bit."""
    g = torch.Generator().manual_seed(34)
    lengths = [700, 1, 333, 1100, 128, 256, 900, 515] * 4
    cu = wl.cu_from_lengths(lengths)
    n = int(cu[-1])
    Q, K, V = (torch.randn(n, h, 128, generator=g).to(torch.bfloat16).to(DEV) for h in (14, 2, 2))
    O = dash.dash_varlen_attention(Q, K, V, cu.to(DEV), max(lengths))
    for s in (0, 1, 2, 3, 5, 31):
        a, b = int(cu[s]), int(cu[s + 1])
        one = dash.dash_varlen_attention(Q[a:b].contiguous(), K[a:b].contiguous(), V[a:b].contiguous(), wl.cu_from_lengths([b - a]).to(DEV), b - a)
        assert torch.equal(one, O[a:b])
    assert dash.dash_check_status() == dash.OK


def test_attention_row_sums_keep_small_weights_beside_a_large_one():
    """Row sums are formed per 64 keys, in four chains of 16: key 0 has weight 1, keys 64 to 127 have 2^-25 each, the others none.  In one chain
    with key 0 a 2^-25 is lost (half a unit of 1 is 2^-24), in chains of their own all 64 count: l = 1 + 2^-19.  A chain of 32 over the whole block
    would leave 16 of them out, 4.8e-7.  Sums that hold key 0 are rounded at most five times, 5 * 2^-24 = 3.0e-7; log and exp add 1e-12."""
    K = torch.full((256, 1, 128), 0.0)
    K[1:64, 0, 0], K[64:128, 0, 0], K[128:, 0, 0] = -1000.0, -25.0, -1000.0
    Q = torch.zeros(256, 1, 128)
    Q[:, 0, 0] = 1.0
    Q, K, V = Q.to(torch.bfloat16).to(DEV), K.to(torch.bfloat16).to(DEV), torch.ones(256, 1, 128, dtype=torch.bfloat16, device=DEV)
    _, lse = dash.dash_varlen_attention(Q, K, V, wl.cu_from_lengths([256]).to(DEV), 256, scale=math.log(2.0), want_lse=True)
    assert float((lse[0, 127:].double() - math.log1p(2.0 ** -19)).abs().max()) < 3.0e-7


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("lengths", [[100, 60, 1, 128, 90, 5] * 25, [100, 300, 5, 1, 257, 128, 40, 200, 129] * 8], ids=["one tile each", "pairs and single tiles"])
def test_attention_of_short_sequences_keeps_their_rows_apart(lengths, D):
    """Items of one tile take the two halves of a CTA in turn, and either half clears the value rows behind a sequence's end: NaN and infinities in every
    second sequence leave the outputs of the others as they are without, bit for bit."""
    g = torch.Generator().manual_seed(35)
    cu = wl.cu_from_lengths(lengths)
    n = int(cu[-1])
    Q, K, V = (torch.randn(n, h, D, generator=g).to(torch.bfloat16).to(DEV) for h in (8, 4, 4))
    odd = torch.cat([torch.full((x,), i % 2, dtype=torch.bool) for i, x in enumerate(lengths)]).to(DEV)
    _attention_case(lengths, 8, 4, D, torch.bfloat16, 36, pad=3)
    clean = dash.dash_varlen_attention(Q, K, V, cu.to(DEV), max(lengths))
    K[odd], V[odd] = float("inf"), float("nan")
    O = dash.dash_varlen_attention(Q, K, V, cu.to(DEV), max(lengths))
    assert torch.equal(O[~odd], clean[~odd]) and bool(torch.isfinite(clean.float()).all())
    assert dash.dash_check_status() == dash.OK


def _entries(lengths, Hq, Hkv, D, n=None, max_seqlen=None, dtype=torch.bfloat16):
    """Entries of the item list that a call leaves in its workspace: tiles, where they go alone, pairs and odd tiles otherwise."""
    cu = wl.cu_from_lengths(lengths).to(DEV)
    n = n or int(cu[-1])
    Q, K, V = (torch.zeros(n, h, D, dtype=dtype, device=DEV) for h in (Hq, Hkv, Hkv))
    ws = dash.workspace(dash.dash_workspace_bytes(dash.WS_ATTENTION, n, len(lengths), Hq, Hkv, D, dash.dtype_code(Q)), DEV)
    dash.dash_varlen_attention(Q, K, V, cu, max_seqlen or max(lengths), ws=ws)
    return int(ws[4:8].view(torch.int32)) // Hq


@pytest.mark.parametrize("lengths,Hq,Hkv,D,rows", [([1000], 16, 16, 64, 8192), ([1000], 28, 4, 128, 8192), ([2000], 4, 4, 64, 16000), ([300], 28, 4, 128, 131072),
                                                   ([900] * 20, 14, 2, 128, 40000), ([200] * 40, 8, 2, 128, 8100)])
def test_attention_items_follow_the_true_lengths(lengths, Hq, Hkv, D, rows):
    """Behind a selection the caller knows bounds only; whether tiles go in pairs hangs on the lengths that are there (20 sequences of 900: pairs)."""
    tiles = [(x + 127) // 128 for x in lengths]
    expect = sum((t + 1) // 2 for t in tiles) if len(lengths) == 20 else sum(tiles)
    assert _entries(lengths, Hq, Hkv, D) == expect and _entries(lengths, Hq, Hkv, D, rows, rows) == expect


@pytest.mark.parametrize("lengths", [[150] * 60 + [1, 128, 40, 7], [700, 130, 1, 300, 900] * 4], ids=["one or two tiles", "pairs"])
@pytest.mark.parametrize("D", [64, 128])
def test_attention_by_index_of_many_sequences(lengths, D):
    """Two warps share every fetch by index, items of one tile and pairs."""
    _indexed_attention_case(lengths, 0.6, 12, 4, D, 37)
