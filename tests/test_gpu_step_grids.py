"""GPU checks of the decode step's per-head kernels over the grids they are launched with: the
sequences of a head in one CTA or spread over several, one or several passes, rows of the new
tokens and queries at any 2-byte alignment, contiguous and paged caches.  The projection sums in the same order whatever the
split, so appended cache bytes agree exactly between the forms."""
import numpy as np
import pytest
import torch

from paper_2609_24298_gb300 import cobra, synth

from .gpu_util import DEV, oracle_head, rel_err, upload

pytestmark = pytest.mark.gpu
ROWS = 4  # code rows per sequence (two pages)


@pytest.fixture(scope="module", autouse=True)
def need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    cobra.lib()


@pytest.fixture(scope="module")
def heads():
    srcs = [synth.HeadSource(61, 0, h, side, (0.3, 2.5)) for side in (0, 1) for h in range(2)]
    return [oracle_head(s, r, b) for s, (r, b) in zip(srcs, [(128, 2), (34, 5), (100, 1), (64, 3)])]


def step(heads, layers, S, G, layer=None, shift=0, paged=False, cap=500, empty=None):
    """One step over `layers` copies of the two heads (or over layer `layer` alone) on a cache of
    constant bytes; inputs are the same whatever the form.  shift: elements the inputs and outputs
    are moved from their 16-byte boundary; paged: the sequences' pages in random order; empty: a
    sequence whose length reads 0 in the attention."""
    n = 2 * layers
    params = heads[:2] * layers + heads[2:] * layers
    n_slots = S * ROWS
    block, offs, total, r, b = upload(params, n_slots)
    cache = torch.full((total,), 0x5A, dtype=torch.uint8, device=DEV)
    g = np.random.default_rng(7)
    draw = lambda *shape: torch.tensor(g.standard_normal(shape), dtype=torch.bfloat16, device=DEV)
    k, v, q = draw(layers, S, 2, 128), draw(layers, S, 2, 128), draw(layers, S, 2 * G, 128)
    lens = g.integers(1, cap + 1, S).astype(np.int32)
    rps, pps, table = ROWS, 0, None
    if paged:
        rps, pps = 0, ROWS // 2
        table = torch.tensor(g.permutation(S * pps).astype(np.int32), device=DEV)
    L, l0 = (layers, 0) if layer is None else (1, layer)

    def moved(t):
        t = t[l0:l0 + L].contiguous()
        buf = torch.zeros(t.numel() + 8, dtype=t.dtype, device=DEV)
        buf[shift:shift + t.numel()] = t.reshape(-1)
        return buf, buf.data_ptr() + 2 * shift

    (kb, kp), (vb, vp), (qb, qp) = moved(k), moved(v), moved(q)
    desc = cobra.decode_desc(k_head0=2 * l0, v_head0=n + 2 * l0, layer_stride=2, n_layers=L, n_kv_heads=2, group=G,
                             n_seqs=S, rows_per_seq=rps, pages_per_seq=pps, q_stride_layer=S * 2 * G * 128,
                             q_stride_seq=2 * G * 128, o_stride_layer=S * 2 * G * 128, o_stride_seq=2 * G * 128)
    side = lambda s: cobra.compress_desc(head0=s * n + 2 * l0, layer_stride=2, n_layers=L, n_kv_heads=2, side=s, n_seqs=S,
                                         rows_per_seq=rps, pages_per_seq=pps, x_stride_layer=S * 256, x_stride_seq=256,
                                         x_stride_tok=256, x_stride_head=128)
    wsb = cobra.cobra_decode_workspace_size(desc, r, b, lens)
    ws = torch.empty(wsb, dtype=torch.uint8, device=DEV)
    info = cobra.cobra_decode_plan(desc, r, b, lens, ws, wsb)
    obuf = torch.full((L * S * 2 * G * 128 + 4,), float("nan"), dtype=torch.float32, device=DEV)
    out = obuf[shift % 4:shift % 4 + obuf.numel() - 4].view(L, S, 2 * G, 128)
    ld, pos = torch.tensor(lens, device=DEV), torch.tensor(lens - 1, device=DEV)
    if empty is not None:
        ld[empty] = 0
    cobra.cobra_decode_step(block, desc, info, side(0), side(1), kp, vp, pos, qp, cache, ld, table, out, ws, wsb)
    assert cobra.cobra_check() == cobra.COBRA_OK
    return cache.cpu().numpy(), out.cpu().numpy(), offs, n_slots, r, b


@pytest.mark.parametrize("G", [4, 8])
@pytest.mark.parametrize("S,paged", [(1, False), (3, True), (41, False), (41, True), (83, False)])
def test_alignment_of_tokens_and_queries(heads, S, G, paged):
    c0, o0, *_ = step(heads, 1, S, G, paged=paged)
    for shift in (1, 2, 4):
        c1, o1, *_ = step(heads, 1, S, G, shift=shift, paged=paged)
        assert np.array_equal(c0, c1) and np.array_equal(o0, o1)
    if paged:  # the same rows wherever their pages lie
        assert np.array_equal(o0, step(heads, 1, S, G)[1])


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("S,G", [(5, 4), (7, 4), (11, 4), (15, 4), (7, 8)])
def test_one_cta_per_head_equals_split_heads(heads, S, G, paged):
    """80 layers x 2 heads fill the GPU (one CTA per head: passes of 8 sequences and a rest, of 7 with
    a warp left over, of 4 with 8 query heads); a layer alone spreads its heads' sequences over CTAs."""
    layers = 80
    c0, o0, offs, n_slots, r, b = step(heads, layers, S, G, paged=paged)
    for layer in (0, 37, 79):
        c1, o1, *_ = step(heads, layers, S, G, layer=layer, paged=paged)
        for h in (2 * layer, 2 * layer + 1, 2 * (layers + layer), 2 * (layers + layer) + 1):
            at = slice(int(offs[h]), int(offs[h]) + n_slots * 16 * int(r[h]) * int(b[h]))
            assert np.array_equal(c0[at], c1[at])
        assert rel_err(o1[0], o0[layer]) < 2e-3  # the chunks of the two plans differ


@pytest.mark.parametrize("S,empty", [(6, None), (7, None), (7, 0)])
def test_combine_of_two_sequences_per_cta(heads, S, empty):
    """80 layers x 2 heads x 6 or 7 sequences of one chunk each are combined two sequences to a CTA
    (the last one alone when S is odd), a layer alone one to a CTA: the same partials, the same
    outputs.  An empty sequence gives zeros in either."""
    layers = 80
    _, o0, *_ = step(heads, layers, S, 4, cap=128, empty=empty)
    for layer in (0, 37, 79):
        _, o1, *_ = step(heads, layers, S, 4, layer=layer, cap=128, empty=empty)
        assert np.array_equal(o1[0], o0[layer])
    assert np.array_equal(o0, step(heads, layers, S, 4, cap=128, empty=empty, shift=1)[1])
    if empty is not None:
        assert np.all(o0[:, empty] == 0) and np.all(o0[:, empty + 1] != 0)
