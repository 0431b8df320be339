"""Whole-encoder parity: the CUDA path through the C ABI against the fp64 oracle, element by element
on the same seeded inputs, for all five workload families; plus the determinism properties."""
import numpy as np
import pytest
import torch

import eas_synth as S
from oracle import encoder_oracle as O
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _make(cfg, profile="plain"):
    import paper_2609_31551_b200 as P
    w = S.make_weights(cfg, profile=profile)
    enc = P.Encoder(cfg, P.weights_to_device(w))
    return w, enc


CASES = {
    # name: (config overrides, item shapes)
    "c0_full": ("c0", {}, [(1, 224, 224)] * 4),
    "c1_2layers": ("c1", dict(n_layers=2), [(1, 336, 336)] * 3),
    "c2_2layers": ("c2", dict(n_layers=2), [(1, 56, 84), (1, 224, 224), (1, 28, 28), (1, 140, 364)]),
    "c3_2layers": ("c3", dict(n_layers=2), [(4, 56, 56), (2, 112, 84)]),
    "c4_2layers": ("c4", dict(n_layers=2, max_pos=1500), [(200, 128, 1), (600, 128, 1), (2, 128, 1)]),
}


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("profile", ["plain", "sharp"])
def test_encoder_parity_small(case, profile):
    name, over, shapes = CASES[case]
    cfg = S.get_config(name, **over)
    w, enc = _make(cfg, profile)
    items = S.make_items(cfg, shapes, seed=2000 + len(shapes))
    ref, cu, _ = O.encode_microbatch(cfg, w, items)
    got, _ = G.run_gpu(enc, cfg, items)
    rel, mabs = G.assert_parity(got, ref, case)
    print(f"{case}/{profile}: row-rel {rel:.3e} max-abs {mabs:.3e}")


@pytest.mark.parametrize("case", ["c0_full", "c1_2layers", "c2_2layers", "c3_2layers", "c4_2layers"])
def test_folded_normalisation_parity_and_determinism(case):
    """eas_encoder_set_norm_fold: the blocks' normalisations applied inside the GEMMs around them (no normalisation
    kernel inside a block).  Same tolerance against the oracle as the default path, the same bytes for every SM
    budget and for an item alone or packed, fewer launches, and switching it off restores the default path's bytes."""
    name, over, shapes = CASES[case]
    cfg = S.get_config(name, **over)
    w, enc = _make(cfg, "sharp")
    items = S.make_items(cfg, shapes, seed=2050 + len(shapes))
    ref, _, _ = O.encode_microbatch(cfg, w, items)
    plain, plain_dev = G.run_gpu(enc, cfg, items)
    n_plain = enc.last_launch_count()
    enc.set_norm_fold(True)
    got, dev = G.run_gpu(enc, cfg, items)
    rel, mabs = G.assert_parity(got, ref, case + " folded")
    G.record_margin(f"{case}, folded normalisation", "sharp", 2050 + len(shapes), rel, mabs)
    assert enc.last_launch_count() == n_plain - 2 * cfg["n_layers"] + 1
    assert np.abs(got - plain).max() <= G.ABS_TOL          # two roundings of the same values
    for budget in (3, 37, 111):
        _, again = G.run_gpu(enc, cfg, items, sm_budget=budget)
        assert torch.equal(dev, again), budget
    sl0 = S.out_tokens_per_item(cfg, G.item_shape(cfg, items[0]))
    _, alone = G.run_gpu(enc, cfg, [items[0]])
    assert torch.equal(alone, dev[:sl0])
    enc.set_norm_fold(False)
    _, back = G.run_gpu(enc, cfg, items)
    assert torch.equal(back, plain_dev)


def test_c0_bit_stability_and_packing_invariance():
    cfg = S.get_config("c0")
    w, enc = _make(cfg)
    items = S.make_items(cfg, [(1, 224, 224)] * 4, seed=2002)
    _, a = G.run_gpu(enc, cfg, items)
    _, b = G.run_gpu(enc, cfg, items)
    assert torch.equal(a, b)                                  # same input twice -> same bytes
    for budget in (37, 74, 111):
        _, c = G.run_gpu(enc, cfg, items, sm_budget=budget)
        assert torch.equal(a, c), budget                      # any sm_budget -> same bytes
    _, alone = G.run_gpu(enc, cfg, [items[2]])
    assert torch.equal(a[2 * 196:3 * 196], alone)             # item alone == item packed


def test_invalid_arguments_are_rejected_before_launch():
    import paper_2609_31551_b200 as P
    cfg = S.get_config("c0")
    w, enc = _make(cfg)
    items = S.make_items(cfg, [(1, 224, 224)], seed=1)
    data, offs = P.pack_items(items)
    with pytest.raises(P.EasError) as e:
        enc.encode_microbatch(data, [(1, 224, 224)], offs, [0, 195])
    assert e.value.status == 1
    with pytest.raises(P.EasError) as e:
        enc.encode_microbatch(data, [(1, 224, 230)], offs, [0, 196])
    assert e.value.status == 1
    with pytest.raises(P.EasError) as e:
        enc.encode_microbatch(data, [(1, 224, 224)], offs, [0, 196], sm_budget=100000)
    assert e.value.status == 1
    small = torch.empty(1024, dtype=torch.uint8, device="cuda")
    with pytest.raises(P.EasError) as e:
        enc.encode_microbatch(data, [(1, 224, 224)], offs, [0, 196], workspace=small)
    assert e.value.status == 3
    # a device cu_seqlens that differs from the host copy is reported by the device check
    bad = torch.tensor([0, 100], dtype=torch.int32, device="cuda")
    enc.encode_microbatch(data, [(1, 224, 224)], offs, [0, 196], cu_seqlens_dev=bad)
    with pytest.raises(P.EasError) as e:
        enc.status()
    assert e.value.status == 7


def test_split_k_is_deterministic_budget_independent_and_optional():
    """Latency path: small micro-batches split the K loop of the residual GEMMs (eas_encoder_set_split_k, off by default).  The result must not depend
    on sm_budget or on the run, must stay within the oracle tolerance, and with the mode off an item's embeddings are
    bit-identical whatever it is packed with."""
    cfg = S.get_config("c1", n_layers=3)
    w, enc = _make(cfg)
    shapes = [(1, 336, 336)] * 2                                  # 1154 tokens: fc2 (K = 4096) splits, proj does not
    items = S.make_items(cfg, shapes, seed=2100)
    ref, _, _ = O.encode_microbatch(cfg, w, items)
    enc.set_split_k(True)
    got, a = G.run_gpu(enc, cfg, items)
    G.assert_parity(got, ref, "split K")
    _, b = G.run_gpu(enc, cfg, items)
    assert torch.equal(a, b)
    for budget in (20, 37, 111):
        _, c = G.run_gpu(enc, cfg, items, sm_budget=budget)
        assert torch.equal(a, c), budget
    enc.set_split_k(False)
    got_off, off = G.run_gpu(enc, cfg, items)
    G.assert_parity(got_off, ref, "split K off")
    assert not torch.equal(a, off)                                # the mode did something (another summation order)
    assert float((a.float() - off.float()).abs().max()) < 0.05
    rows = off.shape[0] // 2
    _, alone = G.run_gpu(enc, cfg, [items[1]])
    assert torch.equal(off[rows:], alone)                         # off: item alone == item packed
    big = items + S.make_items(cfg, [(1, 336, 336)] * 4, seed=2101)    # 3462 tokens: no split either way
    _, packed = G.run_gpu(enc, cfg, big)
    assert torch.equal(packed[rows:2 * rows], alone)
    enc.set_split_k(True)
    _, packed_on = G.run_gpu(enc, cfg, big)
    assert torch.equal(packed_on, packed)


@pytest.mark.parametrize("name,tokens,rows,splits", [("c1", 89, 256, 4), ("c1", 577, 768, 2), ("c1", 1154, 1280, 2), ("c4", 129, 256, 4), ("c4", 1500, 1536, 2), ("c1", 2308, 0, 1)])
def test_split_k_factor(name, tokens, rows, splits):
    """The workspace shows the split factor: s - 1 regions of whole 256-row blocks for the partial sums.  Two where the tiles of two
    splits fill the SMs, four with few tokens, none past the documented line."""
    cfg = S.get_config(name, n_layers=2)
    _, enc = _make(cfg)
    whole = enc.workspace_bytes(tokens, 1)
    enc.set_split_k(True)
    assert enc.workspace_bytes(tokens, 1) - whole == (splits - 1) * rows * cfg["d_model"] * 4


@pytest.mark.parametrize("case", ["c1_2layers", "c2_2layers", "c3_2layers", "c4_2layers"])
def test_split_k_parity_all_families(case):
    """The small cases of every family with split K on (RMSNorm and LayerNorm, SwiGLU and GELU MLPs, d = 1024 and 1280)."""
    name, over, shapes = CASES[case]
    cfg = S.get_config(name, **over)
    w, enc = _make(cfg, "sharp")
    enc.set_split_k(True)
    items = S.make_items(cfg, shapes, seed=2300 + len(shapes))
    ref, _, _ = O.encode_microbatch(cfg, w, items)
    got, dev = G.run_gpu(enc, cfg, items)
    G.assert_parity(got, ref, case + " split K")
    _, again = G.run_gpu(enc, cfg, items, sm_budget=37)
    assert torch.equal(dev, again)


EMBED_CASES = {
    "c0": [(1, 224, 224), (1, 32, 48)],
    "c1": [(1, 336, 336)] * 2,
    "c2": [(1, 56, 84), (1, 364, 140), (1, 28, 28), (1, 224, 1344)],
    "c3": [(4, 56, 56), (2, 112, 84), (6, 28, 28)],
}


@pytest.mark.parametrize("name", list(EMBED_CASES))
def test_fused_patch_embedding_alone(name):
    """An encoder without transformer blocks is the embedding (patch gather fused into the GEMM, bias, position
    rows, CLS) followed by the connector: the gather's index arithmetic for images, clips, raster and
    merge-group-major patch order, several items of different sizes and a ragged last tile, against the oracle."""
    over = dict(n_layers=0)
    if name in ("c0", "c1"):
        over["max_pos"] = 600
    cfg = S.get_config(name, **over)
    if name == "c0":
        cfg = dict(cfg, out_dtype=1)           # final LayerNorm in fp32: nothing but the embedding's own rounding is left
    w, enc = _make(cfg)
    shapes = EMBED_CASES[name]
    items = S.make_items(cfg, shapes, seed=4100)
    ref, _, _ = O.encode_microbatch(cfg, w, items)
    got, dev = G.run_gpu(enc, cfg, items)
    rel, mabs = G.assert_parity(got, ref, f"{name} embedding only")
    if name == "c0":
        assert rel < 2e-3, rel                 # bf16 operands with fp32 accumulation: far inside the tolerance
    for budget in (1, 5, 37):
        _, b = G.run_gpu(enc, cfg, items, sm_budget=budget)
        assert torch.equal(b, dev), budget


@pytest.mark.parametrize("name,over,shapes", [("c3", dict(temporal_patch=3), [(6, 56, 84), (3, 28, 28)]), ("c0", dict(patch=32, max_pos=64), [(1, 224, 224), (1, 32, 64)]),
                                              ("c0", dict(patch=20, max_pos=64), [(1, 100, 60), (1, 20, 20)]), ("c0", dict(patch=32, max_pos=64), [(1, 256, 256)] * 4),
                                              ("c0", dict(patch=33, max_pos=64), [(1, 231, 264), (1, 33, 66)]), ("c0", dict(patch=33, max_pos=64), [(1, 264, 264)] * 4),
                                              ("c0", dict(patch=15, max_pos=64), [(1, 105, 120), (1, 15, 15)]), ("c2", dict(in_channels=1), [(1, 364, 560), (1, 28, 56)])])
def test_patch_embedding_of_other_vector_lengths(name, over, shapes):
    """Embeddings alone against the oracle, and the same bits at budgets of one and a few SMs.  Patch vectors of 28 and 48 k-blocks of 64; 19 (the
    longest whose kernel keeps it resident, and padded); 48 with 256 patches (units of 128 on up to three SMs); odd patch edges (pixel pairs
    that straddle runs) in vectors of 52, in units of 64 and of 128 patches, and of 11; and 4 (units of 128 on few SMs, 32 on all)."""
    cfg = S.get_config(name, n_layers=0, **over)
    w, enc = _make(cfg)
    items = S.make_items(cfg, shapes, seed=4200)
    ref, _, _ = O.encode_microbatch(cfg, w, items)
    got, dev = G.run_gpu(enc, cfg, items)
    G.assert_parity(got, ref, f"{name} patch vector {over}")
    for budget in (1, 3):
        _, b = G.run_gpu(enc, cfg, items, sm_budget=budget)
        assert torch.equal(b, dev), budget


@pytest.mark.parametrize("name", ["c0", "c1", "c2", "c3"])
def test_fused_patch_embedding_same_bits_for_every_block_shape(name):
    """The embedding's units (32 or 64 patches) and column groups follow the micro-batch size and the budget: an
    item's rows must have the same bits alone, packed, and at budgets that take every shape."""
    cfg = S.get_config(name, n_layers=0)
    w, enc = _make(cfg)
    shapes = {"c0": [(1, 224, 224)] * 9, "c1": [(1, 336, 336), (1, 14, 28), (1, 336, 322)] * 2, "c2": [(1, 28, 28), (1, 560, 588), (1, 252, 364)],
              "c3": [(2, 28, 56), (6, 224, 252), (2, 364, 364)]}[name]
    items = S.make_items(cfg, shapes, seed=2070)
    first, rows = None, [S.out_tokens_per_item(cfg, s) for s in shapes]
    for budget in (0, 1, 2, 5, 9, 17, 40):
        _, dev = G.run_gpu(enc, cfg, items, sm_budget=budget)
        first = dev.clone() if first is None else first
        assert torch.equal(dev, first), budget
    for k in range(len(items)):
        _, dev = G.run_gpu(enc, cfg, items[k:k + 1])
        assert torch.equal(dev, first[sum(rows[:k]):sum(rows[:k + 1])]), k


def test_fused_patch_embedding_with_odd_item_offsets():
    """Item offsets that are odd element counts break the 4-byte alignment of pixel pairs: the gather then loads
    single elements.  Same values, same accumulation order: the result must be the same bytes."""
    import paper_2609_31551_b200 as P
    cfg = S.get_config("c2", n_layers=1)
    w, enc = _make(cfg)
    shapes = [(1, 56, 84), (1, 28, 140)]
    items = S.make_items(cfg, shapes, seed=4200)
    _, want = G.run_gpu(enc, cfg, items)
    flat = [torch.from_numpy(np.ascontiguousarray(it).reshape(-1)).to(torch.bfloat16) for it in items]
    offsets = [1, 1 + flat[0].numel() + 2]     # 1 and an odd number: both items start on odd elements
    buf = torch.zeros(offsets[1] + flat[1].numel() + 8, dtype=torch.bfloat16)
    for f, o in zip(flat, offsets):
        buf[o:o + f.numel()] = f
    cu = G.cu_seqlens_of(cfg, items)
    out = enc.encode_microbatch(buf.cuda(), shapes, offsets, cu)
    enc.status()
    assert torch.equal(out, want)


@pytest.mark.parametrize("case", list(CASES))
def test_item_is_untouched_by_a_non_finite_neighbour(case):
    """Items do not interact: with one item of the micro-batch all NaN, the others keep their bits."""
    import paper_2609_31551_b200 as P
    name, over, shapes = CASES[case]
    cfg = S.get_config(name, **over)
    w, enc = _make(cfg)
    items = S.make_items(cfg, shapes, seed=2050)
    _, want = G.run_gpu(enc, cfg, items)
    items[1] = np.full_like(items[1], np.nan)
    _, got = G.run_gpu(enc, cfg, items)
    rows = np.concatenate([[0], np.cumsum([S.out_tokens_per_item(cfg, s) for s in shapes])])
    assert torch.isnan(got[rows[1]:rows[2]].float()).all()
    assert torch.equal(got[:rows[1]], want[:rows[1]]) and torch.equal(got[rows[2]:], want[rows[2]:])


@pytest.mark.parametrize("case", ["c1_2layers", "c2_2layers", "c4_2layers"])
@pytest.mark.parametrize("split", [False, True])
def test_every_gemm_tile_shape_gives_the_same_bits_in_the_forward_pass(case, split):
    """The GEMMs that the single-kernel entry point cannot issue, with their tile shape fixed: convolutions through a row map
    with a position table (shallow 64- and 128-column tiles), rotary epilogues, and residual GEMMs that split K."""
    name, over, shapes = CASES[case]
    cfg = S.get_config(name, **over)
    w, enc = _make(cfg)
    enc.set_split_k(split)
    items = S.make_items(cfg, shapes, seed=2060)
    _, want = G.run_gpu(enc, cfg, items)
    for tile in range(1, 18):
        enc.set_gemm_tile(tile)
        for budget in (0, 7):
            _, got = G.run_gpu(enc, cfg, items, sm_budget=budget)
            assert torch.equal(got, want), (tile, budget)


@pytest.mark.parametrize("d,hd,shape,budgets", [(128, 64, (392, 504), ()), (512, 64, (280, 336), ()), (896, 64, (196, 252), ()), (1408, 64, (224, 280), ()),
                                                (1536, 64, (224, 280), ()), (2048, 64, (112, 140), ()), (1280, 80, (112, 140), range(112, 120))])
def test_rotary_ends_where_the_values_begin_in_every_tile_shape(d, hd, shape, budgets):
    """Half-height tiles have column chunks that start 16 columns off the others, so one of them can hold the last rotated key columns
    and the first value columns.  Widths and token counts where the automatic choice is such a tile (on all SMs, or on the given
    budgets), against the oracle and the bits of the 128x256 tile; and every other shape."""
    cfg = S.get_config("c2", n_layers=1, d_model=d, n_heads=d // hd, d_mlp=256, d_head_hidden=256, d_out=256)
    w, enc = _make(cfg, "sharp")
    items = S.make_items(cfg, [(1,) + shape], seed=2080)
    ref, _, _ = O.encode_microbatch(cfg, w, items)
    got, auto = G.run_gpu(enc, cfg, items)
    enc.set_gemm_tile(1)
    _, want = G.run_gpu(enc, cfg, items)
    G.assert_parity(got, ref, f"rotary at d {d}")
    assert torch.equal(auto, want)
    for tile in range(2, 18):
        enc.set_gemm_tile(tile)
        _, forced = G.run_gpu(enc, cfg, items)
        assert torch.equal(forced, want), tile
    enc.set_gemm_tile(0)
    for budget in budgets:
        _, share = G.run_gpu(enc, cfg, items, sm_budget=budget)
        assert torch.equal(share, want), budget
