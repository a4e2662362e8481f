"""Host logic of the weight-streaming GEMMs' work decomposition (no GPU): every shape of the workloads is covered by its
work items, the tile sizes are ones the kernels can run, and no CTA or cluster gets much more than its share."""
import math

import pytest

from paper_2604_12247_b200 import binding, inputs

SHAPES = [inputs.LLAMA2_7B, inputs.LLAMA3_8B, inputs.LLAMA_13B,
          inputs.scaled(inputs.LLAMA3_8B, name="small", n_layers=4, d_model=512, n_heads=8, n_kv_heads=2, head_dim=64,
                        d_ffn=1416, vocab=2048)]


def _gemms(s):
    qd, kvd = s.n_heads * s.head_dim, s.n_kv_heads * s.head_dim
    return {"qkv": ([qd, kvd, kvd], s.d_model), "o": ([s.d_model], qd), "down": ([s.d_model], s.d_ffn)}


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: s.name)
@pytest.mark.parametrize("mode,units", [(0, 296), (0, 148), (2, 74), (2, 72)])
def test_split_gemm_plans_cover_their_matrices(shape, mode, units):
    per = 2 if mode == 2 else 1                       # CTAs that share a work item
    for name, (n_rows, k) in _gemms(shape).items():
        R, S, items = binding.plan_gemm(mode, n_rows, k, units)
        assert R % 8 == 0 and (8 if mode == 2 else 64) <= R <= 128, (name, R)
        assert (per * R) % 16 == 0 or mode == 0       # the pair kernel's MMA width 2R is a multiple of 16
        kb = math.ceil(k / 64)
        assert 1 <= S <= min(8, kb), (name, S)
        slabs = sum(math.ceil(n / (per * R)) for n in n_rows)
        assert items == slabs * S                     # every row of every matrix lies in exactly one slab, every k block in one split
        # the busiest unit's work (slab rows x k blocks) against a perfectly even share of the matrices
        busiest = math.ceil(items / units) * per * R * math.ceil(kb / S)
        ideal = sum(n_rows) * kb / units
        if shape.name != "small":                     # (a matrix of a few hundred rows cannot fill 296 CTAs)
            assert busiest <= 1.6 * ideal, (name, R, S, items, busiest / ideal)


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: s.name)
@pytest.mark.parametrize("mode,units", [(1, 296), (3, 74)])
def test_gate_up_plans(shape, mode, units):
    h, S, items = binding.plan_gemm(mode, [shape.d_ffn], shape.d_model, units)
    assert S == 1                                     # the SwiGLU epilogue needs whole sums: never split along k
    assert h % 8 == 0 and (32 <= h <= 64 if mode == 1 else 8 <= h <= 128)
    assert items == math.ceil(shape.d_ffn / h)        # every FFN column in exactly one item


def test_plan_query_rejects_bad_arguments():
    with pytest.raises(binding.SBError):
        binding.plan_gemm(4, [4096], 4096, 148)
    with pytest.raises(binding.SBError):
        binding.plan_gemm(0, [4096, 0], 4096, 148)
    with pytest.raises(binding.SBError):
        binding.plan_gemm(2, [4096], 0, 74)
    with pytest.raises(binding.SBError):
        binding.plan_gemm(2, [4096], 4096, 0)


# the decompositions the wide prefill passes launch, one to four tiles of 128 rows: what the kernel can run, the bound on the
# length of a sum, partials that fit their buffer, and everything covered
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: s.name)
@pytest.mark.parametrize("tiles", [1, 2, 3, 4])
@pytest.mark.parametrize("units", [66, 72, 74])
def test_wide_pass_plans(shape, tiles, units):
    for name, (n_rows, k) in _gemms(shape).items():
        R, S, items = binding.plan_gemm(2 + 256 * tiles, n_rows, k, units)
        kb = math.ceil(k / 64)
        assert R % 8 == 0 and 8 <= R <= 128 and 1 <= S <= min(8, kb), (name, R, S)
        assert items == sum(math.ceil(n / (2 * R)) for n in n_rows) * S * tiles
        if tiles > 1:
            assert math.ceil(kb / S) <= (45 if kb > 66 else 22), (name, S)     # k blocks that one accumulator takes in
            least = math.ceil(kb / (45 if kb > 66 else 22))
            assert S <= max(60 * 2**20 // (4 * 128 * tiles * sum(n_rows)), least), (name, S)     # partials the workspace has room for
        else:
            assert (R, S, items) == binding.plan_gemm(2, n_rows, k, units)
        busiest = math.ceil(items / units) * 2 * R * math.ceil(kb / S)
        if shape.name != "small":
            assert busiest <= 1.6 * sum(n_rows) * kb * tiles / units, (name, R, S, items)


@pytest.mark.parametrize("d_ffn", [1408, 1416, 9472, 9480, 11008, 11016, 13824, 14336, 18944, 18952, 28672])
@pytest.mark.parametrize("tiles", [1, 2, 4])
@pytest.mark.parametrize("units", [66, 72, 74])
def test_wide_pass_gate_up_plans(d_ffn, tiles, units):
    h, S, items = binding.plan_gemm(3 + 256 * tiles, [d_ffn], 4096, units)
    assert S == 1 and h % 8 == 0 and 8 <= h <= 256
    assert items == math.ceil(d_ffn / h) * tiles
    if h > 128:                                       # two accumulators: one round of one tile, halves the MMA can take
        assert tiles == 1 and h % 16 == 0 and items <= units
        stage = h * 128 + 16384                       # bytes of a pipeline stage; at least one per producer fits
        assert 4 * stage + 1280 <= 225 * 1024
    else:                                             # and where one round of two parts is the shorter one, it is taken
        rounds = math.ceil(math.ceil(d_ffn / h) / units)
        one = math.ceil(math.ceil(d_ffn / units) / 16) * 16
        assert tiles > 1 or rounds == 1 or one > 256 or one > rounds * max(h, 96)


def test_plan_query_rejects_bad_tile_counts():
    for mode in (256, 257, 2 + 256 * 5, 4 + 256, -254):
        with pytest.raises(binding.SBError):
            binding.plan_gemm(mode, [4096], 4096, 74)
