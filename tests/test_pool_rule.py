"""How a launch deals out its tiles by default, checked on the host (no GPU):
the limits in tiles per CTA, and E4M3 with a scale per tensor, whose CTAs
must not be led through every one of many tensors (each entry recomputes
candidates for the tensor's exact maximum)."""
import pytest

from paper_2607_10611_gb300 import builder as B

CTAS, TILE = 152, 3840
ALL_FORMATS = ("bf16", "e4m3", "e4m3_b32", "nvfp4")


@pytest.fixture(scope="module")
def rule():
    B.build()
    from paper_2607_10611_gb300 import _native as N
    return lambda tiles, tensors, wd, md: N.mpadam_debug_pool_rule(tiles, tensors, CTAS, N.DTYPE[wd], N.DTYPE[md])


@pytest.mark.parametrize("md", ["f32", "bf16"])
@pytest.mark.parametrize("wd", ALL_FORMATS)
def test_limits_of_one_long_tensor(rule, wd, md):
    """One tensor: every format alike."""
    want = [(8, (1024, 4, False)), (16, (768, 4, False)), (128, (256, 1, False)),
            (1 << 20, (0, 1 if md == "f32" else 2, True))]
    lo = 0
    for per_cta, r in want:
        for tiles in (lo, per_cta * CTAS - 1):
            assert rule(tiles, 1, wd, md) == r, tiles
        lo = per_cta * CTAS
    assert rule(2 ** 31 - 1, 1, wd, md)[0] == 1024  # a claim counter of 32 bits


def _tiles(shapes):
    return sum(-(-n // TILE) for n in shapes), len(shapes)


def _llama(layers, d, ffn, vocab):
    return [vocab * d] + ([d * d] * 4 + [d * ffn] * 3 + [d] * 2) * layers + [d, vocab * d]


def _gpt2(layers=12, d=768, vocab=50257, ctx=1024):
    return [vocab * d, ctx * d] + [d, d, 3 * d * d, 3 * d, d * d, d, d, d, 4 * d * d, 4 * d, 4 * d * d, d] * layers + [d, d]


RAGGED = [1 + (i * i * 7919) % 65521 for i in range(4000)]  # 9 tiles on average


@pytest.mark.parametrize("md,shapes,want", [
    ("bf16", _llama(4, 2048, 5632, 16000), (768, 4, False)), ("bf16", _llama(24, 2048, 5632, 32000), (768, 4, False)),
    ("bf16", _gpt2(), (768, 4, False)), ("bf16", RAGGED, (768, 4, False)), ("bf16", RAGGED[:1000], (768, 4, False)),
    ("bf16", _llama(1, 4096, 11008, 32000), (0, 2, True)), ("bf16", [200_000_000], (0, 2, True)),
    ("f32", _llama(24, 2048, 5632, 32000), (0, 1, True)), ("f32", _llama(4, 2048, 5632, 16000), (0, 1, True)),
    ("f32", RAGGED, (768, 4, False)), ("f32", _gpt2(), (256, 1, False)), ("f32", _llama(8, 1024, 2816, 16000), (256, 1, False)),
    ("f32", RAGGED[:1000], (256, 1, False))])
def test_e4m3_keeps_ctas_in_their_tensors(rule, md, shapes, want):
    assert rule(*_tiles(shapes), "e4m3", md) == want


@pytest.mark.parametrize("md", ["f32", "bf16"])
@pytest.mark.parametrize("wd", ["bf16", "e4m3_b32", "nvfp4"])
def test_other_formats_follow_tiles_per_cta(rule, wd, md):
    assert rule(*_tiles(_llama(4, 2048, 5632, 16000)), wd, md) == (0, 1 if md == "f32" else 2, True)
    assert rule(*_tiles(RAGGED), wd, md) == (0, 2, False)
    assert rule(*_tiles(RAGGED[:1000]), wd, md) == (256, 1, False)
