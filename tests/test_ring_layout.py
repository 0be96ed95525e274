"""The step kernel's shared-memory ring, checked on the host (no GPU): regions
that do not overlap and start on 16-byte lines, room for the shift of
misaligned arrays where (and only where) an instance shifts them, and as many
stages as a GB300 block's shared memory holds."""
import itertools

import pytest

from paper_2607_10611_gb300 import builder as B

TILE, SMEM = 3840, 232_448  # elements per tile; shared memory a GB300 block may have
SIZE = {"f32": 4, "bf16": 2}
WEIGHTS = {"bf16": 2 * TILE, "e4m3": TILE, "e4m3_b32": TILE, "nvfp4": TILE // 2}
SCALES = {"e4m3_b32": 240, "nvfp4": 240}


@pytest.fixture(scope="module")
def N():
    B.build()
    from paper_2607_10611_gb300 import _native
    return _native


@pytest.mark.parametrize("wd,gd,md,mis", [x for x in itertools.product(WEIGHTS, SIZE, SIZE, (False, True))
                                          if x[0] != "nvfp4" or not x[3]])
def test_ring(N, wd, gd, md, mis):
    r = N.mpadam_debug_ring_layout(N.make_config(weight_dtype=wd, grad_dtype=gd, moment_dtype=md), mis, SMEM)
    line = 16 if mis else 0
    bounds = [0, r["off_g"], r["off_m"], r["off_v"], r["off_ve"], r["off_s"], r["stage_bytes"]]
    assert all(b % 16 == 0 for b in bounds)
    room = [b - a for a, b in zip(bounds, bounds[1:])]
    assert room == [WEIGHTS[wd] + (line if wd in ("e4m3", "e4m3_b32") else 0), TILE * SIZE[gd] + line,
                    *[TILE * SIZE[md]] * 3, SCALES.get(wd, 0)]
    assert r["static_bytes"] == 1024
    assert r["stages"] == min(8, (SMEM - 1024) // r["stage_bytes"])


def test_stages_of_the_training_formats(N):
    """Aligned lists: four stages with binary32 moments (BF16 weights have room for three), six or seven with BF16."""
    want = {("bf16", "f32"): 3, ("e4m3", "f32"): 4, ("e4m3_b32", "f32"): 4, ("nvfp4", "f32"): 4,
            ("bf16", "bf16"): 6, ("e4m3", "bf16"): 6, ("e4m3_b32", "bf16"): 6, ("nvfp4", "bf16"): 7}
    for (wd, md), n in want.items():
        r = N.mpadam_debug_ring_layout(N.make_config(weight_dtype=wd, grad_dtype="bf16", moment_dtype=md), False, SMEM)
        assert r["stages"] == n, (wd, md)


def test_too_little_shared_memory_is_refused(N):
    with pytest.raises(N.MPAdamError):
        N.mpadam_debug_ring_layout(N.make_config(), False, 48 << 10)
