"""Host-side helpers of bench.py (no GPU)."""
import math

import bench


def test_serve_pool_sizes():
    assert bench.serve_pool_sizes(0, [1 << 18, 1 << 20]) == [0, 0]
    assert bench.serve_pool_sizes(1 << 29, [1 << 18, 1 << 20]) == [1 << 27, 1 << 29]
    # whole blocks of 2^22, at least one block
    assert bench.serve_pool_sizes(1 << 29, [1000, 1 << 20]) == [1 << 22, 1 << 29]
    assert all(x % (1 << 22) == 0 for x in bench.serve_pool_sizes(3 * 10 ** 8, [123457, 999999, 1 << 20]))


def test_same_result_ignores_steps_and_matches_nan():
    a = {"hits": 10, "attempts": 99, "steps": 5, "eps_t": math.nan}
    assert bench.same_result(a, dict(a, steps=7))
    assert not bench.same_result(a, dict(a, attempts=98))
    assert not bench.same_result(a, dict(a, eps_t=0.1))
    assert bench.same_result(dict(a, eps_t=0.25), dict(a, eps_t=0.25))


def test_sampler_hash_covers_the_helpers(tmp_path, monkeypatch):
    """The traffic figure's key changes with every device function that k_sample calls, and with nothing else."""
    import os
    import shutil

    csrc = os.path.join("paper_1702_05854_gb300", "csrc")
    os.makedirs(tmp_path / csrc)
    real = os.path.join(bench.ROOT, csrc)
    before = bench.sampler_hash()
    assert before in {key for key, _ in bench.NCU_TRAFFIC}
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))

    def changed(name, old, new):
        for f in ("sample.cu", "common.cuh"):
            shutil.copy(os.path.join(real, f), tmp_path / csrc / f)
        text = (tmp_path / csrc / name).read_text()
        assert text.count(old) >= 1
        (tmp_path / csrc / name).write_text(text.replace(old, new))
        return bench.sampler_hash() != before

    for name, old in (("sample.cu", "start_rec[w][slot]"), ("common.cuh", "ld.global.nc.v8.b32"),
                      ("common.cuh", "0x1p-20f"), ("common.cuh", "(first >> 2) + v"), ("common.cuh", "min(b, buckets - 1)"),
                      ("common.cuh", "past &= 0xFu"), ("common.cuh", "pos < next"), ("common.cuh", "philox4x32_10_rk")):
        assert changed(name, old, old + " "), old
    assert not changed("common.cuh", "class Slab {", "class Slab  {")
    assert not changed("sample.cu", "k_compact", "k_compact_hits")
