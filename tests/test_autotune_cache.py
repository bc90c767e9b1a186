"""Cached launch options are installed for the matrix and the library's paths that they were
measured for, and not for others."""
import json
import types

from paper_1612_08060_gb300 import autotune
from paper_1612_08060_gb300 import napspmv as nap


def test_options_of_other_paths_are_not_taken(monkeypatch, tmp_path):
    monkeypatch.setattr(autotune, "_cache", {})
    given = []
    monkeypatch.setattr(nap, "napspmv_set_default_opts", lambda plan, opts: given.append(opts))
    plan, row_ptr = types.SimpleNamespace(n_p=4, ppn=2), [0, 2, 5, 7, 9]
    key = autotune.matrix_key(row_ptr, 4, 2, nap.PREC_F64)
    old = key[key.index("n4_"):]  # the matrix alone, as files from before the windows have it
    assert old != key
    best = {"engine": nap.ENGINE_OVERLAP, "vec": 1, "tile_nnz": 1536, "tile_rows": 512}
    cache = tmp_path / "tune.json"
    cache.write_text(json.dumps({old: {"opts": best, "ms": 1.0}}))
    assert autotune.apply_cached(plan, row_ptr, cache_file=str(cache)) is None and not given
    cache.write_text(json.dumps({key: {"opts": best, "ms": 1.0}}))
    assert autotune.apply_cached(plan, row_ptr, cache_file=str(cache)) == best
    assert given[0].engine == nap.ENGINE_OVERLAP and given[0].tile_nnz == 1536
