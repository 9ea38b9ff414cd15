"""Tuning results cached by a library of other sources are not taken over: an entry under another source mark, or under none as
older files have it, is kept in the file but the search runs again; one under this library's mark is used as it stands."""
import json
import re

import numpy as np
import pytest

from synth import SK_CARBON_LIKE, lattice_positions

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("old", ["|kernels=000000000000|", "|"])
def test_entries_of_other_sources(tmp_path, old):
    from paper_1202_0098_gb300 import build, mka
    build.build()
    pos, box = lattice_positions("diamond", 3.567, 3, 0.1, 0.0, 23)
    s = mka.mka_build_system(pos, box, SK_CARBON_LIKE, "bf16", cluster_radius=5.0)
    cache = str(tmp_path / "tune.json")
    sample, prm = np.arange(16, dtype=np.int64), mka.solve_params(3, 3, arith="mixed", cg_tol=1e-7)

    def tune():
        t = mka.mka_autotune(s, prm, sample, 64.0, 0.1, cache)
        return t.threads, t.ctas_per_sm, t.order_by_size

    def batch():
        return mka.mka_autotune_batch(s, prm, mka.tuning(), [16, 32], 0, 4.0, 0.1, cache)

    try:
        tune(), batch()
        mark = f"|kernels={build.source_mark()}|"
        text = open(cache).read()
        assert text.count(mark) == 2
        # this library's entries are believed, whatever they say
        text = re.sub(r'"threads": \d+, "ctas_per_sm": \d+, "order_by_size": \d+', '"threads": 64, "ctas_per_sm": 7, "order_by_size": 1', text)
        text = re.sub(r'"batch": \d+', '"batch": 7', text)
        open(cache, "w").write(text)
        assert tune() == (64, 7, 1) and batch() == 7
        # another library's are not
        open(cache, "w").write(text.replace(mark, old))
        assert tune()[0] in (128, 256, 512) and batch() in (16, 32)
        entries = json.load(open(cache))["entries"]
        assert sum(mark in e["key"] for e in entries) == 2 and len(entries) == 4
    finally:
        mka.mka_system_destroy(s)
