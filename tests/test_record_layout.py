"""Records as dicts: read where the structure's fields are, also when the structure changes."""
import os
import types

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("insert_before", [None, "step", "q", "mass", "uu", "k_cov"])
def test_dict_holds_the_fields(insert_before):
    import paper_2602_16486_gb300.flbm as fb

    text = open(fb.__file__).read()
    if insert_before:
        extra = {"q": '("more", ctypes.c_int32), ("less", ctypes.c_int32),'}.get(insert_before, '("more", ctypes.c_double * 3),')
        text = text.replace('        ("%s", ' % insert_before, '        %s\n        ("%s", ' % (extra, insert_before), 1)
    mod = types.ModuleType("flbm_copy")
    mod.__file__, mod.__package__ = fb.__file__, fb.__package__
    exec(compile(text, fb.__file__, "exec"), mod.__dict__)
    r = mod.flbm_stats_t()
    assert hasattr(r, "more") == bool(insert_before)
    r.step, r.sites, r.nonfinite, r.lattice, r.q, r.mass = 1 << 40, -3, 7, 2, 19, 0.25
    for k, name in enumerate(("mom", "u_mean", "uu", "k_mean", "k_cov")):
        for j in range(len(getattr(r, name))):
            getattr(r, name)[j] = 1000.0 * (k + 1) + j
    d = r.to_dict()
    assert [d[k] for k in ("step", "sites", "nonfinite", "lattice", "q", "mass")] == [1 << 40, -3, 7, 2, 19, 0.25]
    assert all(type(d[k]) is int for k in ("step", "sites", "nonfinite", "lattice", "q"))
    for name, n in (("mom", 3), ("u_mean", 3), ("uu", 6), ("k_mean", 19)):
        assert np.array_equal(d[name], getattr(r, name)[:n]), name
    assert np.array_equal(d["k_cov"], np.reshape(r.k_cov[:361], (19, 19)))
