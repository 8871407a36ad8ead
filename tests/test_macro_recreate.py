"""A new macro mesh has no Dirichlet data until it is given some: the old mesh's dofs and values belong to another numbering
and may lie beyond its rows.  The host code on the CPU, with the stand-in runtime of test_failed_allocations.py."""
import ctypes

import numpy as np

from test_failed_allocations import L, context  # noqa: F401  (L is the fixture)


def test_new_mesh_without_dirichlet_data(L):  # noqa: F811
    h = context(L, 2, 0, [2])
    big, small = np.array([6, 6], dtype=np.int32), np.array([2, 1], dtype=np.int32)
    dofs, values = np.arange(98, dtype=np.int32), np.ones(98)  # every dof of the big mesh
    for n_el, rows in ((small, 12), (big, 98)):
        assert L.fehmm_macro_create(h, big.ctypes.data) == 0
        assert L.fehmm_macro_set_dirichlet(h, dofs.size, dofs.ctypes.data, values.ctypes.data) == 0
        assert L.fehmm_macro_create(h, n_el.ctypes.data) == 0
        # the load of a Dirichlet increment is zero, which the host code writes itself: no kernel reads the old values
        g, K = np.full(rows + 1, 7.0), np.zeros(4000)
        assert L.fehmm_macro_dirichlet_load(h, K.ctypes.data, 1.0, g.ctypes.data, None) == 0
        assert np.all(g[:-1] == 0.0) and g[-1] == 7.0
        u = np.zeros(rows)
        L.fake_watch(5)  # the kernel's number of fixed dofs
        assert L.fehmm_macro_apply_dirichlet(h, u.ctypes.data, None, 1.0, None) == 0
        assert L.fake_watch(-1) == 0
    assert L.fehmm_destroy(h) == 0
