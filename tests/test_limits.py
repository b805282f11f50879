"""The largest context: a list entry names a cluster with 25 bits, so a system
whose clusters would not fit is refused on the host, before anything of its
size is allocated."""

import ctypes
import resource

import numpy as np

from paper_0902_0827_gb300 import nb


def test_more_clusters_than_a_list_entry_can_name():
    sig = np.array([3.0], np.float32)
    p = nb.nb_params()
    p.n_atoms = 1 << 28  # 2^25 clusters, and the partial ones of every column
    for a in range(3):
        p.box[a] = 1400.0
    p.cutoff, p.switch_dist, p.ewald_alpha, p.coulomb_k = 9.0, 7.5, 0.32, 332.0636
    p.n_types = 1
    p.sigma = p.epsilon = sig.ctypes.data_as(ctypes.c_void_p)
    p.scale14_lj, p.scale14_coul = 0.5, 1 / 1.2
    h = ctypes.c_void_p()
    before = resource.getrusage(resource.RUSAGE_SELF).ru_maxrss
    assert nb.lib().nb_create(ctypes.byref(p), None, ctypes.byref(h)) == 11  # NB_ERR_UNSUPPORTED
    assert not h.value
    assert resource.getrusage(resource.RUSAGE_SELF).ru_maxrss - before < 1 << 20  # KB
