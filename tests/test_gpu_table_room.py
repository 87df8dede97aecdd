"""Tables of few qubits grow no further than twice the strings there are, whatever
growth an earlier layer showed, and hold the oracle's strings (needs a GB300)."""
import numpy as np
import pytest

import oracle
import paper_2512_12094_gb300 as pp
import pp_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,block_threads", [(2, 0), (5, 0), (6, 256), (7, 0), (8, 0)])
def test_room_of_small_tables(n, block_threads):
    pp.build()
    pp.load()
    oracle.build()
    wl = pi.config0_heisenberg(n=n, steps=3)
    x, z, c = wl.observable.arrays()
    st = oracle.OracleState(n, x, z, c)
    prop = pp.Propagator.from_workload(wl, symmetry=0, block_threads=block_threads)
    for layer in reversed(range(len(wl.circuit.layers))):
        px, pz, th = wl.circuit.gate_arrays(layer)
        prop.apply_layer(px, pz, th, True)
        st.apply_layer(px, pz, th)
    # capacities are multiples of 1024
    assert prop.stats()["capacity"] <= max(1024, 2 * 4 ** n)
    gx, gz, gc = prop.export()
    ox, oz, oc = st.export()
    a, b = np.lexsort((*gx.T, *gz.T)), np.lexsort((*ox.T, *oz.T))
    np.testing.assert_array_equal(gx[a], ox[b])
    np.testing.assert_array_equal(gz[a], oz[b])
    np.testing.assert_array_equal(gc[a], oc[b])
    prop.close()
