"""A call that runs out of device memory reports it, and the calls after it do not (needs
a GB300)."""
import pytest

import paper_2512_12094_gb300 as pp
import pp_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    pp.build()
    pp.load()


@pytest.mark.parametrize("block_threads", [0, 256])
def test_the_next_call_does_not_fail(block_threads):
    """Headroom of a billion times the strings: terabytes, refused at once.  Another
    context, and the same one by another call, go on."""
    wl = pi.config1_ring(n=32, steps=2, eps=1e-3, max_weight=8)
    gx, gz, th = wl.circuit.gate_arrays(0)
    a = pp.Propagator.from_workload(wl, symmetry=0, room_factor=1e9, block_threads=block_threads)
    with pytest.raises(pp.PPError) as e:
        a.apply_layer(gx, gz, th, True)
    assert e.value.status == 2  # PP_ERR_OOM
    b = pp.Propagator.from_workload(wl, symmetry=0)  # failed with the error of the call before
    b.apply_layer(gx, gz, th, True)
    assert b.num_terms()[0] > 32 and a.num_terms()[0] == 32
    with pytest.raises(pp.PPError):
        a.apply_layer(gx, gz, th, True)
    a.expect(wl.state.bloch)
    a.close()
    b.close()
