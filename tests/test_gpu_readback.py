"""States read back at the lengths where the way to the caller changes (64 KB, 16 KB
for packed rows of single bytes): the bytes that were loaded, in either form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(260, 252), (256, 256), (256, 260), (260, 256),  # 64 KB
                                   (508, 516), (512, 512), (512, 516), (1024, 1024)])
def test_states_come_back_at_every_length(shape):
    import paper_2301_11735_gb300 as cc

    Lx, Ly = shape
    st = np.random.default_rng(Lx + Ly).integers(0, 4, size=(Ly, Lx)).astype(np.uint8)
    c = st.reshape(-1, 4)
    packed = c[:, 0] | (c[:, 1] << 2) | (c[:, 2] << 4) | (c[:, 3] << 6)
    with cc.Lattice(Lx, Ly) as lat:
        lat.set_state_packed(packed, 1, 0)
        for _ in range(2):
            assert np.array_equal(lat.get_state(), st)
            assert np.array_equal(lat.get_state_packed(), packed)
