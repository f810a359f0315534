"""Read-outs of a state that the engine reports: each of them reports it again."""
import pytest

import chaingen
import paper_1001_3764_gb300 as md

pytestmark = pytest.mark.gpu


def test_energy_of_a_state_with_a_force_out_of_range_is_reported_every_time():
    """An atom 0.9 nm off on each axis: a bond force of some 4e5 kJ/mol/nm, beyond the fixed-point range of the mixed form."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    m = chaingen.melt(4, seed=1, L=4.0)
    s = md.System(m, precision=md.MD_MIXED)
    good = s.energy()[0]
    x, v, _ = s.state()
    y = x.copy()
    y[75] += 0.9
    for call in (lambda: s.set_state(y, v), s.energy, s.energy):
        with pytest.raises(md.MDError) as e:
            call()
        assert e.value.code == md.MD_EOVERFLOW
    s.set_state(x, v)
    assert s.energy()[0] == pytest.approx(good)
    s.close()
