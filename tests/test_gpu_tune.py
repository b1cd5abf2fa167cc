"""What lbm_batch_tune returns is what it left in force."""
import pytest

import lbm_cases as lc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_applying_the_returned_choice_changes_nothing(storage):
    """Small cavities, for which several steps per launch win: the kind and
    config that come back keep them."""
    import paper_1510_08224_gb300 as P
    b = P.Batch()
    lats = [P.Lattice(lc.cavity(n=n, Ra=1e4, noise=1e-3), storage=storage) for n in (20, 33, 48)]
    for lat in lats:
        b.add(lat)
    kind, config, ms = b.tune(trial_steps=64)
    assert (kind, config) == ("fused", -1) and len(ms) == 31
    before = b.steps_per_launch()
    assert before > 1
    b.set_kind(kind)
    b.set_config(config, 1)
    assert b.steps_per_launch() == before
    b.close()
