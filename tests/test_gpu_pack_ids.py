"""rtoss_pack takes an id array that starts at any byte (the ids of a model's layers kept back to back): the packed layer is
the one an aligned array gives, bit for bit.  Channel counts whose rows the ordering pass reads as sixteen ids, as four and
one by one; filter counts on both sides of its two forms."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2303_02191_b200 import binding as rt
    from paper_2303_02191_b200 import synth
    import gpu_util as gu


@pytest.mark.parametrize("Cin", [16, 20, 17])
@pytest.mark.parametrize("Cout", [33, 513])
def test_ids_at_any_byte(Cout, Cin):
    c, masks = gu.ctx(), rt.rtoss_pattern_preset(4, rt.PRESET_CENTRE8)
    w = gu.to_dev(synth.kaiming_weights(21, Cout + Cin, Cout, Cin, 3), "f32")
    pid = c.rtoss_select_patterns(w, 3, masks, 4)
    want = c.rtoss_pack(w, 3, masks, 4, pid, rt.BF16)
    store = torch.full((Cout * Cin + 16,), 200, dtype=torch.uint8, device="cuda")
    into = None
    for shift in (1, 2, 3, 4, 15):
        store[shift:shift + Cout * Cin] = pid
        into = c.rtoss_pack(w, 3, masks, 4, store[shift:], rt.BF16, into=into)   # (the first a new handle, then packed again in place)
        a, b = want.export(), into.export()
        assert all(np.array_equal(a[key], b[key]) for key in a), shift
    want.close(), into.close()
