"""The radial walk with two derivative lanes in tensor memory against the same walk with all of them in
shared memory: the operations are the same, so the same point gives the same bits in either."""
import pytest

torch = pytest.importorskip("torch")

import paper_2409_19156_gb300 as zp  # noqa: E402
from paper_2409_19156_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_max,k", [(69, 3), (72, 3), (97, 2), (98, 3), (99, 3), (100, 3), (101, 2), (107, 3), (110, 2)])
def test_wide_walk_has_the_bits_of_the_one_warp_walk(n_max, k):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    wave = 4 * 32 * sms  # one warp per scheduler; the wide form takes whole multiples of two of them
    r = torch.rand(3 * wave, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n_max))
    r[:2] = torch.tensor([0.0, 1.0])
    r[2 * wave:] = r[:wave]
    ns, ms = inputs.radial_modes(n_max)
    out = zp.radial(ns, ms, r, k)
    assert torch.equal(out[:, :, :wave], out[:, :, 2 * wave:])
