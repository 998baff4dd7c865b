"""Channels-first inputs as the kernels keep them: the transposes at the edges of their tiles, exactly."""
import pytest
import torch

from paper_2505_11157_b200 import sna

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [32, 64, 96, 128, 24, 48])
@pytest.mark.parametrize("nlat, nlon", [(5, 20), (16, 32), (9, 36), (8, 33), (3, 17), (13, 20), (2, 2)],
                         ids=["100", "512", "324", "264", "51", "260", "4"])
def test_inputs_are_transposed_exactly(C, nlat, nlon):
    """Planes of 4 to 512 points: less than a tile of 128, whole tiles, a tile of 4 points at the end (260) and nothing else (4), planes
    that are not whole 16-byte pieces (51 points); channels in groups of 32, and others."""
    B, H = 2, 3
    gen = torch.Generator(device="cuda").manual_seed(C + nlon)
    q, k, v = (torch.randn(B, H * C, nlat, nlon, generator=gen, device="cuda") for _ in range(3))
    with sna.Plan(nlat, nlon, nlat, nlon, 0, 0, global_attention=True) as plan:
        _, state = plan.forward_cf(q, k, v, H)
        torch.cuda.synchronize()
    kept = state.view(torch.float32)
    at, count = 0, q.numel()
    for x in (q, k, v):
        want = x.view(B, H, C, nlat, nlon).permute(0, 1, 3, 4, 2).reshape(-1)
        assert torch.equal(kept[at:at + count], want)
        at += (count * 4 + 255) // 256 * 64
