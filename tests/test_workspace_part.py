"""A caller's workspace that is smaller than its own padding to 256 bytes has no usable part: the call is refused for its size."""
import pytest

from paper_2609_32114_b200 import binding


@pytest.mark.parametrize("address,nbytes,part", [(256, 8, (256, 8)), (64, 8, (256, 0)), (64, 192, (256, 0)), (64, 193, (256, 1)),
                                                 (1, 0, (256, 0)), (512, 0, (512, 0)), (511, 4096, (512, 4095))])
def test_aligned_part(address, nbytes, part):
    assert binding._aligned_part(address, nbytes) == part


@pytest.mark.gpu
@pytest.mark.parametrize("lead", [(1,), ()], ids=["native", "marshalled"])
def test_a_small_slice_off_the_boundary_is_refused(lead):
    import torch
    import paper_2609_32114_b200 as ha

    q = torch.zeros(*lead, 3, 1, 128, dtype=torch.bfloat16, device="cuda")
    g = torch.zeros(*lead, 3, 1, device="cuda")
    buf = torch.zeros(4096, dtype=torch.uint8, device="cuda")
    for first, n in ((64, 8), (64, 192), (1, 200), (0, 256)):
        with pytest.raises(ha.HaLaError) as e:
            ha.ha_la_prefill(q, q, q, g, g, workspace=buf[first:first + n])
        assert e.value.status == binding.HA_LA_ERR_WORKSPACE
    torch.cuda.synchronize()
    assert int(buf.max().item()) == 0
