"""Recovery of one stream takes one or two rows a step, by the number of chunks: vectors on both sides of that line, with short codes and with codes
that the table does not resolve, flat and in layers. The state that the compress call itself writes is the reference."""
import pytest
import torch

from test_gpu_parity import DEV

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_13003_b200 import binding

    binding.lib()
    return binding


@pytest.mark.parametrize("nbits,kind", [(2, "gauss"), (4, "rare"), (8, "lognormal"), (9, "uniform")])
@pytest.mark.parametrize("past", [-1, 0, 1])
def test_both_sides_of_the_line(lc, nbits, kind, past):
    from paper_2009_13003_b200 import synth

    warps = 24 * torch.cuda.get_device_properties(0).multi_processor_count  # with one stream, on the device
    n = (5 * warps // 2 + past) * 4096 + (77 if past else 0)
    base = synth.normal(n, 0.02, DEV, 5)
    if kind == "rare":  # stretches of rare exponents: long codes side by side
        delta = synth.normal(n, 1e-4, DEV, 6)
        delta[1_000_000:1_200_000] *= torch.exp2(torch.randint(0, 9, (200_000,), device=DEV, generator=torch.Generator(DEV).manual_seed(1)).float())
    elif kind == "uniform":  # over many exponents
        g = torch.Generator(DEV).manual_seed(2)
        delta = torch.exp2(torch.rand(n, device=DEV, generator=g) * 60 - 70)
    else:
        delta = synth.sweep_delta(kind, n, DEV, 6)
    cur = base + delta
    stream, tracked = lc.compress_update(base, cur, nbits)
    assert torch.equal(lc.recover(base, [stream]), tracked)
    if nbits <= 4:
        seg = [0, 4096 * 3, n // 2 // 4 * 4, n // 4 * 4]
        streams, _ = lc.compress_segments(base[: seg[-1]], cur[: seg[-1]], seg, nbits, tracked_out=tracked)
        assert torch.equal(lc.recover_segments(base[: seg[-1]], [streams], seg, nbits), tracked[: seg[-1]])
