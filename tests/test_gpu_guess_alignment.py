"""Mesh arrays of the caller: read and written in pairs of floats, so that 8
bytes are enough (a guess at any even offset of a buffer gives the same bits)
and less is refused before a launch."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_guess_off_the_16_byte_boundary():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2312_02968_gb300 import binding as B

    n = 32
    gen = torch.Generator().manual_seed(1)
    rho = torch.rand((n, n, n), generator=gen).cuda()
    buf = 0.01 * torch.randn(3 * n ** 3 + 4, generator=gen).cuda()
    guess = buf[:3 * n ** 3].clone()
    h = B.MondPM(n, 1, float(n), 1.0, 1.0, B.MU_DEEP, 1.0, 1)
    for warm in (B.WARM_GUESS, B.WARM_GUESS_RAW):
        fields = []
        for shift in (0, 2):
            at = buf[shift:shift + 3 * n ** 3]
            assert at.data_ptr() % 16 == 4 * shift
            at.copy_(guess)
            torch.cuda.synchronize()
            h.set_density(rho)
            h.solve_field(2, warm, at)
            fields.append(h.get_field(B.FIELD_ACC))
        assert torch.isfinite(fields[0]).all() and torch.equal(fields[0], fields[1])
        for call in (lambda: h.solve_field(2, warm, buf[1:1 + 3 * n ** 3]), lambda: h.smooth(buf[1:1 + 3 * n ** 3])):
            with pytest.raises(B.MondError) as e:
                call()
            assert e.value.code == -1  # MOND_EINVAL
    h.close()
