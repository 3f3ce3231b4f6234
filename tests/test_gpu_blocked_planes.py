"""FP32 meshes with planes of 2 MB or more and z lines of 768 points or more keep
their workspace in blocks of 16 planes.  Their potentials against the float-pair
solve of the same source on plain planes (held to the oracle at 1e-12
elsewhere), with N_z a multiple of the block and not (the last block then holds
planes whose values must reach no potential), on every line length with a
blocked form, in every y-pass form, over a NaN-filled workspace and from host
buffers."""
import numpy as np
import pytest

from paper_1106_0557_gb300 import native

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

# (N, Mz); planes of 2.1 to 2.4 MB
SHAPES = [((1000, 140, 330), 768), ((1000, 140, 384), 768), ((640, 200, 385), 1024), ((1024, 128, 512), 1024),
          ((700, 180, 515), 1152), ((1000, 130, 649), 1536), ((1000, 130, 771), 2048), ((1000, 130, 1025), 2304),
          ((1000, 130, 1040), 2304)]


def _src(N):
    g = torch.Generator(device="cuda").manual_seed(sum(N))
    s = torch.rand((N[2], N[1], N[0]), dtype=torch.float32, device="cuda", generator=g)
    return s * (torch.rand(s.shape, device="cuda", generator=g) < 0.3)


@pytest.mark.parametrize("N,Mz", SHAPES)
def test_blocked_planes_match_float_pairs(N, Mz):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1106_0557_gb300 import Plan
    h = (1.0, 0.5, 0.75)
    src = _src(N)
    # float pairs too block 2304-point lines of whole blocks: one empty plane
    # more keeps the reference on plain planes
    pad = int(Mz == 2304 and N[2] % 16 == 0)
    with Plan((N[0], N[1], N[2] + pad), h, "df64") as p:
        assert p.padded_shape[2] == (Mz if Mz != 768 else 1024)
        ref = p.solve(torch.nn.functional.pad(src.double(), (0, 0, 0, 0, 0, pad)))[:N[2]]
    with Plan(N, h, "f32") as p:
        M = p.padded_shape
        assert M[2] == Mz and M[1] * M[0] // 2 * 8 >= 2 << 20
        assert p.workspace_bytes == -(-N[2] // 16) * 16 * M[1] * (M[0] // 2) * 8
        assert native.ipf_estimate_bytes(N, h, "f32") == p.workspace_bytes  # the spectrum is cached
        phi = p.solve(src)
        host = p.solve_host(src.cpu().numpy())
        p.check()
    # FP32 against 64 bits: a few 1e-7 (the parity tests allow 1e-5)
    err = float((phi.double() - ref).abs().max() / ref.abs().max())
    assert err <= 2e-6, err
    assert np.array_equal(host, phi.cpu().numpy())
    for flags in (native.IPF_FLAG_TEST_CANARY, native.IPF_FLAG_Y_TILES, native.IPF_FLAG_Y_STREAM,
                  native.IPF_FLAG_Y_TILES_NARROW):
        with Plan(N, h, "f32", flags=flags) as p:
            assert torch.equal(p.solve(src), phi), flags
            p.check()
