"""Every doubled length a plan may choose, on every axis that takes it and in
every arithmetic type, against the oracle: the largest and the smallest N that
takes it, with short other axes, and meshes with several lengths at once."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

BASIC = [32, 48, 64, 96, 128, 192, 256, 288, 384, 512, 576, 768, 1024, 1152, 1536, 2048, 2304]
LENGTHS = {("f32", 0): sorted(BASIC + [324, 648, 1296]), ("f32", 1): sorted(BASIC + [324, 432, 648, 1296]),
           ("f32", 2): sorted(BASIC + [324, 1296]),
           ("df64", 2): [m for m in BASIC if m not in (384, 768)]}
for _a in range(3):
    LENGTHS["f64", _a] = sorted(BASIC + [144])
    LENGTHS.setdefault(("df64", _a), LENGTHS["f64", _a])
TOL = {"f32": 1e-5, "f64": 1e-12, "df64": 1e-12}  # the parity tests' tolerances
NP = {"f32": np.float32, "f64": np.float64, "df64": np.float64}


def _src(N, seed):
    g = np.random.default_rng(seed)
    s = g.uniform(0.0, 1.0, (N[2], N[1], N[0]))
    s[g.uniform(size=s.shape) > 0.6] = 0.0
    return s


def _check(N, h, dtype, want):
    from paper_1106_0557_gb300 import Plan
    src = _src(N, sum(N)).astype(NP[dtype])
    with Plan(N, h, dtype) as p:
        assert tuple(m for m, w in zip(p.padded_shape, want) if w) == tuple(w for w in want if w)
        phi = p.solve(torch.from_numpy(src).cuda()).cpu().numpy().astype(np.float64)
        p.check()
    assert oracle.max_rel_error(phi, oracle.solve(src.astype(np.float64), h)) <= TOL[dtype]


@pytest.mark.parametrize("dtype,axis,M", [(d, a, m) for d, a in sorted(LENGTHS) for m in LENGTHS[d, a]])
def test_each_length_matches_oracle(dtype, axis, M):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    below = [m for m in LENGTHS[dtype, axis] if m < M]
    for n in {M // 2, (below[-1] // 2 if below else 0) + 1}:
        N, want = [7, 9, 10], [0, 0, 0]
        N[axis], want[axis] = n, M
        _check(tuple(N), (1.0, 0.5, 2.0), dtype, want)


@pytest.mark.parametrize("dtype", ["f32", "f64", "df64"])
def test_mixed_lengths_with_several_tiles(dtype):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    _check((137, 60, 153), (1.0, 1.0, 1.0), dtype, (288, 128, 0))
    _check((66, 211, 70), (0.5, 1.0, 1.0), dtype, (0, 0, 0))
    _check((300, 40, 270), (1.0, 0.5, 0.5), dtype, (0, 0, 576))
    # z-blocked planes (2304-point z lines of a multiple of 16 planes): y of the
    # 16-byte types keeps to the lengths that have blocked passes
    _check((20, 140, 1040), (1.0, 0.5, 0.5), dtype, (0, 288 if dtype == "f32" else 384, 2304))
    _check((20, 140, 1041), (1.0, 0.5, 0.5), dtype, (0, 288, 2304))


@pytest.mark.parametrize("dtype,M", [(d, m) for d in ("f32", "f64", "df64") for m in LENGTHS[d, 1]
                                     if m in (144, 288, 324, 432, 576, 648, 1152, 1296, 2048)])
def test_y_pass_forms_agree_bitwise(dtype, M):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1106_0557_gb300 import Plan, native
    N = (37, M // 2 - 1, 5)
    src = torch.from_numpy(_src(N, M).astype(NP[dtype])).cuda()
    outs = []
    for flag in (native.IPF_FLAG_Y_TILES, native.IPF_FLAG_Y_STREAM, native.IPF_FLAG_Y_TILES_NARROW):
        with Plan(N, (1.0, 0.5, 1.0), dtype, flags=flag) as p:
            outs.append(p.solve(src))
            p.check()
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
