"""The Green's spectra of the FP64-class types keep full FP64 precision in every
bin.  A source that alternates from cell to cell lives in the highest bins of
every axis, the smallest of the spectrum, so rounding that is relative to
larger bins shows there; its potential is held against direct sums in long
double, through a plan and through the allocation-free call."""
import numpy as np
import pytest

from paper_1106_0557_gb300 import native

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

LD = np.longdouble


def _direct(src, h, cells):
    """Potential at `cells` (z, y, x): sums over every source cell, in long double."""
    nz, ny, nx = src.shape
    r = [np.arange(n).astype(LD) * LD(w) for n, w in zip((nz, ny, nx), (h[2], h[1], h[0]))]
    r2 = (r[0] ** 2)[:, None, None] + (r[1] ** 2)[None, :, None] + (r[2] ** 2)[None, None, :]
    r2[0, 0, 0] = LD(min(h)) ** 2
    pi = LD("3.14159265358979323846264338327950288")
    G = -(LD(h[0]) * LD(h[1]) * LD(h[2]) / (4 * pi)) / np.sqrt(r2)
    s = src.astype(LD)
    out = []
    for z, y, x in cells:
        g = G[np.abs(np.arange(nz) - z)][:, np.abs(np.arange(ny) - y)][:, :, np.abs(np.arange(nx) - x)]
        out.append((g * s).sum())
    return np.array(out)


# One line per transform: 2.7e-15 to 5.1e-15 on these meshes (rms over all
# cells); two lines sharing a transform: 2.4e-14 to 8.5e-14.  The bound is twice
# the former.
BOUND = 1e-14


@pytest.mark.parametrize("N", [(36, 36, 36), (40, 33, 24)])
def test_alternating_sources_keep_fp64_precision(N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1106_0557_gb300 import Plan
    h = (1.0, 1.0, 1.0)
    z, y, x = np.meshgrid(*[np.arange(n) for n in N[::-1]], indexing="ij")
    src = 1.0 - 2.0 * ((x + y + z) & 1)
    g = np.random.default_rng(sum(N))
    cells = [tuple(int(g.integers(n)) for n in src.shape) for _ in range(100)]
    want = _direct(src, h, cells)
    pick = tuple(np.array(c) for c in zip(*cells))

    def err(phi):
        d = phi.cpu().numpy()[pick].astype(LD) - want
        return float(np.sqrt((d * d).sum() / (want * want).sum()))

    s = torch.from_numpy(src).cuda()
    got = {}
    for dtype in ("f64", "df64"):
        with Plan(N, h, dtype) as p:
            got[dtype] = err(p.solve(s))
    out = torch.empty_like(s)
    native.ipf_solve_noalloc(N, h, "f64", s.data_ptr(), out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    got["noalloc"] = err(out)
    assert max(got.values()) <= BOUND, got
