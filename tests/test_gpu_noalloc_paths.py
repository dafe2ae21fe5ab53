"""The allocation-free field where its two kernels' partitions change (rows of
four, source iterations of 64, I blocks of 256 and tiles of 64 per species,
the line between the kernels), against FP64, with inputs at 4-byte alignment."""
import numpy as np
import pytest

import oracle
import paper_2506_09712_gb300 as cts

pytestmark = pytest.mark.gpu
TOL = 1e-5   # of the whole field (the entry point's tests)
# per carrier, of its terms' absolute sum: a pair at distance r inherits the
# FP32 rounding of its coordinates (up to 8 um, 2^-22 um) over r, some 1e-2 um
# for the closest of 2e4 carriers
TOL_TERMS = 1e-5


@pytest.mark.parametrize("n_h,n_e", [(1, 0), (0, 5), (2, 1), (63, 1), (64, 64), (65, 63), (829, 0),
                                     (3000, 2003), (19_999, 1), (20_000, 0), (20_001, 0),
                                     (0, 20_100), (20_000, 129), (257, 20_000), (10_100, 10_037)])
def test_field_matches_fp64(n_h, n_e):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = n_h + n_e
    g = torch.Generator(device="cuda").manual_seed(n)
    buf = torch.randn(3 * n + 3, device="cuda", generator=g) * 2.0
    x, y, z = (buf[1 + c * n:1 + (c + 1) * n] for c in range(3))  # not 16-byte aligned
    out = torch.full((3 * n + 1,), 7.0, device="cuda")
    for _ in range(2):  # the second call starts from what the first left
        rc = cts.cts_field_noalloc(x.data_ptr(), y.data_ptr(), z.data_ptr(), n_h, n_e, 11.7, 1e-6,
                                   out.data_ptr(), torch.cuda.current_stream().cuda_stream)
        assert rc == cts.SIM_OK
    torch.cuda.synchronize()
    assert float(out[-1]) == 7.0
    r = torch.stack([x, y, z]).double()
    q = torch.ones(n, dtype=torch.float64, device="cuda")
    q[n_h:] = -1.0
    ref, terms = torch.empty(3, n, dtype=torch.float64, device="cuda"), torch.empty(n, device="cuda")
    for a in range(0, n, 2048):
        d = r[:, a:a + 2048, None] - r[:, None, :]
        r2 = (d * d).sum(0) + 1e-12
        w = r2.rsqrt() ** 3
        ref[:, a:a + 2048] = (d * (w * q)).sum(2)
        terms[a:a + 2048] = ((r2 - 1e-12).clamp(min=0).sqrt() * w).sum(1).float()
    ref *= oracle.coulomb_k()
    got = out[:3 * n].reshape(3, n).double()
    err, mag = (got - ref).norm(dim=0), ref.norm(dim=0)
    assert bool(torch.isfinite(got).all())
    if n > 1:
        assert float(err.norm() / mag.norm()) <= TOL
        assert float((err / (oracle.coulomb_k() * terms.double())).max()) <= TOL_TERMS
    else:
        assert float(got.abs().max()) == 0.0
