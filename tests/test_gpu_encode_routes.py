"""Routes of the encoder's dispatch, each against the oracle at the sizes where
it can go wrong: the FMA encoder (fp32 rows, and bf16 rows outside the
tensor-core encoder's widths) at partial 32-coordinate blocks, one and two
groups of 8 beam slots, partial scoring tiles and code lists of 1 to 8 words
a lane. Tolerances are the parity rules' (tests/parity.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2607_20652_gb300 import build, dpb, inputs
from test_gpu_parity import _check_all, _gpu, _ref

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    dpb.load()


@pytest.mark.parametrize("d,m_bits,levels,beam,k,dtype,std", [
    (31, 9, 3, 3, 3, "f32", False),       # less than a block; a partial tile
    (64, 12, 3, 4, 64, "f32", False),     # every coordinate in the code
    (65, 12, 4, 5, 40, "f32", True),      # one coordinate in the last block; two tiles, the second partial
    (100, 14, 3, 8, 100, "bf16", False),  # bf16, d not a multiple of 32
    (256, 14, 3, 9, 12, "f32", False),    # two groups, one slot in the second
    (768, 18, 4, 12, 128, "f32", True),   # two groups of a whole and a half
    (1056, 16, 3, 16, 200, "bf16", False),  # bf16 above 1024; the bisection at level 0
    (2048, 16, 3, 8, 32, "f32", False),
])
def test_fma_encoder(d, m_bits, levels, beam, k, dtype, std):
    plan = dpb.Plan(d=d, levels=levels, m_bits=m_bits, children=16, beam=beam, k=k, dtype=dtype)
    ref = _ref(plan)
    x = inputs.gaussian_rows(37, d, 51 + d)
    x[3] = 0.0                  # ties: every score equal
    x[4] = np.sign(x[4])        # level-0 ties throughout
    x = inputs.to_bf16(x) if dtype == "bf16" else x
    mu = sigma = None
    if std:
        mu, sigma = (t.astype(np.float64) for t in inputs.moment_tables(plan.n_features, 5))
    keep = [i for i in range(37) if i != 3]
    g = _gpu(plan, x, mu=mu, sigma=sigma)
    _check_all(plan, ref, x[keep], {n: v[keep] if isinstance(v, np.ndarray) else v for n, v in g.items()},
               mu=mu, sigma=sigma)
    if not std:  # the zero row: the first k coordinates, in order
        assert (g["idx"][3] == np.arange(k)).all() and (g["val"][3] == 0).all() and (g["y"][3] == 0).all()


def test_fma_encoder_groups_of_rows_are_independent():
    """A row's code does not depend on the batch it comes in, bit for bit."""
    plan = dpb.Plan(d=96, levels=3, m_bits=12, children=16, beam=8, k=16, dtype="f32")
    x = torch.from_numpy(inputs.gaussian_rows(1001, 96, 7)).cuda()
    idx, val, xn = dpb.encode(plan, x)
    for n in (1, 2, 3):
        i, v, q = dpb.encode(plan, x[:n].contiguous())
        assert torch.equal(i, idx[:n]) and torch.equal(v, val[:n]) and torch.equal(q, xn[:n])


@pytest.mark.parametrize("beam,k,std", [(8, 64, False), (16, 32, False), (4, 5, True)])
def test_rows_do_not_depend_on_their_batch(beam, k, std):
    """Every share of tokens among the warps (a token or two to a warp, full and
    partial rounds, spread and blockwise grids) gives a row the same bits."""
    plan = dpb.Plan(d=96, levels=4, m_bits=14, children=16, beam=beam, k=k, dtype="bf16")
    mu = sigma = None
    if std:
        mu, sigma = (torch.from_numpy(t).cuda() for t in inputs.moment_tables(plan.n_features, 5))
    base = torch.from_numpy(inputs.gaussian_rows(64, 96, 3)).cuda().to(torch.bfloat16)
    gyb = torch.from_numpy(inputs.normal((64, 96), 4)).cuda().to(torch.bfloat16)
    want = None
    for T in (64, 1, 151, 153, 1375, 3041, 4577, 6081, 9001, 12321):
        rows = torch.arange(T, device="cuda") % 64
        x, gy = base[rows].contiguous(), gyb[rows].contiguous()
        r = torch.empty((T, 96), dtype=torch.float32, device="cuda")
        code = dpb.forward(plan, x, mu, sigma, r_out=r)
        out = code + (r,) + dpb.backward(plan, x, code[0], code[1], gy, sigma=sigma, r=r)
        if want is None:
            want = out
        for w, o in zip(want, out):
            assert torch.equal(w[rows], o), T
    assert plan.status() == 0


@pytest.mark.parametrize("T", [1, 37, 5000])
def test_table_wait_that_gives_up_is_flagged(T):
    """With the wait for the tables bounded at 0 polls the tensor-core encoder
    flags DPB_DEV_TIMEOUT, lets its copies land and returns; the next call is
    whole again."""
    plan = dpb.Plan(d=96, levels=4, m_bits=14, children=16, beam=8, k=64, dtype="bf16")
    x = torch.from_numpy(inputs.gaussian_rows(T, 96, 8)).cuda().to(torch.bfloat16)
    want = dpb.encode(plan, x)
    assert plan.status() == 0
    try:
        dpb.set_wait_limit(0)
        dpb.encode(plan, x)
        torch.cuda.synchronize()
    finally:
        dpb.set_wait_limit(-1)
    assert plan.status() == dpb.DEV_TIMEOUT
    for w, o in zip(want, dpb.encode(plan, x)):
        assert torch.equal(w, o)
    assert plan.status() == 0
