"""The resident PCG's fail word: a lane in which some block has given up a wait must not end as if
nothing had happened.  The word is set from the host, so no wait has to run out on the GPU."""
import ctypes as C

import numpy as np
import pytest

import workloads as wl
from oracle import hamiltonian as ham

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
L, N_UP, K = 10, 5, 32


class PcgDev(C.Structure):
    _fields_ = [("rz", C.c_void_p), ("rz0", C.c_void_p), ("alpha", C.c_void_p), ("beta", C.c_void_p),
                ("active", C.c_void_p), ("tol2", C.c_double), ("partials", C.c_void_p), ("counter", C.c_void_p)]


@pytest.fixture(scope="module")
def mbl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2012_00217_gb300 as m
    m.binding.lib()
    return m


def _run(mbl, blocks, steps, fail, staged):
    """`steps` PCG steps of one lane on `blocks` blocks; returns (w, counter words)."""
    so = C.CDLL(mbl.binding.LIB_PATH)
    n = ham.sector_dim(L, N_UP)
    chain = mbl.make_chain(L, wl.fields(L, 5.0, 4), 1.0, True, N_UP)
    cp, lane = C.create_string_buffer(8192), C.create_string_buffer(8192)
    assert so["_ZN3mbl17make_chain_paramsEPK9mbl_chaindPNS_11ChainParamsE"](C.byref(chain), C.c_double(0.1), cp) == 0
    f32 = dict(dtype=torch.float32, device=DEV)
    r = torch.from_numpy(wl.block(n, K, 7, np.float32)).to(DEV)
    dinv = torch.full((n,), 0.1, **f32)
    p, t, w = dinv[:, None] * r, torch.zeros(n, K, **f32), torch.zeros(n, K, **f32)
    rz = (r.double() * p.double()).sum(0)
    pad = lambda x: torch.nn.functional.pad(x, (0, 64 - K))  # noqa: E731
    scal = [pad(rz), pad(rz).clone(), pad(torch.zeros_like(rz)), pad(torch.zeros_like(rz))]
    active = torch.ones(64, dtype=torch.int32, device=DEV)
    partials = torch.zeros(2 * blocks * K, dtype=torch.float64, device=DEV)
    counter = torch.tensor([0, 0, 0, fail], dtype=torch.int32, device=DEV)
    dev = PcgDev(*[x.data_ptr() for x in scal], active.data_ptr(), 0.0, partials.data_ptr(), counter.data_ptr())
    ptr = lambda x: C.c_void_p(x.data_ptr())  # noqa: E731
    fill = so["_ZN3mbl13pcg_lane_fillEPNS_7PcgLaneERKNS_11ChainParamsEjiiPKvPvS7_S7_S7_RKNS_6PcgDevEjjb"]
    run = so["_ZN3mbl7pcg_runEiPKNS_7PcgLaneES2_iijjiP11CUstream_st"]
    mbl.binding.set_product_schedule(K, torch.float32, 3 if staged else 1)
    try:
        assert fill(lane, cp, C.c_uint32(n), K, 1, ptr(dinv), ptr(r), ptr(p), ptr(t), ptr(w), C.byref(dev),
                    C.c_uint32(0), C.c_uint32(blocks), C.c_bool(True)) == 0
    finally:
        mbl.binding.set_product_schedule(K, torch.float32, 0)
    # the lane ends with n, B, block0, nblocks, items, chunk, stage_bytes
    tail = np.frombuffer(lane.raw, dtype=np.uint32)
    at = [i for i in range(tail.size - 6) if tail[i] == n and tail[i + 3] == blocks and tail[i + 2] == 0]
    assert len(at) == 1
    stage_bytes = int(tail[at[0] + 6])
    assert (stage_bytes > 0) == staged
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert run(1, lane, None, 1, K, C.c_uint32(blocks), C.c_uint32(stage_bytes), steps, st) == 0
    torch.cuda.synchronize()
    return w, counter.tolist()


@pytest.mark.parametrize("staged", [False, True])
@pytest.mark.parametrize("blocks", [1, 3])
@pytest.mark.parametrize("steps", [1, 5])
def test_a_failed_lane_reports_it(mbl, blocks, steps, staged):
    w, words = _run(mbl, blocks, steps, 0, staged)
    assert torch.isfinite(w).all() and (w != 0).any() and words == [0, 0, 0, 0]
    w, words = _run(mbl, blocks, steps, 1, staged)
    assert torch.isnan(w).any(dim=0).all()  # every column: the solve ends as MBL_ERR_NUMERIC
    assert words == [0, 0, 0, 1]
