"""A call that fails with a CUDA error reports it once: the next call does not find it again."""
import ctypes

import pytest
import torch

from paper_2404_10272_gb300 import scenes
from _helpers import assert_same, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    from paper_2404_10272_gb300 import build, hdda
    build.build()
    hdda.load()
    return hdda


def test_next_call_after_a_refused_one(H):
    sc = scenes.tiny_scene()
    o, d = (torch.from_numpy(x[:1000]).cuda() for x in scenes.tiny_camera().rays())
    p = sc.params
    prm = H.make_params(p.near, p.far, p.step, p.cone, p.max_step, p.max_steps)
    grid = H.build_vdb(torch.from_numpy(sc.occ).cuda(), sc.aabbs)
    want = tuple(to_np(x) for x in H.traverse_hdda(o, d, grid, prm).trimmed())
    out = H.alloc_samples(1000, want[1].size)
    torch.cuda.synchronize()
    # a synchronous sampler call cannot be captured: the runtime refuses its wait
    cuda = ctypes.CDLL("libcuda.so.1")
    s = torch.cuda.Stream()
    assert cuda.cuStreamBeginCapture_v2(ctypes.c_void_p(s.cuda_stream), 1) == 0
    try:
        with pytest.raises(H.HddaError) as ex:
            H.traverse_hdda(o, d, grid, prm, out, stream=s)
    finally:
        graph = ctypes.c_void_p()
        cuda.cuStreamEndCapture(ctypes.c_void_p(s.cuda_stream), ctypes.byref(graph))
    assert ex.value.code == H.ERR_CUDA
    got = H.traverse_hdda(o, d, grid, prm, out)
    assert_same(tuple(to_np(x) for x in got.trimmed()), want, "after a refused call")
