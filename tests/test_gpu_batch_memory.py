"""A batch runs its chains on streams of its own, which end with it, while the
chains' states live on: every buffer of theirs is asked for, and given back, in
the order of the caller's stream, never of one of the batch's."""
import pytest
import torch

from paper_1212_0785_gb300 import lqcd

pytestmark = pytest.mark.gpu

SPECS = [((4, 4, 4, 4), 0.150), ((6, 4, 2, 10), 0.153), ((8, 6, 6, 12), 0.157)]


class RecordingAllocator:
    """device memory from PyTorch's caching allocator; records the streams named"""

    def __init__(self):
        self.alloc_streams, self.free_streams, self.live = set(), set(), set()

    def alloc(self, nbytes, stream):
        self.alloc_streams.add(int(stream or 0))
        p = torch.cuda.caching_allocator_alloc(nbytes)
        self.live.add(p)
        return p

    def free(self, ptr, stream):
        self.free_streams.add(int(stream or 0))
        self.live.remove(ptr)
        torch.cuda.caching_allocator_delete(ptr)


@pytest.fixture
def recorder():
    r = RecordingAllocator()
    lqcd.set_allocator(r.alloc, r.free)
    yield r
    lqcd.set_allocator(None, None)


@pytest.mark.parametrize("force_prec", [lqcd.F32, lqcd.F64])
def test_batch_allocates_on_the_callers_stream(recorder, force_prec):
    stream = torch.cuda.Stream()
    cg = lqcd.cg_params(tol=1e-10, sloppy=lqcd.F16N, delta=0.01)
    params = [lqcd.hmc_params(5.8, kappa, 0.3, 4, lqcd.OMELYAN, cg=cg, force_prec=force_prec, chrono=3,
                              chrono_mre=True) for _, kappa in SPECS]
    fields, states = [], []
    for i, (dims, _) in enumerate(SPECS):
        U = lqcd.gauge_field(dims)
        lqcd.gauge_start(U, i + 1, 0.3)
        fields.append(U)
        states.append(lqcd.HmcState(U, seed=i + 1))
    torch.cuda.synchronize()
    batch = lqcd.Batch(states)
    infos = batch.trajectory(params, stream=stream.cuda_stream)
    assert all(f["cg_guesses_refined"] > 0 for f in infos)  # the extrapolation's buffers were used
    stream.synchronize()
    batch.close()
    for st in states:
        st.close()
    for U in fields:
        U.free()
    assert not recorder.live
    assert recorder.alloc_streams <= {0, stream.cuda_stream}
    assert recorder.free_streams <= {0, stream.cuda_stream}
