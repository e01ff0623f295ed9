"""Batches whose splits are large enough for the tensor-core stages: several maps of one split
as one stack, another split beside it, one entry that stays with the lists, and a map that
the two-part split cannot carry.  The stages are the single call's kernels on the same data:
outputs equal those of single calls bit for bit where both stages are theirs, and within
1e-6 of the rms (another contraction of the same sums) where the gather is the lists'."""
import numpy as np
import pytest

from paper_1409_4441_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1409_4441_gb300 import ksconv
    return ksconv


@pytest.mark.parametrize("use_graph", [False, True])
def test_batch_on_the_tensor_core_stages(K, use_graph):
    # belt stage only; both stages; neither
    specs = [(128, 22.0, False), (256, 32.0, True), (32, 6.0, False)]
    sps = [K.make_split_real(inputs.gaussian_beam(2 * ns, np.radians(3 * 58.6 / ns)), ns,
                             np.radians(td)) for ns, td, _ in specs]
    which = [0, 1, 0, 2, 1, 0]
    ins = []
    for k, i in enumerate(which):
        m = inputs.white_noise_map(specs[i][0], 300 + k).astype(np.float32)
        if k == 2:
            m[::7] *= np.float32(1e-9)
        ins.append(torch.tensor(m, device="cuda"))
    ref = []
    for k, i in enumerate(which):
        y = torch.empty_like(ins[k])
        K.conv_real(sps[i], ins[k], y)
        ref.append(y)
    torch.cuda.synchronize()
    with K.Batch([sps[i] for i in which], use_graph=use_graph) as b:
        for _ in range(2):  # other buffers the second time
            outs = [torch.full_like(x, float("nan")) for x in ins]
            b.run([x.clone() for x in ins] if _ else ins, outs)
            b.status()
            for k, i in enumerate(which):
                if specs[i][2]:
                    assert torch.equal(outs[k], ref[k])
                else:
                    rms = ref[k].double().square().mean().sqrt()
                    assert (outs[k] - ref[k]).abs().max() <= 1e-6 * rms
    for s in sps:
        s.close()
