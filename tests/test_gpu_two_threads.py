"""Two host threads with a context and a stream each, whose calls launch the
same kernel with different amounts of shared memory (by the batch's size or by
the model): no launch is refused and every result is that of a call alone."""
import threading

import pytest
import torch

from paper_2201_05213_gb300 import nlc as N

from gpu_util import images, make_codec, to_dev

pytestmark = pytest.mark.gpu


def _run_together(jobs, reps):
    errors, gate = [], threading.Barrier(len(jobs))

    def loop(job):
        try:
            gate.wait()
            for _ in range(reps):
                job()
        except Exception as e:  # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=loop, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]


@pytest.mark.parametrize("prec", [N.NLC_FP32, N.NLC_BF16])
def test_compressors_of_a_large_and_a_small_batch(prec):
    jobs, ends = [], []
    # 16 warps per SM against one; the FP32 kernel's need follows the model
    for cfg, size in (((2, 32, 1, 10), (260, 260)), ((1, 32, 0, 9), (4, 4))):
        codec, _ = make_codec(cfg, prec, seed=1)
        d = [to_dev(images(7, [size])[0])]
        ref, roffs = codec.compress(d, 0)
        out, offs = torch.zeros_like(ref), torch.zeros_like(roffs)
        stream = torch.cuda.Stream()
        jobs.append(lambda c=codec, d=d, o=out, f=offs, s=stream:
                    N.nlc_compress(c.ctx, d, 0, N.NLC_LAYOUT_ROW, o, f, s))
        ends.append((codec, stream, out, offs, ref, roffs))
    torch.cuda.synchronize()
    _run_together(jobs, 2000)
    for codec, stream, out, offs, ref, roffs in ends:
        codec.check(stream)
        end = int(roffs[-1])
        assert torch.equal(offs, roffs) and torch.equal(out[:end], ref[:end])


@pytest.mark.parametrize("prec", [N.NLC_FP32, N.NLC_BF16])
def test_trainers_of_a_large_and_a_small_model(prec):
    jobs, ends = [], []
    for cfg in ((3, 64, 2, 10), (1, 64, 0, 1)):
        codec, _ = make_codec(cfg, prec, seed=1)
        batch = torch.stack([to_dev(i) for i in images(7, [(6, 6)] * 2)])
        ref = codec.loss_grad(batch)
        loss, grad = torch.zeros_like(ref[0]), torch.zeros_like(ref[1])
        stream = torch.cuda.Stream()
        jobs.append(lambda c=codec, b=batch, l=loss, g=grad, s=stream:
                    N.nlc_loss_grad(c.ctx, b, l, g, s))
        ends.append((codec, stream, loss, grad, ref))
    torch.cuda.synchronize()
    _run_together(jobs, 2000)
    for codec, stream, loss, grad, ref in ends:
        codec.check(stream)
        assert torch.equal(loss, ref[0]) and torch.equal(grad, ref[1])
