"""Batch sizes of the learned-guess network at the edges of its buffers.

* A batch too large for the device's memory is refused, and the network goes on with the buffers it had:
  the training steps after it are those of a network that never saw the request, bit for bit.
* One step of a large batch takes the memory of its activations and little more: 64 MB cover the
  indices of its own rows and the allocator's granularity, not those of a chunk of steps (134 MB).
* Steps that go out in several chunks are those of single calls.
* More rows than one grid dimension has tiles for (65,535 x 32): with one training pair every batch has
  the same loss.  Both sides add n equal FP32 terms per thread before the fixed tree, n up to 2^21 x 1024
  / 65,536 = 32,768, each addition rounding to 2^-24 relative: 2^15 x 2^-24 = 2e-3, and as much again for
  the division by the batch size.
"""
import numpy as np
import pytest

from paper_2410_24138_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nls():
    from paper_2410_24138_gb300 import build, nls as binding
    build.build()
    return binding


def harvested(nls, seed=3):
    """A small network with the 16 pairs of one F_x evaluation."""
    p = I.diffusion_problem(32, I.box_partition(32, 4, 4), 16, 1)
    s = nls.make_solver(p, coupling="one")
    net = nls.GuessNet(h1=16, h2=16, seed=seed, capacity=16)
    nls.attach_guess(s, net, nls.GUESS_HARVEST)
    s.eval_Fx(np.zeros(p.n_nodes))
    nls.attach_guess(s, None, 0)
    s.close()
    assert net.pairs() == 16
    return net


def test_failed_growth_keeps_the_buffers(nls):
    a, b = harvested(nls), harvested(nls)
    la, lb = [a.train(3, batch=8)], [b.train(3, batch=8)]
    for _ in range(2):
        with pytest.raises(nls.NLSError):  # 2^31 - 1 rows of 391 inputs: 3.4 TB
            b.train(1, batch=2 ** 31 - 1)
    for batch in (8, 300, 16):
        la.append(a.train(3, batch=batch))
        lb.append(b.train(3, batch=batch))
    assert np.array_equal(np.concatenate(la), np.concatenate(lb))
    assert np.all(np.isfinite(np.concatenate(la))) and np.array_equal(a.params(), b.params())


def test_memory_of_a_large_step(nls):
    import torch
    net = harvested(nls)
    net.train(1, batch=8)
    batch = 1 << 17
    free = torch.cuda.mem_get_info()[0]
    net.train(1, batch=batch)
    used = free - torch.cuda.mem_get_info()[0]
    wide = max(net.h1, net.h2, net.n_out)
    assert used <= 4 * batch * (net.n_in + 2 * net.n_out + 2 * net.h1 + 2 * net.h2 + 2 * wide) + (64 << 20)


def test_chunks_of_steps(nls):
    a, b = harvested(nls), harvested(nls)
    batch = 1 << 20  # four steps to a chunk
    la, lb = a.train(4, batch=batch, seed=5), b.train(6, batch=batch, seed=5)
    assert np.array_equal(la, lb[:4])
    assert np.all(np.isfinite(lb)) and lb[5] < lb[0]


def test_more_rows_than_a_grid_dimension(nls):
    p = I.diffusion_problem(8, I.box_partition(8, 1, 1), 1, 1)
    losses = []
    for batch in (64, 65535 * 32 + 33):
        s = nls.make_solver(p, coupling="one")
        net = nls.GuessNet(h1=16, h2=16, seed=3, capacity=1)
        nls.attach_guess(s, net, nls.GUESS_HARVEST)
        s.eval_Fx(np.zeros(p.n_nodes))
        nls.attach_guess(s, None, 0)
        losses.append(net.train(1, batch=batch)[0])
        net.close()
    assert abs(losses[1] - losses[0]) <= 4e-3 * losses[0]
