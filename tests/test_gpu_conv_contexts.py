"""Network convolutions of two contexts from two host threads: what belongs to a device as a whole must not
pass from one context's calls to the other's."""

import threading

import numpy as np
import pytest

import hhg_inputs as hi
from paper_1908_08666_gb300 import binding as B

from hhg_gpu import torch_cuda

pytestmark = pytest.mark.gpu


class Net:
    """A context with a network on a stream of its own, and an input."""

    def __init__(self, seed, shape):
        self.torch = t = torch_cuda()
        self.stream = t.cuda.Stream()
        self.shape = shape
        self.h = B.hhg_create(0, self.stream.cuda_stream)
        xyz, tets = hi.unit_tet()
        B.hhg_set_macro_mesh(self.h, xyz, tets)
        B.hhg_refine(self.h, 2)
        B.hhg_set_problem(self.h)
        B.hhg_learn_init(self.h, seed)
        self.x = t.as_tensor(np.random.default_rng(seed).normal(size=shape + (7,)), dtype=t.float32, device="cuda")
        self.out = t.empty(shape + (3,), dtype=t.float32, device="cuda")
        t.cuda.synchronize()

    def forward(self):
        B.hhg_learn_forward(self.h, self.x, 7, *self.shape, self.out)

    def close(self):
        B.hhg_destroy(self.h)


def _together(*loops):
    """Runs the functions in a thread each, starting together; returns what they raised."""
    errors, gate = [], threading.Barrier(len(loops))

    def body(f):
        gate.wait()
        try:
            f()
        except BaseException as e:  # noqa: BLE001  (reported by the caller)
            errors.append(e)

    threads = [threading.Thread(target=body, args=(f,)) for f in loops]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    return errors


def test_grids_of_different_tilings_from_two_threads():
    """Grids whose tiles take 104 and 85 KB of shared memory: the limit that one launch needs is not lowered
    by the other context's."""
    nets = [Net(1, (8, 31, 31, 32)), Net(2, (24, 16, 20, 16))]
    try:
        want = []
        for net in nets:
            net.forward()
            want.append(net.out.clone())

        def loop(net):
            for _ in range(400):
                net.forward()

        assert _together(*(lambda net=net: loop(net) for net in nets)) == []
        for net, w in zip(nets, want):
            assert net.torch.equal(net.out, w)
    finally:
        for net in nets:
            net.close()


def test_a_timeout_is_reported_to_its_own_context():
    """One context's wait for its MMAs runs out in every call (bound of zero polls); the other one's calls,
    whose kernel has no such wait, succeed meanwhile."""
    nets = [Net(3, (1, 3, 4, 16)), Net(4, (1, 3, 4, 16))]
    try:
        nets[1].forward()
        want = nets[1].out.clone()
        B.hhg_learn_set_conv_wait(nets[0].h, 0)

        def times_out():
            for _ in range(300):
                B.hhg_learn_set_conv_kernel(nets[0].h, 1)
                with pytest.raises(B.HhgError) as e:
                    nets[0].forward()
                assert e.value.status == 7

        def succeeds():
            for _ in range(300):
                nets[1].forward()

        assert _together(times_out, succeeds) == []
        assert nets[1].torch.equal(nets[1].out, want)
    finally:
        for net in nets:
            net.close()


# grids up to 456 tiles of 4 x 4 x 32 voxels take the warp-level kernel, which has no wait; larger ones the
# grouped tcgen05 kernel, in both of its tile forms, batched and with a ragged march in z
@pytest.mark.parametrize("shape,grouped", [((1, 33, 20, 129), False), ((1, 29, 65, 127), True), ((1, 33, 65, 66), True),
                                           ((24, 16, 20, 16), True), ((1, 5, 160, 165), True)])
def test_default_kernel_timeout_falls_back(shape, grouped):
    """With a bound of zero polls the grouped kernel's wait runs out in every block: the call reports it, the
    next ones run on the warp-level kernel, and choosing the kernel again brings the grouped one back.  All
    results agree to the last bit, as the kernels do."""
    net = Net(5, shape)
    try:
        t = net.torch
        net.forward()
        want = net.out.clone()

        def same():
            net.out.fill_(7.0)
            t.cuda.synchronize()
            net.forward()
            return t.equal(net.out, want)

        B.hhg_learn_set_conv_wait(net.h, 0)
        if not grouped:
            assert same()
            return
        for _ in range(2):
            with pytest.raises(B.HhgError) as e:
                net.forward()
            assert e.value.status == 7 and "timed out" in str(e.value)
            assert same()  # the warp-level kernel: the bound is still zero
            B.hhg_learn_set_conv_kernel(net.h, 0)
        B.hhg_learn_set_conv_wait(net.h, -1)
        assert same()
    finally:
        net.close()
